// 27-point mixed-grid Helmholtz stencil y = A u (Eq. eq1), matrix-free, multi-RHS.
//
// The mixed-grid stencil (rotated-coordinate Laplacians with weights w1..w3
// plus a consistent mass term with weights wm1..wm4) is applied in its exact
// product form with 1-D second differences:
//   A u = h^-2 [sum D_a + a2 sum_{a<b} D_a D_b + a3 D_x D_y D_z] u
//       + [m0 + m1 sum P_a + m2 sum P_a P_b + m3 P_x P_y P_z] (k^2 u)
// with a2 = w2/6 + w3/2, a3 = w3/4, m0 = wm1+6wm2+12wm3+8wm4,
// m1 = wm2+4wm3+4wm4, m2 = wm3+2wm4, m3 = wm4.  D_a is the 3-point second
// difference stretched by the absorbing layer (coefficients cm, c0, cp per
// node, from the grid's 1-D tables); P_a is the plain (1, -2, 1).  Ghost
// neighbours (outside the grid, including the Dirichlet plane above k = 0)
// contribute zero.
//
// The coefficient of neighbour (dx, dy, dz) is a tensor product of the 1-D
// coefficients; per (dy, dz) pair the two partial sums
//   A = e_y e_z + a2 (Y e_z + e_y Z) + a3 Y Z,  B = Y e_z + e_y Z + a2 Y Z
// give the Laplacian coefficient X_dx A + [dx == 0] B, and likewise for the
// real mass coefficient.  Each thread owns one node and RCH consecutive
// right-hand sides, rhs fastest across threads (complex64: RCH = 2, one
// 16-byte vector per thread, so every neighbour load of a warp covers 512
// contiguous bytes; complex128: RCH up to 4, as the FP64 arithmetic and not
// the loads bounds it).  The coefficient is formed once per neighbour and
// reused for the RCH columns.  The grid is (x-line chunks, y, z), so no
// thread divides 64-bit indices.
#include <atomic>
#include <cmath>

#include "internal.h"

namespace {

// Rows whose 1-D coefficients are all the plain (1, -2, 1) and whose 26 neighbours exist
// (inside [lo, hi] on every axis) use the four class constants of the stencil: with
// plain differences the Laplacian coefficient of a neighbour depends only on its class
// (centre, face, edge, corner), Lc = {-6+12a2-8a3, 1-4a2+4a3, a2-2a3, a3}, and the mass
// coefficient is Mc = {wm1, wm2, wm3, wm4}; the neighbour's coefficient is Lc/h^2 + Mc k^2_q,
// real when k^2 is real (REALK).
struct Interior {
    int lo[3], hi[3];
    double Lc[4], Mc[4];
};

// RCH consecutive complex values loaded or stored as one aligned vector
template <typename T, int RCH>
struct __align__(2 * sizeof(T) * RCH) CPack {
    cplx<T> v[RCH];
};

// NR > 0: the column count as a compile-time constant (neighbour addresses become immediate offsets)
template <typename T, int RCH, bool SUB, bool REALK, int NR>
__global__ void __launch_bounds__(128) stencil_kernel(const cplx<T>* __restrict__ u, const cplx<T>* __restrict__ b,
                                                      cplx<T>* __restrict__ y,
                                                      const cplx<T>* __restrict__ k2,
                                                      const cplx<T>* __restrict__ tab, int nx, int ny, int nz,
                                                      int nrhs_rt, StencilW w, Interior in,
                                                      const StencilW* __restrict__ wtab,
                                                      const unsigned char* __restrict__ wbin) {
    // grid: (x-line chunks, y, z); a thread owns node (i, j, k) and columns [ch RCH, ch RCH + RCH)
    const int nrhs = NR > 0 ? NR : nrhs_rt;
    const int nch = nrhs / RCH;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nx * nch) return;
    const int ch = t % nch, i = t / nch;
    const int j = blockIdx.y, k = blockIdx.z;
    const long long p = ((long long)k * ny + j) * nx + i;
    // neighbour offsets: nodes for k^2, entries for the vectors
    const long long nxy = (long long)nx * ny;
    const cplx<T>* up = u + p * nrhs + (long long)ch * RCH;
    const cplx<T>* kp = k2 + p;

    if (wtab) w = wtab[wbin[p]];   // adaptive weights: this row's bin
    const T ih2 = (T)w.inv_h2;
    const cplx<T> zero = mk<T>(0, 0);
    cplx<T> acc[RCH];
#pragma unroll
    for (int r = 0; r < RCH; ++r) acc[r] = zero;

    if (i >= in.lo[0] && i <= in.hi[0] && j >= in.lo[1] && j <= in.hi[1] && k >= in.lo[2] && k <= in.hi[2]) {
        T L[4], M[4];
        if (wtab) {
            // class constants of this row's weights (the same identities as for the grid's constant weights)
            const double Lr[4] = {-6.0 + 12.0 * w.a2 - 8.0 * w.a3, 1.0 - 4.0 * w.a2 + 4.0 * w.a3, w.a2 - 2.0 * w.a3, w.a3};
            const double Mr[4] = {w.m0 - 6.0 * w.m1 + 12.0 * w.m2 - 8.0 * w.m3, w.m1 - 4.0 * w.m2 + 4.0 * w.m3,
                                  w.m2 - 2.0 * w.m3, w.m3};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                L[c] = (T)(Lr[c] * w.inv_h2);
                M[c] = (T)Mr[c];
            }
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                L[c] = (T)(in.Lc[c] * w.inv_h2);
                M[c] = (T)in.Mc[c];
            }
        }
        // one z-plane of 9 neighbours at a time: its 18 loads are issued together, then the FMAs
#pragma unroll
        for (int dz = -1; dz <= 1; ++dz) {
            cplx<T> kq[9];
            CPack<T, RCH> uq[9];
#pragma unroll
            for (int d = 0; d < 9; ++d) {
                const long long dq = dz * nxy + (d / 3 - 1) * nx + (d % 3 - 1);
                kq[d] = kp[dq];
                uq[d] = *reinterpret_cast<const CPack<T, RCH>*>(up + dq * nrhs);
            }
#pragma unroll
            for (int d = 0; d < 9; ++d) {
                const int cls = (d % 3 != 1) + (d / 3 != 1) + (dz != 0);
                if (REALK) {
                    const T cr = L[cls] + M[cls] * kq[d].x;
#pragma unroll
                    for (int r = 0; r < RCH; ++r) {
                        acc[r].x = fma(cr, uq[d].v[r].x, acc[r].x);
                        acc[r].y = fma(cr, uq[d].v[r].y, acc[r].y);
                    }
                } else {
                    const cplx<T> cc = mk<T>(L[cls] + M[cls] * kq[d].x, M[cls] * kq[d].y);
#pragma unroll
                    for (int r = 0; r < RCH; ++r) cmac(acc[r], cc, uq[d].v[r]);
                }
            }
        }
    } else {
    const cplx<T>* tx = tab + 3 * i;
    const cplx<T>* ty = tab + 3 * (nx + j);
    const cplx<T>* tz = tab + 3 * (nx + ny + k);
    cplx<T> X[3], Y[3], Z[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) { X[d] = tx[d]; Y[d] = ty[d]; Z[d] = tz[d]; }

    const T a2 = (T)w.a2, a3 = (T)w.a3, m0 = (T)w.m0, m1 = (T)w.m1, m2 = (T)w.m2, m3 = (T)w.m3;

#pragma unroll
    for (int dz = -1; dz <= 1; ++dz) {
        const int kk = k + dz;
        if (kk < 0 || kk >= nz) continue;
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy) {
            const int jj = j + dy;
            if (jj < 0 || jj >= ny) continue;
            const cplx<T> Yd = Y[dy + 1], Zd = Z[dz + 1];
            const cplx<T> yz = Yd * Zd;
            const cplx<T> ye = (dz == 0) ? Yd : zero;       // Y e_z
            const cplx<T> ez = (dy == 0) ? Zd : zero;       // e_y Z
            const T ee = (dy == 0 && dz == 0) ? (T)1 : (T)0;
            cplx<T> Ac = a3 * yz + a2 * (ye + ez);
            Ac.x += ee;
            const cplx<T> Bc = ye + ez + a2 * yz;
            const T Py = (dy == 0) ? (T)-2 : (T)1, Pz = (dz == 0) ? (T)-2 : (T)1;
            const T pe = (dz == 0) ? Py : (T)0;
            const T ep = (dy == 0) ? Pz : (T)0;
            const T pp = Py * Pz;
            const T Am = m1 * ee + m2 * (pe + ep) + m3 * pp;
            const T Bm = m0 * ee + m1 * (pe + ep) + m2 * pp;
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                const int ii = i + dx;
                if (ii < 0 || ii >= nx) continue;
                cplx<T> lap = X[dx + 1] * Ac;
                T mass = ((dx == 0) ? (T)-2 : (T)1) * Am;
                if (dx == 0) { lap = lap + Bc; mass += Bm; }
                const long long dq = dz * nxy + dy * nx + dx;
                const cplx<T> kq = kp[dq];
                cplx<T> coef = mk<T>(lap.x * ih2 + mass * kq.x, lap.y * ih2 + mass * kq.y);
                const CPack<T, RCH> uq = *reinterpret_cast<const CPack<T, RCH>*>(up + dq * nrhs);
#pragma unroll
                for (int r = 0; r < RCH; ++r) cmac(acc[r], coef, uq.v[r]);
            }
        }
    }
    }
    CPack<T, RCH> out;
    if (SUB) {
        const CPack<T, RCH> bp = *reinterpret_cast<const CPack<T, RCH>*>(b + p * nrhs + (long long)ch * RCH);
#pragma unroll
        for (int r = 0; r < RCH; ++r) out.v[r] = bp.v[r] - acc[r];
    } else {
#pragma unroll
        for (int r = 0; r < RCH; ++r) out.v[r] = acc[r];
    }
    *reinterpret_cast<CPack<T, RCH>*>(y + p * nrhs + (long long)ch * RCH) = out;
}

// ---------------------------------------------------------------- z-march
//
// The same operator grouped by z-planes.  A thread owns MN consecutive x-nodes of one row and one vector V of
// columns (two complex64, one complex64 or one complex128) and walks a run of output planes; for every plane q
// it forms the in-plane terms of its nodes once and adds plane q's contribution to the outputs q - 1 (its last
// term, then stored), q and q + 1 (its first term), so each output costs (MN + 2) * 3 / MN vector loads instead of
// 27 and the sums over the rows and the x-neighbours are shared.  Per plane a warp takes one of three forms:
//
// * class sums with the mass term folded in (all coefficients plain (1, -2, 1), k^2 real): a neighbour's
//   coefficient is a_c = Lc_c / h^2 + Mc_c k^2, c = centre, face, edge, corner, four reals per node formed once
//   per block and plane (shared memory) and used by all columns.  With s_y the sum over the rows j -+ 1:
//     Q1 = s_y (a_3 u) + a_2 u,  Q0 = s_y (a_2 u) + a_1 u,  R0 = s_y (a_1 u) + a_0 u    (per x-column)
//     outputs q -+ 1 += Q1(i - 1) + Q1(i + 1) + Q0(i),   output q += Q0(i - 1) + Q0(i + 1) + R0(i).
//   19 real multiply-adds per complex value at MN = 4 and 17 at MN = 8 (the per-node kernel: 54 and the
//   coefficients).
// * class sums of u and of v = k^2 u apart (plain coefficients, complex k^2).
// * the product form (absorbing layers): with D_a the stretched second differences and a2, a3 the stencil's
//   product weights, S0 = D_x p + D_y u, S1 = D_x r + p, p = u + a2 D_y u, r = a2 u + a3 D_y u, and plane q adds
//   h^-2 (S0 + z_c S1) to output q and h^-2 z_-+ S1 to its neighbours; the mass term in class sums of v.
//
// The choice is made per warp in x and y and per plane in z, so a run may pass from the interior into the bottom
// layer.  A plane's neighbourhood ((GX MN + 2) x (MTY + 2) nodes, PC vectors each, and k^2) is copied into one
// of three shared-memory buffers with cp.async two planes ahead; the source offsets are formed once per thread,
// not per plane.  Ghost nodes are zero-filled by the copy.
//
// complex128 is bound by the FP64 pipe (two lanes per SM and clock): the form with the fewest FP64 operations is
// taken wherever it holds, and plain axes are tested at run time in the product form too.  112^3 x 16: 2.84 ms
// (per-node kernel 5.1 ms), 87 % of the pipe while a block runs; 101 x 93 x 77 x 10: 1.30 (2.54) ms; 48^3 x 1: 0.11
// (0.18) ms.  complex64 is bound by instruction latency at 12 warps per SM (issue 38 to 44 % active on a slab of 24
// planes, DRAM a third of its rate at 112^3): 112^3 x 16 163 us (per-node 361), 160 x 160 x 80 x 128 with complex k^2 1.40
// (5.07) ms, 101 x 93 x 77 x 10 85 (168) us; in brackets the per-node kernel throughout.  MN = 2 (more warps) measured 247
// and MN = 8 171 us at 112^3 x 16 when MN = 4 took 170 (163 since the tile is chosen by total work), so 4.
struct PlainRange {
    int lo[3], hi[3];   // per axis: indices whose stretched coefficients are exactly (1, -2, 1)
};

// Vectors of complex values: float4 (two complex64) and float2 (one), processed as (re, im) pairs by the packed
// FP32 instructions (two lanes per instruction, each rounded like the scalar operation), and double2.
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 cat4(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }
__device__ __forceinline__ float2 sw2(float2 a) { return make_float2(a.y, a.x); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(make_float2(-1.f, -1.f), b, a); }
__device__ __forceinline__ float2 vscal(float s, float2 b) { return __fmul2_rn(make_float2(s, s), b); }
__device__ __forceinline__ float2 vscal(float2 s, float2 b) { return __fmul2_rn(s, b); }
__device__ __forceinline__ float2 vaxpy(float2 s, float2 b, float2 a) { return __ffma2_rn(s, b, a); }
__device__ __forceinline__ float2 vaxpy(float s, float2 b, float2 a) { return __ffma2_rn(make_float2(s, s), b, a); }
__device__ __forceinline__ float4 vadd(float4 a, float4 b) { return cat4(vadd(lo2(a), lo2(b)), vadd(hi2(a), hi2(b))); }
__device__ __forceinline__ float4 vsub(float4 a, float4 b) { return cat4(vsub(lo2(a), lo2(b)), vsub(hi2(a), hi2(b))); }
__device__ __forceinline__ float4 vscal(float s, float4 b) { return cat4(vscal(s, lo2(b)), vscal(s, hi2(b))); }
__device__ __forceinline__ float4 vaxpy(float s, float4 b, float4 a) {
    return cat4(vaxpy(s, lo2(b), lo2(a)), vaxpy(s, hi2(b), hi2(a)));
}
__device__ __forceinline__ float4 vscal(float2 s, float4 b) { return cat4(vscal(s, lo2(b)), vscal(s, hi2(b))); }
__device__ __forceinline__ float4 vaxpy(float2 s, float4 b, float4 a) {
    return cat4(vaxpy(s, lo2(b), lo2(a)), vaxpy(s, hi2(b), hi2(a)));
}
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 vsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 vscal(double s, double2 b) { return make_double2(s * b.x, s * b.y); }
__device__ __forceinline__ double2 vaxpy(double s, double2 b, double2 a) {
    return make_double2(fma(s, b.x, a.x), fma(s, b.y, a.y));
}
// c b and a + c b for a complex coefficient c
__device__ __forceinline__ float2 vcmul(c64 c, float2 b) {
    return __ffma2_rn(make_float2(c.x, c.x), b, __fmul2_rn(make_float2(-c.y, c.y), sw2(b)));
}
__device__ __forceinline__ float2 vcaxpy(c64 c, float2 b, float2 a) {
    return __ffma2_rn(make_float2(c.x, c.x), b, __ffma2_rn(make_float2(-c.y, c.y), sw2(b), a));
}
__device__ __forceinline__ float4 vcmul(c64 c, float4 b) { return cat4(vcmul(c, lo2(b)), vcmul(c, hi2(b))); }
__device__ __forceinline__ float4 vcaxpy(c64 c, float4 b, float4 a) {
    return cat4(vcaxpy(c, lo2(b), lo2(a)), vcaxpy(c, hi2(b), hi2(a)));
}
__device__ __forceinline__ double2 vcmul(c128 c, double2 b) {
    return make_double2(fma(c.x, b.x, -c.y * b.y), fma(c.x, b.y, c.y * b.x));
}
__device__ __forceinline__ double2 vcaxpy(c128 c, double2 b, double2 a) {
    return make_double2(fma(c.x, b.x, fma(-c.y, b.y, a.x)), fma(c.x, b.y, fma(c.y, b.x, a.y)));
}

template <typename V> struct VTraits;
template <> struct VTraits<float4> {
    typedef float T;
    typedef float4 Coef;   // a complex coefficient as (re, re, im, im)
    typedef float2 Real;   // a real coefficient as (a, a), the packed instructions' operand
    static __device__ __forceinline__ float4 zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
};
template <> struct VTraits<float2> {
    typedef float T;
    typedef float4 Coef;
    typedef float2 Real;
    static __device__ __forceinline__ float2 zero() { return make_float2(0.f, 0.f); }
};
template <> struct VTraits<double2> {
    typedef double T;
    typedef c128 Coef;
    typedef double Real;
    static __device__ __forceinline__ double2 zero() { return make_double2(0.0, 0.0); }
};
__device__ __forceinline__ void make_coef(c64 c, float4& o) { o = make_float4(c.x, c.x, c.y, c.y); }
__device__ __forceinline__ void make_coef(c128 c, c128& o) { o = c; }
__device__ __forceinline__ void make_real(float a, float2& o) { o = make_float2(a, a); }
__device__ __forceinline__ void make_real(double a, double& o) { o = a; }

// c0 x0 + c1 x1 + c2 x2 with complex coefficients.  Packed FP32: the real-coefficient and the imaginary-coefficient
// sums are formed first and combined once (one swap instead of three).
__device__ __forceinline__ float2 d3c(const float4* c, float2 x0, float2 x1, float2 x2) {
    const float2 r = __ffma2_rn(lo2(c[2]), x2, __ffma2_rn(lo2(c[1]), x1, __fmul2_rn(lo2(c[0]), x0)));
    const float2 i = __ffma2_rn(hi2(c[2]), x2, __ffma2_rn(hi2(c[1]), x1, __fmul2_rn(hi2(c[0]), x0)));
    return __ffma2_rn(make_float2(-1.f, 1.f), sw2(i), r);
}
__device__ __forceinline__ float4 d3c(const float4* c, float4 x0, float4 x1, float4 x2) {
    return cat4(d3c(c, lo2(x0), lo2(x1), lo2(x2)), d3c(c, hi2(x0), hi2(x1), hi2(x2)));
}
__device__ __forceinline__ double2 d3c(const c128* c, double2 x0, double2 x1, double2 x2) {
    return vcaxpy(c[2], x2, vcaxpy(c[1], x1, vcmul(c[0], x0)));
}
// x0 - 2 x1 + x2
template <typename V> __device__ __forceinline__ V d3p(V x0, V x1, V x2) {
    return vaxpy((typename VTraits<V>::T)-2, x1, vadd(x0, x2));
}

template <int BYTES>
__device__ __forceinline__ void cp_async(void* sdst, const void* gsrc, bool valid) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(sdst));
    if (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(gsrc), "r"(valid ? 16 : 0) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(gsrc), "r"(valid ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

constexpr int MTHREADS = 128;   // threads per block
constexpr int MNBUF = 3;        // plane buffers: q is computed while q + 1 and q + 2 arrive

// The stencil's constants in the working precision, formed on the host (the class constants Lc / h^2 and Mc).
template <typename T>
struct MarchW {
    T L[4], M[4], a2, a3, ih2;
};

// A block's tile: PC column vectors x GX groups of MN x-nodes x MTY rows, one thread each.
struct MarchTile {
    int pc, gx, mty;   // gx groups of MN nodes
    int ncc;           // chunks of the columns
    int threads, mzc;  // threads per block, planes per block
};

// The vectors of one plane buffer a thread copies at most (the tile is chosen within it).
template <typename V> struct MarchCfg;
template <> struct MarchCfg<float4> { static constexpr int MN = 4, NU = 7, BPS = 3, WORK = 110, LAT = 3600; };
template <> struct MarchCfg<float2> { static constexpr int MN = 4, NU = 8, BPS = 5, WORK = 75, LAT = 3600; };
template <> struct MarchCfg<double2> { static constexpr int MN = 4, NU = 8, BPS = 2, WORK = 2900, LAT = 2000; };

template <typename V>
__host__ __device__ constexpr size_t march_smem(int pc, int gx, int mty) {
    typedef typename VTraits<V>::T T;
    const size_t ek = (size_t)(mty + 2) * (gx * MarchCfg<V>::MN + 2);
    return ek * 4 * sizeof(typename VTraits<V>::Real) + MNBUF * ek * pc * sizeof(V) + (size_t)gx * MarchCfg<V>::MN * 3 * sizeof(typename VTraits<V>::Coef) +
           MNBUF * ek * sizeof(cplx<T>);
}

// grid: (x tiles, row tiles, plane chunks x column chunks); the column chunk is the fastest part of blockIdx.z
template <typename V, bool SUB, bool REALK>
__global__ void __launch_bounds__(MTHREADS, MarchCfg<V>::BPS)
    stencil_march(const V* __restrict__ u, const V* __restrict__ b, V* __restrict__ y,
                  const cplx<typename VTraits<V>::T>* __restrict__ k2, const cplx<typename VTraits<V>::T>* __restrict__ tab,
                  int nx, int ny, int nz, int nrs, MarchTile tl, MarchW<typename VTraits<V>::T> w, PlainRange pl) {
    typedef typename VTraits<V>::T T;
    typedef typename VTraits<V>::Coef Coef;
    typedef typename VTraits<V>::Real Real;
    typedef cplx<T> C;
    constexpr int MN = MarchCfg<V>::MN, NU = MarchCfg<V>::NU;
    struct __align__(16) A4 { Real v[4]; };
    extern __shared__ __align__(16) unsigned char march_sm[];
    const int PC = tl.pc, MBX = tl.gx * MN + 2, EK = (tl.mty + 2) * MBX, EU = EK * PC;
    A4* sa = reinterpret_cast<A4*>(march_sm);
    Coef* sx = reinterpret_cast<Coef*>(sa + EK);
    V* su = reinterpret_cast<V*>(sx + tl.gx * MN * 3);
    C* sk = reinterpret_cast<C*>(su + MNBUF * EU);

    const int tid = threadIdx.x;
    // the last planes (the bottom layer, the longer work) first
    const int cc = blockIdx.z % tl.ncc, zc = (gridDim.z - 1 - blockIdx.z) / tl.ncc;
    const int i0 = blockIdx.x * tl.gx * MN, j0 = blockIdx.y * tl.mty;
    const int nth = blockDim.x;
    const int k0 = zc * tl.mzc, k1 = min(k0 + tl.mzc, nz);
    // columns fastest, then rows, then x-groups, so that a warp spans few rows and groups and its form is seldom mixed
    const int pc = tid % PC, jr = (tid / PC) % tl.mty, g = tid / (PC * tl.mty);
    const int j = j0 + jr, ib = i0 + g * MN;
    const bool live = g < tl.gx && j < ny && ib < nx && cc * PC + pc < nrs;
    const int xbs = min(g, tl.gx - 1) * MN;   // nodes read by threads past the tile (their values are never stored)
    const long long pln = (long long)nx * ny * nrs;

    // source offsets of this thread's copies inside a plane
    int off[NU];
    uint32_t ok = 0;
#pragma unroll
    for (int i = 0; i < NU; ++i) {
        const int e = tid + i * nth;
        off[i] = 0;
        if (e < EU) {
            const int c = e % PC, xn = (e / PC) % MBX, yr = e / (PC * MBX);
            const int ii = i0 + xn - 1, jj = j0 + yr - 1;
            if (ii >= 0 && ii < nx && jj >= 0 && jj < ny && cc * PC + c < nrs) {
                off[i] = (jj * nx + ii) * nrs + cc * PC + c;
                ok |= 1u << i;
            }
        }
    }
    int koff[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int e = tid + i * nth;
        const int ii = i0 + e % MBX - 1, jj = j0 + e / MBX - 1;
        const bool in = ii >= 0 && ii < nx && jj >= 0 && jj < ny;
        koff[i] = in ? jj * nx + ii : 0;
        if (in) ok |= 1u << (30 + i);
    }
    auto stage = [&](int buf, int q) {
        if (q >= 0 && q < nz) {
            const V* src = u + q * pln;
            V* dst = su + buf * EU + tid;
#pragma unroll
            for (int i = 0; i < NU; ++i)
                if (tid + i * nth < EU) cp_async<sizeof(V)>(dst + i * nth, src + off[i], (ok >> i) & 1u);
            const C* ks = k2 + (long long)q * nx * ny;
            C* kd = sk + buf * EK;
#pragma unroll
            for (int i = 0; i < 2; ++i)
                if (tid + i * nth < EK) cp_async<sizeof(C)>(kd + tid + i * nth, ks + koff[i], (ok >> (30 + i)) & 1u);
            for (int e = tid + 2 * nth; e < EK; e += nth) {   // few columns: more nodes than two per thread
                const int ii = i0 + e % MBX - 1, jj = j0 + e / MBX - 1;
                const bool in = ii >= 0 && ii < nx && jj >= 0 && jj < ny;
                cp_async<sizeof(C)>(kd + e, ks + (in ? jj * nx + ii : 0), in);
            }
        }
        cp_async_commit();
    };

    // per warp: all its nodes have plain coefficients along x, along y (threads past the grid do not count)
    const bool px = __all_sync(0xffffffffu, !live || (ib >= pl.lo[0] && min(ib + MN, nx) - 1 <= pl.hi[0]));
    const bool py = __all_sync(0xffffffffu, !live || (j >= pl.lo[1] && j <= pl.hi[1]));
    for (int e = tid; e < tl.gx * MN * 3; e += nth) {
        Coef cf;
        make_coef(i0 + e / 3 < nx ? tab[3 * i0 + e] : mk<T>(0, 0), cf);
        sx[e] = cf;
    }
    Coef Y[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) make_coef(j < ny ? tab[3 * (nx + j) + d] : mk<T>(0, 0), Y[d]);
    const C* tz = tab + 3 * (nx + ny);
    V P[MN], N[MN];   // outputs q and q + 1, partial
#pragma unroll
    for (int c = 0; c < MN; ++c) P[c] = N[c] = VTraits<V>::zero();
    stage(0, k0 - 1);
    stage(1, k0);
    for (int q = k0 - 1, buf = 0; q <= k1; ++q, buf = buf == MNBUF - 1 ? 0 : buf + 1) {
        cp_async_wait<1>();   // plane q has arrived (plane q + 1 may still be in flight)
        __syncthreads();      // everyone's copies of q; and every thread is done with plane q - 1's buffer
        {
            const int nb = buf >= 1 ? buf - 1 : MNBUF - 1;
            if (q + 2 <= k1) stage(nb, q + 2);
            else cp_async_commit();
        }
        const bool qin = q >= 0 && q < nz;
        // plain coefficients for every output this plane contributes to
        const bool zp_ = max(q - 1, k0) >= pl.lo[2] && min(q + 1, k1 - 1) <= pl.hi[2];
        const bool plain = px && py && zp_;
        const C* ck = sk + buf * EK;
        if (REALK && zp_ && qin) {
            for (int e = tid; e < EK; e += nth) {
                const T kk = ck[e].x;
                A4 a;
#pragma unroll
                for (int c = 0; c < 4; ++c) make_real(fma(w.M[c], kk, w.L[c]), a.v[c]);
                sa[e] = a;
            }
            __syncthreads();
        }
        const bool out = live && q - 1 >= k0;
        V* yq = y + (q - 1) * pln + ((long long)j * nx + ib) * nrs + cc * PC + pc;
        V bq[MN];
        if (SUB) {
            const V* bp = b + (yq - y);
#pragma unroll
            for (int c = 0; c < MN; ++c) bq[c] = out && ib + c < nx ? __ldcs(bp + c * nrs) : VTraits<V>::zero();
        }
        // plane q's contributions to node c: am to output q - 1, a0 to q, ap to q + 1
        auto emit = [&](int c, V am, V a0, V ap) {
            if (out && ib + c < nx) {
                V o = vadd(P[c], am);
                if (SUB) o = vsub(bq[c], o);
                __stcs(yq + c * nrs, o);
            }
            P[c] = vadd(N[c], a0);
            N[c] = ap;
        };
        const V* cu = su + buf * EU + (jr * MBX + xbs) * PC + pc;
        if (!qin) {
#pragma unroll
            for (int c = 0; c < MN; ++c) emit(c, VTraits<V>::zero(), VTraits<V>::zero(), VTraits<V>::zero());
        } else if (REALK && plain) {
            const A4* ca = sa + jr * MBX + xbs;
            V Q1[3], Q0[3], R0[3];
            auto column = [&](int n, int s) {
                const V u0 = cu[n * PC], u1 = cu[(MBX + n) * PC], u2 = cu[(2 * MBX + n) * PC];
                const A4 a0 = ca[n], a1 = ca[MBX + n], a2 = ca[2 * MBX + n];
                Q1[s] = vaxpy(a1.v[2], u1, vaxpy(a2.v[3], u2, vscal(a0.v[3], u0)));
                Q0[s] = vaxpy(a1.v[1], u1, vaxpy(a2.v[2], u2, vscal(a0.v[2], u0)));
                R0[s] = vaxpy(a1.v[0], u1, vaxpy(a2.v[1], u2, vscal(a0.v[1], u0)));
            };
            column(0, 0);
            column(1, 1);
#pragma unroll
            for (int c = 0; c < MN; ++c) {
                column(c + 2, (c + 2) % 3);
                const int s0 = c % 3, s1 = (c + 1) % 3, s2 = (c + 2) % 3;
                const V A1 = vadd(vadd(Q1[s0], Q1[s2]), Q0[s1]);
                emit(c, A1, vadd(vadd(Q0[s0], Q0[s2]), R0[s1]), A1);
            }
        } else if (!REALK && plain) {
            const C* kp = ck + jr * MBX + xbs;
            V Cu[3], Cv[3], Yu[3], Yv[3];
            auto column = [&](int n, int s) {
                const V u0 = cu[n * PC], u1 = cu[(MBX + n) * PC], u2 = cu[(2 * MBX + n) * PC];
                Cu[s] = u1;
                Cv[s] = vcmul(kp[MBX + n], u1);
                Yu[s] = vadd(u0, u2);
                Yv[s] = vcaxpy(kp[2 * MBX + n], u2, vcmul(kp[n], u0));
            };
            column(0, 0);
            column(1, 1);
#pragma unroll
            for (int c = 0; c < MN; ++c) {
                column(c + 2, (c + 2) % 3);
                const int s0 = c % 3, s1 = (c + 1) % 3, s2 = (c + 2) % 3;
                const V cU = Cu[s1], cV = Cv[s1];
                const V FU = vadd(vadd(Cu[s0], Cu[s2]), Yu[s1]), EU_ = vadd(Yu[s0], Yu[s2]);
                const V FV = vadd(vadd(Cv[s0], Cv[s2]), Yv[s1]), EV = vadd(Yv[s0], Yv[s2]);
                const V A0 = vaxpy(w.M[2], EV, vaxpy(w.M[1], FV, vaxpy(w.M[0], cV, vaxpy(w.L[2], EU_, vaxpy(w.L[1], FU, vscal(w.L[0], cU))))));
                const V A1 = vaxpy(w.M[3], EV, vaxpy(w.M[2], FV, vaxpy(w.M[1], cV, vaxpy(w.L[3], EU_, vaxpy(w.L[2], FU, vscal(w.L[1], cU))))));
                emit(c, A1, A0, A1);
            }
        } else {
            const C* kp = ck + jr * MBX + xbs;
            const T ih2 = w.ih2, a2 = w.a2, a3 = w.a3;
            C zm = mk<T>(0, 0), zz = ih2 * tz[3 * q + 1], zp = mk<T>(0, 0);
            if (q >= 1) zm = ih2 * tz[3 * (q - 1) + 2];
            if (q + 1 < nz) zp = ih2 * tz[3 * (q + 1)];
            V Pw[3], Rw[3], Dy[3], Cv[3], Yv[3];
            auto column = [&](int n, int s) {
                const V u0 = cu[n * PC], u1 = cu[(MBX + n) * PC], u2 = cu[(2 * MBX + n) * PC];
                const V dy = py ? d3p(u0, u1, u2) : d3c(Y, u0, u1, u2);
                Pw[s] = vaxpy(a2, dy, u1);
                Rw[s] = vaxpy(a3, dy, vscal(a2, u1));
                Dy[s] = dy;
                if (REALK) {
                    Cv[s] = vscal(kp[MBX + n].x, u1);
                    Yv[s] = vaxpy(kp[2 * MBX + n].x, u2, vscal(kp[n].x, u0));
                } else {
                    Cv[s] = vcmul(kp[MBX + n], u1);
                    Yv[s] = vcaxpy(kp[2 * MBX + n], u2, vcmul(kp[n], u0));
                }
            };
            column(0, 0);
            column(1, 1);
#pragma unroll
            for (int c = 0; c < MN; ++c) {
                column(c + 2, (c + 2) % 3);
                const int s0 = c % 3, s1 = (c + 1) % 3, s2 = (c + 2) % 3;
                const Coef* X = sx + (xbs + c) * 3;
                V S0, S1;
                if (px) {
                    S0 = d3p(Pw[s0], Pw[s1], Pw[s2]);
                    S1 = d3p(Rw[s0], Rw[s1], Rw[s2]);
                } else {
                    S0 = d3c(X, Pw[s0], Pw[s1], Pw[s2]);
                    S1 = d3c(X, Rw[s0], Rw[s1], Rw[s2]);
                }
                S0 = vadd(S0, Dy[s1]);
                S1 = vadd(S1, Pw[s1]);
                const V FV = vadd(vadd(Cv[s0], Cv[s2]), Yv[s1]), EV = vadd(Yv[s0], Yv[s2]);
                const V B0 = vaxpy(ih2, S0, vaxpy(w.M[2], EV, vaxpy(w.M[1], FV, vscal(w.M[0], Cv[s1]))));
                const V B1 = vaxpy(w.M[3], EV, vaxpy(w.M[2], FV, vscal(w.M[1], Cv[s1])));
                if (zp_) {
                    const V A1 = vaxpy(ih2, S1, B1);
                    emit(c, A1, vaxpy((T)-2 * ih2, S1, B0), A1);
                } else {
                    emit(c, vcaxpy(zm, S1, B1), vcaxpy(zz, S1, B0), vcaxpy(zp, S1, B1));
                }
            }
        }
    }
    cp_async_wait<0>();
}

struct RowW {
    const StencilW* wtab;
    const unsigned char* wbin;
};

template <typename T, int RCH, bool SUB, int NR = 0>
void launch_t(const cplx<T>* u, const cplx<T>* b, cplx<T>* y, const cplx<T>* k2, const cplx<T>* tab,
              const helm_grid_desc& d, int nrhs, const StencilW& w, const Interior& in, bool realk, RowW rw,
              cudaStream_t s) {
    const int threads = 128;
    const dim3 grid((unsigned)((d.nx * (nrhs / RCH) + threads - 1) / threads), (unsigned)d.ny, (unsigned)d.nz);
    if (realk)
        stencil_kernel<T, RCH, SUB, true, NR><<<grid, threads, 0, s>>>(u, b, y, k2, tab, d.nx, d.ny, d.nz, nrhs, w, in,
                                                                       rw.wtab, rw.wbin);
    else
        stencil_kernel<T, RCH, SUB, false, NR><<<grid, threads, 0, s>>>(u, b, y, k2, tab, d.nx, d.ny, d.nz, nrhs, w,
                                                                        in, rw.wtab, rw.wbin);
}

template <typename T, bool SUB>
void dispatch(const cplx<T>* u, const cplx<T>* b, cplx<T>* y, const cplx<T>* k2, const cplx<T>* tab,
              const helm_grid_desc& d, int nrhs, const StencilW& w, const Interior& in, bool realk, RowW rw,
              cudaStream_t s) {
    // complex64: one 16-byte vector per thread and neighbour, two columns when the column count is
    // even and every base address is 16-byte aligned, else one.  complex128 (FP64-pipe bound on this
    // part): up to four columns per thread, so each neighbour's coefficient is formed once for four
    // (a pack of RCH values is loaded as one aligned object: every base address must be aligned to it)
    const auto al = [&](uintptr_t a) {
        return ((uintptr_t)u & (a - 1)) == 0 && ((uintptr_t)y & (a - 1)) == 0 && (!SUB || ((uintptr_t)b & (a - 1)) == 0);
    };
    if constexpr (sizeof(T) == 4) {
        if (nrhs == 16 && al(16))
            launch_t<T, 2, SUB, 16>(u, b, y, k2, tab, d, nrhs, w, in, realk, rw, s);
        else if (nrhs % 2 == 0 && al(16))
            launch_t<T, 2, SUB>(u, b, y, k2, tab, d, nrhs, w, in, realk, rw, s);
        else
            launch_t<T, 1, SUB>(u, b, y, k2, tab, d, nrhs, w, in, realk, rw, s);
    } else {
        if (nrhs % 4 == 0 && al(64)) launch_t<T, 4, SUB>(u, b, y, k2, tab, d, nrhs, w, in, realk, rw, s);
        else if (nrhs % 2 == 0 && al(32)) launch_t<T, 2, SUB>(u, b, y, k2, tab, d, nrhs, w, in, realk, rw, s);
        else launch_t<T, 1, SUB>(u, b, y, k2, tab, d, nrhs, w, in, realk, rw, s);
    }
}

Interior interior_of(helm_grid g) {
    const helm_grid_desc& d = g->d;
    Interior in;
    const int n[3] = {d.nx, d.ny, d.nz};
    for (int a = 0; a < 3; ++a) {
        const bool low = a < 2 || d.top_bc == HELM_TOP_PML;
        in.lo[a] = std::max(1, low && d.npml > 0 ? d.npml + 1 : 1);
        in.hi[a] = n[a] - 2 - (d.npml > 0 ? d.npml : 0);
    }
    const double a2 = g->w.a2, a3 = g->w.a3;
    in.Lc[0] = -6.0 + 12.0 * a2 - 8.0 * a3;
    in.Lc[1] = 1.0 - 4.0 * a2 + 4.0 * a3;
    in.Lc[2] = a2 - 2.0 * a3;
    in.Lc[3] = a3;
    const double m0 = g->w.m0, m1 = g->w.m1, m2 = g->w.m2, m3 = g->w.m3;
    in.Mc[0] = m0 - 6.0 * m1 + 12.0 * m2 - 8.0 * m3;
    in.Mc[1] = m1 - 4.0 * m2 + 4.0 * m3;
    in.Mc[2] = m2 - 2.0 * m3;
    in.Mc[3] = m3;
    return in;
}

// Per axis, the index range whose stretched coefficients are exactly (1, -2, 1) (the table is contiguous-plain in the
// middle and stretched in the absorbing layers); empty if not contiguous.  Tested in complex64 for both types: a stretched
// coefficient has an imaginary part, which only rounds away below 1e-45, where complex128 results do not see it either.
PlainRange plain_range(helm_grid g) {
    PlainRange r;
    const int n[3] = {g->d.nx, g->d.ny, g->d.nz};
    int base = 0;
    for (int a = 0; a < 3; ++a) {
        auto plain = [&](int i) {
            const c128* c = &g->htab[3 * (base + i)];
            return (float)c[0].x == 1.f && (float)c[0].y == 0.f && (float)c[1].x == -2.f && (float)c[1].y == 0.f &&
                   (float)c[2].x == 1.f && (float)c[2].y == 0.f;
        };
        int lo = 0, hi = n[a] - 1;
        while (lo < n[a] && !plain(lo)) ++lo;
        while (hi >= 0 && !plain(hi)) --hi;
        for (int i = lo; i <= hi; ++i)
            if (!plain(i)) {
                lo = 1;
                hi = 0;
                break;
            }
        r.lo[a] = lo;
        r.hi[a] = hi;
        base += n[a];
    }
    return r;
}

// The tile of the z-march: PC column vectors (at most 8, the chunks of equal width), and the x-groups, rows and planes
// per block with the least estimated time on this grid: the blocks' walks (two planes of halo each), a plane costing
// its latency and the schedulers' work on it.
template <typename V>
MarchTile march_tile(const helm_grid_desc& d, int nrs, int sms, int planes) {
    constexpr int MN = MarchCfg<V>::MN;
    MarchTile t{};
    t.ncc = (nrs + 7) / 8;
    t.pc = (nrs + t.ncc - 1) / t.ncc;
    double best = 1e300;
    for (int gx = 1; gx <= 32 && (gx == 1 || (gx - 1) * MN < d.nx); gx *= 2)
        for (int warps = 1; warps <= MTHREADS / 32; warps *= 2) {
            const int rows = std::min(warps * 32 / (t.pc * gx), d.ny);
            if (rows < 1) continue;
            const int threads = (rows * t.pc * gx + 31) / 32 * 32;
            const long long eu = (long long)(rows + 2) * (gx * MN + 2) * t.pc;
            if (eu > (long long)MarchCfg<V>::NU * threads) continue;
            const int per_sm = std::min(MarchCfg<V>::BPS * MTHREADS / threads, (int)(227 * 1024 / (march_smem<V>(t.pc, gx, rows) + 1024)));
            if (per_sm < 1) continue;
            const double xy = (double)((d.nx + gx * MN - 1) / (gx * MN)) * ((d.ny + rows - 1) / rows) * t.ncc;
            for (int nch = 1; nch <= d.nz; ++nch) {
                const int mzc = planes ? std::min(planes, d.nz) : (d.nz + nch - 1) / nch;
                if (!planes && mzc > 64) continue;
                if (!planes && mzc < 4 && nch > 1) break;
                const double blocks = xy * ((d.nz + mzc - 1) / mzc), slots = (double)per_sm * sms;
                // clocks of one plane with res blocks on an SM: a warp's latency, or its scheduler's work
                auto plane = [&](double res) {
                    const double warps = std::ceil(res * (threads / 32) / 4.0);   // per scheduler
                    return MarchCfg<V>::LAT + warps * MarchCfg<V>::WORK * MN;
                };
                // blocks are replaced as they finish, so the total work spread over the slots, but no less than one walk,
                // and a quarter of a walk of tail
                const double walk = (mzc + 2) * plane(std::min((double)per_sm, std::ceil(blocks / sms)));
                const double time = std::max(blocks * (mzc + 2) * plane(per_sm) / slots, walk) + 0.25 * walk;
                if (time < best) {
                    best = time;
                    t.gx = gx;
                    t.mty = rows;
                    t.threads = threads;
                    t.mzc = mzc;
                }
                if (planes) break;
            }
        }
    return t;
}

// Launch of the z-march; false when it does not apply (the per-node kernel then runs).
template <typename V, bool SUB>
bool launch_march(helm_grid g, const void* u, const void* b, void* y, int nrs, cudaStream_t s) {
    typedef typename VTraits<V>::T T;
    const helm_grid_desc& d = g->d;
    if ((long long)d.nx * d.ny * nrs >= (1ll << 31)) return false;   // 32-bit offsets inside a plane
    const MarchTile t = march_tile<V>(d, nrs, std::max(g->ctx->sm_count, 1), g->ctx->stencil_planes);
    if (!t.gx) return false;
    const size_t smem = march_smem<V>(t.pc, t.gx, t.mty);
    const int gx = (d.nx + t.gx * MarchCfg<V>::MN - 1) / (t.gx * MarchCfg<V>::MN), gy = (d.ny + t.mty - 1) / t.mty;
    const long long gz = (long long)((d.nz + t.mzc - 1) / t.mzc) * t.ncc;
    if (gy > 65535 || gz > 65535) return false;
    const PlainRange pl = plain_range(g);
    const cplx<T>* k2 = sizeof(T) == 8 ? (const cplx<T>*)g->k2 : (const cplx<T>*)g->k2f;
    const cplx<T>* tab = sizeof(T) == 8 ? (const cplx<T>*)g->tab : (const cplx<T>*)g->tabf;
    const Interior in = interior_of(g);
    MarchW<T> w;
    for (int c = 0; c < 4; ++c) {
        w.L[c] = (T)(in.Lc[c] * g->w.inv_h2);
        w.M[c] = (T)in.Mc[c];
    }
    w.a2 = (T)g->w.a2;
    w.a3 = (T)g->w.a3;
    w.ih2 = (T)g->w.inv_h2;
    const dim3 grid((unsigned)gx, (unsigned)gy, (unsigned)gz);
    static PerDevice attr;
    if (!attr.done(g->ctx->device)) {
        cudaFuncSetAttribute(stencil_march<V, SUB, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
        cudaFuncSetAttribute(stencil_march<V, SUB, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
        attr.mark(g->ctx->device);
    }
    if (g->k2_real)
        stencil_march<V, SUB, true><<<grid, t.threads, smem, s>>>((const V*)u, (const V*)b, (V*)y, k2, tab, d.nx, d.ny,
                                                                  d.nz, nrs, t, w, pl);
    else
        stencil_march<V, SUB, false><<<grid, t.threads, smem, s>>>((const V*)u, (const V*)b, (V*)y, k2, tab, d.nx, d.ny,
                                                                   d.nz, nrs, t, w, pl);
    return true;
}

template <bool SUB>
helm_status launch_any(helm_grid g, int prec, const void* u, const void* b, void* y, int nrhs, cudaStream_t s) {
    if (nrhs <= 0) return HELM_OK;
    // algorithmic bytes: read u (and b), write y, read k^2 once
    const double es = prec == HELM_PREC_FP64 ? sizeof(c128) : sizeof(c64);
    const double bytes = (double)g->n * es * ((SUB ? 3.0 : 2.0) * nrhs + 1.0);
    const int tok = prof_begin(g->ctx, prec == HELM_PREC_FP64 ? "stencil64" : "stencil");
    const Interior in = interior_of(g);
    const RowW rw{g->wtab, g->wbin};
    const uintptr_t al = (uintptr_t)u | (uintptr_t)y | (SUB ? (uintptr_t)b : 0);
    bool done = false;
    // complex64 calls of fewer than 2^20 values run the per-node kernel: a walk's planes are a serial chain, and too
    // few blocks hide its latency (48^3 x 1: 27 us per call against 38; 64^3 x 4, 2^20 values: 44 against 40;
    // 112^3 x 1: 77 against 74).  complex128 is FP64-bound sooner, and the per-node kernel
    // forms its coefficients per node: below 40,000 nodes and 90,000 values (per-node against walk, us: 30 x 33 x 29 x 1 66,
    // 106; 33 x 40 x 25 x 2 96, 106; 36^3 x 1 118, 107; 40^3 x 1 136, 106; 32^3 x 3 123, 103).
    const bool walk = g->ctx->stencil_march == 2 || g->ctx->stencil_planes ||
                      (prec == HELM_PREC_FP64 ? g->n >= 40000 || g->n * nrhs >= 90000 : g->n * nrhs >= (1 << 20));
    if (g->ctx->stencil_march && !g->wtab && walk) {
        if (prec == HELM_PREC_FP64) done = (al & 15) == 0 && launch_march<double2, SUB>(g, u, b, y, nrhs, s);
        else if (nrhs % 2 == 0 && (al & 15) == 0) done = launch_march<float4, SUB>(g, u, b, y, nrhs / 2, s);
        else done = (al & 7) == 0 && launch_march<float2, SUB>(g, u, b, y, nrhs, s);
    }
    if (done) {
    } else if (prec == HELM_PREC_FP64) {
        dispatch<double, SUB>((const c128*)u, (const c128*)b, (c128*)y, g->k2, g->tab, g->d, nrhs, g->w, in,
                              g->k2_real, rw, s);
    } else {
        dispatch<float, SUB>((const c64*)u, (const c64*)b, (c64*)y, g->k2f, g->tabf, g->d, nrhs, g->w, in,
                             g->k2_real, rw, s);
    }
    prof_end(g->ctx, tok, bytes);
    HELM_LAUNCH_CHECK(g->ctx, "stencil_kernel");
    return HELM_OK;
}

}  // namespace

helm_status launch_stencil(helm_grid g, int prec, const void* u, void* y, int nrhs, cudaStream_t s) {
    return launch_any<false>(g, prec, u, nullptr, y, nrhs, s);
}

helm_status launch_stencil_sub(helm_grid g, int prec, const void* u, const void* b, void* y, int nrhs, cudaStream_t s) {
    return launch_any<true>(g, prec, u, b, y, nrhs, s);
}
