// complex128 plane inverses on the tensor cores: G = S^{-1} in FP64 from the complex64 inverse X0 of the tensor-core
// elimination (planelu_tc.cu) by two Newton steps X <- X + X (I - S X), whose products are sums of small integers.
//
// Why: the FP64 pipe of this part does two multiply-adds per SM and clock, so the block elimination in FP64 (planelu.cu)
// runs at 1.0 TFLOP/s at best and inverts one 32 x 32 block at a time beside it.  The products here run as BF16 MMAs.
//
// Slices (the Ozaki scheme): a row of the left operand, or a column of the right one, is scaled by a power of two so that
// its entries lie in (-1, 1) and written as digits d_0, d_1, ... in base 256, |d_i| <= 128, x = 2^(e-7) sum d_i 256^-i.
// Digits are exact in BF16 and a product of two is an integer of at most 2^14.  Orders are accumulated apart (one TMEM
// accumulator each), the products of the orders kept (i + j < O) are added as 64-bit integers and converted once.
// An FP32 accumulator is exact while its running sum stays below 2^24.  The digits' range does not ensure that (K <= 4608
// products of up to eight digit pairs), their distribution does: leading digits follow |S| |X|, whose rows decay from the
// diagonal (sums below 2^21), the others are as good as random, so that sums have a standard deviation of 2^20 at most
// (2^20 at 320 unknowns in an emulation), 2^24 being sixteen of them.  An accumulator that ends beyond 2^23 sets the flag
// that sends the set to the FP64 elimination; one that went beyond 2^24 and came back would be rounded there unseen.
//
// Precision.  X0 is cut to 3 digits (24 bits of its column's largest entry) and taken as exact.  R0 = I - S X0 with 5
// digits of S (2^-40), X1 = X0 + X0 R0 cut to 5 digits, R1 = I - S X1 with all 8 digits of S (64 bits below its row's largest
// entry) and the orders 0..7, X = X1 + X1 R1.  The error left is |R1|^2 and R1's own, of which the orders left out are the
// larger part: sums of about 2^19 at 2^-64 of the scale 2^14, 2^-59 of |S| |X| (with 7 digits and orders: 2^-51, and
// residuals 20 times an FP64 elimination's).  Where an entry of R1 exceeds 3e-10 (condition numbers of about 3e2 and
// more) the box takes a third step, with all 8 digits of X1: at 5 digits the cut alone leaves a residual of 2^-40 of |S| |X|,
// again above 3e-10, and an inverse up to four times as far off as an FP64 elimination's.  |R0| > 1e-3, |R1| > 1e-4 or a
// third residual above 1e-9 (condition numbers of about 1e5) sets the flag too.
//
// A product costs 36 (8 x 8 digits, 8 orders; third step), 30 (8 x 5 digits), 14, 8 or 6 BF16 MMAs; the matrices of a plane
// are read and written a few times.  Bound: the operands' loads (0.43 of the tensor pipe at 8 boxes of 676 unknowns: 30
// products 814 us, 14 464 us, 8 243 us; with 64-column tiles, half the instruction's rate, and four epilogue warps 1046,
// 593, 264 us), launches for small planes.
#include <cuda.h>
#include <cuda_bf16.h>

#include <atomic>

#include "internal.h"
#include "tc.cuh"
#include "tgj.h"

namespace {

constexpr int SAS = 8;    // digits of S
constexpr int SAX = 3;    // digits of X as a left operand
constexpr int SBM = 8;    // digits of a right operand at most
constexpr int GM = 128, GK = 64;
constexpr int A_SLOT = GM * 128;

__device__ __forceinline__ double pow2(int e) {
    e = min(max(e, -1022), 1023);
    return __longlong_as_double((long long)(e + 1023) << 52);
}

// exponent e with |x| < 2^e for every x whose high word (sign cleared) is at most hi; 0 for a zero row; flags rows that are
// not finite or out of the range in which the scales are normal numbers
__device__ __forceinline__ int exponent_of(uint32_t hi, int* flag) {
    const int E = (int)(hi >> 20);
    if (E == 0) return 0;
    if (E >= 1923 || E <= 123) atomicOr(flag, 4);
    return E - 1022;
}
__device__ __forceinline__ uint32_t high_word(double x) { return (uint32_t)(__double_as_longlong(x) >> 32) & 0x7FFFFFFFu; }

// the s digits of x 2^(8s - 1 - e), most significant first
template <int S>
__device__ __forceinline__ void digits(long long q, int (&d)[S]) {
#pragma unroll
    for (int i = S - 1; i > 0; --i) {
        d[i] = (int)((q + 128) & 255) - 128;
        q = (q - d[i]) >> 8;
    }
    d[0] = (int)q;
}

// Kernels of a step that only some boxes take: gate[box] holds the largest |R1| of the box's plane as float bits (null: all).
__device__ __forceinline__ bool gated_out(const int* gate, int box) {
    return gate && __int_as_float(gate[box]) <= 3e-10f;
}

// Left operand: row I of the matrix (pitch m or ld), S digits into slices [S][nb][Lr][Kp]; with S32 also the row as
// complex64 into the elimination's work matrix.
template <int S>
__global__ void __launch_bounds__(128) dp_slice_rows(const BoxInfo* __restrict__ boxes, const c128* __restrict__ src,
                                                     int from_g, int m_max, __nv_bfloat16* __restrict__ out, int nb, int Lr,
                                                     int Kp, int* __restrict__ eout, c64* __restrict__ S32, int L, int k,
                                                     int* __restrict__ flag, int* __restrict__ clear,
                                                     const int* __restrict__ gate) {
    __shared__ uint32_t red[4];
    const int box = blockIdx.y, I = blockIdx.x;
    const BoxInfo B = boxes[box];
    if (k >= B.dims[2] || I >= B.m || gated_out(gate, box)) return;
    if (clear && I == 0 && threadIdx.x == 0) clear[box] = 0;
    const int m = B.m;
    const c128* row = from_g ? src + B.fac_off + (long long)k * B.pstride + (long long)I * B.ld
                             : src + (size_t)box * m_max * m_max + (size_t)I * m;
    uint32_t hi = 0;
    for (int j = threadIdx.x; j < m; j += 128) hi = max(hi, max(high_word(row[j].x), high_word(row[j].y)));
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = hi;
    __syncthreads();
    hi = max(max(red[0], red[1]), max(red[2], red[3]));
    const int e = exponent_of(hi, flag);
    if (threadIdx.x == 0) eout[box * Lr + I] = e;
    const double sc = pow2(8 * S - 1 - e);
    const size_t plane = (size_t)nb * Lr * Kp;
    __nv_bfloat16* o = out + ((size_t)box * Lr + I) * Kp;
    for (int j = threadIdx.x; j < m; j += 128) {
        const c128 v = row[j];
        int dr[S], di[S];
        digits<S>(__double2ll_rn(v.x * sc), dr);
        digits<S>(__double2ll_rn(v.y * sc), di);
#pragma unroll
        for (int s = 0; s < S; ++s)
            *reinterpret_cast<__nv_bfloat162*>(o + s * plane + 2 * j) = __floats2bfloat162_rn((float)dr[s], (float)di[s]);
        if (S32) S32[((size_t)box * L + I) * L + j] = mk<float>((float)v.x, (float)v.y);
    }
}

// Where a right operand comes from: the complex64 work matrix (pitch L), a complex128 scratch (pitch m), or G.
struct ColSrc {
    const c64* s32;
    const c128* s64;   // [nb][m_max^2]
    const c128* g;
    int L, m_max;
};
__device__ __forceinline__ c128 col_at(const ColSrc& c, const BoxInfo& B, int box, int k, int p, int j) {
    if (c.s32) {
        const c64 v = c.s32[((size_t)box * c.L + p) * c.L + j];
        return mk<double>((double)v.x, (double)v.y);
    }
    if (c.s64) return c.s64[(size_t)box * c.m_max * c.m_max + (size_t)p * B.m + j];
    return c.g[B.fac_off + (long long)k * B.pstride + (long long)p * B.ld + j];
}

// exponents of the columns: 32 columns per block, 32 rows at a time
__global__ void __launch_bounds__(1024) dp_col_exponents(const BoxInfo* __restrict__ boxes, ColSrc src, int* __restrict__ eout,
                                                        int Lc, int k, int* __restrict__ flag,
                                                        const int* __restrict__ gate) {
    __shared__ uint32_t red[32][32];
    const int box = blockIdx.y;
    const BoxInfo B = boxes[box];
    if (k >= B.dims[2] || (int)blockIdx.x * 32 >= B.m || gated_out(gate, box)) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, j = blockIdx.x * 32 + lane;
    uint32_t hi = 0;
    if (j < B.m)
#pragma unroll 4
        for (int p = w; p < B.m; p += 32) {
            const c128 v = col_at(src, B, box, k, p, j);
            hi = max(hi, max(high_word(v.x), high_word(v.y)));
        }
    red[w][lane] = hi;
    __syncthreads();
    if (w == 0 && j < B.m) {
#pragma unroll
        for (int i = 1; i < 32; ++i) hi = max(hi, red[i][lane]);
        eout[box * Lc + j] = exponent_of(hi, flag);
    }
}

// Right operand: S digits of column j as rows 2j and 2j + 1 of the transposed 2x2 real embedding, slices [S][nb][Nr][Kp];
// with gout the values the digits stand for (the operand's exact value) are written back to G.  32 x 32 tiles.
template <int S>
__global__ void __launch_bounds__(256) dp_slice_cols(const BoxInfo* __restrict__ boxes, ColSrc src,
                                                     __nv_bfloat16* __restrict__ out, int nb, int Nr, int Kp,
                                                     const int* __restrict__ ein, c128* __restrict__ gout, int k,
                                                     const int* __restrict__ gate) {
    __shared__ __nv_bfloat162 t[S][32][33];   // [digit][column][row]
    const int box = blockIdx.z;
    const BoxInfo B = boxes[box];
    const int m = B.m, j0 = blockIdx.x * 32, p0 = blockIdx.y * 32;
    if (k >= B.dims[2] || j0 >= m || p0 >= m || gated_out(gate, box)) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, Lc = Nr / 2;
    const int j = j0 + lane;
    const int e = j < m ? ein[box * Lc + j] : 0;
    const double sc = pow2(8 * S - 1 - e), back = pow2(e + 1 - 8 * S);
    for (int i = w; i < 32; i += 8) {
        const int p = p0 + i;
        int dr[S], di[S];
#pragma unroll
        for (int s = 0; s < S; ++s) dr[s] = di[s] = 0;
        if (j < m && p < m) {
            const c128 v = col_at(src, B, box, k, p, j);
            const long long qr = __double2ll_rn(v.x * sc), qi = __double2ll_rn(v.y * sc);
            digits<S>(qr, dr);
            digits<S>(qi, di);
            if (gout) gout[B.fac_off + (long long)k * B.pstride + (long long)p * B.ld + j] = mk<double>((double)qr * back, (double)qi * back);
        }
#pragma unroll
        for (int s = 0; s < S; ++s) t[s][lane][i] = __floats2bfloat162_rn((float)dr[s], (float)di[s]);
    }
    __syncthreads();
    const size_t plane = (size_t)nb * Nr * Kp;
    const int p = p0 + lane;
    for (int i = w; i < 32; i += 8) {
        if (j0 + i >= m || p >= m) continue;
        __nv_bfloat16* o = out + ((size_t)box * Nr + 2 * (j0 + i)) * Kp + 2 * p;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const __nv_bfloat162 v = t[s][i][lane];
            *reinterpret_cast<__nv_bfloat162*>(o + s * plane) = __halves2bfloat162(v.x, __hneg(v.y));
            *reinterpret_cast<__nv_bfloat162*>(o + s * plane + Kp) = __halves2bfloat162(v.y, v.x);
        }
    }
}

// x 2^e for finite x; results below the normal range become 0
__device__ __forceinline__ double scale2(double x, int e) {
    const int hi = __double2hiint(x), E = ((hi >> 20) & 2047) + e;
    if (((hi >> 20) & 2047) == 0 || E <= 0) return 0.0;
    return E >= 2047 ? __hiloint2double((hi & 0x80000000) | 0x7FF00000, 0) : __hiloint2double(hi + e * (1 << 20), __double2loint(x));
}
// the double of an integer below 2^51 in size: one addition on the FP64 pipe
__device__ __forceinline__ double small_double(long long v) {
    return __longlong_as_double(0x4338000000000000ll + v) - 6755399441055744.0;
}

// One pass of dp_gemm: the orders LO <= i + j < HI of the products of digits i < SA and j < SB, which need the digits
// A0 <= i < A1 and B0 <= j < B1.  Each operand has a ring of slots, filled in the order of first use (A digits descend).
template <int SA, int SB, int LO, int HI, int GN>
struct DpPass {
    static constexpr int A0 = LO - SB + 1 > 0 ? LO - SB + 1 : 0, A1 = SA < HI ? SA : HI;
    static constexpr int B0 = LO - SA + 1 > 0 ? LO - SA + 1 : 0, B1 = SB < HI ? SB : HI;
    static constexpr int NA = GN == 64 || A1 - A0 > 7 ? 8 : 7, NB = (14 - NA) * (128 / GN);
    static __device__ constexpr int first(int j) { return HI - 1 - j < A1 - 1 ? HI - 1 - j : A1 - 1; }   // first i that uses B_j
    static __device__ constexpr int last(int j) { return LO - j > A0 ? LO - j : A0; }
};
constexpr int DP_SLOTS = 20;                           // barriers: 8 + 12 slots at 64 columns, 14 at 128
constexpr int dp_smem() { return 14 * A_SLOT + 1024 + 512; }

struct DpPipe {
    unsigned char* base;
    uint64_t *full, *empty, *done, *drained;
    int* err;
    uint32_t phase;   // one bit per slot: producer, the phase of its last load (ones before the first); consumer, the next phase
    bool ok;
};

template <int GN>
__device__ __forceinline__ unsigned char* dp_slot(unsigned char* base, int s, int na) {
    return s < na ? base + s * A_SLOT : base + na * A_SLOT + (s - na) * (GN * 128);
}

template <class P, int GN>
__device__ __forceinline__ void dp_load(DpPipe& p, uint32_t& used, int s, const CUtensorMap& map, int x, int y, int z) {
    if (p.ok) p.ok = tc::mbar_wait(&p.empty[s], (p.phase >> s) & 1, p.err, 32);
    if (!p.ok) return;
    tc::mbar_arrive_expect_tx(&p.full[s], s < P::NA ? A_SLOT : GN * 128);
    tc::tma_load_3d(dp_slot<GN>(p.base, s, P::NA), &map, x, y, z, &p.full[s]);
    p.phase ^= 1u << s;
    used |= 1u << s;
}

template <class P, int GN>
__device__ __forceinline__ void dp_produce(DpPipe& p, uint32_t& used, const CUtensorMap& mA, const CUtensorMap& mB, int nK, int row0,
                                           int n0, int nb, int box) {
    int a = 0, b = 0;
    for (int kc = 0; kc < nK && p.ok; ++kc) {
#pragma unroll
        for (int i = P::A1 - 1; i >= P::A0; --i) {
            dp_load<P, GN>(p, used, a, mA, kc * GK, row0, i * nb + box);
            a = a + 1 == P::NA ? 0 : a + 1;
#pragma unroll
            for (int j = P::B0; j < P::B1; ++j) {
                if (P::first(j) != i) continue;
                dp_load<P, GN>(p, used, P::NA + b, mB, kc * GK, n0, j * nb + box);
                b = b + 1 == P::NB ? 0 : b + 1;
            }
        }
    }
}

template <class P, int LO, int HI, int GN>
__device__ __forceinline__ void dp_consume(DpPipe& p, uint32_t tmem, int nK) {
    constexpr uint32_t idesc = tc::idesc_bf16(GM, GN);
    uint32_t seen = 0;   // orders that hold a product already
    int a = 0, b = 0, bs[P::B1];
    for (int kc = 0; kc < nK && p.ok; ++kc) {
#pragma unroll
        for (int i = P::A1 - 1; i >= P::A0; --i) {
            if (p.ok) p.ok = tc::mbar_wait(&p.full[a], (p.phase >> a) & 1, p.err, 34);
            p.phase ^= 1u << a;
#pragma unroll
            for (int j = P::B0; j < P::B1; ++j) {
                if (P::first(j) != i) continue;
                bs[j] = P::NA + b;
                b = b + 1 == P::NB ? 0 : b + 1;
                if (p.ok) p.ok = tc::mbar_wait(&p.full[bs[j]], (p.phase >> bs[j]) & 1, p.err, 33);
                p.phase ^= 1u << bs[j];
            }
            if (!p.ok) continue;
            tc::fence_after_sync();
            const uint32_t aa = tc::smem_u32(dp_slot<GN>(p.base, a, P::NA));
#pragma unroll
            for (int j = P::B0; j < P::B1; ++j) {
                if (i + j < LO || i + j >= HI) continue;
                const int o = i + j - LO;
                const uint32_t ab = tc::smem_u32(dp_slot<GN>(p.base, bs[j], P::NA));
#pragma unroll
                for (int kk = 0; kk < GK / 16; ++kk)
                    tc::mma_f16(tmem + o * GN, tc::desc_k_sw128(aa + kk * 32), tc::desc_k_sw128(ab + kk * 32), idesc,
                                ((seen >> o) & 1u) | (kk > 0 ? 1u : 0u));
                seen |= 1u << o;
            }
            tc::mma_commit(&p.empty[a]);
            a = a + 1 == P::NA ? 0 : a + 1;
#pragma unroll
            for (int j = P::B0; j < P::B1; ++j)
                if (P::last(j) == i) tc::mma_commit(&p.empty[bs[j]]);
        }
    }
    tc::mma_commit(p.done);
}

// The orders LO .. HI - 1 of the tile as doubles.  ADD: G += them; else R = -them, and with LAST R = I - them + what the pass
// before left there.
template <int LO, int HI, int GN, bool ADD, bool LAST, bool FIRST>
__device__ __forceinline__ void dp_epilogue(uint32_t tmem, int c_begin, int n0, int I, int m, int er, const int* __restrict__ eb,
                                            c128* __restrict__ row, bool& bad, uint32_t& big) {
    constexpr int O = HI - LO, OH = O < 4 ? O : 4;   // orders of the first 64-bit integer
#pragma unroll 1
    for (int c0 = c_begin; c0 < c_begin + GN / 2; c0 += 8) {
        const int j0 = (n0 + c0) / 2;
        uint32_t v[O][8];
#pragma unroll
        for (int o = 0; o < O; ++o) tc::tmem_ld_32x32b_x8(tmem + (uint32_t)(o * GN + c0), v[o]);
        c128 old[4];
        int ej[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const bool in = I < m && j0 + h < m;
            ej[h] = in ? eb[j0 + h] : 0;
            old[h] = (ADD || !FIRST) && in ? row[j0 + h] : mk<double>(0, 0);
        }
        tc::tmem_ld_wait();
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int j = j0 + h;
            if (I >= m || j >= m) continue;
            const int E = er + ej[h];
            double d[2], l[2];
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                long long vh = 0, vl = 0;
#pragma unroll
                for (int o = 0; o < O; ++o) {
                    const float a = __uint_as_float(v[o][2 * h + x]);
                    bad |= !(fabsf(a) < 8388608.f);
                    if (o < OH) vh = vh * 256 + __float2int_rn(a);
                    else vl = vl * 256 + __float2int_rn(a);
                }
                d[x] = scale2(small_double(vh), E - 8 * (LO + OH - 1));
                l[x] = O > 4 ? scale2(small_double(vl), E - 8 * (HI - 1)) : 0.0;
            }
            if (ADD) {
                row[j] = mk<double>(old[h].x + d[0], old[h].y + d[1]);
            } else if (!LAST) {
                row[j] = mk<double>(-d[0], -d[1]);
            } else {
                double re = (I == j ? 1.0 : 0.0) - d[0], im = -d[1];
                if (O > 4) re -= l[0], im -= l[1];
                if (!FIRST) re += old[h].x, im += old[h].y;
                row[j] = mk<double>(re, im);
                big = max(big, max(high_word(re), high_word(im)));
            }
        }
    }
}

// D = (left operand) (right operand) of one 128 x GN (real) tile per CTA, the orders below O.  ADD = false: R = I - D (pitch
// m); true: G += D.  Warp 0 lane 0 loads (TMA), warp 1 lane 0 issues the MMAs, warps 2-9 read the accumulators.  TMEM holds
// 4 orders of 128 columns or 8 of 64: at 128 columns more than four orders take two passes over K, the small orders last
// (the first pass leaves its part in the output).  A digit's slot is free again after its last product of a chunk; the
// order of the products gives each load at least six products' time.  Every wait is bounded.
template <int SA, int SB, int O, bool ADD, int GN>
__global__ void __launch_bounds__(320, 1) dp_gemm(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB,
                                                  const BoxInfo* __restrict__ boxes, const int* __restrict__ ea,
                                                  const int* __restrict__ eb, int nb, int Lr, int Lc, int m_max,
                                                  c128* __restrict__ out, float limit, int k, int* __restrict__ flag,
                                                  int* __restrict__ stat, const int* __restrict__ gate) {
    extern __shared__ __align__(1024) unsigned char dp_raw[];
    constexpr bool TWO = O * GN > 512;
    static_assert(!(TWO && ADD), "an addition is one pass");
    using PL = DpPass<SA, SB, TWO ? 4 : 0, O, GN>;            // the first pass: the large orders, or all
    using PH = DpPass<SA, SB, 0, TWO ? 4 : O, GN>;
    constexpr uint32_t TCOLS = (TWO ? 4 : O) * GN <= 256 ? 256 : 512;
    const int box = blockIdx.z;
    const BoxInfo B = boxes[box];
    const int m = B.m, row0 = blockIdx.y * GM, n0 = blockIdx.x * GN;
    if (k >= B.dims[2] || row0 >= m || n0 >= 2 * m || gated_out(gate, box)) return;
    DpPipe p;
    p.base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(dp_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    p.full = reinterpret_cast<uint64_t*>(p.base + 14 * A_SLOT);
    p.empty = p.full + DP_SLOTS;
    p.done = p.empty + DP_SLOTS;
    p.drained = p.done + 1;
    p.err = flag + 1;
    p.ok = true;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(p.drained + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2 * DP_SLOTS + 1; ++i) tc::mbar_init(&p.full[i], 1);
        tc::mbar_init(p.drained, 8);
        tc::fence_barrier_init();
        tc::prefetch_tmap(&mA);
        tc::prefetch_tmap(&mB);
    }
    if (warp == 1) {
        tc::tmem_alloc(tmem_slot, TCOLS);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    const int nK = (2 * m + GK - 1) / GK;
    if (warp == 0) {
        if (lane == 0) {
            uint32_t used = 0;
            p.phase = 0xFFFFFFFFu;
            dp_produce<PL, GN>(p, used, mA, mB, nK, row0, n0, nb, box);
            if (TWO) dp_produce<PH, GN>(p, used, mA, mB, nK, row0, n0, nb, box);
            // a give-up anywhere: let the loads already issued land before the slots are left
            if (!p.ok || *reinterpret_cast<volatile int*>(p.err) != 0)
                for (int s = 0; s < DP_SLOTS; ++s)
                    if ((used >> s) & 1) tc::mbar_drain(&p.full[s], (p.phase >> s) & 1);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            p.phase = 0;
            dp_consume<PL, TWO ? 4 : 0, O, GN>(p, tmem, nK);
            if (TWO) {
                if (p.ok) p.ok = tc::mbar_wait(p.drained, 0, p.err, 36);
                if (!p.ok) tc::mbar_drain(p.done, 0);   // the first pass's products, before the barrier's next phase
                tc::fence_after_sync();
                dp_consume<PH, 0, 4, GN>(p, tmem, nK);
            }
            // every product issued has completed before this warp meets the CTA's barrier and frees TMEM: an epilogue warp
            // that gave up on the first pass does not wait for the second
            tc::mbar_drain(p.done, TWO ? 1 : 0);
        }
    } else {
        const int q = warp & 3, I = row0 + q * 32 + lane, cb = (warp - 2) / 4 * (GN / 2);
        const int er = I < m ? ea[box * Lr + I] - 14 : 0;
        const uint32_t tm = tmem + ((uint32_t)(q * 32) << 16);
        const int* ebb = eb + box * Lc;
        c128* row = ADD ? out + B.fac_off + (long long)k * B.pstride + (long long)I * B.ld
                        : out + (size_t)box * m_max * m_max + (size_t)I * m;
        bool bad = false, ok = tc::mbar_wait(p.done, 0, p.err, 35);
        uint32_t big = 0;
        if (!ok) tc::mbar_drain(p.done, 0);   // products already issued still write TMEM
        tc::fence_after_sync();
        if (ok) dp_epilogue<TWO ? 4 : 0, O, GN, ADD, !TWO, true>(tm, cb, n0, I, m, er, ebb, row, bad, big);
        if (TWO) {
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(p.drained);
            if (ok && !(ok = tc::mbar_wait(p.done, 1, p.err, 37))) tc::mbar_drain(p.done, 1);
            tc::fence_after_sync();
            if (ok) dp_epilogue<0, 4, GN, ADD, true, false>(tm, cb, n0, I, m, er, ebb, row, bad, big);
        }
        const float f = (float)__hiloint2double((int)big, 0);
        if (ok && (bad || (!ADD && !(f <= limit)))) atomicOr(flag, 4);
        if (ok && !ADD && stat) {   // the largest entry (non-negative floats compare like their bits)
            const int b = __reduce_max_sync(0xffffffffu, __float_as_int(f));
            if (lane == 0) atomicMax(stat + box, b);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, TCOLS);
    }
}

// bf16 [z][rows][cols] with row pitch Kp, boxes of 64 x box_rows, 128-byte swizzle
bool encode_slices(CUtensorMap* map, void* base, uint64_t cols, uint64_t rows, uint64_t z, uint64_t Kp, uint32_t box_rows) {
    const PFN_cuTensorMapEncodeTiled_v12000 fn = tc::tensor_map_encoder();
    if (!fn) return false;
    cuuint64_t dims[3] = {cols, rows, z};
    cuuint64_t strides[2] = {Kp * 2, Kp * 2 * rows};
    cuuint32_t box[3] = {GK, box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int SA, int SB, int O, bool ADD, int GN>
void launch_gemm_n(helm_ctx ctx, const DpWork& D, const CUtensorMap& mA, const CUtensorMap& mB, const int* ea, const BoxInfo* dbox,
                   int nbox, int m_max, c128* out, float limit, int k, int* flag, int* stat, const int* gate) {
    static PerDevice attr;
    if (!attr.done(ctx->device)) {
        cudaFuncSetAttribute(dp_gemm<SA, SB, O, ADD, GN>, cudaFuncAttributeMaxDynamicSharedMemorySize, dp_smem());
        attr.mark(ctx->device);
    }
    const dim3 grid((2 * m_max + GN - 1) / GN, (m_max + GM - 1) / GM, nbox);
    dp_gemm<SA, SB, O, ADD, GN><<<grid, 320, dp_smem(), ctx->stream>>>(mA, mB, dbox, ea, D.eB, D.nb, D.Lr, D.Nr / 2, D.m_max, out,
                                                                       limit, k, flag, stat, gate);
    ctx->launches++;
}

template <int SA, int SB, int O, bool ADD>
void launch_gemm(helm_ctx ctx, const DpWork& D, const CUtensorMap& mA, const int* ea, const BoxInfo* dbox, int nbox, int m_max,
                 c128* out, float limit, int k, int* flag, int* stat = nullptr, const int* gate = nullptr) {
    // 128-column tiles once every SM has one: 8 boxes of 676 unknowns (528 tiles) 814 us with 30 products against 1046;
    // small coarse boxes (fewer tiles than SMs) 37 us, with 64 columns, twice the CTAs and all orders in one pass, 27
    const long long tiles = (long long)((2 * m_max + 127) / 128) * ((m_max + GM - 1) / GM) * nbox;
    if (tiles > ctx->sm_count)
        launch_gemm_n<SA, SB, O, ADD, 128>(ctx, D, mA, D.mB128, ea, dbox, nbox, m_max, out, limit, k, flag, stat, gate);
    else
        launch_gemm_n<SA, SB, O, ADD, 64>(ctx, D, mA, D.mB64, ea, dbox, nbox, m_max, out, limit, k, flag, stat, gate);
}

template <int S>
void slice_rows(helm_ctx ctx, const DpWork& D, const TgjWork& T, const BoxInfo* dbox, int nbox, int m_max, const c128* src,
                bool from_g, void* out, int* e, c64* S32, int k, int* clear = nullptr, const int* gate = nullptr) {
    dp_slice_rows<S><<<dim3(m_max, nbox), 128, 0, ctx->stream>>>(dbox, src, from_g ? 1 : 0, D.m_max, (__nv_bfloat16*)out, D.nb,
                                                                 D.Lr, D.Kp, e, S32, T.L, k, T.flag, clear, gate);
    ctx->launches++;
}

template <int S>
void slice_cols(helm_ctx ctx, const DpWork& D, const TgjWork& T, const BoxInfo* dbox, int nbox, int m_max, const ColSrc& src,
                c128* gout, int k, const int* gate = nullptr) {
    const int t = (m_max + 31) / 32;
    dp_col_exponents<<<dim3(t, nbox), 1024, 0, ctx->stream>>>(dbox, src, D.eB, D.Nr / 2, k, T.flag, gate);
    dp_slice_cols<S><<<dim3(t, t, nbox), 256, 0, ctx->stream>>>(dbox, src, (__nv_bfloat16*)D.B, D.nb, D.Nr, D.Kp, D.eB, gout, k, gate);
    ctx->launches += 2;
}

}  // namespace

static void dp_sizes(int nb, int m_max, DpWork& W) {
    W.nb = nb;
    W.m_max = m_max;
    W.Lr = (m_max + GM - 1) / GM * GM;
    W.Nr = std::max(128, 2 * ((m_max + 31) / 32 * 32));
    W.Kp = (2 * m_max + GK - 1) / GK * GK;
    W.as_bytes = (size_t)SAS * nb * W.Lr * W.Kp * 2;
    W.ax_bytes = (size_t)SAX * nb * W.Lr * W.Kp * 2;
    W.b_bytes = (size_t)SBM * nb * W.Nr * W.Kp * 2;
    W.e_bytes = (size_t)nb * (std::max(W.Lr, W.Nr) + 1) * sizeof(int);   // eB: one more int per box, the largest |R1|
}

size_t dp_bytes(int nb, int m_max) {
    DpWork W;
    dp_sizes(nb, m_max, W);
    return W.as_bytes + W.ax_bytes + W.b_bytes + 3 * W.e_bytes;
}

void dp_free(helm_ctx ctx, DpWork& W) {
    dev_free(ctx, W.AS, W.as_bytes);
    dev_free(ctx, W.AX, W.ax_bytes);
    dev_free(ctx, W.B, W.b_bytes);
    dev_free(ctx, W.eS, W.e_bytes);
    dev_free(ctx, W.eX, W.e_bytes);
    dev_free(ctx, W.eB, W.e_bytes);
    W.AS = W.AX = W.B = nullptr;
    W.eS = W.eX = W.eB = nullptr;
}

helm_status dp_alloc(helm_ctx ctx, int nb, int m_max, DpWork& W) {
    dp_sizes(nb, m_max, W);
    helm_status rc;
    if ((rc = dev_alloc(ctx, &W.AS, W.as_bytes, "digit slices")) || (rc = dev_alloc(ctx, &W.AX, W.ax_bytes, "digit slices")) ||
        (rc = dev_alloc(ctx, &W.B, W.b_bytes, "digit slices")) ||
        (rc = dev_alloc(ctx, (void**)&W.eS, W.e_bytes, "slice exponents")) ||
        (rc = dev_alloc(ctx, (void**)&W.eX, W.e_bytes, "slice exponents")) ||
        (rc = dev_alloc(ctx, (void**)&W.eB, W.e_bytes, "slice exponents"))) {
        dp_free(ctx, W);
        return rc;
    }
    // entries past a box's m x m are never written: they stay zero, so they add nothing to any product
    cudaMemsetAsync(W.AS, 0, W.as_bytes, ctx->stream);
    cudaMemsetAsync(W.AX, 0, W.ax_bytes, ctx->stream);
    cudaMemsetAsync(W.B, 0, W.b_bytes, ctx->stream);
    const uint64_t c = 2ull * m_max;
    if (!encode_slices(&W.mAS, W.AS, c, W.Lr, (uint64_t)SAS * nb, W.Kp, GM) ||
        !encode_slices(&W.mAX, W.AX, c, W.Lr, (uint64_t)SAX * nb, W.Kp, GM) ||
        !encode_slices(&W.mB64, W.B, c, W.Nr, (uint64_t)SBM * nb, W.Kp, 64) ||
        !encode_slices(&W.mB128, W.B, c, W.Nr, (uint64_t)SBM * nb, W.Kp, 128)) {
        dp_free(ctx, W);
        return set_error(ctx, HELM_ECUDA, "cuTensorMapEncodeTiled failed for the digit slices");
    }
    return HELM_OK;
}

void dp_invert(helm_ctx ctx, const TgjWork& T, const DpWork& D, const BoxInfo* dbox, const BoxInfo* hbox, int nbox, int m_max,
               int k, const c128* S, c128* R, c128* G) {
    int* stat = D.eB + (size_t)D.nb * (D.Nr / 2);
    tgj_pad(ctx, T, dbox, nbox);
    slice_rows<SAS>(ctx, D, T, dbox, nbox, m_max, S, false, D.AS, D.eS, (c64*)T.S, k, stat);
    tgj_eliminate(ctx, T, dbox, hbox, nbox, m_max, k);
    const ColSrc x32{(const c64*)T.S, nullptr, nullptr, T.L, D.m_max}, r{nullptr, R, nullptr, 0, D.m_max},
        g{nullptr, nullptr, G, 0, D.m_max};
    // X0 (cut to its digits) into G, R0 = I - S X0
    slice_cols<3>(ctx, D, T, dbox, nbox, m_max, x32, G, k);
    launch_gemm<5, 3, 6, false>(ctx, D, D.mAS, D.eS, dbox, nbox, m_max, R, 1e-3f, k, T.flag);
    // X1 = X0 + X0 R0
    slice_rows<SAX>(ctx, D, T, dbox, nbox, m_max, G, true, D.AX, D.eX, nullptr, k);
    slice_cols<3>(ctx, D, T, dbox, nbox, m_max, r, nullptr, k);
    launch_gemm<3, 3, 4, true>(ctx, D, D.mAX, D.eX, dbox, nbox, m_max, G, 0.f, k, T.flag);
    for (int step = 0; step < 2; ++step) {   // the second time for the boxes that need it
        const int* gate = step ? stat : nullptr;
        // R1 = I - S X1 (X1 cut to its digits), X = X1 + X1 R1
        if (step == 0) {
            slice_cols<5>(ctx, D, T, dbox, nbox, m_max, g, G, k);
            launch_gemm<SAS, 5, 8, false>(ctx, D, D.mAS, D.eS, dbox, nbox, m_max, R, 1e-4f, k, T.flag, stat);
        } else {
            slice_cols<SBM>(ctx, D, T, dbox, nbox, m_max, g, G, k, gate);
            launch_gemm<SAS, SBM, 8, false>(ctx, D, D.mAS, D.eS, dbox, nbox, m_max, R, 1e-9f, k, T.flag, nullptr, gate);
        }
        slice_rows<SAX>(ctx, D, T, dbox, nbox, m_max, G, true, D.AX, D.eX, nullptr, k, nullptr, gate);
        slice_cols<3>(ctx, D, T, dbox, nbox, m_max, r, nullptr, k, gate);
        launch_gemm<3, 3, 3, true>(ctx, D, D.mAX, D.eX, dbox, nbox, m_max, G, 0.f, k, T.flag, nullptr, gate);
    }
}
