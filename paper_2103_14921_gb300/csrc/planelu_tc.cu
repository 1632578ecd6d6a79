// Plane factorisation of the complex64 local operators on the tensor cores (the exact local solves of
// Eq. oras): for every box and plane k, S_0 = D_0, S_k = D_k - L_k S_{k-1}^{-1} U_{k-1} and the dense
// inverse G_k = S_k^{-1}, by blocked Gauss-Jordan whose rank-NB updates run as tcgen05 GEMMs.
//
// Blocked Gauss-Jordan with block pivots.  For the panel J = [j0, j0 + NB) of the m x m matrix A:
//   P      = A[J,J]^{-1}                      (NB x NB, Gauss-Jordan with partial pivoting inside the block)
//   A[J,:] = P A[J,:]  (columns outside J),    A[J,J] = P
//   A[I,:] = A[I,:] - (A[I,J] P) A[J,:]  (rows I outside J, columns outside J; A[J,:] before the step)
//   A[I,J] = -A[I,J] P                      (rows I outside J)
// After the last panel A holds S^{-1}.  With W[I,:] = A[I,J] P outside J, W[J,:] = -P, and R = A[J,:] before the step
// with the identity in columns J, all four lines are one product: A = [row and column outside J] A - W R.  So only
// A[I,J] P (one row of tiles) waits for the block inverse, and it runs on the tensor cores too; R is a copy.
// Pivoting stays inside each diagonal block: for these Helmholtz Schur complements (condition numbers
// 1e0-1e2 at the workload sizes) block pivots give the same accuracy as full partial pivoting, and a block
// pivot below 1e-6 of its block's largest entry (the rows and columns below m, so that the bar has the matrix's own
// scale) is reported so that the caller can fall back to an elimination on the CUDA cores.
//
// The product W R (m x NB times NB x m, complex; W = A[I,J] P is the same with N = 2 NB) is one real GEMM with the 2x2 embedding used by the plane
// sweeps: A operand = rows of W read as 2 NB reals (K-major), B operand = B^T[2j][2c] = Re R[c][j],
// B^T[2j][2c+1] = -Im R[c][j], B^T[2j+1][2c] = Im R[c][j], B^T[2j+1][2c+1] = Re R[c][j].  FP32 accuracy
// from TF32 units: each operand x is split into hi = x with its low 13 mantissa bits cleared (exact in TF32)
// and lo = x - hi, and D = hi*hi + hi*lo + lo*hi (the lo*lo term is below FP32 rounding), accumulated in
// FP32 in TMEM.  Three MMAs (M = 128, N = 256, K = 8) per K step; operands staged by TMA (128-byte swizzle).
//
// Padding: the work matrix of every box is L x L (L = m_max rounded up to 128) with identity rows and
// columns beyond the box's m, written once and never touched again, so the block inverse of a partial last
// panel is that of block-diag(S_JJ, I) and the padding contributes nothing to rows and columns below m.
#include <cuda.h>

#include <atomic>

#include "internal.h"
#include "tc.cuh"
#include "tgj.h"

namespace {

constexpr int NB = 128;              // panel width (complex columns)
constexpr int K2 = 2 * NB;           // real K of the update product
constexpr int UBM = 128;             // output rows per tile
constexpr int UBN = 256;             // output real columns per tile (128 complex)
constexpr int UST = 2;               // operand ring stages
constexpr int A_TILE = UBM * 128;    // 128 rows x 32 fp32 = 16 KB
constexpr int B_TILE = UBN * 128;    // 256 rows x 32 fp32 = 32 KB
constexpr int STAGE = 2 * A_TILE + 2 * B_TILE;
constexpr int DIAG_THREADS = 640;   // 16 warps of the rank steps, 4 of the column chain
constexpr int DP = NB + 1;           // row pitch of the diagonal block in shared memory

__device__ __forceinline__ float tf32_hi(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }

// ------------------------------------------------------------------ Schur complements (pitch L)

// S_0 = D_0: the in-plane couplings of plane 0
__global__ void tgj_schur_init(const BoxInfo* __restrict__ boxes, const c64* __restrict__ coef, c64* __restrict__ S,
                               int L) {
    const BoxInfo B = boxes[blockIdx.y];
    const int m = B.m, bx = B.dims[0];
    c64* Sb = S + (size_t)blockIdx.y * L * L;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * m; e += gridDim.x * blockDim.x) {
        const int p = e / m, q = e % m;
        const int dx = q % bx - p % bx, dy = q / bx - p / bx;
        c64 v = mk<float>(0.f, 0.f);
        if (dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1) v = coef[(B.loc_off + p) * 27 + 9 + (dy + 1) * 3 + (dx + 1)];
        Sb[(size_t)p * L + q] = v;
    }
}

// T = G_{k-1} U_{k-1}, G_{k-1} held in S: T[a][q] = sum_d G[a][q-d] U(node q-d of plane k-1, offset (d, +1))
__global__ void tgj_schur_gu(const BoxInfo* __restrict__ boxes, const c64* __restrict__ coef,
                             const c64* __restrict__ S, c64* __restrict__ T, int L, int k) {
    const BoxInfo B = boxes[blockIdx.y];
    const int m = B.m;
    if (k >= B.dims[2]) return;
    const int bx = B.dims[0], by = B.dims[1];
    const c64* G = S + (size_t)blockIdx.y * L * L;
    c64* Tb = T + (size_t)blockIdx.y * L * L;
    const c64* cU = coef + (B.loc_off + (long long)(k - 1) * m) * 27 + 18;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * m; e += gridDim.x * blockDim.x) {
        const int a = e / m, q = e % m;
        const int qx = q % bx, qy = q / bx;
        c64 acc = mk<float>(0.f, 0.f);
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy) {
            const int py = qy - dy;
            if (py < 0 || py >= by) continue;
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                const int px = qx - dx;
                if (px < 0 || px >= bx) continue;
                const int p = py * bx + px;
                cmac(acc, G[(size_t)a * L + p], cU[(long long)p * 27 + (dy + 1) * 3 + (dx + 1)]);
            }
        }
        Tb[(size_t)a * L + q] = acc;
    }
}

// S = D_k - L_k T: S[p][q] = D_k[p][q] - sum_d L(node p of plane k, offset (d, -1)) T[p+d][q]
__global__ void tgj_schur_lt(const BoxInfo* __restrict__ boxes, const c64* __restrict__ coef,
                             const c64* __restrict__ T, c64* __restrict__ S, int L, int k) {
    const BoxInfo B = boxes[blockIdx.y];
    const int m = B.m;
    if (k >= B.dims[2]) return;
    const int bx = B.dims[0], by = B.dims[1];
    const c64* Tb = T + (size_t)blockIdx.y * L * L;
    c64* Sb = S + (size_t)blockIdx.y * L * L;
    const c64* cK = coef + (B.loc_off + (long long)k * m) * 27;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * m; e += gridDim.x * blockDim.x) {
        const int p = e / m, q = e % m;
        const int px = p % bx, py = p / bx;
        const int dxq = q % bx - px, dyq = q / bx - py;
        c64 acc = mk<float>(0.f, 0.f);
        if (dxq >= -1 && dxq <= 1 && dyq >= -1 && dyq <= 1) acc = cK[(long long)p * 27 + 9 + (dyq + 1) * 3 + (dxq + 1)];
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy) {
            const int ny_ = py + dy;
            if (ny_ < 0 || ny_ >= by) continue;
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                const int nx_ = px + dx;
                if (nx_ < 0 || nx_ >= bx) continue;
                const c64 l = cK[(long long)p * 27 + (dy + 1) * 3 + (dx + 1)];
                const c64 t = Tb[(size_t)(ny_ * bx + nx_) * L + q];
                acc.x -= l.x * t.x - l.y * t.y;
                acc.y -= l.x * t.y + l.y * t.x;
            }
        }
        Sb[(size_t)p * L + q] = acc;
    }
}

// identity on the padding diagonal (the rest of the padding is zero from the initial memset)
__global__ void tgj_pad_diag(const BoxInfo* __restrict__ boxes, c64* __restrict__ S, int L) {
    const BoxInfo B = boxes[blockIdx.y];
    for (int i = B.m + blockIdx.x * blockDim.x + threadIdx.x; i < L; i += gridDim.x * blockDim.x)
        S[(size_t)blockIdx.y * L * L + (size_t)i * L + i] = mk<float>(1.f, 0.f);
}

// ------------------------------------------------------------------ panel: block inverse, operands

// P = A[J,J]^{-1} by in-place Gauss-Jordan in sub-panels of SB columns, pivots by largest modulus among the block's rows not
// used yet.  Rows are not swapped: s_p[c] is the row that column c was eliminated with (s_k its inverse), and
// P[s_k[row]][s_p[col]] = X[row][col] in the end.
//
// X stays in registers: thread (rg, cg) of 32 x 16 holds rows 4 rg .. 4 rg + 3 and columns cg + 16 i.  A sub-panel (slot 0
// of every thread; the slots rotate) goes to shared memory and is eliminated by four warps, a row per thread; per column
// a 32-bit key (|x|^2 in the high bits, the row in the low seven) is reduced with one redux per warp, each warp's best
// row is published with it (and the pivot's reciprocal), and every thread scales by itself: one barrier of four warps per
// column.  The transform W
// then reaches the other columns in a rank-SB step of the other 16 warps, X <- [rows not used here] X + W X[pivot rows]: the
// next sub-panel's columns first, so that the four warps eliminate it during the rest of the step.
// Bound: the serial column chain (670 clocks a column by itself, 1,080 beside the rank steps: 17,300 of a sub-panel's
// 22,000), and the rank-SB steps (128^3 complex multiply-adds on one SM's FP32 lanes, 32 us).  27 boxes: 103 us a panel
// (chain and rank steps one after the other, X in shared memory: 123).
constexpr int SB = 16;
constexpr int SWP = SB + 2;           // row pitch of a sub-panel in shared memory
constexpr int DIAG_SMEM = NB * DP * (int)sizeof(c64);
static_assert(2 * NB * SWP + SB * NB <= NB * DP, "the sub-panels and the pivot rows share the block's memory");

struct DiagShared {
    uint4 key[2];
    c64 row[2][4][SB + 2];   // a warp's best row and 1 / its pivot
    int p[NB], k[NB];
};

// One sub-panel, columns c0 .. c0 + SB - 1 of the block, by 128 threads: Wr is the row'th row.  The columns rotate through
// the registers, so that the loop stays rolled: sixteen copies of its body ran at the speed of instruction fetch.  bar: the
// least |pivot|^2 of the row that is not weak.
__device__ __forceinline__ void diag_columns(c64* Wr, DiagShared& D, bool& used, int row, int c0, float bar, int* flag) {
    const int lane = row & 31, wid = row >> 5;
    c64 a[SB];
#pragma unroll
    for (int j = 0; j < SB; j += 2) {
        const float4 v = *reinterpret_cast<const float4*>(Wr + j);
        a[j] = mk<float>(v.x, v.y);
        a[j + 1] = mk<float>(v.z, v.w);
    }
    float q;
    c64 inv;
    uint32_t key, kw;
    auto candidate = [&]() {
        q = a[0].x * a[0].x + a[0].y * a[0].y;
        const float d = q > 0.f ? 1.f / q : 1.f;
        inv = q > 0.f ? mk<float>(a[0].x * d, -a[0].y * d) : mk<float>(1.f, 0.f);
        // rows not used yet: |x|^2 rounded down to 16 mantissa bits, ties to the smallest row; used: 0
        key = used ? 0u : ((__float_as_uint(q) & 0xFFFFFF80u) | (uint32_t)(NB - 1 - row)) + 1u;
        kw = __reduce_max_sync(0xffffffffu, key);
    };
    candidate();
#pragma unroll 1
    for (int j = 0; j < SB; ++j) {
        const int pb = j & 1;
        if (lane == 0) reinterpret_cast<uint32_t*>(&D.key[pb])[wid] = kw;
        if (key == kw && kw) {
            float4* o = reinterpret_cast<float4*>(D.row[pb][wid]);
#pragma unroll
            for (int i = 0; i < SB / 2; ++i) o[i] = make_float4(a[2 * i].x, a[2 * i].y, a[2 * i + 1].x, a[2 * i + 1].y);
            D.row[pb][wid][SB] = inv;
        }
        __syncwarp();
        tc::named_bar(1, NB);
        const uint4 k4 = D.key[pb];
        const uint32_t km = max(max(k4.x, k4.y), max(k4.z, k4.w));
        const int p = NB - 1 - (int)((km - 1u) & 127u);
        const c64* r = D.row[pb][p >> 5];
        // the pivot row becomes inv r, the others a - (a_0 inv) r; column 0 (inv, or -a_0 inv) rotates to the end
        const c64 ip = r[SB];
        const bool piv = row == p;
        if (piv) {
            if (!(q > 0.f)) atomicOr(flag, 1);
            else if (q < bar) atomicOr(flag, 2);
            used = true;
            D.p[c0 + j] = row;
            D.k[row] = c0 + j;
        }
        const c64 g = piv ? ip : mk<float>(-(a[0].x * ip.x - a[0].y * ip.y), -(a[0].x * ip.y + a[0].y * ip.x));
        auto step = [&](int i, float x, float y) {
            c64 t = piv ? mk<float>(0.f, 0.f) : a[i];
            cmac(t, g, mk<float>(x, y));
            a[i - 1] = t;
        };
        step(1, r[1].x, r[1].y);
        candidate();   // of the next column, while the others are updated
#pragma unroll
        for (int i = 1; i < SB / 2; ++i) {
            const float4 v = reinterpret_cast<const float4*>(r)[i];
            step(2 * i, v.x, v.y);
            step(2 * i + 1, v.z, v.w);
        }
        a[SB - 1] = g;
    }
#pragma unroll
    for (int j = 0; j < SB; j += 2) *reinterpret_cast<float4*>(Wr + j) = make_float4(a[j].x, a[j].y, a[j + 1].x, a[j + 1].y);
}

// slots I0 .. I1 - 1 of X <- [rows not used here] X + W X[pivot rows]
template <int I0, int I1>
__device__ __forceinline__ void diag_step(c64 (&x)[4][8], const c64* W, const c64* Brow, int rg, int cg, uint32_t piv) {
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int i = I0; i < I1; ++i)
            if ((piv >> r) & 1) x[r][i] = mk<float>(0.f, 0.f);
#pragma unroll(I1 - I0 > 1 ? 1 : 4)
    for (int c = 0; c < SB; c += 2) {
        float4 w[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) w[r] = *reinterpret_cast<const float4*>(W + (4 * rg + r) * SWP + c);
#pragma unroll
        for (int i = I0; i < I1; ++i) {
            const c64 b0 = Brow[c * NB + i * 16 + cg], b1 = Brow[(c + 1) * NB + i * 16 + cg];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                cmac(x[r][i], mk<float>(w[r].x, w[r].y), b0);
                cmac(x[r][i], mk<float>(w[r].z, w[r].w), b1);
            }
        }
    }
}

// the inverse P of the 128 x 128 block at A (pitch L) into X (pitch DP); rows and columns from nr on are padding
__device__ __forceinline__ void diag_inverse(const c64* __restrict__ A, int L, int nr, c64* X, DiagShared& D, float* s_max,
                                             int* flag) {
    constexpr int RT = DIAG_THREADS - NB;   // threads of the rank steps
    const int tid = threadIdx.x;
    c64* const Wb = X;                    // [2][NB][SWP]
    c64* const Brow = X + 2 * NB * SWP;   // [SB][NB]
    if (tid >= RT) {
        const int row = tid - RT;
        bool used = false;
        D.k[row] = -1;
        tc::named_bar(2, DIAG_THREADS);
        float amax = 0.f;
        for (int w = 0; w < RT / 32; ++w) amax = fmaxf(amax, s_max[w]);
        // a row of the padding (pivot 1) is never weak; a |pivot|^2 below the normal range has no reciprocal
        const float bar = row < nr ? fmaxf(1e-12f * amax, 1.1754944e-38f) : 0.f;
        diag_columns(Wb + row * SWP, D, used, row, 0, bar, flag);
#pragma unroll 1
        for (int s = 0; s < NB / SB; ++s) {
            for (int i = 0; i < 3; ++i) tc::named_bar(2, DIAG_THREADS);
            if (s + 1 < NB / SB) diag_columns(Wb + (((s + 1) & 1) * NB + row) * SWP, D, used, row, (s + 1) * SB, bar, flag);
        }
        tc::named_bar(2, DIAG_THREADS);
        __syncthreads();
        return;
    }
    const int rg = tid >> 4, cg = tid & 15;
    c64 x[4][8];
    float amax = 0.f;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int i = 0; i < 8; ++i) x[r][i] = A[(size_t)(4 * rg + r) * L + cg + 16 * i];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (4 * rg + r < nr) amax = fmaxf(amax, x[r][i].x * x[r][i].x + x[r][i].y * x[r][i].y);
    amax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(amax)));   // non-negative: ordered like the bits
    if ((tid & 31) == 0) s_max[tid >> 5] = amax;
#pragma unroll
    for (int r = 0; r < 4; ++r) Wb[(4 * rg + r) * SWP + cg] = x[r][0];
    tc::named_bar(2, DIAG_THREADS);
#pragma unroll 1
    for (int s = 0; s < NB / SB; ++s) {
        const c64* W = Wb + (s & 1) * NB * SWP;
        c64* Wn = Wb + ((s + 1) & 1) * NB * SWP;
        const int c0 = s * SB;
        tc::named_bar(2, DIAG_THREADS);   // W is complete
        uint32_t piv = 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int k = D.k[4 * rg + r] - c0;
            if (k >= 0 && k < SB) {
                piv |= 1u << r;
#pragma unroll
                for (int i = 1; i < 8; ++i) Brow[k * NB + i * 16 + cg] = x[r][i];
            }
        }
        __syncwarp();
        tc::named_bar(2, DIAG_THREADS);   // and the pivot rows
        diag_step<1, 2>(x, W, Brow, rg, cg, piv);
#pragma unroll
        for (int r = 0; r < 4; ++r) Wn[(4 * rg + r) * SWP + cg] = x[r][1];
        tc::named_bar(2, DIAG_THREADS);   // the next sub-panel's columns
        diag_step<2, 8>(x, W, Brow, rg, cg, piv);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const c64 own = W[(4 * rg + r) * SWP + cg];
#pragma unroll
            for (int i = 0; i < 7; ++i) x[r][i] = x[r][i + 1];
            x[r][7] = own;
        }
    }
    tc::named_bar(2, DIAG_THREADS);       // X takes the sub-panels' place
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int c = D.k[4 * rg + r];
#pragma unroll
        for (int i = 0; i < 8; ++i) X[c * DP + D.p[cg + 16 * i]] = x[r][i];
    }
    __syncthreads();
}

// hi and lo parts of four values at an operand position
__device__ __forceinline__ void split4(float* h, float* l, size_t at, float a, float b, float c, float d) {
    const float4 v = make_float4(tf32_hi(a), tf32_hi(b), tf32_hi(c), tf32_hi(d));
    *reinterpret_cast<float4*>(h + at) = v;
    *reinterpret_cast<float4*>(l + at) = make_float4(a - v.x, b - v.y, c - v.z, d - v.w);
}

// The panel's first launch, in which nothing depends on anything else: CTA b < nbox inverts the diagonal block of box b
// and writes P as the right operand of W P (Ph, Pl) and -P as rows J of the left operand of the update (Wh, Wl);
// the other CTAs copy W = A[:, J] (rows outside J; zero beyond m) and A[J, :], with the identity in columns J, as the
// update's right operand (Bh, Bl; every column below L, so that the operand is finite everywhere).
__global__ void __launch_bounds__(DIAG_THREADS) tgj_panel(const BoxInfo* __restrict__ boxes, const c64* __restrict__ S,
                                                          int L, int nbox, float* __restrict__ Wh, float* __restrict__ Wl,
                                                          float* __restrict__ Ph, float* __restrict__ Pl,
                                                          float* __restrict__ Bh, float* __restrict__ Bl,
                                                          int* __restrict__ flag, int j0, int k) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ __align__(16) DiagShared s_d;
    __shared__ float s_max[DIAG_THREADS / 32];
    const int tid = threadIdx.x;
    c64* X = reinterpret_cast<c64*>(dsm);   // [NB][DP]
    if ((int)blockIdx.x < nbox) {
        const int box = blockIdx.x;
        const int m = boxes[box].m;
        if (k >= boxes[box].dims[2] || j0 >= m) return;
        diag_inverse(S + (size_t)box * L * L + (size_t)j0 * L + j0, L, min(NB, m - j0), X, s_d, s_max, flag);
        float *wh = Wh + ((size_t)box * L + j0) * K2, *wl = Wl + ((size_t)box * L + j0) * K2;
        float *ph = Ph + (size_t)box * K2 * K2, *pl = Pl + (size_t)box * K2 * K2;
        for (int e = tid; e < NB * NB / 2; e += DIAG_THREADS) {
            const int c = e / (NB / 2), q = 2 * (e % (NB / 2));
            const c64 v0 = X[c * DP + q], v1 = X[c * DP + q + 1];
            split4(wh, wl, (size_t)c * K2 + 2 * q, -v0.x, -v0.y, -v1.x, -v1.y);
            const c64 u0 = X[q * DP + c], u1 = X[(q + 1) * DP + c];   // P[q][c]: rows 2c, 2c + 1 of the right operand, K index q
            split4(ph, pl, (size_t)(2 * c) * K2 + 2 * q, u0.x, -u0.y, u1.x, -u1.y);
            split4(ph, pl, (size_t)(2 * c + 1) * K2 + 2 * q, u0.y, u0.x, u1.y, u1.x);
        }
        return;
    }
    const int t32 = L / 32;   // 32-row pieces of W and 32-column pieces of A[J, :] per box
    for (int it = blockIdx.x - nbox; it < nbox * 2 * t32; it += gridDim.x - nbox) {
        const int box = it / (2 * t32), part = it % (2 * t32);
        const int m = boxes[box].m;
        if (k >= boxes[box].dims[2] || j0 >= m) continue;
        const c64* A = S + (size_t)box * L * L;
        if (part < t32) {
            const int I0 = part * 32;
            if (I0 >= j0 && I0 < j0 + NB) continue;   // rows J: -P, from the block's CTA
            float *wh = Wh + ((size_t)box * L + I0) * K2, *wl = Wl + ((size_t)box * L + I0) * K2;
#pragma unroll 4
            for (int e = tid; e < 32 * NB / 2; e += DIAG_THREADS) {
                const int I = e / (NB / 2), c = 2 * (e % (NB / 2));
                const float4 v = I0 + I < m ? *reinterpret_cast<const float4*>(&A[(size_t)(I0 + I) * L + j0 + c])
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
                split4(wh, wl, (size_t)I * K2 + 2 * c, v.x, v.y, v.z, v.w);
            }
        } else {
            const int jc = (part - t32) * 32;
            __syncthreads();
#pragma unroll 4
            for (int e = tid; e < NB * 16; e += DIAG_THREADS) {
                const int c = e / 16, jj = 2 * (e % 16), j = jc + jj;
                float4 v;
                if (j >= j0 && j < j0 + NB) v = make_float4(c == j - j0 ? 1.f : 0.f, 0.f, c == j + 1 - j0 ? 1.f : 0.f, 0.f);
                else v = *reinterpret_cast<const float4*>(&A[(size_t)(j0 + c) * L + j]);
                X[c * 33 + jj] = mk<float>(v.x, v.y);
                X[c * 33 + jj + 1] = mk<float>(v.z, v.w);
            }
            __syncthreads();
            float *bh = Bh + ((size_t)box * 2 * L + 2 * jc) * K2, *bl = Bl + ((size_t)box * 2 * L + 2 * jc) * K2;
#pragma unroll 2
            for (int e = tid; e < 32 * NB / 2; e += DIAG_THREADS) {
                const int jj = e / (NB / 2), c = 2 * (e % (NB / 2));
                const c64 v = X[c * 33 + jj], w = X[(c + 1) * 33 + jj];
                split4(bh, bl, (size_t)(2 * jj) * K2 + 2 * c, v.x, -v.y, w.x, -w.y);
                split4(bh, bl, (size_t)(2 * jj + 1) * K2 + 2 * c, v.y, v.x, w.y, w.x);
            }
        }
    }
}

// ------------------------------------------------------------------ the rank-NB update on the tensor cores

// The panel's two products, persistent: one CTA per SM takes the launch's tiles in turn (every gridDim.x-th one), with two
// TMEM accumulators so that the epilogue of one tile runs while the products of the next are issued.  Warp 0 lane 0
// loads the operands (TMA, 2-stage ring), warp 1 lane 0 issues the MMAs, warps 2-5 read the accumulator (warp w owns
// TMEM lanes 32 (w mod 4)..) and write it back through shared memory with TMA.
// WP (tile = box, row tile outside J): W <- W P in place, split into hi and lo again: a tile reads only its own rows of W,
//   all before its first store.
// update (tile = box, row tile, column tile): -D with D = W B is added into A (reduce-add) outside rows and columns J,
//   and stored in them (A[I,J] = -W P, A[J,:] = P A[J,:], the left operand's rows J being -P).
// The padding diagonal is restored before the next plane.  Every wait is bounded; on a give-up each role leaves its loop,
// copies and products already issued are waited for, and TMEM is freed.
constexpr int PW = 6;                     // warps: producer, MMA issuer, four epilogue warps
constexpr int STG = 2 * UBM * 128;        // staging: two 128-row x 32-float boxes (32 KB)
constexpr int PSMEM = UST * STAGE + STG + 1024 + 256;

template <bool WP>
__device__ __forceinline__ bool tile_of(const BoxInfo* __restrict__ boxes, int t, int tl, int j0, int k, int& box,
                                        int& row0, int& col0) {
    const int per = WP ? tl : tl * tl;
    box = t / per;
    const int r = t % per;
    row0 = (WP ? r : r / tl) * UBM;
    col0 = WP ? 0 : (r % tl) * (UBN / 2);
    const BoxInfo& B = boxes[box];
    return k < B.dims[2] && j0 < B.m && row0 < B.m && col0 < B.m && !(WP && row0 == j0);
}

template <bool WP>
__global__ void __launch_bounds__(PW * 32, 1) tgj_update_pers(const __grid_constant__ CUtensorMap mWh,
                                                              const __grid_constant__ CUtensorMap mWl,
                                                              const __grid_constant__ CUtensorMap mBh,
                                                              const __grid_constant__ CUtensorMap mBl,
                                                              const __grid_constant__ CUtensorMap mS,
                                                              const BoxInfo* __restrict__ boxes, int nbox, int L,
                                                              int j0, int k, int* __restrict__ err) {
    extern __shared__ __align__(1024) unsigned char psm_raw[];
    unsigned char* base =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(psm_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    unsigned char* stg = base + UST * STAGE;
    uint64_t* full = reinterpret_cast<uint64_t*>(stg + STG);
    uint64_t* empty = full + UST;
    uint64_t* tfull = empty + UST;
    uint64_t* tempty = tfull + 2;
    uint64_t* fin = tempty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fin + 1);
    int* s_go = reinterpret_cast<int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tl = L / UBM;
    const int ntiles = nbox * (WP ? tl : tl * tl);
    if (threadIdx.x == 0) {
        for (int i = 0; i < UST; ++i) {
            tc::mbar_init(&full[i], 1);
            tc::mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&tfull[i], 1);
            tc::mbar_init(&tempty[i], 4);
        }
        tc::mbar_init(fin, 1);
        tc::fence_barrier_init();
        tc::prefetch_tmap(&mWh);
        tc::prefetch_tmap(&mWl);
        tc::prefetch_tmap(&mBh);
        tc::prefetch_tmap(&mBl);
        tc::prefetch_tmap(&mS);
    }
    if (warp == 1) {
        tc::tmem_alloc(tmem_slot, 512);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    constexpr int NKC = K2 / 32;
    int box, row0, col0;
    if (warp == 0) {
        if (lane == 0) {
            uint32_t g = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                if (!tile_of<WP>(boxes, t, tl, j0, k, box, row0, col0)) continue;
                for (int kc = 0; kc < NKC; ++kc, ++g) {
                    const int st = g % UST;
                    if (g >= UST && !tc::mbar_wait(&empty[st], ((g / UST) - 1) & 1, err, 21)) {
                        ok = false;
                        break;
                    }
                    unsigned char* s = base + st * STAGE;
                    tc::mbar_arrive_expect_tx(&full[st], STAGE);
                    tc::tma_load_3d(s, &mWh, kc * 32, row0, box, &full[st]);
                    tc::tma_load_3d(s + A_TILE, &mWl, kc * 32, row0, box, &full[st]);
                    tc::tma_load_3d(s + 2 * A_TILE, &mBh, kc * 32, 2 * col0, box, &full[st]);
                    tc::tma_load_3d(s + 2 * A_TILE + B_TILE, &mBl, kc * 32, 2 * col0, box, &full[st]);
                }
            }
            // a give-up anywhere: let the loads already issued land before the stages are left
            if (!ok || *reinterpret_cast<volatile int*>(err) != 0)
                for (uint32_t q = g > UST ? g - UST : 0; q < g; ++q) tc::mbar_drain(&full[q % UST], (q / UST) & 1);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = tc::idesc_tf32(UBM, UBN);
            uint32_t g = 0, i = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                if (!tile_of<WP>(boxes, t, tl, j0, k, box, row0, col0)) continue;
                const uint32_t a = i & 1, u = i >> 1;
                if (u >= 1 && !tc::mbar_wait(&tempty[a], (u - 1) & 1, err, 22)) break;
                tc::fence_after_sync();
                const uint32_t acc = tmem + a * 256;
                for (int kc = 0; kc < NKC; ++kc, ++g) {
                    const int st = g % UST;
                    if (!tc::mbar_wait(&full[st], (g / UST) & 1, err, 23)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after_sync();
                    const uint32_t sah = tc::smem_u32(base + st * STAGE);
                    const uint32_t sal = sah + A_TILE, sbh = sah + 2 * A_TILE, sbl = sbh + B_TILE;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const uint64_t ah = tc::desc_k_sw128(sah + kk * 32), al = tc::desc_k_sw128(sal + kk * 32);
                        const uint64_t bh = tc::desc_k_sw128(sbh + kk * 32), bl = tc::desc_k_sw128(sbl + kk * 32);
                        tc::mma_tf32(acc, ah, bh, idesc, (kc > 0 || kk > 0) ? 1u : 0u);
                        tc::mma_tf32(acc, ah, bl, idesc, 1u);
                        tc::mma_tf32(acc, al, bh, idesc, 1u);
                    }
                    tc::mma_commit(&empty[st]);
                }
                if (!ok) break;
                tc::mma_commit(&tfull[a]);
                ++i;
            }
            // every product issued has completed before TMEM is freed
            tc::mma_commit(fin);
            tc::mbar_drain(fin, 0);
        }
    } else {
        // epilogue: 128 threads, hardware barrier 1 among them
        const int et = threadIdx.x - 64;
        const int q = warp & 3;                 // TMEM lane quarter of this warp
        const int r = q * 32 + lane;            // tile row of this thread
        uint32_t i = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
            if (!tile_of<WP>(boxes, t, tl, j0, k, box, row0, col0)) continue;
            const uint32_t a = i & 1, u = i >> 1;
            if (et == 0) *s_go = tc::mbar_wait(&tfull[a], u & 1, err, 24) ? 1 : 0;
            tc::named_bar(1, 128);
            if (!*s_go) break;                  // uniform over the four warps
            tc::fence_after_sync();
            const bool store = col0 == j0 || row0 == j0;   // the panel's own rows and columns
            // per trip, update: 64 columns (two boxes of 32); WP: 32 columns, their hi and lo parts
            constexpr int CW = WP ? 32 : 64;
            for (int c = 0; c < UBN / CW; ++c) {
                uint32_t v[2][32];
                const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + a * 256 + c * CW;
                tc::tmem_ld_32x32b_x32(ta, v[0]);
                if (!WP) tc::tmem_ld_32x32b_x32(ta + 32, v[1]);
                tc::tmem_ld_wait();
                if (c == UBN / CW - 1) {
                    // the accumulator has been read: the MMA issuer may reuse it
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&tempty[a]);
                }
                if (et == 0) tc::bulk_wait_read0();   // the staging buffer's last TMA copy has read it
                tc::named_bar(1, 128);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    unsigned char* rowp = stg + h * (UBM * 128) + r * 128;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float x[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            if (WP) {
                                const float f = __uint_as_float(v[0][4 * j + e]), fh = tf32_hi(f);
                                x[e] = h == 0 ? fh : f - fh;
                            } else {
                                x[e] = -__uint_as_float(v[h][4 * j + e]);
                            }
                        }
                        *reinterpret_cast<float4*>(rowp + ((j ^ (r & 7)) << 4)) = make_float4(x[0], x[1], x[2], x[3]);
                    }
                }
                tc::fence_proxy_async_smem();
                tc::named_bar(1, 128);
                if (et == 0) {
                    if (WP) {
                        tc::tma_store_3d(&mWh, stg, c * 32, row0, box);
                        tc::tma_store_3d(&mWl, stg + UBM * 128, c * 32, row0, box);
                    } else {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int x = 2 * col0 + c * 64 + h * 32;
                            if (store) tc::tma_store_3d(&mS, stg + h * (UBM * 128), x, row0, box);
                            else tc::tma_reduce_add_3d(&mS, stg + h * (UBM * 128), x, row0, box);
                        }
                    }
                    tc::bulk_commit();
                }
            }
            ++i;
        }
        if (et == 0) tc::bulk_wait0();
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, 512);
    }
}

// G_k (row pitch ld, complex64) <- the inverse in S
__global__ void tgj_store(const BoxInfo* __restrict__ boxes, const c64* __restrict__ S, int L, c64* __restrict__ G,
                          int k) {
    const BoxInfo B = boxes[blockIdx.y];
    const int m = B.m;
    if (k >= B.dims[2]) return;
    const c64* A = S + (size_t)blockIdx.y * L * L;
    c64* Gk = G + B.fac_off + (size_t)k * B.pstride;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * m; e += gridDim.x * blockDim.x) {
        const int r = e / m, j = e % m;
        Gk[(size_t)r * B.ld + j] = A[(size_t)r * L + j];
    }
}

// the work matrices S as fp32 [nb][L][2L], boxes of 32 floats x 128 rows, 128-byte swizzle (epilogue stores)
bool encode_matrix(CUtensorMap* map, void* base, uint64_t L, uint64_t nb) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tc::tensor_map_encoder();
    if (!enc) return false;
    cuuint64_t dims[3] = {2 * L, L, nb};
    cuuint64_t strides[2] = {2 * L * 4, 2 * L * 4 * L};
    cuuint32_t box[3] = {32, (cuuint32_t)UBM, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// fp32 [nb][rows][K2] operand, boxes of 32 x box_rows, 128-byte swizzle
bool encode_operand(CUtensorMap* map, void* base, uint64_t rows, uint64_t nb, uint32_t box_rows) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tc::tensor_map_encoder();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)K2, rows, nb};
    cuuint64_t strides[2] = {(cuuint64_t)K2 * 4, (cuuint64_t)K2 * 4 * rows};
    cuuint32_t box[3] = {32, box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

size_t tgj_bytes(int nb, int m_max) {
    const size_t L = (m_max + NB - 1) / NB * NB;
    return (size_t)nb * (L * L * sizeof(c64) + 6 * L * K2 * sizeof(float) + 2 * (size_t)K2 * K2 * sizeof(float));
}

void tgj_free(helm_ctx ctx, TgjWork& W) {
    dev_free(ctx, W.S, W.s_bytes);
    dev_free(ctx, W.Wh, W.w_bytes);
    dev_free(ctx, W.Wl, W.w_bytes);
    dev_free(ctx, W.Bh, W.b_bytes);
    dev_free(ctx, W.Bl, W.b_bytes);
    dev_free(ctx, W.Ph, W.p_bytes);
    dev_free(ctx, W.Pl, W.p_bytes);
    dev_free(ctx, W.flag, 2 * sizeof(int));
    W.S = W.Wh = W.Wl = W.Bh = W.Bl = W.Ph = W.Pl = nullptr;
    W.flag = nullptr;
}

helm_status tgj_alloc(helm_ctx ctx, int nbox, int m_max, TgjWork& W) {
    const int L = (m_max + NB - 1) / NB * NB;
    const size_t nb = (size_t)nbox;
    W.nb = nbox;
    W.L = L;
    W.s_bytes = nb * L * L * sizeof(c64);
    W.w_bytes = nb * L * K2 * sizeof(float);
    W.b_bytes = nb * 2 * L * K2 * sizeof(float);
    W.p_bytes = nb * K2 * K2 * sizeof(float);
    helm_status rc;
    if ((rc = dev_alloc(ctx, &W.S, W.s_bytes, "tensor-core factor work S")) ||
        (rc = dev_alloc(ctx, &W.Wh, W.w_bytes, "factor operand W")) ||
        (rc = dev_alloc(ctx, &W.Wl, W.w_bytes, "factor operand W")) ||
        (rc = dev_alloc(ctx, &W.Bh, W.b_bytes, "factor operand B")) ||
        (rc = dev_alloc(ctx, &W.Bl, W.b_bytes, "factor operand B")) ||
        (rc = dev_alloc(ctx, &W.Ph, W.p_bytes, "block pivots")) || (rc = dev_alloc(ctx, &W.Pl, W.p_bytes, "block pivots")) ||
        (rc = dev_alloc(ctx, (void**)&W.flag, 2 * sizeof(int), "factor flags"))) {
        tgj_free(ctx, W);
        return rc;
    }
    if (!encode_operand(&W.mWh, W.Wh, L, nb, UBM) || !encode_operand(&W.mWl, W.Wl, L, nb, UBM) ||
        !encode_operand(&W.mBh, W.Bh, 2ull * L, nb, UBN) || !encode_operand(&W.mBl, W.Bl, 2ull * L, nb, UBN) ||
        !encode_operand(&W.mPh, W.Ph, K2, nb, UBN) || !encode_operand(&W.mPl, W.Pl, K2, nb, UBN) ||
        !encode_matrix(&W.mS, W.S, L, nb)) {
        tgj_free(ctx, W);
        return set_error(ctx, HELM_ECUDA, "cuTensorMapEncodeTiled failed for the tensor-core factorisation");
    }
    static PerDevice attr;
    if (!attr.done(ctx->device)) {
        cudaFuncSetAttribute(tgj_update_pers<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, PSMEM);
        cudaFuncSetAttribute(tgj_update_pers<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, PSMEM);
        cudaFuncSetAttribute(tgj_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, DIAG_SMEM);
        attr.mark(ctx->device);
    }
    cudaMemsetAsync(W.S, 0, W.s_bytes, ctx->stream);
    cudaMemsetAsync(W.flag, 0, 2 * sizeof(int), ctx->stream);
    return HELM_OK;
}

void tgj_pad(helm_ctx ctx, const TgjWork& W, const BoxInfo* dbox, int nbox) {
    tgj_pad_diag<<<dim3(1, nbox), 128, 0, ctx->stream>>>(dbox, (c64*)W.S, W.L);
    ctx->launches++;
}

void tgj_eliminate(helm_ctx ctx, const TgjWork& W, const BoxInfo* dbox, const BoxInfo* hbox, int nbox, int m_max, int k) {
    cudaStream_t st = ctx->stream;
    const int tl = W.L / NB, sms = std::max(1, ctx->sm_count);
    const int pgrid = std::min(sms, nbox * tl * tl), wgrid = std::min(sms, nbox * tl);
    // the block inverses (one CTA each) and the copying CTAs beside them: the SMs the blocks leave free, half of them at
    // least
    const int cgrid = nbox + std::max(sms - nbox, sms / 2);
    // algorithmic bytes of one update launch: every active box reads and writes the rows outside J (below m) of its
    // matrix once; of one panel: the block, the rows J, the column block J and the operands written
    for (int j0 = 0; j0 < m_max; j0 += NB) {
        double ub = 0, pb = 0;
        for (int i = 0; i < nbox; ++i) {
            const BoxInfo& b = hbox[i];
            if (k < b.dims[2] && j0 < b.m) {
                const double rows = b.m - std::min(NB, b.m - j0);
                ub += 2.0 * rows * b.m * sizeof(c64);
                pb += (2.0 * NB * b.m + (double)NB * b.m) * sizeof(c64) + (2.0 * 2 * b.m + b.m) * K2 * sizeof(float);
            }
        }
        int t = prof_begin(ctx, "gj_panel_tc");
        tgj_panel<<<cgrid, DIAG_THREADS, DIAG_SMEM, st>>>(dbox, (const c64*)W.S, W.L, nbox, (float*)W.Wh, (float*)W.Wl,
                                                          (float*)W.Ph, (float*)W.Pl, (float*)W.Bh, (float*)W.Bl, W.flag, j0,
                                                          k);
        if (tl > 1) {   // W P is empty when the panel is the whole matrix
            tgj_update_pers<true><<<wgrid, PW * 32, PSMEM, st>>>(W.mWh, W.mWl, W.mPh, W.mPl, W.mS, dbox, nbox, W.L, j0, k,
                                                                 W.flag + 1);
            ctx->launches++;
        }
        prof_end(ctx, t, pb);
        t = prof_begin(ctx, "gj_update_tc");
        tgj_update_pers<false><<<pgrid, PW * 32, PSMEM, st>>>(W.mWh, W.mWl, W.mBh, W.mBl, W.mS, dbox, nbox, W.L, j0, k,
                                                              W.flag + 1);
        prof_end(ctx, t, ub);
        ctx->launches += 2;
    }
}

// Tensor-core factorisation of a padded complex64 plane set (the fine sets of TF32 / BF16 factors).
// *singular: a zero block pivot; *weak: a block pivot below 1e-6 of its block (the caller then factors the
// set again with full partial pivoting).  Returns HELM_ETIMEOUT if a bounded wait of the update gave up.
helm_status planeset_factor_tc(helm_ctx ctx, PlaneSet& P, int* singular, int* weak) {
    *singular = *weak = 0;
    if (P.prec != HELM_PREC_FP32 || !P.padded)
        return set_error(ctx, HELM_EINVAL, "planeset_factor_tc: needs a padded complex64 set");
    cudaStream_t st = ctx->stream;
    TgjWork W;
    HELM_TRY(tgj_alloc(ctx, P.nbox, P.m_max, W));
    void* T = nullptr;
    helm_status rc = dev_alloc(ctx, &T, W.s_bytes, "tensor-core factor work T");
    auto cleanup = [&]() {
        dev_free(ctx, T, W.s_bytes);
        tgj_free(ctx, W);
    };
    if (rc) {
        cleanup();
        return rc;
    }
    const c64* coef = (const c64*)P.coef;
    c64* S = (c64*)W.S;
    const unsigned eb = (unsigned)std::min<long long>(((long long)P.m_max * P.m_max + 255) / 256, 2048);
    const dim3 egrid(eb, P.nbox);
    for (int k = 0; k < P.bz_max; ++k) {
        tgj_pad(ctx, W, P.dbox, P.nbox);
        if (k == 0) {
            tgj_schur_init<<<egrid, 256, 0, st>>>(P.dbox, coef, S, W.L);
            ctx->launches++;
        } else {
            tgj_schur_gu<<<egrid, 256, 0, st>>>(P.dbox, coef, S, (c64*)T, W.L, k);
            tgj_schur_lt<<<egrid, 256, 0, st>>>(P.dbox, coef, (const c64*)T, S, W.L, k);
            ctx->launches += 2;
        }
        tgj_eliminate(ctx, W, P.dbox, P.hbox.data(), P.nbox, P.m_max, k);
        tgj_store<<<egrid, 256, 0, st>>>(P.dbox, S, W.L, (c64*)P.G, k);
        ctx->launches++;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) {
            cleanup();
            return cuda_check(ctx, e, "tensor-core plane factorisation launch");
        }
    }
    int hflag[2] = {0, 0};
    cudaMemcpyAsync(hflag, W.flag, 2 * sizeof(int), cudaMemcpyDeviceToHost, st);
    rc = cuda_check(ctx, cudaStreamSynchronize(st), "tensor-core plane factorisation");
    cleanup();
    if (rc) return rc;
    if (hflag[1]) return set_error(ctx, HELM_ETIMEOUT, "tensor-core plane factorisation: a bounded wait gave up");
    *singular = hflag[0] & 1;
    *weak = (hflag[0] >> 1) & 1;
    return HELM_OK;
}
