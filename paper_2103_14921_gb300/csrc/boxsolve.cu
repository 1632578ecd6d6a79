// One-level ORAS on small boxes in one launch: out = sum_i R_i^T D_i A_i^{-1} R_i v for boxes whose local vector and
// plane inverses fit in shared memory (the coarse boxes of the inexact coarse solve: about 8 x 8 x 8 nodes).
//
// A CTA owns one box and cc columns and walks the 2 n_z - 1 steps of the plane sweeps (y_k = G_k (b_k - L_k y_{k-1}),
// then x_k = y_k - G_k U_k x_{k+1}): b_k is gathered from v, the plane of the last step stays in shared memory, y_k
// waits for the backward sweep in loc, and core nodes of x_k go straight to out.  So the 2 n_z - 1 pairs of launches of the
// general sweeps, with a few microseconds of work each, and the two transfers become one.  G_k and the coupling
// coefficients of the next step arrive by cp.async while a step runs (two buffers when they fit, else one).
// A thread of the product owns two rows and CT columns over one of ks slices of K (two shared loads of G and CT of
// the right-hand side for 2 CT complex multiply-adds); the slices are added in a fixed order, so results do not
// depend on scheduling.
//
// Bound: the product's FP32 multiply-adds (8 x 8-node planes, 16 columns: 4,300 clocks per step and SM with two CTAs, 4,100
// at full rate); around it the items of a plane belong to fixed threads, so that their indices are formed once and what
// they read from global memory is loaded a step ahead (with the indices and loads in the loops a step took 14,500).
#include <atomic>

#include "internal.h"

namespace {

constexpr int BS_THREADS = 256;
constexpr int BS_ITEMS = 4;   // (node, column) items of a plane per thread at most

template <int BYTES>
__device__ __forceinline__ void bs_copy(void* s, const void* g) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(s);
    if (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(g) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(g) : "memory");
}

struct BoxPlan {
    int cc = 0, nbuf = 0, ks = 0, gp = 0;
    bool wide = false;   // 16-byte copies of G
    size_t smem = 0;
};

template <typename TV, typename TL, int CT>
__global__ void __launch_bounds__(BS_THREADS, 2) box_solve(const BoxInfo* __restrict__ boxes,
                                                        const cplx<TL>* __restrict__ coef,
                                                        const cplx<TL>* __restrict__ G, const cplx<TV>* __restrict__ v,
                                                        cplx<TV>* __restrict__ out, cplx<TL>* __restrict__ loc, int nx,
                                                        int ny, int nrhs, int m_max, BoxPlan pl) {
    typedef cplx<TL> C;
    extern __shared__ __align__(16) unsigned char bs_sm[];
    const BoxInfo B = boxes[blockIdx.y];
    const int m = B.m, bx = B.dims[0], by = B.dims[1], bz = B.dims[2], cc = pl.cc, gp = pl.gp;
    C* gs = reinterpret_cast<C*>(bs_sm);                     // [nbuf][m][gp]
    C* win = gs + (size_t)pl.nbuf * m_max * gp;              // [m][cc]: the plane of the last step
    C* rb = win + (size_t)m_max * cc;                        // [m][cc]
    C* part = rb + (size_t)m_max * cc;                       // [ks][m][cc]
    C* cs = part + (size_t)pl.ks * m_max * cc;               // [nbuf][m][9]
    const int r0 = blockIdx.x * cc, tid = threadIdx.x;
    const int nsteps = 2 * bz - 1;
    auto plane_of = [&](int t) { return t < bz ? t : 2 * bz - 2 - t; };
    auto fetch = [&](int t) {
        const int k = plane_of(t), buf = pl.nbuf == 2 ? t & 1 : 0;
        const C* Gk = G + B.fac_off + (long long)k * B.pstride;
        C* gd = gs + (size_t)buf * m_max * gp;
        if (sizeof(C) == 8 && pl.wide) {
            // rows of an even length start on 16 bytes: two entries per copy
            for (int i = tid / 32; i < m; i += BS_THREADS / 32)
                for (int q = 2 * (tid % 32); q < m; q += 64) bs_copy<16>(gd + i * gp + q, Gk + (long long)i * B.ld + q);
        } else {
            for (int i = tid / 32; i < m; i += BS_THREADS / 32)
                for (int q = tid % 32; q < m; q += 32) bs_copy<sizeof(C)>(gd + i * gp + q, Gk + (long long)i * B.ld + q);
        }
        if (t > 0) {
            const C* ck = coef + (B.loc_off + (long long)k * m) * 27 + (t < bz ? 0 : 18);
            C* cd = cs + (size_t)buf * m_max * 9;
            for (int e = tid; e < m * 9; e += BS_THREADS) bs_copy<sizeof(C)>(cd + e, ck + (e / 9) * 27 + e % 9);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(0);
    // this thread's items of a plane: column r0 + (tid mod cc), nodes tid / cc + i (256 / cc); per item the in-plane
    // node (-1: none), its grid offset in plane 0 of the box, and whether the box's core holds it
    const int cl = tid & (cc - 1), col = r0 + cl, p_first = tid / cc, p_step = BS_THREADS / cc;
    const bool has = col < nrhs;
    int px_[BS_ITEMS], py_[BS_ITEMS];
    uint32_t core = 0;
#pragma unroll
    for (int i = 0; i < BS_ITEMS; ++i) {
        const int p = p_first + i * p_step;
        px_[i] = p < m ? p % bx : -1;
        py_[i] = p / bx;
        const int gi = B.lo[0] + px_[i], gj = B.lo[1] + py_[i];
        if (p < m && gi >= B.core_lo[0] && gi < B.core_hi[0] && gj >= B.core_lo[1] && gj < B.core_hi[1]) core |= 1u << i;
    }
    auto at_grid = [&](int i, int k) {
        return (((long long)(B.lo[2] + k) * ny + B.lo[1] + py_[i]) * nx + B.lo[0] + px_[i]) * nrhs + col;
    };
    auto at_loc = [&](int i, int k) { return (B.loc_off + (long long)k * m + p_first + i * p_step) * nrhs + col; };
    // b of the next forward plane, loaded a step ahead; backward, y of the current one, loaded before its product
    C nxt[BS_ITEMS];
#pragma unroll
    for (int i = 0; i < BS_ITEMS; ++i) {
        nxt[i] = mk<TL>(0, 0);
        if (px_[i] >= 0 && has) {
            const cplx<TV> a = v[at_grid(i, 0)];
            nxt[i] = mk<TL>((TL)a.x, (TL)a.y);
        }
    }
    const int mh = (m + 1) / 2, ncg = cc / CT, units = mh * ncg, kw = (m + pl.ks - 1) / pl.ks;
    for (int t = 0; t < nsteps; ++t) {
        const bool fwd = t < bz;
        const int k = plane_of(t), buf = pl.nbuf == 2 ? t & 1 : 0;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();   // step t's G and coefficients, the previous step's plane of win
        if (pl.nbuf == 2 && t + 1 < nsteps) fetch(t + 1);
        // the prepared right-hand side; couplings that leave the box have zero coefficients, their index is clamped
        const C* ck = cs + (size_t)buf * m_max * 9;
#pragma unroll
        for (int i = 0; i < BS_ITEMS; ++i) {
            if (px_[i] < 0) break;
            const int p = p_first + i * p_step;
            C acc = fwd ? nxt[i] : mk<TL>(0, 0);
            if (t > 0) {
                const int xo[3] = {max(px_[i] - 1, 0), px_[i], min(px_[i] + 1, bx - 1)};
#pragma unroll
                for (int d = 0; d < 9; ++d) {
                    const int qy = min(max(py_[i] + d / 3 - 1, 0), by - 1);
                    C c = ck[p * 9 + d];
                    if (fwd) c = mk<TL>(-c.x, -c.y);
                    cmac(acc, c, win[(qy * bx + xo[d % 3]) * cc + cl]);
                }
            }
            rb[p * cc + cl] = acc;
        }
#pragma unroll
        for (int i = 0; i < BS_ITEMS; ++i) {
            if (px_[i] < 0 || !has) break;
            if (t + 1 < bz) {
                const cplx<TV> a = v[at_grid(i, t + 1)];
                nxt[i] = mk<TL>((TL)a.x, (TL)a.y);
            } else if (!fwd) {
                nxt[i] = loc[at_loc(i, k)];
            }
        }
        __syncthreads();
        const C* gk = gs + (size_t)buf * m_max * gp;
        for (int u = tid; u < units * pl.ks; u += BS_THREADS) {
            const int s = u / units, w = u % units, c0 = (w % ncg) * CT, i0 = w / ncg, i1 = min(i0 + mh, m - 1);
            const int q1 = min(m, (s + 1) * kw);
            C a0[CT], a1[CT];
#pragma unroll
            for (int c = 0; c < CT; ++c) a0[c] = a1[c] = mk<TL>(0, 0);
            const C *g0 = gk + i0 * gp, *g1 = gk + i1 * gp;
#pragma unroll 4
            for (int q = s * kw; q < q1; ++q) {
                const C x0 = g0[q], x1 = g1[q];
#pragma unroll
                for (int c = 0; c < CT; ++c) {
                    const C bv = rb[q * cc + c0 + c];
                    cmac(a0[c], x0, bv);
                    cmac(a1[c], x1, bv);
                }
            }
            C* ps = part + (size_t)s * m_max * cc;
#pragma unroll
            for (int c = 0; c < CT; ++c) {
                ps[i0 * cc + c0 + c] = a0[c];
                if (i0 + mh < m) ps[(i0 + mh) * cc + c0 + c] = a1[c];
            }
        }
        __syncthreads();
        if (pl.nbuf == 1 && t + 1 < nsteps) fetch(t + 1);
        // y_k (kept for the backward sweep), or x_k: written by the box whose core holds the node (owner partition of
        // unity; the last forward plane is also the first of the backward sweep)
        const bool core_z = t >= bz - 1 && B.lo[2] + k >= B.core_lo[2] && B.lo[2] + k < B.core_hi[2];
#pragma unroll
        for (int i = 0; i < BS_ITEMS; ++i) {
            if (px_[i] < 0) break;
            const int e = (p_first + i * p_step) * cc + cl;
            C x = part[e];
            for (int s = 1; s < pl.ks; ++s) x = x + part[(size_t)s * m_max * cc + e];
            if (has) {
                if (t < bz - 1) loc[at_loc(i, k)] = x;
                if (!fwd) x = nxt[i] - x;
                if (core_z && ((core >> i) & 1u)) out[at_grid(i, k)] = mk<TV>((TV)x.x, (TV)x.y);
            }
            win[e] = x;
        }
    }
}

// Columns per CTA: the most (at most 16) that still give every SM a CTA; two buffers when two CTAs fit per SM with them
// or no SM gets a second CTA anyway, else one.  cc = 0: the boxes are too large.
template <typename TL>
BoxPlan box_plan(helm_ctx ctx, const PlaneSet& P, int nrhs) {
    BoxPlan best;
    const size_t es = sizeof(cplx<TL>);
    const int m = P.m_max, mh = (m + 1) / 2;
    for (int cc = 16; cc >= 1; cc >>= 1) {
        if ((cc > 1 && cc >= 2 * nrhs) || m * cc > BS_ITEMS * BS_THREADS) continue;
        BoxPlan p;
        p.cc = cc;
        // pitch: the rows a warp reads fall in different banks (odd, or 2 mod 4 where 16-byte copies need an even one)
        p.wide = es == 8 && P.hbox.size() > 0;
        for (const auto& b : P.hbox) p.wide = p.wide && b.m % 2 == 0;
        p.gp = p.wide ? m + (m % 4 == 0 ? 2 : 0) : (m | 1);
        const int units = mh * (cc / std::min(cc, 4));
        p.ks = std::max(1, std::min({BS_THREADS / units, m / 8, 8}));
        for (p.nbuf = 2; p.nbuf >= 1; --p.nbuf) {
            p.smem = ((size_t)(2 + p.ks) * m * cc + (size_t)p.nbuf * m * (p.gp + 9)) * es;
            const bool one = (long long)P.nbox * ((nrhs + cc - 1) / cc) <= ctx->sm_count;
            if (p.smem <= (size_t)(p.nbuf == 2 && !one ? 110 : 200) * 1024) break;
        }
        if (p.nbuf < 1) continue;
        best = p;
        if ((long long)P.nbox * ((nrhs + cc - 1) / cc) >= ctx->sm_count) break;
    }
    return best;
}

template <typename TV, typename TL, int CT>
cudaError_t launch_ct(helm_ctx ctx, const PlaneSet& P, const cplx<TV>* v, cplx<TV>* out, cplx<TL>* loc, int nx, int ny, int nrhs,
                      const BoxPlan& p, cudaStream_t st) {
    static PerDevice attr;
    if (!attr.done(ctx->device)) {
        const cudaError_t e = cudaFuncSetAttribute(box_solve<TV, TL, CT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   200 * 1024);
        if (e != cudaSuccess) return e;
        attr.mark(ctx->device);
    }
    box_solve<TV, TL, CT><<<dim3((nrhs + p.cc - 1) / p.cc, P.nbox), BS_THREADS, p.smem, st>>>(
        P.dbox, (const cplx<TL>*)P.coef, (const cplx<TL>*)P.G, v, out, loc, nx, ny, nrhs, P.m_max, p);
    return cudaGetLastError();
}

template <typename TV, typename TL>
helm_status run(helm_ctx ctx, const PlaneSet& P, const void* v, void* out, void* loc, int nx, int ny, int nrhs,
                cudaStream_t st, bool* done) {
    if (P.nbox > 65535) return HELM_OK;
    const BoxPlan p = box_plan<TL>(ctx, P, nrhs);
    if (!p.cc) return HELM_OK;
    const cplx<TV>* vv = (const cplx<TV>*)v;
    cplx<TV>* oo = (cplx<TV>*)out;
    cplx<TL>* ll = (cplx<TL>*)loc;
    const cudaError_t e = p.cc >= 4   ? launch_ct<TV, TL, 4>(ctx, P, vv, oo, ll, nx, ny, nrhs, p, st)
                          : p.cc == 2 ? launch_ct<TV, TL, 2>(ctx, P, vv, oo, ll, nx, ny, nrhs, p, st)
                                      : launch_ct<TV, TL, 1>(ctx, P, vv, oo, ll, nx, ny, nrhs, p, st);
    HELM_CUDA(ctx, e);
    ctx->launches++;
    *done = true;
    return HELM_OK;
}

}  // namespace

// out = M^{-1} v of a set of small boxes (cores partition the nx x ny x ... grid), vectors in precision wp; loc: nloc x
// nrhs entries of the set's precision (scratch).  *done = false when a box does not fit in shared memory (the caller then runs the general sweeps).
helm_status boxes_solve_smem(helm_ctx ctx, const PlaneSet& P, int wp, const void* v, void* out, void* loc, int nx, int ny,
                             int nrhs, cudaStream_t st, bool* done) {
    *done = false;
    if (P.padded || P.packed || P.prec == HELM_PREC_BF16 || nrhs < 1) return HELM_OK;
    const bool l64 = P.prec == HELM_PREC_FP64;
    if (wp == HELM_PREC_FP64)
        return l64 ? run<double, double>(ctx, P, v, out, loc, nx, ny, nrhs, st, done)
                   : run<double, float>(ctx, P, v, out, loc, nx, ny, nrhs, st, done);
    return l64 ? run<float, double>(ctx, P, v, out, loc, nx, ny, nrhs, st, done)
               : run<float, float>(ctx, P, v, out, loc, nx, ny, nrhs, st, done);
}
