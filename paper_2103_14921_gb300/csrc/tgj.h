// Workspace and driver of the tensor-core block Gauss-Jordan elimination (planelu_tc.cu), shared by the complex64
// factorisation and by the complex128 one (planelu_dp.cu), which starts from its inverses.
#pragma once
#include <cuda.h>

#include "internal.h"

struct TgjWork {
    int nb = 0, L = 0;                       // boxes; pitch of the work matrices (m_max rounded up to 128)
    size_t s_bytes = 0, w_bytes = 0, b_bytes = 0, p_bytes = 0;
    void *S = nullptr, *Wh = nullptr, *Wl = nullptr, *Bh = nullptr, *Bl = nullptr, *Ph = nullptr, *Pl = nullptr;
    int* flag = nullptr;                     // [0] pivots (bit 0 zero, bit 1 tiny) and bit 2 of dp_invert, [1] bounded waits
    CUtensorMap mWh, mWl, mBh, mBl, mPh, mPl, mS;
};

size_t tgj_bytes(int nb, int m_max);
helm_status tgj_alloc(helm_ctx ctx, int nb, int m_max, TgjWork& W);   // S and the flags zeroed
void tgj_free(helm_ctx ctx, TgjWork& W);
// identity on the padding diagonal of every box's work matrix (before each plane)
void tgj_pad(helm_ctx ctx, const TgjWork& W, const BoxInfo* dbox, int nbox);
// S <- S^{-1} of plane k of the boxes (device and host tables of nbox <= W.nb boxes, planes of at most m_max unknowns)
void tgj_eliminate(helm_ctx ctx, const TgjWork& W, const BoxInfo* dbox, const BoxInfo* hbox, int nbox, int m_max, int k);

// complex128 plane inverses from complex64 ones (planelu_dp.cu)
struct DpWork {
    int nb = 0, m_max = 0, Lr = 0, Nr = 0, Kp = 0;
    size_t as_bytes = 0, ax_bytes = 0, b_bytes = 0, e_bytes = 0;
    void *AS = nullptr, *AX = nullptr, *B = nullptr;   // digit slices of S and X (left operands) and of a right operand
    int *eS = nullptr, *eX = nullptr, *eB = nullptr;   // their row and column exponents
    CUtensorMap mAS, mAX, mB64, mB128;   // (right operand: boxes of 64 and of 128 rows)
};
size_t dp_bytes(int nb, int m_max);
helm_status dp_alloc(helm_ctx ctx, int nb, int m_max, DpWork& W);
void dp_free(helm_ctx ctx, DpWork& W);
// G_k <- S^{-1} (FP64) of plane k of the boxes: S is [nbox][m_max^2] with pitch m, R a scratch of the same size, G the
// factor storage.  flag bit 2 is set when the result is not good to FP64 (the caller then eliminates in FP64).
void dp_invert(helm_ctx ctx, const TgjWork& T, const DpWork& D, const BoxInfo* dbox, const BoxInfo* hbox, int nbox, int m_max,
               int k, const c128* S, c128* R, c128* G);
