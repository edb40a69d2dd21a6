// Blocked Householder QR of batched tall matrices (m >= n) with diag(R) >= 0: the QR
// fallback of Algorithm 1 (Appendix A.2) and the QR preprocessing of rectangular inputs
// (Section 4.1, rectangular matrices).
#pragma once
#include "ops.cuh"

namespace psvd {

constexpr int kQrMaxRows = 23024;
// Panel width nb (64 or 32) for m rows; false above kQrMaxRows.
bool qr_shape(int m, int *nb);

constexpr int kQrSplit = 8;   // largest K split of the X^T Y products of a block

// The columns are normalized by powers of two (norms <= 1), so every array below is bounded and kept as
// split-FP16 halves; matrices with very small rows (fine[b]) as split TF32 in the same memory.
struct QrWS {
    int B = 0, m = 0, n = 0, nb = 0, npan = 0, nsup = 0, ks = 1;
    long long ldm = 0, ldn = 0;
    float *UThi = nullptr, *UTlo = nullptr;   // [B][n][ldm] the matrix transposed, being factored (kF16X)
    float *YThi = nullptr, *YTlo = nullptr;   // [B][n][ldm] reflector j as row j (1 at j, 0 above) (kF16V)
    float *Yhi = nullptr, *Ylo = nullptr;     // [B][m][ldn] the same reflectors as columns (kF16V)
    float *QThi = nullptr, *QTlo = nullptr;   // [B][n][ldm] Q^T being accumulated (kF16X)
    float *tau = nullptr, *beta = nullptr;     // [B][n]
    float *Tm = nullptr;                       // [B][npan][nb][nb] compact-WY T of every panel
    float *Wp = nullptr;                       // [ks][B][nb][n] partial Y^T X of a panel (K split)
    float *W2hi = nullptr, *W2lo = nullptr;   // [B][n][kWY] (op(T) Y^T X)^T (kF16S2)
    float *Ts = nullptr;                       // [B][nsup][kWY][kWY] T of blocks of kWY columns
    float *Sp = nullptr;                       // [kQrSplit][B][n][kWY] partial X^T Y, or Y^T Y, of a block
    unsigned *amax = nullptr;                  // [B][n] max |a| of every column (float bits)
    float *scale = nullptr, *iscale = nullptr; // [B][n] 2^e and 2^-e of every column
    int *fine = nullptr;                       // [B] PREC_F16X3 or PREC_TF32X3
    int *skip = nullptr;                       // [B] 1 = matrix not factored (flag[b] == 0)
    unsigned *err = nullptr;

    template <class C>
    void carve(C &cv, int B_, int m_, int n_) {
        B = B_; m = m_; n = n_;
        if (!qr_shape(m, &nb)) nb = 64;
        npan = (n + nb - 1) / nb;
        nsup = (n + kWY - 1) / kWY;
        ldm = pad_ld(m); ldn = pad_ld(n);
        ks = 16;
        const long long B64 = B, nm = (long long)n * ldm;
        UThi = cv.template take<float>(B64 * nm); UTlo = cv.template take<float>(B64 * nm);
        YThi = cv.template take<float>(B64 * nm); YTlo = cv.template take<float>(B64 * nm);
        Yhi = cv.template take<float>(B64 * m * ldn); Ylo = cv.template take<float>(B64 * m * ldn);
        QThi = cv.template take<float>(B64 * nm); QTlo = cv.template take<float>(B64 * nm);
        tau = cv.template take<float>(B64 * n); beta = cv.template take<float>(B64 * n);
        Tm = cv.template take<float>(B64 * npan * nb * nb);
        Wp = cv.template take<float>((long long)ks * B64 * nb * std::min(n, kWY));
        W2hi = cv.template take<float>(B64 * n * kWY); W2lo = cv.template take<float>(B64 * n * kWY);
        Ts = cv.template take<float>(B64 * nsup * kWY * kWY);
        Sp = cv.template take<float>((long long)kQrSplit * B64 * n * kWY);
        amax = cv.template take<unsigned>(B64 * n);
        scale = cv.template take<float>(B64 * n);
        iscale = cv.template take<float>(B64 * n);
        skip = cv.template take<int>(B64);
        fine = cv.template take<int>(B64);
        err = cv.template take<unsigned>(4);
    }
};

// Q R = A for the matrices with flag[b] != 0 (flag may be null: all), diag(R) >= 0.
// A: batch x m x n (user layout, read), Q: batch x m x n out (may alias A; written only for
// flagged matrices), R: batch x n x n out (upper triangular; may be null).  Asynchronous.
int qr_factor(const float *A, float *Q, float *R, const int *flag, QrWS &w, cudaStream_t st);

}  // namespace psvd
