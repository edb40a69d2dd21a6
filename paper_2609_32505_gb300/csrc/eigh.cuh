// Symmetric eigensolver for H = V Sigma V^T (the EVD of Algorithm 1).
#pragma once
#include <algorithm>

#include "ops.cuh"

namespace psvd {

// Largest n.  The kernels whose shared memory goes with n have their limit set for this one: the limit is the
// function's, for all threads, and a call that set it for its own n could lower it between another thread's setting
// and launch.
constexpr int kEighMaxN = 16384;
constexpr int kTrdChipMin = 3, kTrdChipMax = 4096;   // sizes whose tridiagonalization runs on chip (trd.cu)
constexpr int kBtSplit = 8; // largest K split of the back-transform's V^T Y products

constexpr int kIvJ = 8;     // rows per stage of inverse iteration's ring
// rows of its arrays: half the matrix from either end, and what the last stage reads past it
inline int iv_rows(int n) { return (int)round_up((n - 1) / 2 + kIvJ + 1, 2); }
// doubles of one of them for a matrix: 16 vectors per warp, two lanes each
inline long long iv_doubles(int n) { return (long long)((n + 15) / 16) * iv_rows(n) * 32; }
// Matrices whose vectors are worked on at once: as many as fit 3 GB (five such arrays and the FP32 vectors), one at
// least.  Four matrices of 4096 fit; one at a time leaves most of the chip idle.  (A matrix of 16384 takes 11.8 GB;
// counted as 44 bytes an entry, without the padding to whole warps and stages, 65535 matrices of 33 took 6.4 GB.)
constexpr long long kIvBytes = 3000000000LL;
inline int iv_matrices(int B, int n) {
    const long long per = 5 * 8 * iv_doubles(n) + 4LL * n * n;
    return (int)std::max<long long>(1, std::min<long long>(B, kIvBytes / per));
}

struct EighWS {
    int B = 0, n = 0, nblk = 0, chunk = 0, nrp = 0;   // nrp: rows of Vh, padded to kWY
    long long ldn = 0, ll_ld = 0;
    float *Aw = nullptr;          // working copy of H (n x n per matrix)
    float *Vh = nullptr;          // Householder vectors as rows (n x ldn), v_k[k+1] = 1
    float *tau = nullptr;         // [B][n]
    double *d = nullptr, *e = nullptr, *lam = nullptr;   // tridiagonal and eigenvalues [B][n]
    float *pbuf = nullptr;        // [groups][2][n]
    unsigned long long *ll = nullptr;   // [groups][4][ll_ld] exchange words of the on-chip tridiagonalization
    unsigned *bar = nullptr;      // [groups] barrier counters
    // split-FP16 operands of the back-transform
    __half *Vhi = nullptr, *Vlo = nullptr;     // Householder rows (n x ldn), scaled by kF16V
    __half *Yhi = nullptr, *Ylo = nullptr;     // Householder vectors as columns (n x ldn), scaled by kF16V
    __half *VThi = nullptr, *VTlo = nullptr;   // current V^T (n x ldn), scaled by kF16X
    float *S = nullptr;                        // V^T Y for a pair of blocks (n x 2 kWY), K-split slices
    __half *S2hi = nullptr, *S2lo = nullptr;   // the pair's S2 (n x 2 kWY), scaled by kF16S2
    float4 *sturm = nullptr;                   // [B][n] float-float T for the Sturm counts
    float4 *tabf = nullptr;                    // [B][iv_rows][2] T for inverse iteration, float-float
    double2 *tabd = nullptr;                   // the same in FP64
    double *tn = nullptr;                      // [B] ||T||
    float *Tm = nullptr;                       // [B][nblk][kWY][kWY]
    float *Gm = nullptr;                       // [B][nrp / kWY][kWY][kWY]  Y^T Y per block
    float *Gab = nullptr;                      // the same for neighbouring blocks, Y_{a+1}^T Y_a
    double *xs = nullptr, *lm = nullptr, *u = nullptr;   // inverse-iteration vectors, multipliers, pivot rows
    float *xf = nullptr;                       // the normalized eigenvectors of T, interleaved [n][chunk]
    unsigned *err = nullptr;
    int groups = 0;

    template <class C>
    void carve(C &cv, int B_, int n_, int groups_) {
        B = B_; n = n_; groups = groups_;
        ldn = pad_ld(n);
        nblk = n > 2 ? (n - 2 + kWY - 1) / kWY : 0;
        nrp = (int)round_up(n < 1 ? 1 : n, kWY);
        const long long B64 = B, nn = (long long)n * ldn, np = (long long)nrp * ldn;
        chunk = n * iv_matrices(B, n);
        Aw = cv.template take<float>(B64 * n * ldn);
        Vh = cv.template take<float>(B64 * np);
        tau = cv.template take<float>(B64 * n);
        d = cv.template take<double>(B64 * n);
        e = cv.template take<double>(B64 * n);
        lam = cv.template take<double>(B64 * n);
        pbuf = cv.template take<float>((long long)groups * 2 * ldn);
        ll_ld = 128;
        while (ll_ld < n && n <= kTrdChipMax) ll_ld *= 2;
        ll = cv.template take<unsigned long long>((long long)groups * 4 * ll_ld);
        bar = cv.template take<unsigned>((long long)groups * (2 * 160 + 1) + 1);   // release + arrival flags per group
        Vhi = cv.template take<__half>(B64 * np);
        Vlo = cv.template take<__half>(B64 * np);
        Yhi = cv.template take<__half>(B64 * nn);
        Ylo = cv.template take<__half>(B64 * nn);
        VThi = cv.template take<__half>(B64 * nn);
        VTlo = cv.template take<__half>(B64 * nn);
        S = cv.template take<float>(kBtSplit * B64 * n * 2 * kWY);
        S2hi = cv.template take<__half>(B64 * n * 2 * kWY);
        S2lo = cv.template take<__half>(B64 * n * 2 * kWY);
        sturm = cv.template take<float4>(B64 * n);
        tabf = cv.template take<float4>(B64 * iv_rows(n) * 2);
        tabd = cv.template take<double2>(B64 * iv_rows(n) * 2);
        tn = cv.template take<double>(B64);
        Tm = cv.template take<float>(B64 * (nblk > 0 ? nblk : 1) * kWY * kWY);
        Gm = cv.template take<float>(B64 * nrp * kWY);
        Gab = cv.template take<float>(B64 * nrp * kWY);
        xf = cv.template take<float>((long long)n * chunk);
        const long long iv = (chunk / n) * iv_doubles(n);
        xs = cv.template take<double>(iv);
        lm = cv.template take<double>(iv);
        u = cv.template take<double>(3 * iv);
        err = cv.template take<unsigned>(4);
    }
};

int eigh_groups(int B, int n);

// Tridiagonalization of the B matrices Hs (n x n) on chip where the sizes allow it (*ran tells): fills
// w.Vh (pre-zeroed), w.tau, w.d, w.e; w.bar zeroed by the caller.
int trd_chip(const float *Hs, EighWS &w, cudaStream_t st, bool *ran);

// Eigendecomposition of the symmetric matrices Hs (B x n x n, FP32, full storage).
// Writes eigenvalues descending to S (B x n, may be null) and V^T as split-FP16 halves in
// ws.VThi / ws.VTlo (rows = eigenvectors, largest-|.| entry positive), V^T to VT (B x n x n, may be
// null) and V^T as split TF32 to vt_hi / vt_lo (B x n x ldn, may be null), of the matrices whose vt_prec is
// PREC_TF32X3 only if that is given.
int eigh_forward(const float *Hs, float *S, float *VT, EighWS &ws, cudaStream_t st, float *vt_hi = nullptr,
                 float *vt_lo = nullptr, const int *vt_prec = nullptr);

}  // namespace psvd
