// Regularized SVD / polar backward (Algorithm 4, Algorithm 3) from cached factors.
//
// Algorithm 4 evaluated in the eigenbasis of H = V Sigma V^T (V^T V = I):
//   A_U = U^T Ubar, B_V = V^T Vbar, Y = M V, Z = Y^T Ubar      (= V^T M^T Wbar V, as Wbar V = Ubar)
//   B   = skew(B_V + A_U)                                       (= (V^T Vbar_tot - Vbar_tot^T V)/2)
//   V^T Hbar V = diag(Sbar) + K_eps^T o B
//   V^T C V    = sym(V^T Hbar V - D_R Z D_R),  D_R = Sigma (Sigma^2 + eps^(1/2))^-1
//   V^T X V    = T_eps o V^T C V
//   Mbar       = (Ubar D_R + 2 Y (V^T X V)) V^T                 (= Wbar R_eps + 2 M X)
// Algorithm 3 (polar) is the same chain with V^T Hbar V computed from Hbar and
// G = Wbar V in place of Ubar.  Six products on the split-FP16 tcgen05 kernel plus
// one elementwise kernel that holds every mask (K_eps, T_eps, D_R).  The products are bound by the tensor
// cores: at 4096 x 4096 each takes 345 us in split FP16 (0.40 PFLOP/s of FP32-accurate work, three FP16
// products each) and took 700 us in split TF32; the whole backward 4.10 -> 2.43 ms, its error against
// 64 bits unchanged at 2.2e-6.
#include <cmath>
#include <cstring>

#include "eigh.cuh"

namespace psvd {

// Split-FP16 operands need a power of two per matrix.  The inputs' come from their largest entries and, for
// V, the largest column norm (both 1 for orthonormal factors, whatever else a caller hands over stays in
// range); Y = M V, T1 = V^T sym(Hbar) and Wbar V are bounded by sqrt(n) times the largest entry of the one
// and the column norm of the other; X and Q are written in FP32 with their largest entries recorded, then split.
// A matrix M with rows or columns so small that halves of them lose bits has all its operands in split TF32
// (fine[b]; the same memory): the rows of the gradient are of the sizes of M's.
enum BwdMax { AM_M = 0, AM_G, AM_B, AM_U, AM_V, AM_IN, AM_X = AM_IN, AM_Q, AM_N };   // slots of amax; inputs first
enum BwdScale {                                                        // slots of es, each [B]
    ES_M = 0, ES_G, ES_B, ES_U, ES_V, ES_X, ES_Q,      // 2^e (operands are divided by it)
    ES_IM, ES_IG,                          // 2^-e
    ES_AU, ES_BV, ES_Y, ES_Z, ES_QP, ES_DA, ES_T1, ES_EH, ES_WV,      // product scales, 2^-28 included
    ES_N
};

struct BwdWS {
    int B = 0, m = 0, n = 0;
    long long ldn = 0, ldm = 0;
    float *UThi = nullptr, *UTlo = nullptr;      // U^T (n x m)
    float *GThi = nullptr, *GTlo = nullptr;      // Ubar^T or (Wbar V)^T (n x m)
    float *G = nullptr;                           // Wbar V row-major FP32 (m x n) for the epilogue (polar)
    float *Mhi = nullptr, *Mlo = nullptr;        // M (m x n)
    float *VThi = nullptr, *VTlo = nullptr;      // V^T (n x n)
    float *Vhi = nullptr, *Vlo = nullptr;        // V (n x n)
    float *dVThi = nullptr, *dVTlo = nullptr;    // Vbar^T (n x n) or sym(Hbar) (polar)
    float *Yhi = nullptr, *Ylo = nullptr;        // Y = M V (m x n)
    float *YThi = nullptr, *YTlo = nullptr;      // Y^T (n x m)
    float *AU = nullptr, *BV = nullptr, *Z = nullptr;   // n x n FP32
    float *X = nullptr;                           // V^T X V (n x n)
    float *Xhi = nullptr, *Xlo = nullptr;
    float *Q = nullptr;                           // (m x n)
    float *Qhi = nullptr, *Qlo = nullptr;
    float *Wbhi = nullptr, *Wblo = nullptr;      // Wbar (m x n), polar only
    float *S = nullptr;                           // sigma FP32 (polar: eigenvalues of H)
    float *T1 = nullptr;                          // polar: V^T, then V^T Hbar
    float *T1hi = nullptr, *T1lo = nullptr;
    unsigned *amax = nullptr;                     // [AM_N][B]
    unsigned *ext = nullptr;                      // [B][m + n] largest entries of M's rows and columns
    int *fine = nullptr;                          // [B] PREC_F16X3 or PREC_TF32X3
    float *es = nullptr;                          // [ES_N][B]
    unsigned *err = nullptr;
    EighWS ew;
    bool polar = false;
    const float *esp(int slot) const { return es + (long long)slot * B; }

    template <class C>
    void carve(C &cv, int B_, int m_, int n_, bool polar_) {
        B = B_; m = m_; n = n_; polar = polar_;
        ldn = pad_ld(n); ldm = pad_ld(m);
        const long long B64 = B, mn = (long long)m * ldn, nm = (long long)n * ldm, nn = (long long)n * ldn;
        auto pair = [&](float *&hi, float *&lo, long long k) {
            hi = cv.template take<float>(B64 * k);
            lo = cv.template take<float>(B64 * k);
        };
        pair(UThi, UTlo, nm); pair(GThi, GTlo, nm); pair(Mhi, Mlo, mn); pair(VThi, VTlo, nn); pair(Vhi, Vlo, nn);
        pair(dVThi, dVTlo, nn); pair(Yhi, Ylo, mn); pair(YThi, YTlo, nm); pair(Xhi, Xlo, nn); pair(Qhi, Qlo, mn);
        AU = cv.template take<float>(B64 * n * n); BV = cv.template take<float>(B64 * n * n);
        Z = cv.template take<float>(B64 * n * n);
        X = cv.template take<float>(B64 * n * n); Q = cv.template take<float>(B64 * m * n);
        S = cv.template take<float>(B64 * n);
        amax = cv.template take<unsigned>(B64 * (AM_N + m + n));
        ext = amax ? amax + B64 * AM_N : nullptr;
        fine = cv.template take<int>(B64);
        es = cv.template take<float>(B64 * ES_N);
        err = cv.template take<unsigned>(4);
        if (polar) {
            G = cv.template take<float>(B64 * m * n);
            pair(Wbhi, Wblo, mn);
            T1 = cv.template take<float>(B64 * n * n);
            pair(T1hi, T1lo, nn);
            ew.carve(cv, B, n, eigh_groups(B, n));
        }
    }
};

// 2^e above the largest entry (times `grow`); 1 for zero and non-finite arrays.
PSVD_DEV int bwd_exp(unsigned amax, double grow) {
    const float v = __uint_as_float(amax);
    return v > 0.f && v < INFINITY ? min(127, max(-100, ilogb((double)v * grow) + 1)) : 0;
}
// largest entry of a factor (or norm of its columns) above the [1, 2] of an orthonormal one
PSVD_DEV int bwd_exp_factor(unsigned amax) {
    const float v = __uint_as_float(amax);
    return v > 2.f && v < INFINITY ? ilogbf(v) : 0;
}
// stage 0: the scales of the inputs; 1: of X; 2: of Q
PSVD_DEV void bwd_scale(const unsigned *amax, int B, int b, int n, int stage, int polar, float *es) {
    auto put = [&](int slot, int e) { es[(long long)slot * B + b] = ldexpf(1.f, e); };
    const double rn = sqrt((double)n);
    const int eM = bwd_exp(amax[AM_M * B + b], 1.0), eV = bwd_exp_factor(amax[AM_V * B + b]);
    const int eY = bwd_exp(amax[AM_M * B + b], rn) + eV;
    if (stage == 0) {
        const int eG = bwd_exp(amax[AM_G * B + b], polar ? rn : 1.0), eB = bwd_exp(amax[AM_B * B + b], polar ? rn : 1.0);
        const int eU = bwd_exp_factor(amax[AM_U * B + b]);
        put(ES_M, eM); put(ES_G, eG); put(ES_B, eB); put(ES_U, eU); put(ES_V, eV); put(ES_IM, -eY); put(ES_IG, -eG);
        put(ES_AU, eU + eG - 28); put(ES_BV, eV + eB - 28); put(ES_Y, eM + eV - 28); put(ES_Z, eY + eG - 28);
        put(ES_T1, eB - 28); put(ES_EH, eB - 28); put(ES_WV, eG - 28);
    } else if (stage == 1) {
        const int eX = bwd_exp(amax[AM_X * B + b], 1.0);
        put(ES_X, eX); put(ES_QP, eY + eX - 28);
    } else {
        const int eQ = bwd_exp(amax[AM_Q * B + b], 1.0);
        put(ES_Q, eQ); put(ES_DA, eQ + eV - 28);
    }
}

__global__ void bwd_scale_kernel(const unsigned *amax, int B, int n, int stage, float *es) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) bwd_scale(amax, B, b, n, stage, 0, es);
}
// stage 0, and fine[b]: halves of M / 2^eM hold 22 bits down to 2^-28, so a row with a largest entry above sqrt(n)
// 2^(eM - 28), or a column above sqrt(m) 2^(eM - 28), has no more rounding error in them than in split TF32
__global__ void __launch_bounds__(256) bwd_fine_kernel(const unsigned *amax, const unsigned *ext, int B, int m, int n,
                                                       int polar, float *es, int *fine) {
    const int b = blockIdx.x;
    const float lim = ldexpf(1.f, bwd_exp(amax[AM_M * B + b], 1.0)) * 0x1p-28f;
    const float lr = sqrtf((float)n) * lim, lc = sqrtf((float)m) * lim;
    bool small = false;
    for (int i = threadIdx.x; i < m + n; i += blockDim.x) {
        const float v = __uint_as_float(ext[(long long)b * (m + n) + i]);
        small |= v > 0.f && v < (i < m ? lr : lc);
    }
    small = __syncthreads_or(small);
    if (threadIdx.x) return;
    fine[b] = small ? PREC_TF32X3 : PREC_F16X3;
    bwd_scale(amax, B, b, n, 0, polar, es);
}

// The AM_ slots of the inputs, one launch for all of them (grid.z = slot): entries, or for V^T the 2-norm
// of its rows, a warp at a time.  For M also the largest entries of its rows and columns, by tiles of 8 x 128 a
// warp (ext).
struct BwdMaxIn { const float *x[AM_IN]; long long len[AM_IN]; };
__global__ void __launch_bounds__(256) bwd_max_kernel(BwdMaxIn in, int B, int m, int n, unsigned *amax, unsigned *ext) {
    __shared__ unsigned red[8];
    const int b = blockIdx.y, slot = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (!in.x[slot]) return;
    const long long len = in.len[slot];
    const float *a = in.x[slot] + b * len;
    unsigned v = 0;
    if (slot == AM_M) {
        const int tn = (n + 127) / 128, tiles = tn * ((m + 7) / 8);
        for (int t = blockIdx.x * 8 + warp; t < tiles; t += gridDim.x * 8) {
            const int r0 = t / tn * 8, c0 = t % tn * 128 + lane;
            unsigned y[8][4];                      // all loads ahead of the reductions
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    y[r][q] = r0 + r < m && c0 + 32 * q < n
                                  ? __float_as_uint(fabsf(a[(long long)(r0 + r) * n + c0 + 32 * q])) : 0u;
            unsigned cm[4] = {0u, 0u, 0u, 0u}, rm = 0u;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
#pragma unroll
                for (int q = 0; q < 4; ++q) cm[q] = max(cm[q], y[r][q]);
                const unsigned x = __reduce_max_sync(0xffffffffu, max(max(y[r][0], y[r][1]), max(y[r][2], y[r][3])));
                if (lane == r) rm = x;
            }
            unsigned *e = ext + (long long)b * (m + n);
            if (lane < 8 && r0 + lane < m) atomicMax(&e[r0 + lane], rm);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (c0 + 32 * q < n) atomicMax(&e[m + c0 + 32 * q], cm[q]);
            v = max(v, rm);
        }
    } else if (slot == AM_V) {
        for (int r = blockIdx.x * 8 + warp; r < n; r += gridDim.x * 8) {
            float s = 0.f;
#pragma unroll 8
            for (int c = lane; c < n; c += 32) { const float t = a[(long long)r * n + c]; s += t * t; }
#pragma unroll
            for (int d = 16; d; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
            v = max(v, __float_as_uint(sqrtf(s)));
        }
    } else {
        const bool vec = ((uintptr_t)a & 15) == 0;
        const long long n4 = vec ? len / 4 : 0;
        const long long t0 = (long long)blockIdx.x * 256 + threadIdx.x, dt = (long long)gridDim.x * 256;
#pragma unroll 4
        for (long long t = t0; t < n4; t += dt) {
            const float4 q = reinterpret_cast<const float4 *>(a)[t];
            v = max(max(v, __float_as_uint(fabsf(q.x))), max(__float_as_uint(fabsf(q.y)),
                    max(__float_as_uint(fabsf(q.z)), __float_as_uint(fabsf(q.w)))));
        }
        for (long long t = 4 * n4 + t0; t < len; t += dt) v = max(v, __float_as_uint(fabsf(a[t])));
    }
    v = __reduce_max_sync(0xffffffffu, v);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) v = max(v, red[w]);
        if (v) atomicMax(&amax[slot * B + b], v);
    }
}

// D_R entry: sigma / (sigma^2 + eps^(1/2)), or the pseudo-inverse 1/sigma (eps = 0)
PSVD_DEV float dr_of(float s, float sqrt_eps, int exact) {
    if (exact) return s > 0.f ? 1.f / s : 0.f;
    return s / (s * s + sqrt_eps);
}

// V^T X V = T o sym(E_H - D_R Z D_R) with E_H = diag(Sbar) + K^T o skew(B_V + A_U)
// (svd) or E_H = the given V^T Hbar V (polar, `EH`).  The result is symmetric: one block of 32 x 8 threads
// per pair of mirrored 32 x 32 tiles (block (x, y) with x >= y) reads both tiles of every input once,
// rows coalesced, and writes both tiles of X; the largest |X| of the matrix goes to xmax.  (141 us at
// n = 4096, 1.8 TB/s: divisions and the latency of one batch of loads per block.)
__global__ void __launch_bounds__(256) bwd_core_kernel(const float *AU, const float *BV, const float *Z, const float *EH,
                                                       const float *S, const float *dS, int n, float eps, int kreg_mode,
                                                       float tie_tol, float *X, unsigned *xmax) {
    if (blockIdx.x < blockIdx.y) return;
    __shared__ float mt[32][33], mz[32][33];       // the mirrored tile of E_H (or B_V + A_U) and of Z
    __shared__ unsigned red[8];
    const int b = blockIdx.z, i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const long long bo = (long long)b * n * n;
    auto rd = [&](int i, int j, float &t, float &z) {
        t = z = 0.f;
        if (i >= n || j >= n) return;
        const long long o = bo + (long long)i * n + j;
        if (EH) t = EH[o];
        else t = (BV ? BV[o] : 0.f) + (AU ? AU[o] : 0.f);
        if (Z) z = Z[o];
    };
    float tij[4], zij[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        rd(i0 + ty + 8 * q, j0 + tx, tij[q], zij[q]);
        float t, z;
        rd(j0 + ty + 8 * q, i0 + tx, t, z);
        mt[ty + 8 * q][tx] = t;
        mz[ty + 8 * q][tx] = z;
    }
    __syncthreads();
    const float *s = S + (long long)b * n;
    const int exact = kreg_mode == 2;
    const float sq = sqrtf(eps), q4 = sqrtf(sq);
    const int j = j0 + tx;
    const float sj = j < n ? s[j] : 0.f, dj = dr_of(sj, sq, exact);
    float x[4];
    unsigned bits = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = i0 + ty + 8 * q;
        x[q] = 0.f;
        if (i >= n || j >= n) continue;
        const float si = s[i], di = dr_of(si, sq, exact);
        const float tji = mt[tx][ty + 8 * q], zji = mz[tx][ty + 8 * q];
        float eh_ij, eh_ji;
        if (EH) {
            eh_ij = tij[q];
            eh_ji = tji;
        } else {
            const float bij = 0.5f * (tij[q] - tji);    // B = skew part
            // K_ij = (s_i - s_j) / ((s_i - s_j)^2 + reg); (K^T)_ij = K_ji = -K_ij
            float kij;
            const float d = si - sj;
            if (kreg_mode == 0) kij = d / (d * d + sq);
            else if (kreg_mode == 1) kij = d / (d * d + eps * eps);
            else {
                const float smax = fmaxf(fabsf(s[0]), fabsf(s[n - 1]));
                kij = fabsf(d) <= tie_tol * smax ? 0.f : 1.f / d;
            }
            // (K^T o B)_ij = K_ji B_ij = -K_ij B_ij; symmetric, since K and B are both skew
            eh_ij = -kij * bij;
            if (i == j && dS) eh_ij += dS[(long long)b * n + i];
            eh_ji = eh_ij;
        }
        const float c = 0.5f * ((eh_ij - di * zij[q] * dj) + (eh_ji - dj * zji * di));
        const float ssum = si + sj;
        float t;
        if (exact) t = ssum > 0.f ? 1.f / ssum : 0.f;
        else t = ssum / (ssum * ssum + q4);
        x[q] = t * c;
        X[bo + (long long)i * n + j] = x[q];
        bits = max(bits, __float_as_uint(fabsf(x[q])));
    }
    __syncthreads();                               // the mirrored tile has been read
    if (i0 != j0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) mt[ty + 8 * q][tx] = x[q];
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = j0 + ty + 8 * q, c = i0 + tx;
            if (r < n && c < n) X[bo + (long long)r * n + c] = mt[tx][ty + 8 * q];
        }
    }
    bits = __reduce_max_sync(0xffffffffu, bits);
    if (tx == 0) red[ty] = bits;
    __syncthreads();
    if (tx == 0 && ty == 0) {
        for (int w = 1; w < 8; ++w) bits = max(bits, red[w]);
        atomicMax(&xmax[b], bits);
    }
}

// Q = G D_R + 2 acc (acc = Y (V^T X V)), row-major FP32, its largest |entry| recorded per matrix
struct EpiQ {
    int m, n;
    const float *G;      // m x n FP32 (nullable = zero)
    const float *S;
    float sqrt_eps;
    int exact;
    float *Q;
    unsigned *qmax;
    struct Acc { unsigned mx; };
    PSVD_DEV bool row16(Acc &a, int b, int r0, int lane, int c0, float (&v)[16], float *) const {
        if (r0 >= m || c0 >= n) return true;
        if (c0 + 16 > n || (n & 7) || ((uintptr_t)Q & 31) || (G && ((uintptr_t)G & 31))) return false;
        const int r = r0 + lane;
        // D_R of the 16 columns: one lane each
        const float dr = G && lane < 16 ? dr_of(S[(long long)b * n + c0 + lane], sqrt_eps, exact) : 0.f;
        const long long o = (long long)b * m * n + (long long)r * n + c0;
        uint32_t w[16], g[8];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            float x = 2.f * v[i];
            if (G) {
                if ((i & 7) == 0) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) g[q] = 0u;
                    if (r < m) ld_v8(G + o + i, g);
                }
                x += __uint_as_float(g[i & 7]) * __shfl_sync(0xffffffffu, dr, i);
            }
            w[i] = __float_as_uint(x);
            if (r < m) a.mx = max(a.mx, __float_as_uint(fabsf(x)));
        }
        if (r < m) st_v8x2(Q + o, w);
        return true;
    }
    PSVD_DEV void begin(Acc &a) const { a.mx = 0u; }
    PSVD_DEV void chunk(Acc &a, int b, int r, int c0, float (&v)[16]) const {
        if (r >= m) return;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int c = c0 + i;
            if (c >= n) break;
            const long long o = (long long)b * m * n + (long long)r * n + c;
            float x = 2.f * v[i];
            if (G) x += G[o] * dr_of(S[(long long)b * n + c], sqrt_eps, exact);
            Q[o] = x;
            a.mx = max(a.mx, __float_as_uint(fabsf(x)));
        }
    }
    PSVD_DEV void finish(Acc &a, int b, int, int) const {
        const unsigned v = __reduce_max_sync(0xffffffffu, a.mx);
        if ((threadIdx.x & 31) == 0 && v) atomicMax(&qmax[b], v);
    }
};

// sym(H) / scale, split
__global__ void sym_split_kernel(const float *H, const float *scale, const int *fine, int n, float *hi, float *lo,
                                 long long ld) {
    const int b = blockIdx.z;
    const int i = blockIdx.y * 16 + threadIdx.y, j = blockIdx.x * 16 + threadIdx.x;
    if (i >= n || j >= n) return;
    const float *h = H + (long long)b * n * n;
    const float x = 0.5f * (h[(long long)i * n + j] + h[(long long)j * n + i]);
    split_store(fine[b] == PREC_TF32X3, hi, lo, (long long)b * n * ld, (long long)i * ld + j, x / scale[b], kF16X);
}

// split TF32 (the EVD backward, whose factors E and Z have no bound known in advance)
template <class Epi>
static int g3(const float *ahi, const float *alo, int M, int K, long long lda, long long bsa, const float *bhi,
              const float *blo, int N, long long ldb, long long bsb, int B, const Epi &e, unsigned *err,
              cudaStream_t st) {
    MatView vah = view_of(ahi, M, K, lda, bsa, B), val = view_of(alo, M, K, lda, bsa, B);
    MatView vbh = view_of(bhi, N, K, ldb, bsb, B), vbl = view_of(blo, N, K, ldb, bsb, B);
    GemmShape s;
    memset(&s, 0, sizeof(s));
    s.M = M; s.N = N; s.K = K; s.prec_uniform = PREC_TF32X3; s.err = err;
    return launch_gemm(nullptr, nullptr, &vah, &val, &vbh, &vbl, s, B, e, st) == cudaSuccess ? PSVD_OK : PSVD_ERR_CUDA;
}
// split arrays in the formats of w.fine, scaled by es slot `scale` (which has the halves' 2^-28 in it)
template <class Epi>
static int g16(const float *ahi, const float *alo, int M, int K, long long lda, long long bsa, const float *bhi,
               const float *blo, int N, long long ldb, long long bsb, const BwdWS &w, int scale, const Epi &e,
               cudaStream_t st) {
    GemmShape s;
    memset(&s, 0, sizeof(s));
    s.M = M; s.N = N; s.K = K; s.prec = w.fine; s.err = w.err;
    s.f16_scale = 1.f;
    s.tf32_scale = kF16X * kF16X;
    s.scale_b = w.esp(scale);
    s.prof_as = PREC_TF32X3 + 1;
    return launch_split(SplitView(ahi, alo, 0, M, K, lda, bsa, w.B), SplitView(bhi, blo, 0, N, K, ldb, bsb, w.B), s, w.B, e,
                        st) == cudaSuccess ? PSVD_OK : PSVD_ERR_CUDA;
}

static SplitOut so(float *hi, float *lo, long long ld, long long bs) {
    SplitOut s;
    s.hi = hi; s.lo = lo; s.ld = ld; s.bstride = bs;
    return s;
}
// Largest entries of the inputs (null: none) and the scales that follow from them.
static int bwd_scales(BwdWS &w, const float *A, const float *G, const float *Bm, const float *U, const float *VT,
                      cudaStream_t st) {
    const int B = w.B, m = w.m, n = w.n;
    const long long mn = (long long)m * n, nn = (long long)n * n;
    PSVD_TRY(cudaMemsetAsync(w.amax, 0, sizeof(unsigned) * (size_t)B * (AM_N + m + n), st));
    const BwdMaxIn in = {{A, G, Bm, U, VT}, {mn, mn, nn, mn, nn}};
    const long long per = std::max(1, 8 * num_sms() / std::min(B, 8));
    bwd_max_kernel<<<dim3((unsigned)std::min<long long>((mn + 4095) / 4096, per), B, AM_IN), 256, 0, st>>>(in, B, m, n, w.amax, w.ext);
    bwd_fine_kernel<<<B, 256, 0, st>>>(w.amax, w.ext, B, m, n, w.polar ? 1 : 0, w.es, w.fine);
    count_launch(2);
    PSVD_TRY(cudaGetLastError());
    return PSVD_OK;
}

// Shared tail: Y = M V (row-major + transposed), Z = Y^T G, core, Q, dA = Q V^T.  G: Ubar or Wbar V, FP32 (null: zero).
static int bwd_tail(BwdWS &w, const float *G, const float *EH, const float *AU, const float *BV, const float *dS,
                    float eps, int kreg, float *dA, cudaStream_t st) {
    const int B = w.B, m = w.m, n = w.n;
    const long long ldn = w.ldn, ldm = w.ldm, mn = (long long)m * ldn, nm = (long long)n * ldm, nn = (long long)n * ldn;
    {   // Y = M V : B operand B[j][k] = V[k][j] = V^T[j][k]
        EpiHalf e;
        memset(&e, 0, sizeof(e));
        e.rows = m; e.cols = n; e.inv = w.esp(ES_IM); e.fine = w.fine;
        e.hi = w.Yhi; e.lo = w.Ylo; e.ldh = ldn; e.bsh = mn;
        e.hi_t = w.YThi; e.lo_t = w.YTlo; e.ldht = ldm; e.bsht = nm;
        PSVD_TRY_RC(g16(w.Mhi, w.Mlo, m, n, ldn, mn, w.VThi, w.VTlo, n, ldn, nn, w, ES_Y, e, st));
    }
    if (G) {   // Z = Y^T G
        EpiStore e = epi_store_plain(w.Z, n, (long long)n * n, n, n);
        PSVD_TRY_RC(g16(w.YThi, w.YTlo, n, m, ldm, nm, w.GThi, w.GTlo, n, ldm, nm, w, ES_Z, e, st));
    }
    const unsigned nt = (n + 31) / 32;
    bwd_core_kernel<<<dim3(nt, nt, B), dim3(32, 8), 0, st>>>(AU, BV, G ? w.Z : nullptr, EH, w.S, dS, n, eps, kreg, 1e-6f,
                                                            w.X, w.amax + AM_X * B);
    bwd_scale_kernel<<<(B + 127) / 128, 128, 0, st>>>(w.amax, B, n, 1, w.es);
    count_launch(2);
    PSVD_TRY(prepare_operand(w.X, n, (long long)n * n, B, n, n, false, 1.f, w.esp(ES_X), split_out(w.Xhi, w.Xlo, ldn, nn, kF16X, w.fine), st));
    {   // Q = G D_R + 2 Y (V^T X V)  (B operand = V^T X V, symmetric)
        EpiQ e;
        e.m = m; e.n = n; e.G = G; e.S = w.S; e.sqrt_eps = sqrtf(eps); e.exact = kreg == 2;
        e.Q = w.Q; e.qmax = w.amax + AM_Q * B;
        PSVD_TRY_RC(g16(w.Yhi, w.Ylo, m, n, ldn, mn, w.Xhi, w.Xlo, n, ldn, nn, w, ES_QP, e, st));
    }
    bwd_scale_kernel<<<(B + 127) / 128, 128, 0, st>>>(w.amax, B, n, 2, w.es);
    count_launch(1);
    PSVD_TRY(prepare_operand(w.Q, n, (long long)m * n, B, m, n, false, 1.f, w.esp(ES_Q), split_out(w.Qhi, w.Qlo, ldn, mn, kF16X, w.fine), st));
    {   // dA = Q V^T : B operand B[j][k] = V^T[k][j] = V[j][k]
        EpiStore e = epi_store_plain(dA, n, (long long)m * n, m, n);
        PSVD_TRY_RC(g16(w.Qhi, w.Qlo, m, n, ldn, mn, w.Vhi, w.Vlo, n, ldn, nn, w, ES_DA, e, st));
    }
    return cudaGetLastError() == cudaSuccess ? PSVD_OK : PSVD_ERR_CUDA;
}

int svd_backward(const float *A, const float *U, const float *S, const float *VT, const float *dU, const float *dS,
                 const float *dVT, float *dA, BwdWS &w, double eps, int kreg, cudaStream_t st) {
    const int B = w.B, m = w.m, n = w.n;
    const long long ldn = w.ldn, ldm = w.ldm, mn = (long long)m * ldn, nm = (long long)n * ldm, nn = (long long)n * ldn;
    const long long umn = (long long)m * n, unn = (long long)n * n;
    const float feps = kreg == 2 ? 0.f : (float)eps;
    PSVD_TRY(cudaMemcpyAsync(w.S, S, sizeof(float) * (size_t)B * n, cudaMemcpyDeviceToDevice, st));
    PSVD_TRY_RC(bwd_scales(w, A, dU, dVT, dU ? U : nullptr, VT, st));
    PSVD_TRY(prepare_operand(A, n, umn, B, m, n, false, 1.f, w.esp(ES_M), split_out(w.Mhi, w.Mlo, ldn, mn, kF16X, w.fine), st));
    PSVD_TRY(prepare_operand(VT, n, unn, B, n, n, false, 1.f, w.esp(ES_V), split_out(w.VThi, w.VTlo, ldn, nn, kF16X, w.fine), st));
    PSVD_TRY(prepare_operand(VT, n, unn, B, n, n, true, 1.f, w.esp(ES_V), split_out(w.Vhi, w.Vlo, ldn, nn, kF16X, w.fine), st));
    if (dU) {
        PSVD_TRY(prepare_operand(U, n, umn, B, m, n, true, 1.f, w.esp(ES_U), split_out(w.UThi, w.UTlo, ldm, nm, kF16X, w.fine), st));
        PSVD_TRY(prepare_operand(dU, n, umn, B, m, n, true, 1.f, w.esp(ES_G), split_out(w.GThi, w.GTlo, ldm, nm, kF16X, w.fine), st));
        EpiStore e = epi_store_plain(w.AU, n, unn, n, n);       // A_U = U^T Ubar
        PSVD_TRY_RC(g16(w.UThi, w.UTlo, n, m, ldm, nm, w.GThi, w.GTlo, n, ldm, nm, w, ES_AU, e, st));
    }
    if (dVT) {
        PSVD_TRY(prepare_operand(dVT, n, unn, B, n, n, false, 1.f, w.esp(ES_B), split_out(w.dVThi, w.dVTlo, ldn, nn, kF16X, w.fine), st));
        EpiStore e = epi_store_plain(w.BV, n, unn, n, n);       // B_V = V^T Vbar
        PSVD_TRY_RC(g16(w.VThi, w.VTlo, n, n, ldn, nn, w.dVThi, w.dVTlo, n, ldn, nn, w, ES_BV, e, st));
    }
    return bwd_tail(w, dU, nullptr, dU ? w.AU : nullptr, dVT ? w.BV : nullptr, dS, feps, kreg, dA, st);
}

int polar_backward(const float *A, const float *H, const float *dW, const float *dH, float *dA, BwdWS &w, double eps,
                   cudaStream_t st) {
    const int B = w.B, m = w.m, n = w.n;
    const long long ldn = w.ldn, ldm = w.ldm, mn = (long long)m * ldn, nm = (long long)n * ldm, nn = (long long)n * ldn;
    const long long umn = (long long)m * n, unn = (long long)n * n;
    // EVD of H (symmetrized by the eigensolver's reads of the full matrix); V^T plain in T1
    PSVD_TRY_RC(eigh_forward(H, w.S, w.T1, w.ew, st));
    PSVD_TRY_RC(bwd_scales(w, A, dW, dH, nullptr, nullptr, st));
    PSVD_TRY(prepare_operand(A, n, umn, B, m, n, false, 1.f, w.esp(ES_M), split_out(w.Mhi, w.Mlo, ldn, mn, kF16X, w.fine), st));
    PSVD_TRY(prepare_operand(w.T1, n, unn, B, n, n, false, 1.f, nullptr, split_out(w.VThi, w.VTlo, ldn, nn, kF16X, w.fine), st));
    PSVD_TRY(prepare_operand(w.T1, n, unn, B, n, n, true, 1.f, nullptr, split_out(w.Vhi, w.Vlo, ldn, nn, kF16X, w.fine), st));
    const float *EH = w.BV;
    if (dH) {
        dim3 g16x((n + 15) / 16, (n + 15) / 16, B), b16(16, 16);
        sym_split_kernel<<<g16x, b16, 0, st>>>(dH, w.esp(ES_B), w.fine, n, w.dVThi, w.dVTlo, ldn);    // sym(Hbar)
        count_launch(1);
        // T1 = V^T sym(Hbar)  (B operand B[j][k] = Hs[k][j] = Hs[j][k])
        EpiStore e = epi_store_plain(w.T1, n, unn, n, n);
        PSVD_TRY_RC(g16(w.VThi, w.VTlo, n, n, ldn, nn, w.dVThi, w.dVTlo, n, ldn, nn, w, ES_T1, e, st));
        PSVD_TRY(prepare_operand(w.T1, n, unn, B, n, n, false, 1.f, w.esp(ES_B), split_out(w.T1hi, w.T1lo, ldn, nn, kF16X, w.fine), st));
        // E_H = T1 V  (B operand B[j][k] = V[k][j] = V^T[j][k])
        EpiStore e2 = epi_store_plain(w.BV, n, unn, n, n);
        PSVD_TRY_RC(g16(w.T1hi, w.T1lo, n, n, ldn, nn, w.VThi, w.VTlo, n, ldn, nn, w, ES_EH, e2, st));
    } else {
        PSVD_TRY(cudaMemsetAsync(w.BV, 0, sizeof(float) * (size_t)B * n * n, st));
    }
    if (dW) {
        // G = Wbar V (row-major FP32 for the epilogue, and transposed halves for Z)
        PSVD_TRY(prepare_operand(dW, n, umn, B, m, n, false, 1.f, w.esp(ES_G), split_out(w.Wbhi, w.Wblo, ldn, mn, kF16X, w.fine), st));
        EpiHalf e;
        memset(&e, 0, sizeof(e));
        e.rows = m; e.cols = n; e.inv = w.esp(ES_IG); e.fine = w.fine;
        e.out = w.G; e.ld = n; e.bs = umn;
        e.hi_t = w.GThi; e.lo_t = w.GTlo; e.ldht = ldm; e.bsht = nm;
        PSVD_TRY_RC(g16(w.Wbhi, w.Wblo, m, n, ldn, mn, w.VThi, w.VTlo, n, ldn, nn, w, ES_WV, e, st));
    }
    return bwd_tail(w, dW ? w.G : nullptr, EH, nullptr, nullptr, nullptr, (float)eps, eps == 0.0 ? 2 : 0, dA, st);
}


// ------------------------------------------------------------ EVD backward (Theorem 4.3)
// Hbar = V (diag(Sbar) + 1/2 K^T o (P - P^T)) V^T with P = V^T Vbar, K replaced by its
// Tikhonov regularization K_eps (Section 5.2) in modes 0 and 1.  The middle factor E is
// symmetric (K^T and P - P^T are both skew), so V E and (V E) V^T are both TN products
// with V row-major as an operand.
struct EvdBwdWS {
    int B = 0, n = 0;
    long long ldn = 0;
    float *VThi = nullptr, *VTlo = nullptr, *Vhi = nullptr, *Vlo = nullptr;
    float *dVThi = nullptr, *dVTlo = nullptr, *P = nullptr;
    float *Ehi = nullptr, *Elo = nullptr, *Zhi = nullptr, *Zlo = nullptr;
    unsigned *err = nullptr;
    template <class C>
    void carve(C &cv, int B_, int n_) {
        B = B_; n = n_; ldn = pad_ld(n);
        const long long B64 = B, nn = (long long)n * ldn;
        VThi = cv.template take<float>(B64 * nn); VTlo = cv.template take<float>(B64 * nn);
        Vhi = cv.template take<float>(B64 * nn); Vlo = cv.template take<float>(B64 * nn);
        dVThi = cv.template take<float>(B64 * nn); dVTlo = cv.template take<float>(B64 * nn);
        P = cv.template take<float>(B64 * n * n);
        Ehi = cv.template take<float>(B64 * nn); Elo = cv.template take<float>(B64 * nn);
        Zhi = cv.template take<float>(B64 * nn); Zlo = cv.template take<float>(B64 * nn);
        err = cv.template take<unsigned>(4);
    }
};

// E_ij = delta_ij Sbar_i - 1/2 K_ij (P_ij - P_ji)   ((K^T)_ij = K_ji = -K_ij), split TF32.
__global__ void evd_core_kernel(const float *P, const float *S, const float *dS, int n, float eps, int kreg_mode,
                                float tie_tol, float *Ehi, float *Elo, long long ld) {
    const int b = blockIdx.z;
    const int i = blockIdx.y * 16 + threadIdx.y, j = blockIdx.x * 16 + threadIdx.x;
    if (i >= n || j >= n) return;
    const long long bo = (long long)b * n * n;
    const float *s = S + (long long)b * n;
    const float d = s[i] - s[j];
    float kij;
    if (kreg_mode == 0) kij = d / (d * d + sqrtf(eps));
    else if (kreg_mode == 1) kij = d / (d * d + eps * eps);
    else {
        const float smax = fmaxf(fabsf(s[0]), fabsf(s[n - 1]));
        kij = fabsf(d) <= tie_tol * smax ? 0.f : 1.f / d;
    }
    const float pij = P ? P[bo + (long long)i * n + j] : 0.f, pji = P ? P[bo + (long long)j * n + i] : 0.f;
    float e = -0.5f * kij * (pij - pji);
    if (i == j) e = dS ? dS[(long long)b * n + i] : 0.f;
    float h, l;
    split_tf32(e, h, l);
    Ehi[(long long)b * n * ld + (long long)i * ld + j] = h;
    Elo[(long long)b * n * ld + (long long)i * ld + j] = l;
}

int eigh_backward(const float *S, const float *VT, const float *dS, const float *dVT, float *dH, EvdBwdWS &w,
                  double eps, int kreg, cudaStream_t st) {
    const int B = w.B, n = w.n;
    const long long ldn = w.ldn, nn = (long long)n * ldn;
    PSVD_TRY(prepare_operand(VT, n, (long long)n * n, B, n, n, false, 1.f, nullptr, so(w.VThi, w.VTlo, ldn, nn), st));
    PSVD_TRY(prepare_operand(VT, n, (long long)n * n, B, n, n, true, 1.f, nullptr, so(w.Vhi, w.Vlo, ldn, nn), st));
    if (dVT) {
        PSVD_TRY(prepare_operand(dVT, n, (long long)n * n, B, n, n, false, 1.f, nullptr, so(w.dVThi, w.dVTlo, ldn, nn),
                                 st));
        // P = V^T Vbar: P[i][k] = sum_j VT[i][j] dVT[k][j]
        EpiStore e = epi_store_plain(w.P, n, (long long)n * n, n, n);
        PSVD_TRY_RC(g3(w.VThi, w.VTlo, n, n, ldn, nn, w.dVThi, w.dVTlo, n, ldn, nn, B, e, w.err, st));
    }
    dim3 g16((n + 15) / 16, (n + 15) / 16, B), b16(16, 16);
    evd_core_kernel<<<g16, b16, 0, st>>>(dVT ? w.P : nullptr, S, dS, n, kreg == 2 ? 0.f : (float)eps, kreg, 1e-6f,
                                         w.Ehi, w.Elo, ldn);
    count_launch(1);
    PSVD_TRY(cudaGetLastError());
    {   // Z = V E (E symmetric, so the B operand B[k][j] = E[j][k] is E itself)
        EpiStore e;
        memset(&e, 0, sizeof(e));
        e.rows = n; e.cols = n;
        e.hi = w.Zhi; e.lo = w.Zlo; e.ldh = ldn; e.bsh = nn;
        PSVD_TRY_RC(g3(w.Vhi, w.Vlo, n, n, ldn, nn, w.Ehi, w.Elo, n, ldn, nn, B, e, w.err, st));
    }
    {   // Hbar = Z V^T: B operand B[k][j] = V^T[j][k] = V[k][j], V row-major
        EpiStore e = epi_store_plain(dH, n, (long long)n * n, n, n);
        PSVD_TRY_RC(g3(w.Zhi, w.Zlo, n, n, ldn, nn, w.Vhi, w.Vlo, n, ldn, nn, B, e, w.err, st));
    }
    return cudaGetLastError() == cudaSuccess ? PSVD_OK : PSVD_ERR_CUDA;
}

}  // namespace psvd

using namespace psvd;

extern "C" size_t psvd_eigh_bwd_workspace_bytes(int64_t batch, int64_t n) {
    if (batch <= 0 || n <= 0) return 0;
    Sizer s;
    EvdBwdWS w;
    w.carve(s, (int)batch, (int)n);
    return s.used + 256;
}

extern "C" int psvd_eigh_bwd(const float *S, const float *VT, const float *dS, const float *dVT, float *dH,
                             int64_t batch, int64_t n, double eps, int kreg_mode, void *ws, size_t ws_bytes,
                             void *stream) {
    if (!S || !VT || !dH || batch <= 0 || n <= 0 || batch > 65535 || n > 16384 || kreg_mode < 0 || kreg_mode > 2 ||
        !(eps >= 0.0) || (eps == 0.0 && kreg_mode != 2))
        return PSVD_ERR_ARG;
    if (int e = check_device()) return e;
    if (ws_bytes < psvd_eigh_bwd_workspace_bytes(batch, n)) return PSVD_ERR_WORKSPACE;
    Carver cv(ws, ws_bytes);
    EvdBwdWS w;
    w.carve(cv, (int)batch, (int)n);
    if (cv.overflow) return PSVD_ERR_WORKSPACE;
    return eigh_backward(S, VT, dS, dVT, dH, w, eps, kreg_mode, static_cast<cudaStream_t>(stream));
}

extern "C" size_t psvd_svd_bwd_workspace_bytes(int64_t batch, int64_t m, int64_t n) {
    if (batch <= 0 || m <= 0 || n <= 0) return 0;
    Sizer s;
    BwdWS w;
    w.carve(s, (int)batch, (int)m, (int)n, false);
    return s.used + 256;
}

extern "C" size_t psvd_polar_bwd_workspace_bytes(int64_t batch, int64_t m, int64_t n) {
    if (batch <= 0 || m <= 0 || n <= 0) return 0;
    Sizer s;
    BwdWS w;
    w.carve(s, (int)batch, (int)m, (int)n, true);
    return s.used + 256;
}

extern "C" int psvd_svd_bwd(const float *A, const float *U, const float *S, const float *VT, const float *dU,
                            const float *dS, const float *dVT, float *dA, int64_t batch, int64_t m, int64_t n,
                            double eps, int kreg_mode, void *ws, size_t ws_bytes, void *stream) {
    if (!A || !U || !S || !VT || !dA || batch <= 0 || n <= 0 || m < n || batch > 65535 || n > 16384 ||
        kreg_mode < 0 || kreg_mode > 2 || !(eps >= 0.0) || (eps == 0.0 && kreg_mode != 2))
        return PSVD_ERR_ARG;
    if (int e = check_device()) return e;
    if (ws_bytes < psvd_svd_bwd_workspace_bytes(batch, m, n)) return PSVD_ERR_WORKSPACE;
    Carver cv(ws, ws_bytes);
    BwdWS w;
    w.carve(cv, (int)batch, (int)m, (int)n, false);
    if (cv.overflow) return PSVD_ERR_WORKSPACE;
    return svd_backward(A, U, S, VT, dU, dS, dVT, dA, w, eps, kreg_mode, static_cast<cudaStream_t>(stream));
}

extern "C" int psvd_polar_bwd(const float *A, const float *W, const float *H, const float *dW, const float *dH,
                              float *dA, int64_t batch, int64_t m, int64_t n, double eps, void *ws, size_t ws_bytes,
                              void *stream) {
    (void)W;
    if (!A || !H || !dA || batch <= 0 || n <= 0 || m < n || batch > 65535 || n > 16384 || !(eps >= 0.0))
        return PSVD_ERR_ARG;
    if (int e = check_device()) return e;
    if (ws_bytes < psvd_polar_bwd_workspace_bytes(batch, m, n)) return PSVD_ERR_WORKSPACE;
    Carver cv(ws, ws_bytes);
    BwdWS w;
    w.carve(cv, (int)batch, (int)m, (int)n, true);
    if (cv.overflow) return PSVD_ERR_WORKSPACE;
    return polar_backward(A, H, dW, dH, dA, w, eps, static_cast<cudaStream_t>(stream));
}
