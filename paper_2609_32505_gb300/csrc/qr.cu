// Blocked Householder QR (m >= n, diag(R) >= 0) for the QR fallback of Algorithm 1
// (Appendix A.2) and the QR preprocessing of rectangular inputs (Section 4.1).
//
// The matrix is scaled by a power of two to columns of norm <= 1 and kept transposed and split into
// FP16 hi/lo halves (UT: row j = column j).  Panels of nb columns are factored by one thread-block
// cluster per matrix: each of the cl CTAs holds a slab of the panel's rows in shared memory, and the
// per-column dot products (the norm below the diagonal and the projections of the later panel
// columns) are summed across the cluster through distributed shared memory -- one cluster barrier
// per column, where the unblocked kernel needed three grid barriers.
// The reflectors act in compact-WY form on two levels: those of a panel on the rest of its block of
// kWY = 128 columns, H_j0 ... = I - Y T Y^T as W = Y^T X (K split over CTAs), X -= Y (T^T W); those of a
// whole block on everything to its right, as S = X^T Y, S2 = S T, X^T -= S2 Y^T.  The trailing matrix is
// what costs: updated panel by panel (32 columns for 14336 rows) it was read and rewritten four times as
// often and in split TF32, 249 of the 634 ms of 4 x 14336 x 4096 (with 81 ms of Y^T X products).
// Q = H_0 ... H_{n-1} [I; 0] is accumulated backwards block by block with T in place of T^T.  Finally Q and
// R get the signs that make diag(R) >= 0.
#include <cooperative_groups.h>

#include <cmath>
#include <cstring>

#include "qr.cuh"

namespace psvd {

namespace cg = cooperative_groups;

constexpr int kQrThreads = 512;
constexpr size_t kQrSlabMax = 180 * 1024;   // shared memory for one CTA's slab of the panel

// Slab column stride: odd, so that the lanes of a warp (consecutive columns, same row) fall
// in distinct shared-memory banks.
__host__ __device__ inline int qr_slab_stride(int S) { return (S & 1) ? S : S + 1; }

static size_t qr_panel_smem(int m, int nb, int cl) {
    const int S = qr_slab_stride((m + cl - 1) / cl);
    const size_t slab = std::max<size_t>((size_t)S * nb, (size_t)2 * nb * (nb + 1)) * sizeof(float);
    const size_t red = sizeof(float) * (size_t)kQrThreads;
    return sizeof(double) * ((size_t)2 * cl * 2 * nb + 5 * nb) + red + slab;
}

bool qr_shape(int m, int *nb, int *cl) {
    const int nbs[2] = {64, 32}, cls[2] = {8, 16};
    for (int a = 0; a < 2; ++a)
        for (int c = 0; c < 2; ++c) {
            const int S = qr_slab_stride((m + cls[c] - 1) / cls[c]);
            if ((size_t)S * nbs[a] * sizeof(float) <= kQrSlabMax) { *nb = nbs[a]; *cl = cls[c]; return true; }
        }
    return false;
}

struct PanelArgs {
    __half *UThi, *UTlo, *YThi, *YTlo, *Yhi, *Ylo;
    float *tau, *beta, *Tm, *Gpart;
    const int *skip;
    int m, n, j0, pw, panel, npan, nb, cl;
    long long ldm, ldn;
};

// One cluster per matrix factors columns j0 .. j0 + pw - 1 (rows j0 .. m - 1).  CTA q of the
// cluster owns rows [j0 + q S, j0 + (q + 1) S), S = ceil((m - j0) / cl), column-major in
// shared memory.  For column j every CTA contributes, over its rows r > j, the partial sums
// P_c' = sum x_r y_c',r (c' = j: the squared norm below the diagonal) and, from the owner of
// row j, the row-j values; each CTA writes its vector into a slot of every CTA of the cluster,
// and after the barrier every CTA adds the slots in rank order (so all get the same totals,
// bit for bit) and builds the reflector redundantly: beta = -sign(alpha) sqrt(alpha^2 + s2),
// tau = (beta - alpha) / beta, v = [1; x / (alpha - beta)].  Slots are double-buffered by
// column parity, which makes one barrier per column enough.  The slots and their sums are
// FP32, like the partial sums they hold (FP64 sums of the cluster's 8 or 16 partials took
// ~40% of a column's time on the narrow FP64 pipe, measured, and added no accuracy that
// the FP32 partial sums had).
__global__ void __launch_bounds__(kQrThreads, 1) qr_panel_kernel(PanelArgs P) {
    cg::cluster_group cluster = cg::this_cluster();
    const int CL = P.cl, rank = (int)cluster.block_rank();
    const int b = blockIdx.x / CL;
    if (P.skip[b]) return;                       // uniform across the cluster
    extern __shared__ __align__(16) double qsm[];
    const int nb = P.nb, pw = P.pw, j0 = P.j0, m = P.m, n = P.n;
    float *xch = reinterpret_cast<float *>(qsm); // [2][CL][2 nb] slots, double-buffered by column parity
    double *part = qsm + 2 * CL * 2 * nb;        // [2 nb] doubles of room
    float *vec = reinterpret_cast<float *>(part); // [2 nb] this CTA's vector of the column
    float *coef = reinterpret_cast<float *>(part + 4 * nb);   // [nb] f_c' of this column, then [2] scal, beta
    float *scal_s = coef + nb;
    float *red = reinterpret_cast<float *>(part + 5 * nb);    // [kQrThreads] row-block partial sums
    float *slab = red + kQrThreads;                           // [pw][Sp] column-major, Sp odd
    const int S = (m - j0 + CL - 1) / CL;
    const int Sp = qr_slab_stride(S);
    const int r0 = j0 + rank * S;
    const int nr = max(0, min(m, r0 + S) - r0);
    const int tid = threadIdx.x;
    const long long ubase = (long long)b * n * P.ldm;
    // thread -> (column cc, row block rb): the lanes of a warp share rb and hold consecutive columns
    const int nrb = kQrThreads / nb, cc = tid % nb, rb = tid / nb;
    const int rbs = (nr + nrb - 1) / nrb;
    const int rlo = rb * rbs, rhi = min(nr, rlo + rbs);

    for (int c = 0; c < pw; ++c) {
        const __half *hi = P.UThi + ubase + (long long)(j0 + c) * P.ldm + r0;
        const __half *lo = P.UTlo + ubase + (long long)(j0 + c) * P.ldm + r0;
        for (int rr = tid; rr < nr; rr += blockDim.x) slab[c * Sp + rr] = join_f16(hi[rr], lo[rr]) * (1.f / kF16X);
    }
    __syncthreads();

    for (int c = 0; c < pw; ++c) {
        const int j = j0 + c, par = c & 1;
        const int jl = j - r0;
        const bool own = jl >= 0 && jl < nr;
        const int start = max(0, jl + 1);
        const int live = pw - c;                 // entries c .. pw-1 of the vectors are needed
        const float *x = slab + c * Sp;
        // partial dot products of column c with columns cc >= c over rows r > j of this block
        if (cc >= c && cc < pw) {
            const float *y = slab + cc * Sp;
            float a0 = 0.f, a1 = 0.f;
            int rr = max(rlo, start);
            for (; rr + 1 < rhi; rr += 2) {
                a0 = fmaf(x[rr], y[rr], a0);
                a1 = fmaf(x[rr + 1], y[rr + 1], a1);
            }
            if (rr < rhi) a0 = fmaf(x[rr], y[rr], a0);
            red[rb * nb + cc] = a0 + a1;
        }
        // the previous column becomes its reflector (v below the diagonal, beta on it); no
        // thread reads it in this phase (the dot products above start at column c)
        if (c > 0) {
            const int jlp = j - 1 - r0;
            float *xp = slab + (c - 1) * Sp;
            const float fsp = scal_s[0];
            for (int rr = max(0, jlp + 1) + tid; rr < nr; rr += blockDim.x) xp[rr] *= fsp;
            if (jlp >= 0 && jlp < nr && tid == 0) xp[jlp] = scal_s[1];
        }
        __syncthreads();
        // this CTA's vector (sum over the row blocks; the row-j values from its owner), formed
        // once in shared memory, then copied into a slot of every CTA of the cluster
        for (int k = tid; k < 2 * live; k += blockDim.x) {
            if (k < live) {
                const int e = c + k;
                float sum = 0.f;
                for (int q = 0; q < nrb; ++q) sum += red[q * nb + e];
                vec[e] = sum;
            } else {
                const int e = nb + c + (k - live);
                vec[e] = own ? slab[(e - nb) * Sp + jl] : 0.f;
            }
        }
        __syncthreads();
        // the row-j values are nonzero only in the CTA that owns row j: only it sends them,
        // and the readers take them from its slot
        const int nsend = own ? 2 * live : live;
        for (int t = tid; t < CL * nsend; t += blockDim.x) {
            const int peer = t / nsend, k = t - peer * nsend;
            const int e = k < live ? c + k : nb + c + (k - live);
            float *dst = cluster.map_shared_rank(xch + ((long long)par * CL + rank) * 2 * nb, peer);
            dst[e] = vec[e];
        }
        cluster.sync();
        // warp 0: the cluster totals, the reflector (FP32, as single-precision Householder QR
        // computes it) and the coefficient f_c' = tau (v^T y_c') = tau (y_c',j + scal P_c')
        if (tid < 32) {
            const int lane = tid;
            const float *slots = xch + (long long)par * CL * 2 * nb;
            const float *oslot = slots + (long long)((j - j0) / S) * 2 * nb;   // the owner of row j
            float s2 = 0.f;
            for (int q = 0; q < CL; ++q) s2 += slots[q * 2 * nb + c];
            const float alpha = oslot[nb + c];
            const float fa = alpha, f2 = s2;
            float beta, tau, scal;
            if (f2 == 0.f) { beta = fa; tau = 0.f; scal = 0.f; }
            else {
                beta = -copysignf(sqrtf(fmaf(fa, fa, f2)), fa);
                tau = (beta - fa) / beta;
                scal = 1.f / (fa - beta);
            }
            for (int k = c + 1 + lane; k < pw; k += 32) {
                float pc = 0.f;
                for (int q = 0; q < CL; ++q) pc += slots[q * 2 * nb + k];
                coef[k] = tau * (oslot[nb + k] + pc * scal);
            }
            if (lane == 0) {
                scal_s[0] = scal;
                scal_s[1] = beta;
                if (rank == 0) {
                    P.tau[(long long)b * n + j] = tau;
                    P.beta[(long long)b * n + j] = beta;
                }
            }
        }
        __syncthreads();
        // y -= f_c' v for the later panel columns, v = [1; x * scal]
        if (cc > c && cc < pw) {
            float *y = slab + cc * Sp;
            const float f = coef[cc] * scal_s[0];
            for (int rr = max(rlo, start); rr < rhi; ++rr) y[rr] = fmaf(-f, x[rr], y[rr]);
            if (own && jl >= rlo && jl < rhi) y[jl] -= coef[cc];
        }
        __syncthreads();
    }
    if (pw > 0) {                                // the last column's reflector
        const int jlp = j0 + pw - 1 - r0;
        float *xp = slab + (pw - 1) * Sp;
        const float fsp = scal_s[0];
        for (int rr = max(0, jlp + 1) + tid; rr < nr; rr += blockDim.x) xp[rr] *= fsp;
        if (jlp >= 0 && jlp < nr && tid == 0) xp[jlp] = scal_s[1];
        __syncthreads();
    }

    // the factored panel back to UT (R entries above the diagonal, beta on it, v below);
    // the reflectors also as clean rows (YT: 0 above, 1 on the diagonal) and columns (Y)
    for (int c = 0; c < pw; ++c) {
        const int j = j0 + c;
        const long long o = ubase + (long long)j * P.ldm + r0;
        for (int rr = tid; rr < nr; rr += blockDim.x) {
            const int r = r0 + rr;
            const float v = slab[c * Sp + rr];
            __half h, l;
            split_f16(v * kF16X, h, l);
            P.UThi[o + rr] = h;
            P.UTlo[o + rr] = l;
            split_f16((r < j ? 0.f : (r == j ? 1.f : v)) * kF16V, h, l);
            P.YThi[o + rr] = h;
            P.YTlo[o + rr] = l;
        }
    }
    const long long ybase = (long long)b * m * P.ldn;
    for (int t = tid; t < nr * pw; t += blockDim.x) {
        const int rr = t / pw, c = t - rr * pw;
        const int r = r0 + rr, j = j0 + c;
        const float v = slab[c * Sp + rr];
        __half h, l;
        split_f16((r < j ? 0.f : (r == j ? 1.f : v)) * kF16V, h, l);
        P.Yhi[ybase + (long long)r * P.ldn + j] = h;
        P.Ylo[ybase + (long long)r * P.ldn + j] = l;
    }
    // zeros above the panel's first row, down from the first row of its block (the block's products read them)
    const int s0 = j0 - j0 % kWY;
    if (rank == CL - 1)
        for (int t = tid; t < (j0 - s0) * pw; t += blockDim.x) {
            const int rr = t / pw, c = t - rr * pw;
            const __half z = __float2half_rn(0.f);
            P.Yhi[ybase + (long long)(s0 + rr) * P.ldn + j0 + c] = z;
            P.Ylo[ybase + (long long)(s0 + rr) * P.ldn + j0 + c] = z;
            const long long o = ubase + (long long)(j0 + c) * P.ldm + s0 + rr;
            P.YThi[o] = z;
            P.YTlo[o] = z;
        }
    // partial G = Y^T Y over this CTA's rows (upper triangle), summed by CTA 0 into T
    float *gp = P.Gpart + ((long long)b * CL + rank) * nb * nb;
    for (int t = tid; t < pw * pw; t += blockDim.x) {
        const int i = t / pw, k = t - i * pw;
        if (k < i) continue;
        const int ji = j0 + i, jk = j0 + k;
        float acc = 0.f;
        for (int rr = max(0, jk - r0); rr < nr; ++rr) {      // Y_r,k = 0 above its diagonal (jk >= ji)
            const int r = r0 + rr;
            const float yi = r == ji ? 1.f : slab[i * Sp + rr];
            const float yk = r == jk ? 1.f : slab[k * Sp + rr];
            acc = fmaf(yi, yk, acc);
        }
        gp[i * nb + k] = acc;
    }
    __threadfence();
    cluster.sync();
    if (rank != 0) return;
    const int ldt = nb + 1;                          // padded rows: conflict-free column access
    float *G = slab, *T = slab + nb * ldt;           // the slab is no longer needed
    __syncthreads();
    for (int t = tid; t < pw * pw; t += blockDim.x) {
        const int i = t / pw, k = t - i * pw;
        float s = 0.f;
        if (k >= i)
            for (int q = 0; q < CL; ++q) s += P.Gpart[((long long)b * CL + q) * nb * nb + i * nb + k];
        G[i * ldt + k] = s;
        T[i * ldt + k] = 0.f;
    }
    __syncthreads();
    // T[c][c] = tau_c, T[:c, c] = -tau_c T[:c, :c] G[:c, c]  (G upper triangle)
    const float *tb = P.tau + (long long)b * n + j0;
    if (tid == 0) T[0] = tb[0];
    __syncthreads();
    for (int c = 1; c < pw; ++c) {
        float v = 0.f;
        if (tid < c)
            for (int l = tid; l < c; ++l) v += T[tid * ldt + l] * G[l * ldt + c];
        __syncthreads();
        if (tid < c) T[tid * ldt + c] = -tb[c] * v;
        if (tid == 0) T[c * ldt + c] = tb[c];
        __syncthreads();
    }
    float *out = P.Tm + ((long long)b * P.npan + P.panel) * nb * nb;
    for (int t = tid; t < nb * nb; t += blockDim.x) out[t] = t / nb < pw && t % nb < pw ? T[(t / nb) * ldt + t % nb] : 0.f;
}

// W2^T[c][i] = sum_l T^T[i][l] W[l][c], W = sum of the ks K-split slices of Y^T X, for the ncol <= 96
// columns that a panel still has to its right in its block.  Tm holds the nb x nb T of every (matrix,
// panel).  One block of 8 warps per kTaCols columns: the block's columns of W (slices summed) are
// staged in shared memory with coalesced loads, warp g forms outputs i = g, g + 8, ... of every
// column (lane = column); rows of W2^T have stride kWY.
constexpr int kTaCols = 32, kTaWarps = 8;
__global__ void __launch_bounds__(32 * kTaWarps) qr_tapply_kernel(const float *Wp, int ks, int B, int nb, int pw,
                                                                  int n, int ldw, int ncol, const float *Tm, int npan,
                                                                  int panel, const int *skip, __half *W2hi,
                                                                  __half *W2lo) {
    __shared__ float Ts[64 * 65];                   // T^T, rows padded
    __shared__ float ws[64][kTaCols + 1];           // W[l][c] for the block's columns
    const int b = blockIdx.y;
    if (skip[b]) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * kTaCols + lane;
    const float *T = Tm + ((long long)b * npan + panel) * nb * nb;
    for (int t = threadIdx.x; t < pw * pw; t += blockDim.x) {
        const int i = t / pw, l = t - i * pw;
        Ts[i * 65 + l] = T[l * nb + i];
    }
    for (int l = warp; l < pw; l += kTaWarps) {
        float sum = 0.f;
        if (c < ncol)
            for (int kc = 0; kc < ks; ++kc) sum += Wp[(((long long)kc * B + b) * nb + l) * ldw + c];
        ws[l][lane] = sum;
    }
    __syncthreads();
    for (int i = warp; i < pw; i += kTaWarps) {
        float sum = 0.f;
        for (int l = 0; l < pw; ++l) sum += Ts[i * 65 + l] * ws[l][lane];
        if (c >= ncol) continue;
        __half h, lo;
        split_f16(sum * kF16S2, h, lo);
        const long long o = ((long long)b * n + c) * kWY + i;
        W2hi[o] = h;
        W2lo[o] = lo;
    }
}

// S2 = S T (trans = 0) or S T^T (trans = 1) of a block of kWY columns, S (ncol x kWY) the sum of ks K-split
// slices in slice order, S2 split into FP16 halves.  One block of 2 kWY threads per kQsRows rows: op(T)^T
// staged with rows padded to kQsLd floats (thread j of a half reads row j as float4), the rows of S
// as float4 broadcasts.  T is zero outside its triangle and past the block's width.
constexpr int kQsRows = 32, kQsLd = kWY + 4;
constexpr size_t kQsSmem = sizeof(float) * ((size_t)kWY * kQsLd + (size_t)kQsRows * kWY);
__global__ void __launch_bounds__(2 * kWY) qr_stapply_kernel(const float *Sp, int ks, int B, int n, int ncol, int ws,
                                                             const float *Ts, int nsup, int sup, int trans,
                                                             const int *skip, __half *W2hi, __half *W2lo) {
    extern __shared__ __align__(16) float qsm2[];
    float *Ms = qsm2, *sr = qsm2 + kWY * kQsLd;
    const int b = blockIdx.y, t = threadIdx.x, i0 = blockIdx.x * kQsRows;
    if (skip[b]) return;
    const float *T = Ts + ((long long)b * nsup + sup) * kWY * kWY;
    for (int e = t; e < kWY * kWY; e += 2 * kWY) {
        const int r = e / kWY, c = e % kWY;
        if (trans) Ms[r * kQsLd + c] = T[e];        // column j of T^T = row j of T
        else Ms[c * kQsLd + r] = T[e];
    }
    const long long slice = (long long)B * n * kWY;
    for (int e = t; e < kQsRows * kWY; e += 2 * kWY) {
        const int i = i0 + e / kWY, c = e % kWY;
        float sum = 0.f;
        if (i < ncol && c < ws) {
            const float *q = Sp + ((long long)b * n + i) * kWY + c;
            for (int k = 0; k < ks; ++k) sum += q[k * slice];
        }
        sr[e] = sum;
    }
    __syncthreads();
    constexpr int kH = kQsRows / 2;
    const int j = t % kWY, rh = (t / kWY) * kH;
    float acc[kH];
#pragma unroll
    for (int r = 0; r < kH; ++r) acc[r] = 0.f;
    for (int l = 0; l < kWY; l += 4) {
        const float4 m = *reinterpret_cast<const float4 *>(Ms + j * kQsLd + l);
#pragma unroll
        for (int r = 0; r < kH; ++r) {
            const float4 x = *reinterpret_cast<const float4 *>(sr + (rh + r) * kWY + l);
            acc[r] += x.x * m.x + x.y * m.y + x.z * m.z + x.w * m.w;
        }
    }
#pragma unroll
    for (int r = 0; r < kH; ++r) {
        const int i = i0 + rh + r;
        if (i >= ncol) break;
        __half h, lo;
        split_f16(acc[r] * kF16S2, h, lo);
        const long long o = ((long long)b * n + i) * kWY + j;
        W2hi[o] = h;
        W2lo[o] = lo;
    }
}

// max |A| of every factored matrix (float bits; a NaN compares above every finite value)
__global__ void qr_absmax_kernel(const float *A, long long mn, const int *skip, unsigned *amax) {
    __shared__ unsigned red[8];
    const int b = blockIdx.y;
    if (skip[b]) return;
    const float *a = A + b * mn;
    unsigned v = 0;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < mn; t += (long long)gridDim.x * blockDim.x)
        v = max(v, __float_as_uint(fabsf(a[t])));
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) v = max(v, red[w]);
        atomicMax(&amax[b], v);
    }
}
// 2^e >= sqrt(m) max |A| >= every column norm (1 where there is none: a zero or non-finite matrix)
__global__ void qr_scale_kernel(const unsigned *amax, int B, int m, float *scale) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const float v = __uint_as_float(amax[b]);
    const bool ok = v > 0.f && v < INFINITY;
    scale[b] = ok ? ldexpf(1.f, min(127, max(-100, ilogb((double)v * sqrt((double)m)) + 1))) : 1.f;
}

__global__ void qr_skip_kernel(const int *flag, int B, int *skip) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) skip[b] = flag ? (flag[b] ? 0 : 1) : 0;
}

// Q^T = [I 0] (split: hi = identity, lo = 0) for the factored matrices
__global__ void qr_qinit_kernel(int n, int m, long long ldm, const int *skip, __half *QThi, __half *QTlo) {
    const int b = blockIdx.z;
    if (skip[b]) return;
    const int c = blockIdx.y, r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= m) return;
    const long long o = ((long long)b * n + c) * ldm + r;
    QThi[o] = __float2half_rn(r == c ? kF16X : 0.f);
    QTlo[o] = __float2half_rn(0.f);
}

// Q[r][c] = sign(beta_c) Q^T[c][r] (transposed through a shared tile) and, if R is given,
// R[r][c] = 2^e sign(beta_r) (r < c ? UT[c][r] : r == c ? beta_c : 0).
__global__ void qr_store_kernel(const __half *QThi, const __half *QTlo, const __half *UThi, const __half *UTlo,
                                const float *beta, const float *scale, int m, int n, long long ldm, const int *skip,
                                float *Q, float *R) {
    __shared__ float tile[32][33];
    const int b = blockIdx.z;
    if (skip[b]) return;
    const int c0 = blockIdx.y * 32, r0 = blockIdx.x * 32;   // c: column of Q (row of Q^T)
    const float *bb = beta + (long long)b * n;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int c = c0 + i, r = r0 + threadIdx.x;
        float v = 0.f;
        if (c < n && r < m) {
            const long long o = ((long long)b * n + c) * ldm + r;
            v = (bb[c] < 0.f ? -1.f : 1.f) * (join_f16(QThi[o], QTlo[o]) * (1.f / kF16X));
        }
        tile[i][threadIdx.x] = v;
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int r = r0 + i, c = c0 + threadIdx.x;
        if (r < m && c < n) Q[((long long)b * m + r) * n + c] = tile[threadIdx.x][i];
    }
    if (!R) return;
    // R rows r < n: reads UT[c][r] (row c of UT, coalesced over r = threadIdx.x), same tile shape
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int c = c0 + i, r = r0 + threadIdx.x;
        float v = 0.f;
        if (c < n && r < n) {
            const long long o = ((long long)b * n + c) * ldm + r;
            v = r < c ? join_f16(UThi[o], UTlo[o]) * (1.f / kF16X) : (r == c ? fabsf(bb[c]) : 0.f);
            if (r < c && bb[r] < 0.f) v = -v;
            v *= scale[b];
        }
        tile[i][threadIdx.x] = v;
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int r = r0 + i, c = c0 + threadIdx.x;
        if (r < n && c < n) R[((long long)b * n + r) * n + c] = tile[threadIdx.x][i];
    }
}

// X^T[c][j0 + r] -= sum_i W2^T[c][i] Y[j0 + r][j0 + i] for rows c0 .. c0 + ncol - 1 of X^T and the pw reflectors
// from j0 on, W2^T in w.W2hi / w.W2lo.
static int qr_update(QrWS &w, int j0, int pw, int c0, int ncol, __half *Xhi, __half *Xlo, cudaStream_t st) {
    const int B = w.B, m = w.m, n = w.n, K = m - j0;
    F16Views f;
    f.ah = view_f16(w.W2hi, ncol, pw, kWY, (long long)n * kWY, B);
    f.al = view_f16(w.W2lo, ncol, pw, kWY, (long long)n * kWY, B);
    f.bh = view_f16(w.Yhi + (long long)j0 * w.ldn + j0, K, pw, w.ldn, (long long)m * w.ldn, B);
    f.bl = view_f16(w.Ylo + (long long)j0 * w.ldn + j0, K, pw, w.ldn, (long long)m * w.ldn, B);
    GemmShape s;
    memset(&s, 0, sizeof(s));
    s.M = ncol; s.N = K; s.K = pw; s.prec_uniform = PREC_F16X3; s.skip = w.skip; s.err = w.err;
    s.f16_scale = 1.f / (kF16S2 * kF16V);
    EpiSubHalf e;
    e.rows = ncol; e.cols = K; e.hi = Xhi + (long long)c0 * w.ldm + j0; e.lo = Xlo + (long long)c0 * w.ldm + j0;
    e.ld = w.ldm; e.bs = (long long)n * w.ldm; e.scale = kF16X; e.inv = 1.f / kF16X;
    PSVD_TRY(launch_gemm(nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, s, B, e, st, &f));
    return PSVD_OK;
}

// The reflectors of one panel on the ncol columns from c0 on, the rest of its block.
static int qr_apply_panel(QrWS &w, int j0, int pw, int panel, int c0, int ncol, cudaStream_t st) {
    const int B = w.B, m = w.m, n = w.n, nb = w.nb, ldw = std::min(n, kWY);
    const int K = m - j0;
    const long long nm = (long long)n * w.ldm;
    // W = Y^T X: A = Y^T rows of the panel (pw x K), B = X^T rows (ncol x K), split over K
    F16Views f;
    f.ah = view_f16(w.YThi + (long long)j0 * w.ldm + j0, pw, K, w.ldm, nm, B);
    f.al = view_f16(w.YTlo + (long long)j0 * w.ldm + j0, pw, K, w.ldm, nm, B);
    f.bh = view_f16(w.UThi + (long long)c0 * w.ldm + j0, ncol, K, w.ldm, nm, B);
    f.bl = view_f16(w.UTlo + (long long)c0 * w.ldm + j0, ncol, K, w.ldm, nm, B);
    GemmShape s;
    memset(&s, 0, sizeof(s));
    s.M = pw; s.N = ncol; s.K = K; s.prec_uniform = PREC_F16X3; s.skip = w.skip; s.err = w.err;
    s.f16_scale = 1.f / (kF16V * kF16X);
    s.ksplit = std::max(1, std::min(std::min(w.ks, (num_sms() + B - 1) / B), (K + 127) / 128));
    EpiStore e = epi_store_plain(w.Wp, ldw, (long long)nb * ldw, pw, ncol);
    PSVD_TRY(launch_gemm(nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, s, B, e, st, &f));
    qr_tapply_kernel<<<dim3((ncol + kTaCols - 1) / kTaCols, B), 32 * kTaWarps, 0, st>>>(
        w.Wp, s.ksplit, B, nb, pw, n, ldw, ncol, w.Tm, w.npan, panel, w.skip, w.W2hi, w.W2lo);
    count_launch(1);
    PSVD_TRY(cudaGetLastError());
    return qr_update(w, j0, pw, c0, ncol, w.UThi, w.UTlo, st);
}

// T of the block of ws <= kWY columns from j0 on.
static int qr_block_t(QrWS &w, int j0, int ws, int sup, cudaStream_t st) {
    const int B = w.B, K = w.m - j0;
    const long long nm = (long long)w.n * w.ldm, ts = (long long)w.nsup * kWY * kWY;
    F16Views f;
    f.ah = f.bh = view_f16(w.YThi + (long long)j0 * w.ldm + j0, ws, K, w.ldm, nm, B);
    f.al = f.bl = view_f16(w.YTlo + (long long)j0 * w.ldm + j0, ws, K, w.ldm, nm, B);
    GemmShape s;
    memset(&s, 0, sizeof(s));
    s.M = ws; s.N = ws; s.K = K; s.prec_uniform = PREC_F16X3; s.skip = w.skip; s.err = w.err;
    s.f16_scale = 1.f / (kF16V * kF16V);
    EpiStore e = epi_store_plain(w.Gs + (long long)sup * kWY * kWY, kWY, ts, ws, ws);
    PSVD_TRY(launch_gemm(nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, s, B, e, st, &f));
    return larft_blocks(w.Gs, w.tau, w.n, w.n, w.nsup, sup, 1, B, w.Ts, st);
}

// The reflectors of a whole block on rows c0 .. c0 + ncol - 1 of X^T: trans = 0 in the factorization
// (X <- (I - Y T Y^T)^T X), 1 in the accumulation of Q (X <- (I - Y T Y^T) X).
static int qr_apply_block(QrWS &w, int j0, int ws, int sup, int c0, int ncol, __half *Xhi, __half *Xlo, int trans,
                          cudaStream_t st) {
    const int B = w.B, n = w.n, K = w.m - j0;
    const long long nm = (long long)n * w.ldm;
    F16Views f;
    f.ah = view_f16(Xhi + (long long)c0 * w.ldm + j0, ncol, K, w.ldm, nm, B);
    f.al = view_f16(Xlo + (long long)c0 * w.ldm + j0, ncol, K, w.ldm, nm, B);
    f.bh = view_f16(w.YThi + (long long)j0 * w.ldm + j0, ws, K, w.ldm, nm, B);
    f.bl = view_f16(w.YTlo + (long long)j0 * w.ldm + j0, ws, K, w.ldm, nm, B);
    GemmShape s;
    memset(&s, 0, sizeof(s));
    s.M = ncol; s.N = ws; s.K = K; s.prec_uniform = PREC_F16X3; s.skip = w.skip; s.err = w.err;
    s.f16_scale = 1.f / (kF16X * kF16V);
    const int tiles = ((ncol + kBM - 1) / kBM) * B;
    s.ksplit = std::max(1, std::min(std::min(kQrSplit, (num_sms() + tiles - 1) / tiles), (K + 255) / 256));
    EpiStore e = epi_store_plain(w.Sp, kWY, (long long)n * kWY, ncol, ws);
    PSVD_TRY(launch_gemm(nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, s, B, e, st, &f));
    PSVD_TRY(cudaFuncSetAttribute(qr_stapply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQsSmem));
    qr_stapply_kernel<<<dim3((ncol + kQsRows - 1) / kQsRows, B), 2 * kWY, kQsSmem, st>>>(
        w.Sp, s.ksplit, B, n, ncol, ws, w.Ts, w.nsup, sup, trans, w.skip, w.W2hi, w.W2lo);
    count_launch(1);
    PSVD_TRY(cudaGetLastError());
    return qr_update(w, j0, ws, c0, ncol, Xhi, Xlo, st);
}

int qr_factor(const float *A, float *Q, float *R, const int *flag, QrWS &w, cudaStream_t st) {
    const int B = w.B, m = w.m, n = w.n, nb = w.nb, CL = w.cl;
    const long long nm = (long long)n * w.ldm;
    qr_skip_kernel<<<(B + 127) / 128, 128, 0, st>>>(flag, B, w.skip);
    PSVD_TRY(cudaMemsetAsync(w.amax, 0, sizeof(unsigned) * (size_t)B, st));
    const long long mn = (long long)m * n;
    qr_absmax_kernel<<<dim3((unsigned)std::min<long long>((mn + 2047) / 2048, 8 * num_sms()), B), 256, 0, st>>>(
        A, mn, w.skip, w.amax);
    qr_scale_kernel<<<(B + 127) / 128, 128, 0, st>>>(w.amax, B, m, w.scale);
    count_launch(3);
    {
        SplitOut t;
        t.fhi = w.UThi; t.flo = w.UTlo; t.ld = w.ldm; t.bstride = t.fbstride = nm; t.fscale = kF16X;
        PSVD_TRY(prepare_operand(A, n, mn, B, m, n, true, 1.f, w.scale, t, st, w.skip));
    }
    const size_t smem = qr_panel_smem(m, nb, CL);
    PSVD_TRY(cudaFuncSetAttribute(qr_panel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (CL > 8) PSVD_TRY(cudaFuncSetAttribute(qr_panel_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(B * CL));
    cfg.blockDim = dim3(kQrThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    for (int sp = 0; sp < w.nsup; ++sp) {
        const int s0 = sp * kWY, s1 = std::min(n, s0 + kWY);
        for (int j0 = s0; j0 < s1; j0 += nb) {
            const int pw = std::min(nb, s1 - j0), p = j0 / nb;
            PanelArgs a;
            a.UThi = w.UThi; a.UTlo = w.UTlo; a.YThi = w.YThi; a.YTlo = w.YTlo; a.Yhi = w.Yhi; a.Ylo = w.Ylo;
            a.tau = w.tau; a.beta = w.beta; a.Tm = w.Tm; a.Gpart = w.Gpart; a.skip = w.skip;
            a.m = m; a.n = n; a.j0 = j0; a.pw = pw; a.panel = p; a.npan = w.npan; a.nb = nb; a.cl = CL;
            a.ldm = w.ldm; a.ldn = w.ldn;
            PSVD_TRY(cudaLaunchKernelEx(&cfg, qr_panel_kernel, a));
            count_launch(1);
            if (j0 + pw < s1) PSVD_TRY_RC(qr_apply_panel(w, j0, pw, p, j0 + pw, s1 - j0 - pw, st));
        }
        PSVD_TRY_RC(qr_block_t(w, s0, s1 - s0, sp, st));
        if (s1 < n) PSVD_TRY_RC(qr_apply_block(w, s0, s1 - s0, sp, s1, n - s1, w.UThi, w.UTlo, 0, st));
    }
    {
        dim3 g((m + 127) / 128, n, B);
        qr_qinit_kernel<<<g, 128, 0, st>>>(n, m, w.ldm, w.skip, w.QThi, w.QTlo);
        count_launch(1);
        PSVD_TRY(cudaGetLastError());
    }
    for (int sp = w.nsup - 1; sp >= 0; --sp) {
        const int s0 = sp * kWY, s1 = std::min(n, s0 + kWY);
        PSVD_TRY_RC(qr_apply_block(w, s0, s1 - s0, sp, s0, n - s0, w.QThi, w.QTlo, 1, st));
    }
    {
        dim3 g((m + 31) / 32, (n + 31) / 32, B), blk(32, 8);
        qr_store_kernel<<<g, blk, 0, st>>>(w.QThi, w.QTlo, w.UThi, w.UTlo, w.beta, w.scale, m, n, w.ldm, w.skip, Q, R);
        count_launch(1);
        PSVD_TRY(cudaGetLastError());
    }
    return PSVD_OK;
}

}  // namespace psvd

using namespace psvd;

extern "C" size_t psvd_qr_workspace_bytes(int64_t batch, int64_t m, int64_t n) {
    if (batch <= 0 || m <= 0 || n <= 0) return 0;
    Sizer s;
    QrWS w;
    w.carve(s, (int)batch, (int)m, (int)n);
    return s.used + 256;
}

extern "C" int psvd_qr(const float *A, float *Q, float *R, int64_t batch, int64_t m, int64_t n, void *ws,
                       size_t ws_bytes, void *stream) {
    int nb = 0, cl = 0;
    if (!A || !Q || batch <= 0 || n <= 0 || m < n || batch > 65535 || n > 16384 || (long long)m * n > (1LL << 31))
        return PSVD_ERR_ARG;
    if (!qr_shape((int)m, &nb, &cl))
        return fail_msg(PSVD_ERR_ARG, "psvd_qr: m = %lld rows exceed the cluster panel", (long long)m);
    if (int e = check_device()) return e;
    if (ws_bytes < psvd_qr_workspace_bytes(batch, m, n)) return PSVD_ERR_WORKSPACE;
    Carver cv(ws, ws_bytes);
    QrWS w;
    w.carve(cv, (int)batch, (int)m, (int)n);
    if (cv.overflow) return PSVD_ERR_WORKSPACE;
    return qr_factor(A, Q, R, nullptr, w, static_cast<cudaStream_t>(stream));
}
