// Blocked Householder QR (m >= n, diag(R) >= 0) for the QR fallback of Algorithm 1
// (Appendix A.2) and the QR preprocessing of rectangular inputs (Section 4.1).
//
// Every column is scaled by its own power of two to a norm <= 1 (A D = Q (R D), exactly, so the scales only come
// back on R's columns, and a small column beside large ones keeps its accuracy) and the matrix kept transposed
// and split into FP16 hi/lo halves (UT: row j = column j), or, with rows of very small size, into split TF32.  Panels of nb columns are factored by one thread-block
// cluster per matrix: each of its CTAs holds a slab of the panel's rows in registers, and the
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

constexpr int kQrWarps = 16, kQrThreads = 32 * kQrWarps;
constexpr int kQrMaxCl = 16;
constexpr int kQrRows8 = 2048;            // panels of 64 columns up to here: 256 rows per CTA

// Panels are 64 columns wide as far as 16 CTAs hold 512 of their rows each in registers, and 32 above (1536 rows each).
// kQrMaxRows is the interface's limit (psvd.h), within that.
constexpr int kQrRows64 = kQrMaxCl * 512, kQrRows32 = kQrMaxCl * 1536;
static_assert(kQrMaxRows <= kQrRows32, "panel registers");
bool qr_shape(int m, int *nb) {
    *nb = m <= kQrRows64 ? 64 : 32;
    return m <= kQrMaxRows;
}

// four consecutive elements of a split array
PSVD_DEV void split_load4(bool wide, const float *hi, const float *lo, long long bo, long long o, float inv, float (&x)[4]) {
    if (wide) {
        const float4 h = *reinterpret_cast<const float4 *>(hi + bo + o), l = *reinterpret_cast<const float4 *>(lo + bo + o);
        x[0] = h.x + l.x; x[1] = h.y + l.y; x[2] = h.z + l.z; x[3] = h.w + l.w;
    } else {
        __align__(8) __half h[4], l[4];
        *reinterpret_cast<uint2 *>(h) = *reinterpret_cast<const uint2 *>(as_half(hi) + 2 * bo + o);
        *reinterpret_cast<uint2 *>(l) = *reinterpret_cast<const uint2 *>(as_half(lo) + 2 * bo + o);
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = join_f16(h[e], l[e]) * inv;
    }
}
PSVD_DEV void split_store4(bool wide, float *hi, float *lo, long long bo, long long o, const float (&x)[4], float fs) {
    if (wide) {
        float h[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) split_tf32(x[e], h[e], l[e]);
        *reinterpret_cast<float4 *>(hi + bo + o) = make_float4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<float4 *>(lo + bo + o) = make_float4(l[0], l[1], l[2], l[3]);
    } else {
        __align__(8) __half h[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) split_f16(x[e] * fs, h[e], l[e]);
        *reinterpret_cast<uint2 *>(as_half(hi) + 2 * bo + o) = *reinterpret_cast<const uint2 *>(h);
        *reinterpret_cast<uint2 *>(as_half(lo) + 2 * bo + o) = *reinterpret_cast<const uint2 *>(l);
    }
}

struct PanelArgs {
    float *UThi, *UTlo, *YThi, *YTlo, *Yhi, *Ylo;    // (split arrays, formats by fine)
    float *tau, *beta, *Tm;
    const int *skip, *fine;
    int m, n, j0, pw, panel, npan, cl;
    long long ldm, ldn;
};

// Shared memory of the panel kernel: NB columns of S = 32 RPL rows per CTA.
template <int RPL, int C>
struct PanelSmem {
    static constexpr int S = 32 * RPL, NB = kQrWarps * C;
    static constexpr int kSlot = NB + 4;              // a slot's stride: spreads the CTAs' slots over the banks
    alignas(16) float x[2][S];                        // column c, rows above and at the diagonal zeroed
    float slot[2][kQrMaxCl][kSlot];                   // every CTA's partial sums of the column
    float row[2][kSlot];                              // the row-j entries, from CTA 0
    float G[NB][NB + 1];                              // Y^T Y above its diagonal
    float tau[NB];
    float slab[NB][S + 1];                            // the factored panel, for the outputs
};

// One cluster of cl CTAs per matrix factors columns j0 .. j0 + pw - 1 (rows j0 .. m - 1).  CTA q owns rows
// [j0 + q S, j0 + (q + 1) S), in registers: lane l of warp w holds rows 4 l + 128 i + (0..3) of columns
// w, w + 16, ..., so a column's update and its dot products touch nothing but registers and the one
// column x = column c that its warp has put into shared memory.  For column c every warp forms, over
// its rows r > j, the sums P_k = sum x_r a_r,k of its C columns (of column c itself: the squared norm below the
// diagonal; of the finished ones: what Y^T Y needs) and writes them into a slot of every CTA of the
// cluster, CTA 0, which holds all diagonal rows, also the row-j entries a_j,k; after the cluster's barrier
// every warp adds the slots of its columns (the same order everywhere, so all get the same totals bit
// for bit) and builds the reflector redundantly: beta = -sign(alpha) sqrt(alpha^2 + s2), tau = (beta -
// alpha) / beta, v = [1; x / (alpha - beta)].  With g_k = a_j,k + scal P_k a later column takes
// -= tau g_k v, and g_k of an earlier one is (Y^T Y)_kc.  The warp of column c + 1 then writes it out.  Slots
// and columns are double-buffered by column parity, which makes one cluster barrier and one block
// barrier per column enough.
//
// A panel is a chain of pw such columns, so its time is latency: with the panel in shared memory (5 block
// barriers per column, every multiply-add fed from shared memory, the Gram matrix and T formed
// afterwards) a column took 2.9 us at 256 rows, 6.2 at 4096 (8 matrices) and 7.4 at 14336 (4 matrices); it
// takes 1.4, 2.7 and 3.2 us, everything included.
template <int RPL, int C>
__global__ void __launch_bounds__(kQrThreads, 1) qr_panel_kernel(PanelArgs P) {
    using Sm = PanelSmem<RPL, C>;
    constexpr int S = Sm::S, NB = Sm::NB, Q = RPL / 4;
    constexpr bool kKeepX = RPL <= 16;               // x stays in registers between its two uses
    cg::cluster_group cluster = cg::this_cluster();
    const int CL = P.cl, rank = CL > 1 ? (int)cluster.block_rank() : 0;
    const int b = blockIdx.x / CL;
    if (P.skip[b]) return;                       // uniform across the cluster
    extern __shared__ __align__(16) unsigned char qsm[];
    Sm &sm = *reinterpret_cast<Sm *>(qsm);
    const int pw = P.pw, j0 = P.j0, m = P.m, n = P.n;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int r0 = j0 + rank * S;                    // multiple of 4
    const long long ubase = (long long)b * n * P.ldm;
    const bool wide = P.fine[b] == PREC_TF32X3;

    float a[C][RPL];
#pragma unroll
    for (int k = 0; k < C; ++k)
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int c = k * kQrWarps + w, r = r0 + 128 * i + 4 * lane;
            float x[4] = {0.f, 0.f, 0.f, 0.f};
            if (c < pw && r < m) split_load4(wide, P.UThi, P.UTlo, ubase, (long long)(j0 + c) * P.ldm + r, 1.f / kF16X, x);
#pragma unroll
            for (int e = 0; e < 4; ++e) a[k][4 * i + e] = r + e < m ? x[e] : 0.f;   // (the padding of a row takes part as zeros)
        }
    // column c (this warp's index k) to shared memory, zero in rows <= c of CTA 0
    auto publish = [&](const float (&col)[RPL], int c) {
        float *x = sm.x[c & 1];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            float4 v = make_float4(col[4 * i], col[4 * i + 1], col[4 * i + 2], col[4 * i + 3]);
            if (i == 0 && rank == 0) {
                const int r = 4 * lane;
                if (r <= c) v.x = 0.f;
                if (r + 1 <= c) v.y = 0.f;
                if (r + 2 <= c) v.z = 0.f;
                if (r + 3 <= c) v.w = 0.f;
            }
            *reinterpret_cast<float4 *>(x + 128 * i + 4 * lane) = v;
        }
    };
    if (w == 0) publish(a[0], 0);
    if (CL > 1) cluster.sync();                      // every CTA runs before its shared memory is written to
    else __syncthreads();

#pragma unroll
    for (int kc = 0; kc < C; ++kc) {
#pragma unroll 1
        for (int wc = 0; wc < kQrWarps; ++wc) {
            const int c = kc * kQrWarps + wc, par = c & 1;
            if (c >= pw) break;
            const float *xs = sm.x[par] + 4 * lane;
            // the sums of this warp's columns
            float x[kKeepX ? RPL : 1];
            float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const float4 v = *reinterpret_cast<const float4 *>(xs + 128 * i);
                if constexpr (kKeepX) { x[4 * i] = v.x; x[4 * i + 1] = v.y; x[4 * i + 2] = v.z; x[4 * i + 3] = v.w; }
#pragma unroll
                for (int k = 0; k < C; ++k) {
                    s[k] = fmaf(v.x, a[k][4 * i], s[k]);
                    s[k] = fmaf(v.y, a[k][4 * i + 1], s[k]);
                    s[k] = fmaf(v.z, a[k][4 * i + 2], s[k]);
                    s[k] = fmaf(v.w, a[k][4 * i + 3], s[k]);
                }
            }
            // lanes 8 v .. 8 v + 7 get the sum of column index v over the warp
            const bool up = lane & 16, up8 = lane & 8;
            float t0 = (up ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, up ? s[0] : s[2], 16);
            float t1 = (up ? s[3] : s[1]) + __shfl_xor_sync(0xffffffffu, up ? s[1] : s[3], 16);
            float t = (up8 ? t1 : t0) + __shfl_xor_sync(0xffffffffu, up8 ? t0 : t1, 8);
            t += __shfl_xor_sync(0xffffffffu, t, 4);
            t += __shfl_xor_sync(0xffffffffu, t, 2);
            t += __shfl_xor_sync(0xffffffffu, t, 1);
            const int v = lane >> 3, q = lane & 7, e = v * kQrWarps + w;
            float rv = 0.f;
            if (rank == 0) {                         // row j = local row c, in lane c / 4
                const int ce = c & 3, cl4 = c >> 2;
#pragma unroll
                for (int k = 0; k < C; ++k) {
                    const float y = ce == 0 ? a[k][0] : (ce == 1 ? a[k][1] : (ce == 2 ? a[k][2] : a[k][3]));
                    const float z = __shfl_sync(0xffffffffu, y, cl4);
                    if (k == v) rv = z;
                }
            }
            if (v < C) {
                if (CL == 1) {
                    if (q == 0) { sm.slot[par][0][e] = t; sm.row[par][e] = rv; }
                } else {
                    for (int peer = q; peer < CL; peer += 8) {
                        *cluster.map_shared_rank(&sm.slot[par][rank][e], peer) = t;
                        if (rank == 0) *cluster.map_shared_rank(&sm.row[par][e], peer) = rv;
                    }
                }
            }
            if (CL == 1) __syncthreads();
            else cluster.sync();
            // totals of this warp's columns (lanes 8 v ..) and of column c
            float pt = 0.f, s2 = 0.f;
            for (int p = q; p < CL; p += 8) {
                if (v < C) pt += sm.slot[par][p][e];
                s2 += sm.slot[par][p][c];
            }
#pragma unroll
            for (int d = 4; d; d >>= 1) {
                pt += __shfl_xor_sync(0xffffffffu, pt, d);
                s2 += __shfl_xor_sync(0xffffffffu, s2, d);
            }
            const float fa = sm.row[par][c];
            float beta, tau, scal;
            if (s2 == 0.f) { beta = fa; tau = 0.f; scal = 0.f; }
            else {
                beta = -copysignf(sqrtf(fmaf(fa, fa, s2)), fa);
                tau = (beta - fa) / beta;
                scal = 1.f / (fa - beta);
            }
            const float g = v < C ? fmaf(pt, scal, sm.row[par][e]) : 0.f;
            if (rank == 0) {
                if (q == 0 && v < C && e < c) sm.G[e][c] = g;
                if (tid == 0) {
                    sm.tau[c] = tau;
                    P.tau[(long long)b * n + j0 + c] = tau;
                    P.beta[(long long)b * n + j0 + c] = beta;
                }
            }
            // y -= f v for the later columns, v = [1; x scal]; column c becomes its reflector
#pragma unroll
            for (int k = kc; k < C; ++k) {
                const float f = tau * __shfl_sync(0xffffffffu, g, 8 * k);
                if (k > kc || w > wc) {
                    const float fs = f * scal;
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        float4 xv;
                        if constexpr (kKeepX) xv = make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
                        else xv = *reinterpret_cast<const float4 *>(xs + 128 * i);
                        a[k][4 * i] = fmaf(-fs, xv.x, a[k][4 * i]);
                        a[k][4 * i + 1] = fmaf(-fs, xv.y, a[k][4 * i + 1]);
                        a[k][4 * i + 2] = fmaf(-fs, xv.z, a[k][4 * i + 2]);
                        a[k][4 * i + 3] = fmaf(-fs, xv.w, a[k][4 * i + 3]);
                    }
                    if (rank == 0 && lane == c >> 2) {
#pragma unroll
                        for (int ee = 0; ee < 4; ++ee)
                            if ((c & 3) == ee) a[k][ee] -= f;
                    }
                } else if (w == wc) {
#pragma unroll
                    for (int i = 0; i < RPL; ++i) {
                        const int r = rank * S + 128 * (i / 4) + 4 * lane + (i & 3);      // row - j0
                        a[k][i] = r > c ? a[k][i] * scal : (r == c ? beta : a[k][i]);
                    }
                }
            }
            if (wc + 1 < kQrWarps) {
                if (w == wc + 1) publish(a[kc], c + 1);
            } else if (kc + 1 < C) {
                if (w == 0) publish(a[kc + 1 < C ? kc + 1 : kc], c + 1);
            }
            __syncthreads();
        }
    }

    // the factored panel back to UT (R entries above the diagonal, beta on it, v below); the
    // reflectors also as clean rows (YT: 0 above, 1 on the diagonal) and columns (Y)
#pragma unroll
    for (int k = 0; k < C; ++k) {
        const int c = k * kQrWarps + w;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int rl = 128 * i + 4 * lane, r = r0 + rl;
            float u[4], y[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                u[e] = a[k][4 * i + e];
                const int d = r + e - (j0 + c);
                y[e] = d < 0 ? 0.f : (d == 0 ? 1.f : u[e]);
                sm.slab[c][rl + e] = y[e];
            }
            if (c < pw && r < m) {                   // rows of UT and YT are padded to multiples of 32
                const long long o = (long long)(j0 + c) * P.ldm + r;
                split_store4(wide, P.UThi, P.UTlo, ubase, o, u, kF16X);
                split_store4(wide, P.YThi, P.YTlo, ubase, o, y, kF16V);
            }
        }
    }
    __syncthreads();
    const long long ybase = (long long)b * m * P.ldn;
    {
        const int c = 2 * (tid % (NB / 2)), nr = min(S, m - r0);
        for (int rl = tid / (NB / 2); rl < nr; rl += kQrThreads / (NB / 2)) {
            if (c >= pw) continue;
            const long long o = (long long)(r0 + rl) * P.ldn + j0 + c;
            if (!wide && c + 1 < pw) {
                __half h0, l0, h1, l1;
                split_f16(sm.slab[c][rl] * kF16V, h0, l0);
                split_f16(sm.slab[c + 1][rl] * kF16V, h1, l1);
                *reinterpret_cast<__half2 *>(as_half(P.Yhi) + 2 * ybase + o) = __halves2half2(h0, h1);
                *reinterpret_cast<__half2 *>(as_half(P.Ylo) + 2 * ybase + o) = __halves2half2(l0, l1);
            } else {
                split_store(wide, P.Yhi, P.Ylo, ybase, o, sm.slab[c][rl], kF16V);
                if (c + 1 < pw) split_store(wide, P.Yhi, P.Ylo, ybase, o + 1, sm.slab[c + 1][rl], kF16V);
            }
        }
    }
    // zeros above the panel's first row, down from the first row of its block (the block's products read them)
    const int s0 = j0 - j0 % kWY;
    if (rank == CL - 1)
        for (int t = tid; t < (j0 - s0) * pw; t += blockDim.x) {
            const int rr = t / pw, c = t - rr * pw;
            split_store(wide, P.Yhi, P.Ylo, ybase, (long long)(s0 + rr) * P.ldn + j0 + c, 0.f, 1.f);
            split_store(wide, P.YThi, P.YTlo, ubase, (long long)(j0 + c) * P.ldm + s0 + rr, 0.f, 1.f);
        }
    if (rank != 0 || 4 * w >= NB) return;
    // T[c][c] = tau_c, T[:c, c] = -tau_c T[:c, :c] G[:c, c].  Row i needs nothing of the other rows: 8 lanes
    // per row, lane q with entries q, q + 8, ...
    const int i = 4 * w + (lane >> 3), q = lane & 7;
    float *out = P.Tm + ((long long)b * P.npan + P.panel) * NB * NB + (long long)i * NB;
    float tr[NB / 8];
#pragma unroll
    for (int cb = 0; cb < NB / 8; ++cb) tr[cb] = 0.f;
#pragma unroll
    for (int cb = 0; cb < NB / 8; ++cb)
#pragma unroll 1
        for (int cq = 0; cq < 8; ++cq) {
            const int c = 8 * cb + cq;
            float v = 0.f;
            if (c < pw) {
#pragma unroll
                for (int lb = 0; lb <= cb; ++lb)
                    if (8 * lb + q < c) v = fmaf(tr[lb], sm.G[8 * lb + q][c], v);
#pragma unroll
                for (int d = 4; d; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
                const float tc = sm.tau[c];
                v = i < c ? -tc * v : (i == c ? tc : 0.f);
                if (q == cq) tr[cb] = v;
            }
        }
#pragma unroll
    for (int cb = 0; cb < NB / 8; ++cb) out[8 * cb + q] = i < pw ? tr[cb] : 0.f;
}

// Launch of one panel: the fewest CTAs whose registers hold its m - j0 rows, 256 rows each as far as 8 CTAs
// reach (64 columns), else 512; 1024 or 1536 for panels of 32 columns.
template <int RPL, int C>
static int qr_launch_panel(PanelArgs &a, int B, cudaStream_t st) {
    using Sm = PanelSmem<RPL, C>;
    a.cl = (a.m - a.j0 + Sm::S - 1) / Sm::S;
    if (a.cl > kQrMaxCl || a.pw > Sm::NB) return PSVD_ERR_ARG;
    static_assert(sizeof(Sm) <= 227 * 1024, "panel too large");
    PSVD_TRY(cudaFuncSetAttribute(qr_panel_kernel<RPL, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Sm)));
    if (a.cl > 8)
        PSVD_TRY(cudaFuncSetAttribute(qr_panel_kernel<RPL, C>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(B * a.cl));
    cfg.blockDim = dim3(kQrThreads);
    cfg.dynamicSmemBytes = sizeof(Sm);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = a.cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    PSVD_TRY(cudaLaunchKernelEx(&cfg, qr_panel_kernel<RPL, C>, a));
    count_launch(1);
    return PSVD_OK;
}

// W2^T[c][i] = sum_l T^T[i][l] W[l][c], W = sum of the ks K-split slices of Y^T X, for the ncol <= 96
// columns that a panel still has to its right in its block.  Tm holds the nb x nb T of every (matrix,
// panel).  One block of 8 warps per kTaCols columns: the block's columns of W (slices summed) are
// staged in shared memory with coalesced loads, warp g forms outputs i = g, g + 8, ... of every
// column (lane = column); rows of W2^T have stride kWY.
constexpr int kTaCols = 32, kTaWarps = 8;
__global__ void __launch_bounds__(32 * kTaWarps) qr_tapply_kernel(const float *Wp, int ks, int B, int nb, int pw,
                                                                  int n, int ldw, int ncol, const float *Tm, int npan,
                                                                  int panel, const int *skip, const int *fine,
                                                                  float *W2hi, float *W2lo) {
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
        split_store(fine[b] == PREC_TF32X3, W2hi, W2lo, (long long)b * n * kWY, (long long)c * kWY + i, sum, kF16S2);
    }
}

// S2 = S T (trans = 0) or S T^T (trans = 1) of a block of kWY columns, S (ncol x kWY) the sum of ks K-split
// slices in slice order, S2 split.  One block of 2 kWY threads per kQsRows rows: op(T)^T
// staged with rows padded to kQsLd floats (thread j of a half reads row j as float4), the rows of S
// as float4 broadcasts.  T is zero outside its triangle and past the block's width.
constexpr int kQsRows = 32, kQsLd = kWY + 4;
constexpr size_t kQsSmem = sizeof(float) * ((size_t)kWY * kQsLd + (size_t)kQsRows * kWY);
__global__ void __launch_bounds__(2 * kWY) qr_stapply_kernel(const float *Sp, int ks, int B, int n, int ncol, int ws,
                                                             const float *Ts, int nsup, int sup, int trans,
                                                             const int *skip, const int *fine, float *W2hi,
                                                             float *W2lo) {
    extern __shared__ __align__(16) float qsm2[];
    float *Ms = qsm2, *sr = qsm2 + kWY * kQsLd;
    const int b = blockIdx.y, t = threadIdx.x, i0 = blockIdx.x * kQsRows;
    if (skip[b]) return;
    const bool wide = fine[b] == PREC_TF32X3;
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
        split_store(wide, W2hi, W2lo, (long long)b * n * kWY, (long long)i * kWY + j, acc[r], kF16S2);
    }
}

// max |a| of every column of the factored matrices (float bits; a NaN compares above every finite value): one
// block of 32 x 8 threads per 32 columns and kCmRows rows
constexpr int kCmRows = 512;
__global__ void __launch_bounds__(256) qr_colmax_kernel(const float *A, int m, int n, const int *skip, unsigned *amax) {
    __shared__ unsigned red[8][32];
    const int b = blockIdx.z, tx = threadIdx.x & 31, ty = threadIdx.x >> 5, c = blockIdx.x * 32 + tx;
    if (skip[b]) return;
    unsigned v = 0;
    if (c < n) {
        const float *a = A + (long long)b * m * n + c;
        const int r1 = min(m, ((int)blockIdx.y + 1) * kCmRows);
#pragma unroll 8
        for (int r = blockIdx.y * kCmRows + ty; r < r1; r += 8) v = max(v, __float_as_uint(fabsf(a[(long long)r * n])));
    }
    red[ty][tx] = v;
    __syncthreads();
    if (ty == 0 && c < n) {
#pragma unroll
        for (int w = 1; w < 8; ++w) v = max(v, red[w][tx]);
        atomicMax(&amax[(long long)b * n + c], v);
    }
}
// 2^e >= sqrt(m) max |a| >= the norm of column c (1 where there is none: a zero or non-finite column), and 2^-e
__global__ void qr_scale_kernel(const unsigned *amax, long long cols, int m, float *scale, float *iscale) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cols) return;
    const float v = __uint_as_float(amax[c]);
    const bool ok = v > 0.f && v < INFINITY;
    const int e = ok ? min(126, max(-100, ilogb((double)v * sqrt((double)m)) + 1)) : 0;
    scale[c] = ldexpf(1.f, e);
    iscale[c] = ldexpf(1.f, -e);
}

__global__ void qr_skip_kernel(const int *flag, int B, int *skip, int *fine) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    skip[b] = flag ? (flag[b] ? 0 : 1) : 0;
    fine[b] = PREC_F16X3;
}

// Q^T = [I 0] (split: hi = identity, lo = 0) for the factored matrices
__global__ void qr_qinit_kernel(int n, int m, long long ldm, const int *skip, const int *fine, float *QThi, float *QTlo) {
    const int b = blockIdx.z;
    if (skip[b]) return;
    const int c = blockIdx.y, r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= m) return;
    split_store(fine[b] == PREC_TF32X3, QThi, QTlo, (long long)b * n * ldm, (long long)c * ldm + r, r == c ? 1.f : 0.f, kF16X);
}

// Q[r][c] = sign(beta_c) Q^T[c][r] (transposed through a shared tile) and, if R is given,
// R[r][c] = 2^e_c sign(beta_r) (r < c ? UT[c][r] : r == c ? beta_c : 0).
__global__ void qr_store_kernel(const float *QThi, const float *QTlo, const float *UThi, const float *UTlo,
                                const float *beta, const float *scale, int m, int n, long long ldm, const int *skip,
                                const int *fine, float *Q, float *R) {
    __shared__ float tile[32][33];
    const int b = blockIdx.z;
    if (skip[b]) return;
    const int c0 = blockIdx.y * 32, r0 = blockIdx.x * 32;   // c: column of Q (row of Q^T)
    const float *bb = beta + (long long)b * n;
    const bool wide = fine[b] == PREC_TF32X3;
    const long long ub = (long long)b * n * ldm;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int c = c0 + i, r = r0 + threadIdx.x;
        float v = 0.f;
        if (c < n && r < m) {
            v = (bb[c] < 0.f ? -1.f : 1.f) * split_load(wide, QThi, QTlo, ub, (long long)c * ldm + r, 1.f / kF16X);
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
            v = r < c ? split_load(wide, UThi, UTlo, ub, (long long)c * ldm + r, 1.f / kF16X) : (r == c ? fabsf(bb[c]) : 0.f);
            if (r < c && bb[r] < 0.f) v = -v;
            v *= scale[(long long)b * n + c];
        }
        tile[i][threadIdx.x] = v;
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int r = r0 + i, c = c0 + threadIdx.x;
        if (r < n && c < n) R[((long long)b * n + r) * n + c] = tile[threadIdx.x][i];
    }
}

// a product of split arrays whose halves carry `scale`
static GemmShape qr_shape_of(const QrWS &w, int M, int N, int K, float scale) {
    GemmShape s;
    memset(&s, 0, sizeof(s));
    s.M = M; s.N = N; s.K = K; s.prec = w.fine; s.skip = w.skip; s.err = w.err;
    s.f16_scale = 1.f / scale;
    s.prof_as = PREC_TF32X3 + 1;
    return s;
}

// X^T[c][j0 + r] -= sum_i W2^T[c][i] Y[j0 + r][j0 + i] for rows c0 .. c0 + ncol - 1 of X^T and the pw reflectors
// from j0 on, W2^T in w.W2hi / w.W2lo.
static int qr_update(QrWS &w, int j0, int pw, int c0, int ncol, float *Xhi, float *Xlo, cudaStream_t st) {
    const int B = w.B, m = w.m, n = w.n, K = m - j0;
    GemmShape s = qr_shape_of(w, ncol, K, pw, kF16S2 * kF16V);
    const long long off = (long long)c0 * w.ldm + j0;
    EpiSubHalf e;
    e.rows = ncol; e.cols = K; e.ld = w.ldm; e.scale = kF16X; e.inv = 1.f / kF16X;
    e.fine = w.fine; e.fhi = Xhi + off; e.flo = Xlo + off; e.fbs = (long long)n * w.ldm;
    e.hi = as_half(Xhi) + off; e.lo = as_half(Xlo) + off; e.bs = 2 * e.fbs;
    PSVD_TRY(launch_split(SplitView(w.W2hi, w.W2lo, 0, ncol, pw, kWY, (long long)n * kWY, B),
                          SplitView(w.Yhi, w.Ylo, (long long)j0 * w.ldn + j0, K, pw, w.ldn, (long long)m * w.ldn, B), s, B,
                          e, st));
    return PSVD_OK;
}

// The reflectors of one panel on the ncol columns from c0 on, the rest of its block.
static int qr_apply_panel(QrWS &w, int j0, int pw, int panel, int c0, int ncol, cudaStream_t st) {
    const int B = w.B, m = w.m, n = w.n, nb = w.nb, ldw = std::min(n, kWY);
    const int K = m - j0;
    const long long nm = (long long)n * w.ldm;
    // W = Y^T X: A = Y^T rows of the panel (pw x K), B = X^T rows (ncol x K), split over K
    GemmShape s = qr_shape_of(w, pw, ncol, K, kF16V * kF16X);
    s.ksplit = std::max(1, std::min(std::min(w.ks, (num_sms() + B - 1) / B), (K + 127) / 128));
    EpiStore e = epi_store_plain(w.Wp, ldw, (long long)nb * ldw, pw, ncol);
    PSVD_TRY(launch_split(SplitView(w.YThi, w.YTlo, (long long)j0 * w.ldm + j0, pw, K, w.ldm, nm, B),
                          SplitView(w.UThi, w.UTlo, (long long)c0 * w.ldm + j0, ncol, K, w.ldm, nm, B), s, B, e, st));
    qr_tapply_kernel<<<dim3((ncol + kTaCols - 1) / kTaCols, B), 32 * kTaWarps, 0, st>>>(
        w.Wp, s.ksplit, B, nb, pw, n, ldw, ncol, w.Tm, w.npan, panel, w.skip, w.fine, w.W2hi, w.W2lo);
    count_launch(1);
    PSVD_TRY(cudaGetLastError());
    return qr_update(w, j0, pw, c0, ncol, w.UThi, w.UTlo, st);
}

// T of the block of ws <= kWY columns from j0 on.
static int qr_block_t(QrWS &w, int j0, int ws, int sup, cudaStream_t st) {
    const int B = w.B, K = w.m - j0;
    const long long nm = (long long)w.n * w.ldm, gbs = (long long)w.n * kWY;
    GemmShape s = qr_shape_of(w, ws, ws, K, kF16V * kF16V);
    // one tile with all of K: split (4 matrices of 14336 rows 185 -> 29 us, and 38 -> 64 in the T kernel that adds the slices)
    s.ksplit = std::max(1, std::min(kQrSplit, (K + 255) / 256));
    EpiStore e = epi_store_plain(w.Sp, kWY, gbs, ws, ws);
    const SplitView y(w.YThi, w.YTlo, (long long)j0 * w.ldm + j0, ws, K, w.ldm, nm, B);
    PSVD_TRY(launch_split(y, y, s, B, e, st));
    return larft_blocks(w.Sp, s.ksplit, gbs, w.tau, w.n, w.n, w.nsup, sup, 1, B, w.Ts, st);
}

// The reflectors of a whole block on rows c0 .. c0 + ncol - 1 of X^T: trans = 0 in the factorization
// (X <- (I - Y T Y^T)^T X), 1 in the accumulation of Q (X <- (I - Y T Y^T) X).
static int qr_apply_block(QrWS &w, int j0, int ws, int sup, int c0, int ncol, float *Xhi, float *Xlo, int trans,
                          cudaStream_t st) {
    const int B = w.B, n = w.n, K = w.m - j0;
    const long long nm = (long long)n * w.ldm;
    GemmShape s = qr_shape_of(w, ncol, ws, K, kF16X * kF16V);
    const int tiles = ((ncol + kBM - 1) / kBM) * B;
    s.ksplit = std::max(1, std::min(std::min(kQrSplit, (num_sms() + tiles - 1) / tiles), (K + 255) / 256));
    EpiStore e = epi_store_plain(w.Sp, kWY, (long long)n * kWY, ncol, ws);
    PSVD_TRY(launch_split(SplitView(Xhi, Xlo, (long long)c0 * w.ldm + j0, ncol, K, w.ldm, nm, B),
                          SplitView(w.YThi, w.YTlo, (long long)j0 * w.ldm + j0, ws, K, w.ldm, nm, B), s, B, e, st));
    PSVD_TRY(cudaFuncSetAttribute(qr_stapply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQsSmem));
    qr_stapply_kernel<<<dim3((ncol + kQsRows - 1) / kQsRows, B), 2 * kWY, kQsSmem, st>>>(
        w.Sp, s.ksplit, B, n, ncol, ws, w.Ts, w.nsup, sup, trans, w.skip, w.fine, w.W2hi, w.W2lo);
    count_launch(1);
    PSVD_TRY(cudaGetLastError());
    return qr_update(w, j0, ws, c0, ncol, Xhi, Xlo, st);
}

int qr_factor(const float *A, float *Q, float *R, const int *flag, QrWS &w, cudaStream_t st) {
    const int B = w.B, m = w.m, n = w.n, nb = w.nb;
    const long long nm = (long long)n * w.ldm;
    qr_skip_kernel<<<(B + 127) / 128, 128, 0, st>>>(flag, B, w.skip, w.fine);
    const long long mn = (long long)m * n, bn = (long long)B * n;
    PSVD_TRY(cudaMemsetAsync(w.amax, 0, sizeof(unsigned) * (size_t)bn, st));
    qr_colmax_kernel<<<dim3((n + 31) / 32, (m + kCmRows - 1) / kCmRows, B), 256, 0, st>>>(A, m, n, w.skip, w.amax);
    qr_scale_kernel<<<(unsigned)((bn + 127) / 128), 128, 0, st>>>(w.amax, bn, m, w.scale, w.iscale);
    count_launch(3);
    {
        PSVD_TRY(fine_rows(A, B, m, n, w.iscale, w.skip, w.fine, st));
        SplitOut t = split_out(w.UThi, w.UTlo, w.ldm, nm, kF16X, w.fine);
        t.colscale = w.iscale;
        PSVD_TRY(prepare_operand(A, n, mn, B, m, n, true, 1.f, nullptr, t, st, w.skip));
    }
    for (int sp = 0; sp < w.nsup; ++sp) {
        const int s0 = sp * kWY, s1 = std::min(n, s0 + kWY);
        for (int j0 = s0; j0 < s1; j0 += nb) {
            const int pw = std::min(nb, s1 - j0), p = j0 / nb;
            PanelArgs a;
            a.UThi = w.UThi; a.UTlo = w.UTlo; a.YThi = w.YThi; a.YTlo = w.YTlo; a.Yhi = w.Yhi; a.Ylo = w.Ylo;
            a.tau = w.tau; a.beta = w.beta; a.Tm = w.Tm; a.skip = w.skip; a.fine = w.fine;
            a.m = m; a.n = n; a.j0 = j0; a.pw = pw; a.panel = p; a.npan = w.npan;
            a.ldm = w.ldm; a.ldn = w.ldn;
            const int rows = m - j0;
            if (nb == 64) PSVD_TRY_RC(rows <= kQrRows8 ? (qr_launch_panel<8, 4>(a, B, st)) : (qr_launch_panel<16, 4>(a, B, st)));
            else PSVD_TRY_RC(rows <= 16384 ? (qr_launch_panel<32, 2>(a, B, st)) : (qr_launch_panel<48, 2>(a, B, st)));
            if (j0 + pw < s1) PSVD_TRY_RC(qr_apply_panel(w, j0, pw, p, j0 + pw, s1 - j0 - pw, st));
        }
        PSVD_TRY_RC(qr_block_t(w, s0, s1 - s0, sp, st));
        if (s1 < n) PSVD_TRY_RC(qr_apply_block(w, s0, s1 - s0, sp, s1, n - s1, w.UThi, w.UTlo, 0, st));
    }
    {
        dim3 g((m + 127) / 128, n, B);
        qr_qinit_kernel<<<g, 128, 0, st>>>(n, m, w.ldm, w.skip, w.fine, w.QThi, w.QTlo);
        count_launch(1);
        PSVD_TRY(cudaGetLastError());
    }
    for (int sp = w.nsup - 1; sp >= 0; --sp) {
        const int s0 = sp * kWY, s1 = std::min(n, s0 + kWY);
        PSVD_TRY_RC(qr_apply_block(w, s0, s1 - s0, sp, s0, n - s0, w.QThi, w.QTlo, 1, st));
    }
    {
        dim3 g((m + 31) / 32, (n + 31) / 32, B), blk(32, 8);
        qr_store_kernel<<<g, blk, 0, st>>>(w.QThi, w.QTlo, w.UThi, w.UTlo, w.beta, w.scale, m, n, w.ldm, w.skip, w.fine,
                                            Q, R);
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
    int nb = 0;
    if (!A || !Q || batch <= 0 || n <= 0 || m < n || batch > 65535 || n > 16384 || (long long)m * n > (1LL << 31))
        return PSVD_ERR_ARG;
    if (!qr_shape((int)m, &nb))
        return fail_msg(PSVD_ERR_ARG, "psvd_qr: m = %lld rows exceed the cluster panel", (long long)m);
    if (int e = check_device()) return e;
    if (ws_bytes < psvd_qr_workspace_bytes(batch, m, n)) return PSVD_ERR_WORKSPACE;
    Carver cv(ws, ws_bytes);
    QrWS w;
    w.carve(cv, (int)batch, (int)m, (int)n);
    if (cv.overflow) return PSVD_ERR_WORKSPACE;
    return qr_factor(A, Q, R, nullptr, w, static_cast<cudaStream_t>(stream));
}
