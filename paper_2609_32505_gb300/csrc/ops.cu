// Operand preparation (scale, transpose, TF32 hi/lo split, BF16 cast) and the
// generic batched TN product entry point.
#include <cstring>

#include "ops.cuh"

namespace psvd {

__global__ void prepare_kernel(const float *__restrict__ src, long long lds, long long bss, int rows, int cols,
                               int trans, float scale, const float *__restrict__ scale_ptr, SplitOut dst,
                               const int *__restrict__ skip) {
    __shared__ float tile[32][33];
    const int b = blockIdx.z;
    if (skip && skip[b]) return;
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
    float sc = scale;
    if (scale_ptr) {
        const float s = scale_ptr[b];
        sc = s > 0.f ? 1.f / s : 0.f;
    }
    const float *S = src + b * bss;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int r = r0 + i, c = c0 + threadIdx.x;
        float x = 0.f;
        if (r < rows && c < cols) {
            x = S[(long long)r * lds + c] * sc;
            if (dst.colscale) x *= dst.colscale[(long long)b * cols + c];
        }
        tile[i][threadIdx.x] = x;
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        int r, c;
        float x;
        if (trans) { r = c0 + i; c = r0 + threadIdx.x; x = tile[threadIdx.x][i]; if (r >= cols || c >= rows) continue; }
        else { r = r0 + i; c = c0 + threadIdx.x; x = tile[i][threadIdx.x]; if (r >= rows || c >= cols) continue; }
        const long long o = b * dst.bstride + (long long)r * dst.ld + c;
        const int p = dst.prec ? dst.prec[b] : -1;
        if (dst.fhi && (p < 0 || p == PREC_F16X3)) {
            const long long of = b * dst.fbstride + (long long)r * dst.ld + c;
            __half h, l;
            split_f16(x * dst.fscale, h, l);
            dst.fhi[of] = h;
            dst.flo[of] = l;
        }
        if (dst.hi && (p < 0 || p == PREC_TF32 || p == PREC_TF32X3)) {
            if (dst.lo && p != PREC_TF32) { float h, l; split_tf32(x, h, l); dst.hi[o] = h; dst.lo[o] = l; }
            else dst.hi[o] = p == PREC_TF32 ? tf32_round(x) : x;
        }
        if (dst.h16 && (p < 0 || p == PREC_BF16)) dst.h16[o] = __float2bfloat16_rn(x);
    }
}

// The same in 16-byte pieces, for destinations whose rows are padded to multiples of 8 elements: 8 values
// of one destination row per thread.  Rows as they are: a thread reads its 8 values (two float4 where the
// source allows, kVec) and writes them.  Transposed: 64 x 32 tiles through shared memory.
// Bound by memory: 4096^2 to split TF32 takes 42 us (rows 36, transposed 48), the
// kernel above, element by element in 32 x 32 tiles, 59 us; to split FP16 rows 20 us (6.4 TB/s), transposed 30 us.
PSVD_DEV void prepare_store8(const SplitOut &d, int p, int b, int r, int c, int nv, const float (&x)[8]) {
    const long long o = b * d.bstride + (long long)r * d.ld + c;
    if (d.fhi && (p < 0 || p == PREC_F16X3)) {
        const long long of = b * d.fbstride + (long long)r * d.ld + c;
        __align__(16) __half h[8], l[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) split_f16(x[i] * d.fscale, h[i], l[i]);
        if (nv == 8) {
            *reinterpret_cast<uint4 *>(d.fhi + of) = *reinterpret_cast<const uint4 *>(h);
            *reinterpret_cast<uint4 *>(d.flo + of) = *reinterpret_cast<const uint4 *>(l);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < nv) { d.fhi[of + i] = h[i]; d.flo[of + i] = l[i]; }
        }
    }
    if (d.hi && (p < 0 || p == PREC_TF32 || p == PREC_TF32X3)) {
        const bool two = d.lo && p != PREC_TF32;
        float h[8], l[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (two) split_tf32(x[i], h[i], l[i]);
            else h[i] = p == PREC_TF32 ? tf32_round(x[i]) : x[i];
        }
        if (nv == 8) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                reinterpret_cast<float4 *>(d.hi + o)[q] = make_float4(h[4 * q], h[4 * q + 1], h[4 * q + 2], h[4 * q + 3]);
                if (two)
                    reinterpret_cast<float4 *>(d.lo + o)[q] = make_float4(l[4 * q], l[4 * q + 1], l[4 * q + 2], l[4 * q + 3]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < nv) { d.hi[o + i] = h[i]; if (two) d.lo[o + i] = l[i]; }
        }
    }
    if (d.h16 && (p < 0 || p == PREC_BF16)) {
        __align__(16) __nv_bfloat16 h[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) h[i] = __float2bfloat16_rn(x[i]);
        if (nv == 8) *reinterpret_cast<uint4 *>(d.h16 + o) = *reinterpret_cast<const uint4 *>(h);
        else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < nv) d.h16[o + i] = h[i];
        }
    }
}

template <bool kTrans, bool kVec>
__global__ void __launch_bounds__(256) prepare_vec_kernel(const float *__restrict__ src, long long lds, long long bss,
                                                          int rows, int cols, float scale,
                                                          const float *__restrict__ scale_ptr, SplitOut dst,
                                                          const int *__restrict__ skip) {
    __shared__ float tile[kTrans ? 64 : 1][33];
    const int b = blockIdx.z;
    if (skip && skip[b]) return;
    float sc = scale;
    if (scale_ptr) {
        const float s = scale_ptr[b];
        sc = s > 0.f ? 1.f / s : 0.f;
    }
    const int p = dst.prec ? dst.prec[b] : -1;
    const float *S = src + b * bss;
    float x[8];
    if constexpr (kTrans) {
        const int r0 = blockIdx.y * 64, c0 = blockIdx.x * 32;
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        if (dst.colscale && c0 + lane < cols) sc *= dst.colscale[(long long)b * cols + c0 + lane];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = r0 + w + 8 * i, c = c0 + lane;
            tile[w + 8 * i][lane] = (r < rows && c < cols) ? S[(long long)r * lds + c] * sc : 0.f;
        }
        __syncthreads();
        const int c = c0 + (threadIdx.x >> 3), r = r0 + 8 * (threadIdx.x & 7);
        if (c >= cols || r >= rows) return;
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = tile[8 * (threadIdx.x & 7) + i][threadIdx.x >> 3];
        prepare_store8(dst, p, b, c, r, min(8, rows - r), x);
    } else {
        const int c8 = (cols + 7) / 8;
        const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        if (t >= (long long)rows * c8) return;
        const int r = (int)(t / c8), c = 8 * (int)(t % c8), nv = min(8, cols - c);
        const float *q = S + (long long)r * lds + c;
        if (kVec && nv == 8) {
            const float4 u = reinterpret_cast<const float4 *>(q)[0], v = reinterpret_cast<const float4 *>(q)[1];
            x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w; x[4] = v.x; x[5] = v.y; x[6] = v.z; x[7] = v.w;
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = i < nv ? q[i] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] *= sc;
        if (dst.colscale) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < nv) x[i] *= dst.colscale[(long long)b * cols + c + i];
        }
        prepare_store8(dst, p, b, r, c, nv, x);
    }
}

cudaError_t prepare_operand(const float *src, long long lds, long long bss, int batch, int rows, int cols,
                            bool trans, float scale, const float *scale_ptr, const SplitOut &dst,
                            cudaStream_t st, const int *skip) {
    if (batch <= 0 || rows <= 0 || cols <= 0) return cudaSuccess;
    const uintptr_t at = (uintptr_t)dst.hi | (uintptr_t)dst.lo | (uintptr_t)dst.h16 | (uintptr_t)dst.fhi |
                         (uintptr_t)dst.flo;
    if ((at & 15) == 0 && ((dst.ld | dst.bstride | dst.fbstride) & 7) == 0) {
        const bool vec = ((uintptr_t)src & 15) == 0 && ((lds | bss) & 3) == 0;
        if (trans) {
            const dim3 g((cols + 31) / 32, (rows + 63) / 64, batch);
            prepare_vec_kernel<true, false><<<g, 256, 0, st>>>(src, lds, bss, rows, cols, scale, scale_ptr, dst, skip);
        } else {
            const long long n = (long long)rows * ((cols + 7) / 8);
            const dim3 g((unsigned)((n + 255) / 256), 1, batch);
            if (vec) prepare_vec_kernel<false, true><<<g, 256, 0, st>>>(src, lds, bss, rows, cols, scale, scale_ptr, dst, skip);
            else prepare_vec_kernel<false, false><<<g, 256, 0, st>>>(src, lds, bss, rows, cols, scale, scale_ptr, dst, skip);
        }
    } else {
        dim3 grid((cols + 31) / 32, (rows + 31) / 32, batch), block(32, 8);
        prepare_kernel<<<grid, block, 0, st>>>(src, lds, bss, rows, cols, trans ? 1 : 0, scale, scale_ptr, dst, skip);
    }
    count_launch(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) cuda_fail(e, __FILE__, __LINE__);
    return e;
}

__global__ void fine_reset_kernel(int *fine, int B) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) fine[b] = PREC_F16X3;
}
cudaError_t fine_reset(int *fine, int B, cudaStream_t st) {
    fine_reset_kernel<<<(B + 127) / 128, 128, 0, st>>>(fine, B);
    count_launch(1);
    return cudaGetLastError();
}
// One warp per row.  Entries x 2^14 are held to 22 bits down to 2^-28 (split_f16), so a row with a largest
// entry above sqrt(n) 2^-28 has no more rounding error in halves than in split TF32.
__global__ void __launch_bounds__(256) fine_rows_kernel(const float *A, int m, int n, const float *colscale,
                                                        const int *skip, float lim, int *fine) {
    const int b = blockIdx.y, lane = threadIdx.x & 31, r = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (r >= m || (skip && skip[b])) return;
    const float *a = A + ((long long)b * m + r) * n, *cs = colscale ? colscale + (long long)b * n : nullptr;
    float v = 0.f;
#pragma unroll 8
    for (int c = lane; c < n; c += 32) v = fmaxf(v, fabsf(a[c]) * (cs ? cs[c] : 1.f));
    v = warp_max(v);
    if (lane == 0 && v > 0.f && v < lim) fine[b] = PREC_TF32X3;
}
cudaError_t fine_rows(const float *A, int B, int m, int n, const float *colscale, const int *skip, int *fine,
                      cudaStream_t st) {
    fine_rows_kernel<<<dim3((m + 7) / 8, B), 256, 0, st>>>(A, m, n, colscale, skip, sqrtf((float)n) * 0x1p-28f, fine);
    count_launch(1);
    return cudaGetLastError();
}

// out = Q X for the preprocessed route (Q: B x M x N, X: B x N x N, both with orthonormal columns), operands
// split FP16 (split TF32 where rows of Q are very small) in scratch carved from cv.  (4 x 14336 x 4096 x 4096: 3.8 ms, in
// split TF32 7.0 ms.)
int orth_product(Carver &cv, const float *Q, const float *X, float *out, int B, int M, int N, cudaStream_t st) {
    const long long ld = pad_ld(N), qs = (long long)M * ld, xs = (long long)N * ld;
    float *qhi = cv.take<float>((size_t)B * qs), *qlo = cv.take<float>((size_t)B * qs);
    float *xhi = cv.take<float>((size_t)B * xs), *xlo = cv.take<float>((size_t)B * xs);
    int *fine = cv.take<int>(B);
    unsigned *err = cv.take<unsigned>(4);
    if (cv.overflow) return PSVD_ERR_WORKSPACE;
    PSVD_TRY(fine_reset(fine, B, st));
    PSVD_TRY(fine_rows(Q, B, M, N, nullptr, nullptr, fine, st));
    SplitOut a = split_out(qhi, qlo, ld, qs, kF16X, fine), bt = split_out(xhi, xlo, ld, xs, kF16X, fine);
    PSVD_TRY(prepare_operand(Q, N, (long long)M * N, B, M, N, false, 1.f, nullptr, a, st));
    // B operand B[k][j] = X[j][k] (X transposed)
    PSVD_TRY(prepare_operand(X, N, (long long)N * N, B, N, N, true, 1.f, nullptr, bt, st));
    GemmShape s;
    memset(&s, 0, sizeof(s));
    s.M = M; s.N = N; s.K = N; s.prec = fine; s.err = err;
    s.f16_scale = 1.f / (kF16X * kF16X);
    s.prof_as = PREC_TF32X3 + 1;
    EpiStore e = epi_store_plain(out, N, (long long)M * N, M, N);
    PSVD_TRY(launch_split(SplitView(qhi, qlo, 0, M, N, ld, qs, B), SplitView(xhi, xlo, 0, N, N, ld, xs, B), s, B, e, st));
    return PSVD_OK;
}

}  // namespace psvd

using namespace psvd;

extern "C" {

size_t psvd_gemm_workspace_bytes(int64_t batch, int64_t M, int64_t N, int64_t K) {
    const long long ld = pad_ld(K);
    return (size_t)(batch * (M + N) * ld) * (2 * sizeof(float) + sizeof(__nv_bfloat16)) + 4096;
}

int psvd_gemm_tn(const float *A, const float *B, float *D, int64_t batch, int64_t M, int64_t N, int64_t K,
                 int precision, void *ws, size_t ws_bytes, void *stream) {
    if (!A || !B || !D || batch <= 0 || M <= 0 || N <= 0 || K <= 0 || precision < 0 || precision > 2)
        return PSVD_ERR_ARG;
    if (int e = check_device()) return e;
    if (ws_bytes < psvd_gemm_workspace_bytes(batch, M, N, K)) return PSVD_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const long long ld = pad_ld(K);
    Carver cv(ws, ws_bytes);
    float *ahi = cv.take<float>(batch * M * ld), *alo = cv.take<float>(batch * M * ld);
    float *bhi = cv.take<float>(batch * N * ld), *blo = cv.take<float>(batch * N * ld);
    __nv_bfloat16 *a16 = cv.take<__nv_bfloat16>(batch * M * ld), *b16 = cv.take<__nv_bfloat16>(batch * N * ld);
    if (cv.overflow) return PSVD_ERR_WORKSPACE;
    SplitOut da, db;
    da.ld = db.ld = ld;
    da.bstride = M * ld; db.bstride = N * ld;
    if (precision == PREC_BF16) { da.h16 = a16; db.h16 = b16; }
    else { da.hi = ahi; db.hi = bhi; if (precision == PREC_TF32X3) { da.lo = alo; db.lo = blo; } }
    if (prepare_operand(A, K, M * K, (int)batch, (int)M, (int)K, false, 1.f, nullptr, da, st) != cudaSuccess ||
        prepare_operand(B, K, N * K, (int)batch, (int)N, (int)K, false, 1.f, nullptr, db, st) != cudaSuccess)
        return PSVD_ERR_CUDA;
    MatView va16 = view_of16(a16, (int)M, (int)K, ld, M * ld, (int)batch);
    MatView vb16 = view_of16(b16, (int)N, (int)K, ld, N * ld, (int)batch);
    MatView vah = view_of(ahi, (int)M, (int)K, ld, M * ld, (int)batch), val = view_of(alo, (int)M, (int)K, ld, M * ld, (int)batch);
    MatView vbh = view_of(bhi, (int)N, (int)K, ld, N * ld, (int)batch), vbl = view_of(blo, (int)N, (int)K, ld, N * ld, (int)batch);
    GemmShape shp;
    memset(&shp, 0, sizeof(shp));
    shp.M = (int)M; shp.N = (int)N; shp.K = (int)K; shp.prec_uniform = precision;
    EpiStore epi = epi_store_plain(D, N, M * N, (int)M, (int)N);
    cudaError_t e;
    if (precision == PREC_BF16) e = launch_gemm(&va16, &vb16, nullptr, nullptr, nullptr, nullptr, shp, (int)batch, epi, st);
    else if (precision == PREC_TF32) e = launch_gemm(nullptr, nullptr, &vah, nullptr, &vbh, nullptr, shp, (int)batch, epi, st);
    else e = launch_gemm(nullptr, nullptr, &vah, &val, &vbh, &vbl, shp, (int)batch, epi, st);
    return cuda_status(e);
}

}  // extern "C"
