// Operand preparation kernels and the generic store epilogue, shared by the
// polar, SVD and backward drivers.
#pragma once
#include "gemm.cuh"
#include "runtime.h"

namespace psvd {

// Internal buffers keep rows padded to a multiple of 32 elements (128 B of fp32)
// so that every TMA row stride is 16-byte aligned.
inline long long pad_ld(long long cols) { return round_up(cols < 1 ? 1 : cols, 32); }

// The column L1 norms of the normalization (Algorithm 2) are summed in slabs of kL1Rows
// rows; the buffer of column sums holds batch x l1_slabs(m) x n partial sums.
constexpr int kL1Rows = 256;
constexpr int kNormThreads = 1024;   // threads of the block that finishes the norms of one matrix
__host__ __device__ inline int l1_slabs(int m) { return m < 1 ? 1 : (m + kL1Rows - 1) / kL1Rows; }

constexpr int kWY = 128;   // reflectors per compact-WY block (back-transform, QR's trailing updates)
// T (upper triangular, kWY x kWY) of compact-WY blocks from G = Y^T Y and tau (eigh.cu).
int larft_blocks(const float *Gm, int ks, long long gbs, const float *tau, int n, int nrefl, int nblk, int blk0,
                 int count, int B, float *Tm, cudaStream_t st);

// Output format of an operand-preparation pass.
struct SplitOut {
    float *hi = nullptr, *lo = nullptr;   // fp32 split (lo may be null: TF32 rounding only)
    __nv_bfloat16 *h16 = nullptr;         // bf16 copy
    __half *fhi = nullptr, *flo = nullptr;   // fp16 split of x * fscale (strides below, in elements)
    float fscale = 1.f;
    const float *colscale = nullptr;      // factors of the source's columns [batch][cols], or null
    const int *prec = nullptr;            // per matrix: write the one format its precision reads
    long long ld = 0, bstride = 0, fbstride = 0;
};

// Both split formats of arrays with room for floats (batch stride bs floats), by prec[b].
inline SplitOut split_out(float *hi, float *lo, long long ld, long long bs, float fscale, const int *prec) {
    SplitOut s;
    s.hi = hi; s.lo = lo; s.fhi = reinterpret_cast<__half *>(hi); s.flo = reinterpret_cast<__half *>(lo);
    s.ld = ld; s.bstride = bs; s.fbstride = 2 * bs;
    s.fscale = fscale; s.prec = prec;
    return s;
}

// Powers of two that bring split-FP16 operands below 2^16: polar iterates (singular values <= 2 at
// every step of every schedule) and orthonormal factors; the step polynomial c1 I + c3 G
// (entries <= 5.2: c1 = 3 sqrt(3) on [0, 1]); Householder vectors (entries <= 1); the back-transform's S2 = S T^T.
constexpr float kF16X = 0x1p14f, kF16P = 0x1p13f, kF16V = 0x1p14f, kF16S2 = 0x1p10f;

// src (batch x rows x cols, leading dim lds, batch stride bss) scaled by `scale`
// (or by 1/scale_ptr[b] when scale_ptr != nullptr) -> dst in its padded layout,
// transposed when `trans` (dst is then cols x rows).
cudaError_t prepare_operand(const float *src, long long lds, long long bss, int batch, int rows, int cols,
                            bool trans, float scale, const float *scale_ptr, const SplitOut &dst,
                            cudaStream_t st, const int *skip = nullptr);

// MatViews of a SplitOut for TMA.
inline MatView view_of(const float *p, int rows, int cols, long long ld, long long bs, int batch) {
    MatView v; v.ptr = p; v.rows = rows; v.cols = cols; v.ld = ld; v.bstride = bs; v.batch = batch; v.bf16 = false;
    return v;
}
inline MatView view_of16(const __nv_bfloat16 *p, int rows, int cols, long long ld, long long bs, int batch) {
    MatView v; v.ptr = p; v.rows = rows; v.cols = cols; v.ld = ld; v.bstride = bs; v.batch = batch; v.bf16 = true;
    return v;
}

inline MatView view_f16(const __half *p, int rows, int cols, long long ld, long long bs, int batch) {
    MatView v; v.ptr = p; v.rows = rows; v.cols = cols; v.ld = ld; v.bstride = bs; v.batch = batch; v.f16 = true;
    return v;
}

// A split array whose matrices are each in one of the two split formats (fine[b] = PREC_F16X3 or PREC_TF32X3) has
// room for floats; halves lie at the start of their matrix's space, so their batch stride is twice that of floats.
__host__ __device__ inline __half *as_half(float *p) { return reinterpret_cast<__half *>(p); }
__host__ __device__ inline const __half *as_half(const float *p) { return reinterpret_cast<const __half *>(p); }
// element o of the matrix that starts at float bo: x * fs as halves, or x as it is
PSVD_DEV void split_store(bool wide, float *hi, float *lo, long long bo, long long o, float x, float fs) {
    if (wide) {
        float h, l;
        split_tf32(x, h, l);
        hi[bo + o] = h;
        lo[bo + o] = l;
    } else {
        __half h, l;
        split_f16(x * fs, h, l);
        as_half(hi)[2 * bo + o] = h;
        as_half(lo)[2 * bo + o] = l;
    }
}
PSVD_DEV float split_load(bool wide, const float *hi, const float *lo, long long bo, long long o, float inv) {
    return wide ? hi[bo + o] + lo[bo + o] : join_f16(as_half(hi)[2 * bo + o], as_half(lo)[2 * bo + o]) * inv;
}
// the two pairs of views of a split array, `off` elements into every matrix
struct SplitView {
    MatView h, l, fh, fl;
    SplitView(const float *hi, const float *lo, long long off, int rows, int cols, long long ld, long long bs, int batch)
        : h(view_f16(as_half(hi) + off, rows, cols, ld, 2 * bs, batch)),
          l(view_f16(as_half(lo) + off, rows, cols, ld, 2 * bs, batch)),
          fh(view_of(hi + off, rows, cols, ld, bs, batch)), fl(view_of(lo + off, rows, cols, ld, bs, batch)) {}
};
// product of two of them, s.prec = fine
template <class Epi>
cudaError_t launch_split(const SplitView &a, const SplitView &b, const GemmShape &s, int batch, const Epi &e,
                         cudaStream_t st) {
    const F16Views f{a.h, a.l, b.h, b.l};
    return launch_gemm(nullptr, nullptr, &a.fh, &a.fl, &b.fh, &b.fl, s, batch, e, st, &f);
}

// fine[b] = PREC_F16X3 for all b; then PREC_TF32X3 for matrices with a nonzero row of A (B x m x n, columns times
// colscale) whose entries are so small that FP16 halves of them, bound 1, lose bits.
cudaError_t fine_reset(int *fine, int B, cudaStream_t st);
cudaError_t fine_rows(const float *A, int B, int m, int n, const float *colscale, const int *skip, int *fine,
                      cudaStream_t st);

// D = acc, row-major, plain (out, may be null) and/or split TF32 (hi and lo, may be null).
struct EpiStore {
    int rows, cols;
    float *out; long long ld, bs;
    float *hi, *lo; long long ldh, bsh;
    struct Acc {};
    static constexpr bool kElem = true;
    PSVD_DEV bool row16(Acc &, int b, int r0, int lane, int c0, float (&v)[16], float *) const {
        if (r0 >= rows || c0 >= cols) return true;
        if (c0 + 16 > cols || (out && ((((uintptr_t)out & 31) != 0) || ((ld | bs) & 7) != 0))) return false;
        const int r = r0 + lane;
        if (r >= rows) return true;
        uint32_t h[16], l[16];
        if (out) {
#pragma unroll
            for (int i = 0; i < 16; ++i) h[i] = __float_as_uint(v[i]);
            st_v8x2(out + b * bs + (long long)r * ld + c0, h);
        }
        if (!hi) return true;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            float a, c;
            split_tf32(v[i], a, c);
            h[i] = __float_as_uint(a);
            l[i] = __float_as_uint(c);
        }
        const long long o = b * bsh + (long long)r * ldh + c0;
        st_v8x2(hi + o, h);
        st_v8x2(lo + o, l);
        return true;
    }
    PSVD_DEV void elem(Acc &, int b, int r, int c, float v) const {
        if (r >= rows || c >= cols) return;
        if (out) out[b * bs + (long long)r * ld + c] = v;
        if (hi) {
            const long long o = b * bsh + (long long)r * ldh + c;
            split_tf32(v, hi[o], lo[o]);
        }
    }
    PSVD_DEV void begin(Acc &) const {}
    PSVD_DEV void finish(Acc &, int, int, int) const {}
};

// In place: X[r][c] -= acc for a matrix kept as FP16 halves of x * scale (the eigensolver's back-transform,
// the QR's trailing updates), or as split TF32 at fhi / flo where fine[b] says so.
struct EpiSubHalf {
    int rows, cols;
    __half *hi, *lo;
    long long ld, bs;
    float scale, inv;
    const int *fine;              // null: halves
    float *fhi, *flo;
    long long fbs;
    struct Acc {};
    static constexpr bool kElem = true;
    PSVD_DEV bool row16(Acc &, int b, int r0, int lane, int c0, float (&v)[16], float *) const {
        if (r0 >= rows || c0 >= cols) return true;
        if (fine && fine[b] == PREC_TF32X3) return false;
        if (c0 + 16 > cols || (((uintptr_t)hi | (uintptr_t)lo) & 31) || ((ld | bs) & 15)) return false;
        if (r0 + lane >= rows) return true;
        const long long o = b * bs + (long long)(r0 + lane) * ld + c0;
        uint32_t h[8], l[8];
        ld_v8(hi + o, h);
        ld_v8(lo + o, l);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&h[i]));
            const float2 c = __half22float2(*reinterpret_cast<const __half2 *>(&l[i]));
            v[2 * i] = __fmaf_rn(c.x, kF16LoInv, a.x) * inv - v[2 * i];
            v[2 * i + 1] = __fmaf_rn(c.y, kF16LoInv, a.y) * inv - v[2 * i + 1];
        }
        split_f16x16(v, scale, h, l);
        st_v8(hi + o, h);
        st_v8(lo + o, l);
        return true;
    }
    PSVD_DEV void elem(Acc &, int b, int r, int c, float v) const {
        if (r >= rows || c >= cols) return;
        if (fine && fine[b] == PREC_TF32X3) {
            const long long o = b * fbs + (long long)r * ld + c;
            split_tf32((fhi[o] + flo[o]) - v, fhi[o], flo[o]);
            return;
        }
        const long long o = b * bs + (long long)r * ld + c;
        __half h, l;
        split_f16((join_f16(hi[o], lo[o]) * inv - v) * scale, h, l);
        hi[o] = h;
        lo[o] = l;
    }
    PSVD_DEV void begin(Acc &) const {}
    PSVD_DEV void finish(Acc &, int, int, int) const {}
};

// 16 values of one row as split-FP16 halves of v * fs: along the row at rhi / rlo when `rowv`, transposed
// (this lane's 16 rows of column c0 + lane / 2) at chi / clo when `colv`; all lanes call it.
PSVD_DEV void f16_row16(const float (&v)[16], float fs, __half *rhi, __half *rlo, bool rowv, __half *chi, __half *clo,
                        bool colv, float *sw) {
    uint32_t w[16], o[16], h[8], l[8];
    split_f16x16(v, fs, h, l);
    if (rowv) {
        st_v8(rhi, h);
        st_v8(rlo, l);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {                  // (hi, lo) of one value per word
        w[2 * i] = __byte_perm(h[i], l[i], 0x5410);
        w[2 * i + 1] = __byte_perm(h[i], l[i], 0x7632);
    }
    warp_transpose16(sw, w, o);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        h[i] = __byte_perm(o[2 * i], o[2 * i + 1], 0x5410);
        l[i] = __byte_perm(o[2 * i], o[2 * i + 1], 0x7632);
    }
    if (colv) {
        st_v8(chi, h);
        st_v8(clo, l);
    }
}

// Split output of v * inv[b] in the format fine[b] (halves times kF16X), row-major (hi, may be null) and
// transposed (hi_t), optionally with the plain values (out).
struct EpiHalf {
    int rows, cols;
    const float *inv;
    const int *fine;
    float *out;
    long long ld, bs;
    float *hi, *lo;
    long long ldh, bsh;
    float *hi_t, *lo_t;
    long long ldht, bsht;
    struct Acc {};
    PSVD_DEV bool row16(Acc &, int b, int r0, int lane, int c0, float (&v)[16], float *sw) const {
        if (r0 >= rows || c0 >= cols) return true;
        if (fine[b] == PREC_TF32X3) return false;
        if (c0 + 16 > cols || (out && ((((uintptr_t)out & 31) != 0) || ((ld | bs) & 7) != 0))) return false;
        const int r = r0 + lane, ct = c0 + (lane >> 1);
        if (out && r < rows) {
            uint32_t w[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = __float_as_uint(v[i]);
            st_v8x2(out + b * bs + (long long)r * ld + c0, w);
        }
        const long long o = 2 * b * bsh + (long long)r * ldh + c0;
        const long long t = 2 * b * bsht + (long long)ct * ldht + r0 + 16 * (lane & 1);    // (padding past `rows`: zeros)
        f16_row16(v, inv[b] * kF16X, as_half(hi) + o, as_half(lo) + o, hi && r < rows, as_half(hi_t) + t, as_half(lo_t) + t,
                  true, sw);
        return true;
    }
    PSVD_DEV void begin(Acc &) const {}
    PSVD_DEV void chunk(Acc &, int b, int r, int c0, float (&v)[16]) const {
        if (r >= rows) return;
        const float iv = inv[b];
        auto store = [&](auto wide) {              // (the format decided once, not per value)
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int c = c0 + i;
                if (c >= cols) break;
                if (out) out[b * bs + (long long)r * ld + c] = v[i];
                if (hi) split_store(wide, hi, lo, b * bsh, (long long)r * ldh + c, v[i] * iv, kF16X);
                split_store(wide, hi_t, lo_t, b * bsht, (long long)c * ldht + r, v[i] * iv, kF16X);
            }
        };
        if (fine[b] == PREC_TF32X3) store(std::true_type{});
        else store(std::false_type{});
    }
    PSVD_DEV void finish(Acc &, int, int, int) const {}
};

int orth_product(Carver &cv, const float *Q, const float *X, float *out, int B, int M, int N, cudaStream_t st);

inline EpiStore epi_store_plain(float *out, long long ld, long long bs, int rows, int cols) {
    EpiStore e;
    memset(&e, 0, sizeof(e));
    e.rows = rows; e.cols = cols;
    e.out = out; e.ld = ld; e.bs = bs;
    return e;
}

}  // namespace psvd
