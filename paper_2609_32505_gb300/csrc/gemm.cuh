// tcgen05 "TN" GEMM for sm_103a:  D[b][i][j] = sum_k A[b][i][k] * B[b][j][k]
// with both operands K-major (row-major with K contiguous) in global memory.
//
// Every product of the method is put in this form by keeping transposed copies
// where needed (X and X^T for the polynomial steps, U^T, V, ... in the backward),
// so one well-tested kernel serves the Gram matrix, the polynomial apply, H, U and
// the backward chain.
//
// Persistent kernel: one CTA per SM walks a static list of output tiles of
// 128 x BN, UMMA M = 128, N = BN, cta_group::1.  BN = 256, or 128 when N <= 128: 128-wide tiles
// cost about twice as much per flop as 256-wide ones on GB300 (a fixed cost per MMA instruction; measured
// with one mainloop version, BF16 at 8192^3: 559 against 1049 TFLOP/s); halved down to 32 while a launch
// leaves half of the SMs idle (plan_gemm).
// Shared memory holds a 192 KB ring of units (4 x 48 KB at BN = 256, 6 x 32 KB at
// BN = 128, 9 x 20 KB at 32), each one TMA'd k-block: an A sub-tile (128 rows x 128 B) and a B sub-tile
// (BN rows x 128 B), both in the canonical 128-byte-swizzled K-major layout:
//   PREC_BF16   : 64 bf16 of K per unit, one unit per k-block
//   PREC_TF32   : 32 fp32 of K per unit, one unit per k-block
//   PREC_TF32X3 : 32 fp32 of K, two units per k-block (hi parts, lo parts);
//                 hi*hi + hi*lo + lo*hi (split-TF32, FP32-accurate products)
//   PREC_F16X3  : 64 fp16 of K, two units per k-block: the same three products of split FP16 halves
//                 (operands scaled by powers of two, undone by GemmShape::f16_scale; the low halves by
//                 2^kF16LoBits more, undone by the first hi*hi of a k-block).  An FP16 MMA
//                 covers twice the K of a TF32 one in the same time and its operands are half the
//                 bytes (a 4096^3 polar step product: 780 us in split TF32, 474 us with the
//                 same epilogue)
// Two accumulators of 128 x 256 FP32 in TMEM (all 512 columns) let the MMA warp
// run the next tile (or the next k-block of a split one) while the epilogue drains the
// previous one.  The tensor core accumulates with truncation; split tiles are
// therefore flushed into round-to-nearest FP32 registers after every k-block.
// Warp roles: warps 0-7 epilogue (warp w reads TMEM lanes 32 (w % 4) .. + 31 and
// the column half w / 4), warp 8 TMA producer, warp 9 MMA issuer.  The precision is
// chosen per tile at run time from the tile's batch entry, which lets the polar
// iteration switch precision matrix by matrix.
#pragma once
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "common.cuh"

namespace psvd {

enum Prec : int { PREC_BF16 = 0, PREC_TF32 = 1, PREC_TF32X3 = 2, PREC_F16X3 = 3 };

constexpr int kBM = 128;
constexpr int kUnitA = 16384;                  // 128 rows x 128 B
constexpr int kUnitB = 32768;                  // up to 256 rows x 128 B
constexpr int kUnitBytes = kUnitA + kUnitB;    // 48 KB
constexpr int kStages = 4;                     // ring units at BN = 256
constexpr int kRingBytes = kStages * kUnitBytes;
constexpr int kMinBN = 32;
static_assert(kMinBN >= 32 && kMinBN % 32 == 0, "the two column halves of a tile are read and stored 16 columns at a time");
constexpr int kMaxStages = kRingBytes / (kUnitA + kMinBN * 128);   // ring units at BN = 32 (9)
constexpr int kEpiWarps = 8;
constexpr int kGemmThreads = (kEpiWarps + 2) * 32;
constexpr int kStageRow = 17;                  // staging row stride (floats): conflict-free
constexpr int kTransRow = 36;                  // row stride of the 16 x 32 transpose: 16-byte rows, conflict-free
constexpr int kStageWarp = 16 * kTransRow;     // floats per warp (also 32 x kStageRow <= this)
static_assert(32 * kStageRow <= kStageWarp, "staging area");
constexpr int kStageBytes = kEpiWarps * kStageWarp * 4;
constexpr int kGemmSmem = kRingBytes + 1024 /*align*/ + 256 /*barriers*/ + kStageBytes;
static_assert((2 * kMaxStages + 4) * 8 + 4 <= 256, "barrier area");
constexpr int kAccCols = 256;                  // TMEM columns per accumulator
constexpr uint32_t kTmemCols = 512;

struct GemmMaps {
    CUtensorMap a_bf16, b_bf16;  // used by PREC_BF16 tiles
    CUtensorMap a_hi, a_lo;      // fp32 (TF32 uses a_hi only)
    CUtensorMap b_hi, b_lo;
    CUtensorMap a_h16, a_l16, b_h16, b_l16;   // split FP16
};

struct GemmShape {
    int M, N, K;            // logical sizes
    int tiles_m, tiles_n;   // ceil(M/128), ceil(N/BN)
    int bn;                 // 32, 64, 128 or 256
    int batch;
    int sym;                // 1: only tiles that reach the upper triangle (col >= row); requires A == B
    int ksplit;             // > 1: every tile repeated over ksplit disjoint k-block ranges; the
                            // epilogue of range kc gets batch index b + kc * batch (partial sums)
    int prec_uniform;       // used when prec == nullptr
    const int *prec;        // [batch] per-matrix precision, or nullptr
    const int *skip;        // [batch] nonzero = matrix finished, its tiles are skipped (or nullptr)
    const int *gate;        // nullptr, or a device counter: 0 = nothing left to do, the whole launch
                            // returns at once (written by an earlier kernel on the same stream)
    unsigned *ticket;       // nullptr, or a zeroed counter: the last CTA to finish runs epi.tail()
    unsigned *err;          // device error word
    float f16_scale;        // PREC_F16X3: the product of the operands' inverse scales
    float tf32_scale;       // PREC_TF32X3: the same (0: 1)
    const float *scale_b;   // split precisions: another factor for each matrix (nullptr: 1)
    int prof_as;            // profiling class + 1 for the launch timing (0: by precision)
};

// First tile column of row ti that reaches the upper triangle.
PSVD_DEV int sym_first_col(int ti, int bn) { return (kBM * ti) / bn; }

// Tile t of one matrix -> (ti, tj).
PSVD_DEV void tile_coords(const GemmShape &s, int t, int &ti, int &tj) {
    if (!s.sym) { ti = t / s.tiles_n; tj = t % s.tiles_n; return; }
    int row = 0;
    for (;;) {
        const int cnt = s.tiles_n - sym_first_col(row, s.bn);
        if (t < cnt || row == s.tiles_m - 1) break;
        t -= cnt;
        ++row;
    }
    ti = row;
    tj = sym_first_col(row, s.bn) + t;
}

PSVD_DEV int tiles_per_matrix(const GemmShape &s) {
    if (!s.sym) return s.tiles_m * s.tiles_n;
    int c = 0;
    for (int r = 0; r < s.tiles_m; ++r) c += s.tiles_n - sym_first_col(r, s.bn);
    return c;
}

// k-blocks of a tile and accumulation phases (flush points) per tile.
PSVD_DEV int kblocks(const GemmShape &s, int prec) {
    const int kstep = prec == PREC_BF16 || prec == PREC_F16X3 ? 64 : 32;
    return (s.K + kstep - 1) / kstep;
}

// One work item of the persistent tile list: matrix b, k range kc (of ksplit), tile (ti, tj),
// k-blocks [kb0, kb0 + nkb).
struct TileJob { int b, kc, ti, tj, kb0, nkb, prec; };
PSVD_DEV TileJob tile_job(const GemmShape &s, int t, int tpm) {
    TileJob j;
    const int ks = s.ksplit > 1 ? s.ksplit : 1;
    const int per = tpm * ks;
    j.b = t / per;
    const int rem = t % per;
    j.kc = rem / tpm;
    tile_coords(s, rem % tpm, j.ti, j.tj);
    j.prec = s.prec ? s.prec[j.b] : s.prec_uniform;
    const int all = kblocks(s, j.prec);
    const int each = (all + ks - 1) / ks;
    j.kb0 = j.kc * each;
    j.nkb = max(0, min(all, j.kb0 + each) - j.kb0);
    return j;
}

// Epilogues that define a per-element elem(acc, b, r, c, v) get their values through a per-warp shared-memory transpose, so that each store instruction
// of a warp covers two rows x 16 consecutive columns instead of 32 rows x 1 column.
template <class E, class = void> struct EpiHasElem : std::false_type {};
template <class E> struct EpiHasElem<E, std::void_t<decltype(E::kElem)>> : std::integral_constant<bool, E::kElem> {};
// Staged epilogues that also write a transposed copy define trans(acc, b, r, c0, v[16]):
// it runs on the thread's own row (lanes = consecutive rows, so the transposed stores of a
// warp are coalesced) next to the staged row-major element pass.
template <class E, class = void> struct EpiHasTrans : std::false_type {};
template <class E> struct EpiHasTrans<E, std::void_t<decltype(E::kTrans)>> : std::integral_constant<bool, E::kTrans> {};
// Epilogues with a tail() run it once per launch, in the last CTA to finish (shp.ticket set),
// after every CTA's epilogue writes and atomics are visible: a per-launch reduction step
// (the polar iteration's per-matrix decision) without a launch of its own.
template <class E, class = void> struct EpiHasTail : std::false_type {};
template <class E> struct EpiHasTail<E, std::void_t<decltype(E::kTail)>> : std::integral_constant<bool, E::kTail> {};

// row16(acc, b, r0, lane, c0, v, sw) of every epilogue gets the 16 columns c0 .. c0 + 15 of the thread's row
// r0 + lane as they are and store them in 32-byte pieces: along the row directly (a whole sector per
// lane), transposed through the warp's shared memory `sw` (warp_transpose16).  It returns false
// (uniformly) for pieces it does not handle -- ragged edges, the diagonal, unaligned outputs -- which
// then take the element-wise paths above, or chunk(acc, b, r, c0, v) on the thread's own row where there is no
// elem; kTotal: it handles every piece.  (Element by element a polar step's tile cost ~17,000
// instructions per warp, about half the time of a 4096^3 split product: 474 -> 310 us with the pieces.)
template <class E, class = void> struct EpiIsTotal : std::false_type {};
template <class E> struct EpiIsTotal<E, std::void_t<decltype(E::kTotal)>> : std::integral_constant<bool, E::kTotal> {};

// 32 bytes at a 32-byte aligned address
PSVD_DEV void st_v8(void *p, const uint32_t (&r)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]),
                 "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
PSVD_DEV void st_v8x2(void *p, const uint32_t (&r)[16]) {       // 64 bytes
    const uint32_t a[8] = {r[0], r[1], r[2], r[3], r[4], r[5], r[6], r[7]};
    const uint32_t b[8] = {r[8], r[9], r[10], r[11], r[12], r[13], r[14], r[15]};
    st_v8(p, a);
    st_v8(static_cast<char *>(p) + 32, b);
}
// (an ordinary load: the in-place epilogues write what they read, which the read-only path does not allow)
PSVD_DEV void ld_v8(const void *p, uint32_t (&r)[8]) {
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "l"(p)
                 : "memory");
}
// Lane l gives word w[i] of column i of its row; it gets the 16 words of rows 16 (l & 1) .. + 15 of
// column l >> 1.
PSVD_DEV void warp_transpose16(float *sw, const uint32_t (&w)[16], uint32_t (&o)[16]) {
    const int lane = threadIdx.x & 31;
    uint32_t *s = reinterpret_cast<uint32_t *>(sw);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) s[i * kTransRow + lane] = w[i];
    __syncwarp();
    const uint4 *q = reinterpret_cast<const uint4 *>(s + (lane >> 1) * kTransRow + (lane & 1) * 16);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint4 x = q[i];
        o[4 * i] = x.x; o[4 * i + 1] = x.y; o[4 * i + 2] = x.z; o[4 * i + 3] = x.w;
    }
}
// the warp's values, lane = row, into its staging area (rows of kStageRow)
PSVD_DEV void stage_piece(const float (&v)[16], float *sw) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) sw[(threadIdx.x & 31) * kStageRow + i] = v[i];
    __syncwarp();
}
// Sums of 16 per-lane values over the warp: lane l returns the sum of value l >> 1.
PSVD_DEV float warp_sum16(float (&a)[16]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 8, o = 16; h > 0; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < h) {
                const float send = up ? a[i] : a[i + h], keep = up ? a[i + h] : a[i];
                a[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
    }
    return a[0] + __shfl_xor_sync(0xffffffffu, a[0], 1);
}
// 16 values -> packed FP16 halves of x * fs (split_f16)
PSVD_DEV void split_f16x16(const float (&v)[16], float fs, uint32_t (&h)[8], uint32_t (&l)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float x0 = v[2 * i] * fs, x1 = v[2 * i + 1] * fs;
        const __half2 hh = __floats2half2_rn(x0, x1);
        const float2 f = __half22float2(hh);
        const __half2 ll = __floats2half2_rn((x0 - f.x) * kF16Lo, (x1 - f.y) * kF16Lo);
        h[i] = *reinterpret_cast<const uint32_t *>(&hh);
        l[i] = *reinterpret_cast<const uint32_t *>(&ll);
    }
}

// Consumer side of the operand ring, as seen by the MMA issuer: shared-memory address of
// unit 0, unit size, unit count, barriers, and the position of the next unit with the
// parity of its current fill.
struct MmaRing {
    uint32_t base, unit_bytes, nst;
    uint64_t *full, *empty;
    unsigned *err;
    uint32_t stage, phase;
    PSVD_DEV uint32_t take() {                 // returns the stage, advances the position
        const uint32_t s = stage;
        if (++stage == nst) { stage = 0; phase ^= 1; }
        return s;
    }
};

// Descriptor of the k-th 32-byte K step inside a 128-byte swizzled row: the start address
// field (bits 0-13, in 16-byte units) advances by 2; a unit ends below 228 KB, so the
// field never carries.
PSVD_DEV uint64_t sdesc_step(uint64_t d, int k) { return d + (uint64_t)(2 * k); }

// One BF16 or TF32 tile: all its k-blocks accumulate into `tacc` (one phase).
template <bool kTF32>
PSVD_DEV bool mma_tile(MmaRing &r, int nkb, uint32_t tacc, uint32_t id) {
    for (int kb = 0; kb < nkb; ++kb) {
        const uint32_t par = r.phase;
        const uint32_t s = r.take();
        if (!mbar_wait(&r.full[s], par, r.err)) return false;
        tc_fence_after();
        const uint32_t a0 = r.base + s * r.unit_bytes;
        const uint64_t ad = sdesc_k128(a0), bd = sdesc_k128(a0 + kUnitA);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t en = (kb > 0 || k > 0) ? 1u : 0u;
            if constexpr (kTF32) umma_tf32(tacc, sdesc_step(ad, k), sdesc_step(bd, k), id, en);
            else umma_f16(tacc, sdesc_step(ad, k), sdesc_step(bd, k), id, en);
        }
        umma_commit(&r.empty[s]);
    }
    return true;
}

// One split-TF32 or split-FP16 tile: every k-block (hi unit, lo unit) is its own phase in the next
// accumulator, flushed by the epilogue into round-to-nearest FP32 registers.
template <bool kF16>
PSVD_DEV bool mma_tile_x3(MmaRing &r, int nkb, uint32_t tmem, uint64_t *acc_full, uint64_t *acc_empty, uint32_t &q,
                          uint32_t id) {
    for (int kb = 0; kb < nkb; ++kb) {
        const uint32_t buf = q & 1;
        if (q >= 2 && !mbar_wait(&acc_empty[buf], ((q >> 1) - 1) & 1, r.err)) return false;
        const uint32_t tacc = tmem + buf * kAccCols;
        const uint32_t p0 = r.phase;
        const uint32_t s0 = r.take();
        const uint32_t p1 = r.phase;
        const uint32_t s1 = r.take();
        if (!mbar_wait(&r.full[s0], p0, r.err) || !mbar_wait(&r.full[s1], p1, r.err)) return false;
        tc_fence_after();
        const uint32_t a0 = r.base + s0 * r.unit_bytes, a1 = r.base + s1 * r.unit_bytes;
        const uint64_t ahi = sdesc_k128(a0), bhi = sdesc_k128(a0 + kUnitA);
        const uint64_t alo = sdesc_k128(a1), blo = sdesc_k128(a1 + kUnitA);
        // the cross products first: the accumulator truncates at its current magnitude, so while it
        // holds only them (2^-11 of the result) their eight additions cost nothing, and four
        // truncations per k-block remain instead of twelve
        auto mma = [&](uint64_t a, uint64_t b, uint32_t en) {
            if constexpr (kF16) umma_f16(tacc, a, b, id, en);
            else umma_tf32(tacc, a, b, id, en);
        };
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            mma(sdesc_step(alo, k), sdesc_step(bhi, k), k != 0);
            mma(sdesc_step(ahi, k), sdesc_step(blo, k), 1);
        }
        // (the low halves of split FP16 carry 2^kF16LoBits, which the first hi*hi takes out of their sum)
        if constexpr (kF16) umma_f16_lo(tacc, ahi, bhi, id);
        else mma(ahi, bhi, 1);
#pragma unroll
        for (int k = 1; k < 4; ++k) mma(sdesc_step(ahi, k), sdesc_step(bhi, k), 1);
        umma_commit(&r.empty[s0]);
        umma_commit(&r.empty[s1]);
        umma_commit(&acc_full[buf]);
        ++q;
    }
    return true;
}

template <class Epi>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_tn_kernel(const __grid_constant__ GemmMaps maps, const GemmShape shp, Epi epi) {
    // Launched ahead of its predecessor's end (programmatic dependent launch): let the next launch
    // come, then wait until everything before this one has completed and is visible.  Every thread of every
    // launch waits, also of one with nothing to do: only then does the completion of a launch stand for that of
    // all before it, which whatever follows relies on (a reset of the counters, a graph's next node, a reuse of
    // the workspace).
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // A gated launch with nothing left to do returns before any allocation (uniform: every
    // thread reads the same word, final since the kernel that wrote it has completed).
    if (shp.gate && *shp.gate == 0) return;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kRingBytes);
    uint64_t *empty = full + kMaxStages;
    uint64_t *acc_full = empty + kMaxStages;   // [2] accumulator phase complete (tcgen05.commit)
    uint64_t *acc_empty = acc_full + 2;        // [2] accumulator drained by the epilogue (8 warps)
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + 2);
    float *stage = reinterpret_cast<float *>(smem + kRingBytes + 256);
    __shared__ volatile int s_abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bn = shp.bn;
    const uint32_t unit_bytes = (uint32_t)(kUnitA + bn * 128);   // also the ring stride (1024-aligned)
    const uint32_t nst = kRingBytes / unit_bytes;                // 4 .. 9
    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], kEpiWarps); }
        fence_barrier_init();
        s_abort = 0;
    }
    if (warp == 0) tmem_alloc(tmem_slot, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    const int tpm = tiles_per_matrix(shp);
    const int total = tpm * (shp.ksplit > 1 ? shp.ksplit : 1) * shp.batch;

    if (warp == kEpiWarps) {
        // ------------------------------------------------------------ TMA producer
        // The ring position (stage) and its parity advance by counting: this thread and the
        // MMA issuer sit on the tensor pipe's critical path, where even an integer division
        // per k-block shows up in the MMA rate.
        if (lane == 0) {
            uint32_t ps = 0, pphase = 0;
            for (int t = blockIdx.x; t < total && !s_abort; t += gridDim.x) {
                const TileJob jb = tile_job(shp, t, tpm);
                const int b = jb.b, prec = jb.prec, nkb = jb.nkb;
                if (shp.skip && shp.skip[b]) continue;
                const int row_a = jb.ti * kBM, row_b = jb.tj * bn;
                const CUtensorMap *ma0 = &maps.a_hi, *mb0 = &maps.b_hi, *ma1 = &maps.a_lo, *mb1 = &maps.b_lo;
                if (prec == PREC_BF16) { ma0 = &maps.a_bf16; mb0 = &maps.b_bf16; }
                if (prec == PREC_F16X3) { ma0 = &maps.a_h16; mb0 = &maps.b_h16; ma1 = &maps.a_l16; mb1 = &maps.b_l16; }
                const int kstep = prec == PREC_BF16 || prec == PREC_F16X3 ? 64 : 32;
                const int nu = prec >= PREC_TF32X3 ? 2 : 1;
                for (int kb = 0; kb < nkb; ++kb) {
                    const int k0 = (jb.kb0 + kb) * kstep;
                    for (int h = 0; h < nu; ++h) {
                        if (!mbar_wait(&empty[ps], pphase ^ 1, shp.err)) { s_abort = 1; break; }
                        uint8_t *st = smem + ps * unit_bytes;
                        mbar_arrive_expect_tx(&full[ps], unit_bytes);
                        tma_load_3d(st, h ? ma1 : ma0, &full[ps], k0, row_a, b);
                        tma_load_3d(st + kUnitA, h ? mb1 : mb0, &full[ps], k0, row_b, b);
                        if (++ps == nst) { ps = 0; pphase ^= 1; }
                    }
                    if (s_abort) break;
                }
            }
        }
    } else if (warp == kEpiWarps + 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t id_tf32 = idesc_f32acc(kFmtTF32, kBM, bn);
            const uint32_t id_f16 = idesc_f32acc(kFmtF16, kBM, bn);
            const uint32_t id_bf16 = idesc_f32acc(kFmtBF16, kBM, bn);
            MmaRing ring{smem_u32(smem), unit_bytes, nst, full, empty, shp.err, 0u, 0u};
            uint32_t q = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
                const TileJob jb = tile_job(shp, t, tpm);
                if ((shp.skip && shp.skip[jb.b]) || jb.nkb <= 0) continue;
                if (jb.prec == PREC_F16X3) {
                    ok = mma_tile_x3<true>(ring, jb.nkb, tmem, acc_full, acc_empty, q, id_f16);
                } else if (jb.prec == PREC_TF32X3) {
                    ok = mma_tile_x3<false>(ring, jb.nkb, tmem, acc_full, acc_empty, q, id_tf32);
                } else {
                    const uint32_t buf = q & 1;
                    if (q >= 2 && !mbar_wait(&acc_empty[buf], ((q >> 1) - 1) & 1, shp.err)) { ok = false; break; }
                    const uint32_t tacc = tmem + buf * kAccCols;
                    ok = jb.prec == PREC_TF32 ? mma_tile<true>(ring, jb.nkb, tacc, id_tf32)
                                              : mma_tile<false>(ring, jb.nkb, tacc, id_bf16);
                    if (!ok) break;
                    umma_commit(&acc_full[buf]);
                    ++q;
                }
            }
            if (!ok) {
                s_abort = 1;
                mbar_arrive(&acc_full[0]);          // release the epilogue
                mbar_arrive(&acc_full[1]);
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        // thread owns output row ti*128 + 32 (warp % 4) + lane and BN/2 columns
        // starting at (warp / 4) * BN/2, kept in round-to-nearest FP32 registers
        const int quad = warp & 3, half = warp >> 2;
        const int ncols = bn >> 1;
        const uint32_t lane_base = uint32_t(quad * 32) << 16;
        uint32_t q = 0;
        for (int t = blockIdx.x; t < total; t += gridDim.x) {
            const TileJob jb = tile_job(shp, t, tpm);
            const int b = jb.b, prec = jb.prec, nkb = jb.nkb, ti = jb.ti, tj = jb.tj;
            if (shp.skip && shp.skip[b]) continue;
            const int be = b + jb.kc * shp.batch;     // epilogue's batch index (partial-sum slice)
            const int nph = nkb == 0 ? 0 : (prec >= PREC_TF32X3 ? nkb : 1);
            float fs = 1.f;                       // undoes the operands' powers of two (exact)
            if (prec == PREC_F16X3) fs = shp.f16_scale;
            if (prec == PREC_TF32X3 && shp.tf32_scale != 0.f) fs = shp.tf32_scale;
            if (prec >= PREC_TF32X3 && shp.scale_b) fs *= shp.scale_b[b];
            float acc[128];
#pragma unroll
            for (int c = 0; c < 128; ++c) acc[c] = 0.f;
            bool ok = true;
            for (int ph = 0; ph < nph; ++ph, ++q) {
                const uint32_t buf = q & 1;
                ok = mbar_wait(&acc_full[buf], (q >> 1) & 1, shp.err) && !s_abort;
                tc_fence_after();
                if (ok) {
                    const uint32_t tb = tmem + lane_base + buf * kAccCols + half * ncols;
#pragma unroll
                    for (int c = 0; c < 128; c += 16) {
                        if (c < ncols) {
                            float v[16];
                            tmem_ld16(tb + c, v);
#pragma unroll
                            for (int i = 0; i < 16; ++i) acc[c + i] = __fmaf_rn(v[i], fs, acc[c + i]);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[buf]);
                if (!ok) break;
            }
            if (!ok) break;
            const int r = ti * kBM + quad * 32 + lane;
            const int cbase = tj * bn + half * ncols;
            typename Epi::Acc ea;
            epi.begin(ea);
            float *sw = stage + warp * kStageWarp;
            const int r0 = ti * kBM + quad * 32, rr0 = lane >> 4, cc = lane & 15;
#pragma unroll
            for (int c = 0; c < 128; c += 16) {
                if (c >= ncols) continue;
                float v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = acc[c + i];
                if (epi.row16(ea, be, r0, lane, cbase + c, v, sw)) continue;
                if constexpr (EpiHasElem<Epi>::value) {
                    stage_piece(v, sw);
#pragma unroll 1
                    for (int k = 0; k < 16; ++k) {
                        const int rr = 2 * k + rr0;
                        epi.elem(ea, be, r0 + rr, cbase + c + cc, sw[rr * kStageRow + cc]);
                    }
                    __syncwarp();
                    if constexpr (EpiHasTrans<Epi>::value) epi.trans(ea, be, r, cbase + c, v);
                } else if constexpr (!EpiIsTotal<Epi>::value) {
                    epi.chunk(ea, be, r, cbase + c, v);
                }
            }
            epi.finish(ea, be, ti, tj);
        }
        tc_fence_before();
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
    if constexpr (EpiHasTail<Epi>::value) {
        if (shp.ticket) {
            __shared__ int s_last;
            if (threadIdx.x == 0) {
                __threadfence();                                  // this CTA's writes before its ticket
                s_last = atomicAdd(shp.ticket, 1u) == gridDim.x - 1;
                if (s_last) __threadfence();                      // every other CTA's, before the tail
            }
            __syncthreads();
            if (s_last) epi.tail();
        }
    }
}

// ---------------------------------------------------------------- host side
// A 3-D view of a batch of row-major matrices with a padded leading dimension.
struct MatView {
    const void *ptr = nullptr;
    int rows = 0, cols = 0;     // logical
    long long ld = 0;           // elements between rows
    long long bstride = 0;      // elements between batch entries
    int batch = 1;
    bool bf16 = false, f16 = false;
};

// The four split-FP16 views of a product (PREC_F16X3).
struct F16Views {
    MatView ah, al, bh, bl;
};

// Encodes a TMA descriptor: box = box_rows rows x 128 B (32 fp32 / 64 bf16), 128-byte
// swizzle, zero fill outside [cols] x [rows].  Returns false if the driver rejects it.
bool make_tmap(CUtensorMap *out, const MatView &v, int box_rows = 128);

void count_launch(int n = 1);
int cuda_fail(cudaError_t e, const char *file, int line);
int num_sms();

// Optional per-launch timing of the product kernel (CUDA events on the launching
// stream); `flops` is the algorithmic count of the launch, `prec` its class.
void prof_begin(cudaStream_t st);
void prof_end(cudaStream_t st, double flops, int prec);
bool prof_on();

// Host copy of the tile count (same enumeration as the device).
inline int host_tiles_per_matrix(const GemmShape &s) {
    if (!s.sym) return s.tiles_m * s.tiles_n;
    int c = 0;
    for (int r = 0; r < s.tiles_m; ++r) c += s.tiles_n - (kBM * r) / s.bn;
    return c;
}

// What a launch needs besides its epilogue: the tensor maps and the tile list.  A loop that launches the
// same product many times plans it once.
struct GemmPlan {
    GemmMaps maps;
    GemmShape shp;
    int grid = 0;
};

inline cudaError_t plan_gemm(GemmPlan &plan, const MatView *a16, const MatView *b16, const MatView *ahi,
                             const MatView *alo, const MatView *bhi, const MatView *blo, const GemmShape &shape,
                             int batch, const F16Views *f16) {
    GemmShape &shp = plan.shp;
    shp = shape;
    shp.bn = shp.N > 128 ? 256 : 128;
    // A launch with fewer tiles than half the SMs is bound by one tile's serial chain, above all its
    // epilogue: narrower tiles put more CTAs to work on it.  (Whole polar decompositions with
    // tiles down to 128 / 64 / 32 columns, us: 256 x 256 684 / 614 / 564, 1024 x 256 814 / 748 / 679, two of
    // 1500 x 700 1045 / 1007 / 965.)
    while (shp.bn > kMinBN) {
        GemmShape t = shp;
        t.tiles_m = (t.M + kBM - 1) / kBM;
        t.tiles_n = (t.N + t.bn - 1) / t.bn;
        const long long tiles = (long long)host_tiles_per_matrix(t) * (shp.ksplit > 1 ? shp.ksplit : 1) * batch;
        if (2 * tiles > num_sms()) break;
        shp.bn /= 2;
    }
    GemmMaps &maps = plan.maps;
    memset(&maps, 0, sizeof(maps));
    // A map that is not supplied stays zero; the kernel only reads those of the precisions its tiles have.
    auto encode = [&](CUtensorMap *m, const MatView *v, int rows) { return !v || make_tmap(m, *v, rows); };
    if (!(ahi && bhi) && !(a16 && b16) && !f16) {
        cuda_fail(cudaErrorInvalidValue, "launch_gemm: missing operand", __LINE__);
        return cudaErrorInvalidValue;
    }
    if (!encode(&maps.a_hi, ahi, kBM) || !encode(&maps.a_lo, alo, kBM) || !encode(&maps.a_bf16, a16, kBM) ||
        !encode(&maps.b_hi, bhi, shp.bn) || !encode(&maps.b_lo, blo, shp.bn) || !encode(&maps.b_bf16, b16, shp.bn) ||
        (f16 && (!make_tmap(&maps.a_h16, f16->ah) || !make_tmap(&maps.a_l16, f16->al) ||
                 !make_tmap(&maps.b_h16, f16->bh, shp.bn) || !make_tmap(&maps.b_l16, f16->bl, shp.bn)))) {
        cuda_fail(cudaErrorInvalidValue, "tensor map encode", __LINE__);
        return cudaErrorInvalidValue;
    }
    shp.tiles_m = (shp.M + kBM - 1) / kBM;
    shp.tiles_n = (shp.N + shp.bn - 1) / shp.bn;
    shp.batch = batch;
    plan.grid = 0;
    if (shp.tiles_m == 0 || shp.tiles_n == 0 || batch == 0) return cudaSuccess;
    const long long total = (long long)host_tiles_per_matrix(shp) * (shp.ksplit > 1 ? shp.ksplit : 1) * batch;
    plan.grid = (int)std::min<long long>(total, num_sms());
    return cudaSuccess;
}

// `configure`: set the kernel's shared memory limit (needed once before a loop of launches).  It is set through
// the same kernel handle the launch below uses: each .cu file that instantiates this template registers its own
// copy of the kernel, so a process-wide "already configured" flag, or a function of its own, would leave other
// copies unconfigured.
template <class Epi>
cudaError_t launch_plan(const GemmPlan &plan, const Epi &epi, cudaStream_t st, bool configure = true) {
    const GemmShape &shp = plan.shp;
    if (plan.grid == 0) return cudaSuccess;
    if (configure) {
        cudaError_t e = cudaFuncSetAttribute(gemm_tn_kernel<Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kGemmSmem);
        if (e != cudaSuccess) { cuda_fail(e, __FILE__, __LINE__); return e; }
    }
    const bool prof = prof_on();
    if (prof) prof_begin(st);
    // Programmatic dependent launch: the grid is set up while the kernel before it still runs (its
    // CTAs wait at their first instruction), which takes the launch latency out of the chains of
    // short products of small matrices and of the polar steps that find nothing to do.
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)plan.grid);
    cfg.blockDim = dim3(kGemmThreads);
    cfg.dynamicSmemBytes = kGemmSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    {
        cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_tn_kernel<Epi>, plan.maps, shp, epi);
        if (e != cudaSuccess) { cuda_fail(e, __FILE__, __LINE__); return e; }
    }
    count_launch();
    if (prof) {
        // algorithmic flops: 2 M N K per matrix (M (M + 1) K for the symmetric Gram)
        const double f = shp.sym ? (double)shp.M * (shp.M + 1) * shp.K : 2.0 * shp.M * shp.N * (double)shp.K;
        prof_end(st, f * shp.batch, shp.prof_as > 0 ? shp.prof_as - 1 : (shp.prec ? -1 : std::min(shp.prec_uniform, (int)PREC_TF32X3)));
    }
    cudaError_t le = cudaGetLastError();
    if (le != cudaSuccess) cuda_fail(le, __FILE__, __LINE__);
    return le;
}

template <class Epi>
cudaError_t launch_gemm(const MatView *a16, const MatView *b16, const MatView *ahi, const MatView *alo,
                        const MatView *bhi, const MatView *blo, const GemmShape &shp, int batch, const Epi &epi,
                        cudaStream_t st, const F16Views *f16 = nullptr) {
    GemmPlan plan;
    const cudaError_t e = plan_gemm(plan, a16, b16, ahi, alo, bhi, blo, shp, batch, f16);
    return e != cudaSuccess ? e : launch_plan(plan, epi, st);
}

}  // namespace psvd
