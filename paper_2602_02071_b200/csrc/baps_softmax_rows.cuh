// Row softmax by Algorithm 1 with one query row per "tile" and no value product (the
// non-fused path).  One CTA owns one row at a time:
//   pass 1  read the row from HBM, reduce the maximum of every block_k block into shared memory;
//   scan    one warp walks the blocks in order and applies the max bookkeeping of Algorithm 1
//           (block 0: m = ceil(max); later blocks: T = HiF8(max - m), restart if T > lambda,
//           else m += max(0, ceil(T))).  The state is one integer per row and only changes
//           at blocks whose maximum exceeds it, so the warp tests 32 blocks per ballot;
//   pass 2  form the 8-bit weights, reduce d;
//   pass 3  write p = w * 2^(m_block - m_final) / d.
// Rows of up to 1152 columns are handled by one warp each (softmax_rows_warp_kernel), rows of up to 8K columns
// by groups of threads that share a CTA and its tables (softmax_rows_group_kernel), rows of up to 32K by one
// CTA each, fed through a shared-memory ring by bulk asynchronous copies so that the read of the next row
// overlaps the passes over the current one, longer rows by one CTA that keeps half the row in registers and
// half in the shared-memory pieces it arrived in.  In all of these the row stays on chip between the passes,
// so HBM traffic is exactly one read and one write of the row (8 bytes per element).  FULL instances know
// the row length (a power of two, or up to 1152 columns) at compile time; the others take it as an
// argument and leave out the 128-column chunks past the end.  (Measured on 2^27 logits against a variant that
// re-read every row twice from L2: 640 columns 720 -> 167 us, 3200 397 -> 179, 12800 304 -> 180, 49152 280 -> 217.)
// Blocks whose T are all <= 0 (nearly all of them) take the weights from a bank-replicated table keyed
// by the top bits of -T * 2^-120, as the fused attention kernel does.  What a block's weights need --
// the max its T are taken against, the power of two that moves them to the final max, which table --
// is worked out once per block by one lane and handed round by shuffles.
#pragma once
#include "baps_common.cuh"
#include "baps_hif8.cuh"
#include "baps_tables.cuh"
#include "baps_sm100.cuh"

namespace baps {

// Max bookkeeping of Algorithm 1 for one block of a single row: given the running max m
// (integer valued, or -inf before block 0) and the block's largest logit xmax (base-2 score
// xmax * log2(e)), return the new max.  *restart is set when the restart branch was taken.
// T of the maximum is formed exactly as for every other element (one fused multiply-add).
// (The max may be -0, which ceilf gives for scores in (-1, 0).)
__device__ __forceinline__ float row_block_update(float m, float xmax, bool first, int lambda,
                                                  bool *restart, float *delta)
{
    *restart = false; *delta = 0.f;
    if (first) return fmaxf(m, ceilf(xmax * kLog2e));
    const float u = fmaf(xmax, kLog2e, -m);
    if (u <= 0.f) return m;                     // T8 <= 0: no restart, delta = 0 (the common case)
    const float t8 = hif8_round(u);
    if (t8 > (float)lambda) { *restart = true; return fmaxf(m, ceilf(xmax * kLog2e)); }
    const float d = fmaxf(0.f, ceilf(t8));
    *delta = d;
    return m + d;
}

// Maximum over the LPB lanes that hold one block.  LPB = 32 (the whole warp): one reduction instruction
// (REDUX) or five shuffles -- which of the two is faster depends on the kernel around it (measured: the
// instruction wins by 5 to 10 % in most variants and loses as much in the 4K-column group variant and the
// 16K-column ring variant), so the callers choose.  LPB = 16: the two halves of the warp, by shuffles.
template <int LPB, bool REDUX = true>
__device__ __forceinline__ float lanes_max(float mx)
{
    if constexpr (LPB == 32 && REDUX) {
        float r;
        asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(mx));
        return r;
    } else {
#pragma unroll
        for (int o = LPB / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        return mx;
    }
}

// What the weights pass needs to know about the blocks a warp holds, worked out once per block by one lane
// (block j, if `mine`; gm: the max before its group, see scan_groups, or NaN) and left in place of the block's maximum
// and the max before it:
//   x = (the max the block's T are taken against: after a restart or in block 0 the new one, otherwise the old
//       one) * 2^-120, the addend of the table key (exact: that max is an integer; + 0, because against -0 the key of
//       a logit of exactly 0 would be that of -0, a positive T's);
//   y = the power of two that moves the block's weights to the row's final max; with the old max as the
//       reference, 2^-delta 2^(m_after - m_final) = 2^(m_before - m_final).
// Read back with one 8-byte load per vector, the same address in all lanes of a block (three shuffles per
// vector before: the row kernels are bound by instructions issued, not by HBM).  8-bit output: also the
// block's integer exponent.  Returns, as a mask over the lanes' blocks, which of them hold a positive T -- for
// BPW = 2 (two blocks per vector) which of them share a vector with such a block.
constexpr float kTiny = 7.52316384526264e-37f, kHuge = 1.329227995784916e36f;       // 2^-120, 2^120
constexpr float kNoGroup = __builtin_nanf("");
template <int BPW, bool CODES>
__device__ __forceinline__ unsigned prepare_blocks(float2 *s_blk, float gm, int j, bool mine, int lambda, float mfinal, int32_t *block_exp)
{
    bool pos = false;
    if (mine) {
        float2 b = s_blk[j];
        if (gm == gm) b.y = gm;                     // no block of the group moved the max
        const bool first = j == 0;
        bool rs; float dl;
        const float ma = row_block_update(b.y, b.x, first, lambda, &rs, &dl);
        const float mref = (first || rs) ? ma : b.y;
        s_blk[j] = make_float2(fmaf(mref, kTiny, 0.f), exp2f(mref - mfinal));
        if (CODES) block_exp[j] = (int)(mref - mfinal);
        pos = (CODES || !first) && fmaf(b.x, kLog2e, -mref) > 0.f;
    }
    unsigned mask = __ballot_sync(0xffffffffu, pos);
    if (BPW == 2) mask |= ((mask & 0x55555555u) << 1) | ((mask >> 1) & 0x55555555u);
    __syncwarp();
    return mask;
}

// Table words of one 16-byte vector (float output: the fp32 pattern of w0; 8-bit output: the pattern with the
// code in its low byte); mtiny = the block's max * 2^-120.  Blocks whose T are all <= 0: x = -T * 2^-120 by
// packed fused multiply-adds with flush-to-zero (|T| < 2^-6 becomes +0, weight 1), the top bits of x select
// the entry of the bank-replicated table (everything from |T| >= 32 on is the entry 0; rep = the lane's copy).
__device__ __forceinline__ uint4 table_words(const float4 &x, float mtiny, bool any_pos, uint32_t rep, const uint32_t *s_lut)
{
    uint4 e;
    if (!any_pos) {
        const uint64_t cn2 = pack2(-kLog2e * kTiny, -kLog2e * kTiny), mn2 = pack2(mtiny, mtiny);
        float t0, t1, t2, t3;
        unpack2(fma2_ftz(pack2(x.x, x.y), cn2, mn2), t0, t1);
        unpack2(fma2_ftz(pack2(x.z, x.w), cn2, mn2), t2, t3);
        e.x = lds_u32(min(__float_as_uint(t0) >> 19, 192u) * 128u + rep);
        e.y = lds_u32(min(__float_as_uint(t1) >> 19, 192u) * 128u + rep);
        e.z = lds_u32(min(__float_as_uint(t2) >> 19, 192u) * 128u + rep);
        e.w = lds_u32(min(__float_as_uint(t3) >> 19, 192u) * 128u + rep);
    } else {
        const float mref = mtiny * kHuge;
        e.x = s_lut[w0_index(fmaf(x.x, kLog2e, -mref))]; e.y = s_lut[w0_index(fmaf(x.y, kLog2e, -mref))];
        e.z = s_lut[w0_index(fmaf(x.z, kLog2e, -mref))]; e.w = s_lut[w0_index(fmaf(x.w, kLog2e, -mref))];
    }
    return e;
}

// Float output: weights of one vector against its block's own max.  block0: the vector belongs to block 0
// of the row, which is kept in high precision.
__device__ __forceinline__ float4 vector_weights(const float4 &x, float mtiny, bool any_pos, bool block0, uint32_t rep,
                                                 const uint32_t *s_lut)
{
    if (block0) {
        const float mref = mtiny * kHuge;
        return make_float4(exp2f(fmaf(x.x, kLog2e, -mref)), exp2f(fmaf(x.y, kLog2e, -mref)),
                           exp2f(fmaf(x.z, kLog2e, -mref)), exp2f(fmaf(x.w, kLog2e, -mref)));
    }
    const uint4 e = table_words(x, mtiny, any_pos, rep, s_lut);
    return make_float4(__uint_as_float(e.x), __uint_as_float(e.y), __uint_as_float(e.z), __uint_as_float(e.w));
}
__device__ __forceinline__ float sum4(const float4 &w) { return (w.x + w.y) + (w.z + w.w); }
__device__ __forceinline__ void store_scaled(float4 *dst, const float4 &w, float f)
{
    const uint64_t f2 = pack2(f, f);
    float4 o;
    unpack2(mul2(pack2(w.x, w.y), f2), o.x, o.y);
    unpack2(mul2(pack2(w.z, w.w), f2), o.z, o.w);
    __stcs(dst, o);
}

// The scan of Algorithm 1's max bookkeeping over the nb block maxima of one row (s_blk[j].x), by one warp:
// writes the running max before every block (s_blk[j].y) and the final max.  The state is one integer per row and only changes at
// blocks whose maximum exceeds it, so the warp tests 32 blocks per ballot.  (The loop over the groups of
// 32 blocks is kept rolled: unrolled, with the inner loop and the update inlined four or more times, the
// same kernel ran 20 % slower.)
__device__ __forceinline__ void scan_blocks(int nb, float2 *s_blk, float *s_mfinal, int lambda, int lane)
{
    bool rs; float dl;
    float m = row_block_update(-INFINITY, s_blk[0].x, true, lambda, &rs, &dl);
    if (lane == 0) s_blk[0].y = -INFINITY;
#pragma unroll 1
    for (int base = 1; base < nb; base += 32) {
        const int j = base + lane;
        const bool valid = j < nb;
        const float mj = valid ? s_blk[j].x : -INFINITY;
        bool pending = valid;
        while (true) {
            // HiF8(T) > 0  <=>  T >= 2^-23 (smaller magnitudes round to zero)
            const bool pred = pending && fmaf(mj, kLog2e, -m) >= 1.1920928955078125e-07f;
            const unsigned b = __ballot_sync(0xffffffffu, pred);
            if (b == 0u) { if (pending) s_blk[j].y = m; break; }
            const int l = __ffs(b) - 1;
            if (pending && lane <= l) { s_blk[j].y = m; pending = false; }
            const float ml = __shfl_sync(0xffffffffu, mj, l);
            m = row_block_update(m, ml, false, lambda, &rs, &dl);
        }
    }
    if (lane == 0) *s_mfinal = m;
}

// The same scan for rows of several hundred blocks: the warp looks for the blocks that change the max -- a
// handful per row -- among the maxima of whole groups first (a group: the consecutive blocks of one warp, s_gmax[g] their largest maximum;
// 32 groups per ballot) and goes through the blocks of a group only where there is one.  Writes the running max
// before every group (s_gm[g]) -- for the groups with such a block NaN, which m never is, and the max before
// each of their blocks to s_blk[j].y instead -- and the final max.  Block j has group j / bpg.  Measured on 2^27
// logits: 64K columns 197 -> 191 us, 8-bit output 136 -> 126; up to 256 blocks the plain scan is the faster one
// (16K columns with 8-bit output 112 against 129 us).
__device__ __forceinline__ void scan_groups(int ngroups, int bpg, int nb, float2 *s_blk, const float *s_gmax, float *s_gm,
                                            float *s_mfinal, int lambda, int lane)
{
    constexpr float kUp = 1.1920928955078125e-07f;      // HiF8(T) > 0  <=>  T >= 2^-23 (smaller magnitudes round to zero)
    bool rs; float dl;
    float m = row_block_update(-INFINITY, s_blk[0].x, true, lambda, &rs, &dl);
    if (lane == 0) s_blk[0].y = -INFINITY;
#pragma unroll 1
    for (int base = 0; base < ngroups; base += 32) {
        const int g = base + lane;
        bool pending = g < ngroups;
        const float gx = pending ? s_gmax[g] : -INFINITY;
#pragma unroll 1
        while (true) {
            const unsigned b = __ballot_sync(0xffffffffu, pending && (g == 0 || fmaf(gx, kLog2e, -m) >= kUp));
            if (b == 0u) { if (pending) s_gm[g] = m; break; }
            const int l = __ffs(b) - 1;
            if (pending && lane <= l) { s_gm[g] = lane < l ? m : __int_as_float(0x7fc00000); pending = false; }
            const int j = (base + l) * bpg + lane;
            bool in = lane < bpg && j < nb && j > 0;
            const float bx = in ? s_blk[j].x : -INFINITY;
#pragma unroll 1
            while (true) {
                const unsigned bb = __ballot_sync(0xffffffffu, in && fmaf(bx, kLog2e, -m) >= kUp);
                if (bb == 0u) { if (in) s_blk[j].y = m; break; }
                const int ll = __ffs(bb) - 1;
                if (in && lane <= ll) { s_blk[j].y = m; in = false; }
                m = row_block_update(m, __shfl_sync(0xffffffffu, bx, ll), false, lambda, &rs, &dl);
            }
        }
    }
    if (lane == 0) *s_mfinal = m;
}

// Float output of whole power-of-two rows in 128-column blocks: these kernels run at the copy bandwidth, and what the
// fewer instructions of the form above save them they lose in HBM.  With the weights moved to the final max in the second
// pass (not together with the division in the third) and the block parameters handed round by shuffles, 2^27 / 2^28
// logits take at 4K columns 167 / 337 us instead of 172 / 348, at 16K 176 / 351 instead of 178 / 359, at 32K 170 / 327
// instead of 175 / 353.  64-column blocks, 8-bit output and other lengths lose 2 to 5 % by it (3200 columns 175 -> 180).
template <int BK, bool CODES, bool FULL>
constexpr bool kScaledEarly = !CODES && BK == 128 && FULL;

// Largest maximum of a warp's vector (mx: the lane's block), kept by the lanes for the group's.
template <int BPW>
__device__ __forceinline__ float whole_warp_max(float mx)
{
    return BPW == 1 ? mx : fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
}

// Bulk asynchronous copy of one row (or part of one) into shared memory, completion counted on an
// mbarrier: in pieces of at most 32 KB, all on the same barrier.
__device__ __forceinline__ void bulk_load_row(uint32_t dst, const float *src, uint32_t bytes, uint32_t bar)
{
    for (uint32_t off = 0; off < bytes; off += 32768u) {
        const uint32_t n = bytes - off < 32768u ? bytes - off : 32768u;
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(dst + off), "l"(reinterpret_cast<const float *>(src) + off / 4), "r"(n), "r"(bar)
                     : "memory");
    }
}

// Table words of the 8-bit-output kernels: the fp32 pattern of w0(T) with its HiF8 code in the low byte.
__device__ __forceinline__ uint32_t w0_word(float w) { return __float_as_uint(w) | (uint32_t)hif8_pack(w); }

// Where a row kernel writes: probabilities (float output), or codes, block exponents and denominators
// (8-bit output; see the description further down).
struct RowsOut {
    float *probs;
    uint8_t *codes;
    int32_t *block_exp;
    float *row_d;
};

// Tables of a CTA in shared memory, as words (w0_word above for the 8-bit output).
template <bool CODES>
__device__ __forceinline__ void fill_tables(uint32_t *s_lut, uint32_t *s_rep, int t, int nthreads)
{
    for (int i = t; i < kLutN; i += nthreads) s_lut[i] = CODES ? w0_word(g_w0.v[i]) : __float_as_uint(g_w0.v[i]);
    for (int e = t; e < 16 + kLutNegN; e += nthreads) {
        const float w = (e < 16) ? 1.f : g_w0.v[e - 16];
        const uint32_t u = CODES ? w0_word(w) : __float_as_uint(w);
        const uint4 u4 = make_uint4(u, u, u, u);
#pragma unroll
        for (int i = 0; i < 8; ++i) reinterpret_cast<uint4 *>(s_rep)[e * 8 + i] = u4;
    }
}

// 8-bit output of one vector: its table words -> four codes (stored), returns the sum of the decoded weights.
__device__ __forceinline__ float emit_codes(uint32_t *dst, const uint4 &e)
{
    __stcs(dst, __byte_perm(__byte_perm(e.x, e.y, 0x0040), __byte_perm(e.z, e.w, 0x0040), 0x5410));
    return (__uint_as_float(e.x & 0xFFFFFF00u) + __uint_as_float(e.y & 0xFFFFFF00u)) +
           (__uint_as_float(e.z & 0xFFFFFF00u) + __uint_as_float(e.w & 0xFFFFFF00u));
}

__device__ __forceinline__ float warp_sum(float x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Long rows (up to 16K, 32K columns): one CTA per row at a time with the row in registers (32 floats per
// thread: 512 threads for 16K, two CTAs per SM; 1024 threads for 32K), fed through a one-row
// shared-memory ring by bulk asynchronous copies (cp.async.bulk, completion on an mbarrier) that one
// thread issues as soon as the current row sits in registers, i.e. after the first barrier of the row:
// the HBM read of the next row overlaps the scan, the weights and the write of the current one.
// Three barriers per row.  CODES: 8-bit output.
template <int BK, int THREADS, bool CODES, bool REDUX = true, bool FULL = true>
__global__ void __launch_bounds__(THREADS, 2048 / THREADS / 2)
softmax_rows_ring_kernel(const float *__restrict__ logits, RowsOut out, int64_t rows, int lambda, int cols_)
{
    constexpr int NV = 8, kCols = NV * THREADS * 4;
    constexpr int LPB = BK / 4, BPW = 32 / LPB;
    const int cols = FULL ? kCols : cols_, nch = cols / 128, nb = cols / BK;
    const int nwarps = FULL ? THREADS / 32 : blockDim.x / 32;    // a warp per NV chunks
    const uint32_t row_bytes = (uint32_t)cols * 4u;
    static_assert(NV * BPW <= 32, "one block per lane");
    extern __shared__ __align__(128) uint8_t sr_ring[];          // one row
    __shared__ __align__(8) uint64_t s_full;
    __shared__ int s_abort;
    __shared__ float2 s_blk[kCols / BK];
    __shared__ uint32_t s_lut[kLutN];
    __shared__ __align__(16) uint32_t s_rep[(16 + kLutNegN) * 32];
    __shared__ float s_red[THREADS / 32];
    __shared__ float s_mfinal;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rep = sm100::smem_u32(s_rep) + (uint32_t)lane * 4u;
    allow_next_kernel();
    fill_tables<CODES>(s_lut, s_rep, tid, nwarps * 32);
    logits = await_previous_kernel(logits);
    if (tid == 0) {
        sm100::mbar_init(sm100::smem_u32(&s_full), 1);
        sm100::mbar_fence_init();
        s_abort = 0;
    }
    __syncthreads();
    if (tid == 0 && (int64_t)blockIdx.x < rows) {
        sm100::mbar_arrive_expect_tx(sm100::smem_u32(&s_full), row_bytes);
        bulk_load_row(sm100::smem_u32(sr_ring), logits + (int64_t)blockIdx.x * cols, row_bytes, sm100::smem_u32(&s_full));
    }
    // my warp's k-th chunk of 128 columns; with a run-time number of warps consecutive ones, so that every
    // address is the warp's plus a constant (dealt out round-robin they cost 20 % there; with a compile-time
    // number of warps round-robin is 1 to 3 % the faster)
    auto chunk = [&](int k) { return FULL ? warp + k * nwarps : warp * NV + k; };
    auto has = [&](int k) { return FULL || chunk(k) < nch; };

    int it = 0;
    for (int64_t row = blockIdx.x; row < rows; row += gridDim.x, ++it) {
        float4 v[NV];
        // ---- pass 1: the row into registers, block maxima ----------------------------------------------
        // bounded wait; after a time-out the kernel runs on (on stale data) so that every thread keeps
        // meeting the same barriers, and the status word reports the failure
        sm100::mbar_wait(sm100::smem_u32(&s_full), (uint32_t)(it & 1), &s_abort, &g_async_status, 0x400);
        {
            const float4 *ring4 = reinterpret_cast<const float4 *>(sr_ring);
#pragma unroll
            for (int k = 0; k < NV; ++k)
                if (has(k)) v[k] = ring4[chunk(k) * 32 + lane];
        }
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            if (!has(k)) break;
            const float mx = lanes_max<LPB, REDUX>(fmaxf(fmaxf(v[k].x, v[k].y), fmaxf(v[k].z, v[k].w)));
            if ((lane % LPB) == 0) s_blk[chunk(k) * BPW + lane / LPB].x = mx;
        }
        __syncthreads();
        if (tid == 0) {
            const int64_t rn = row + gridDim.x;             // the ring takes the next row
            if (rn < rows) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                sm100::mbar_arrive_expect_tx(sm100::smem_u32(&s_full), row_bytes);
                bulk_load_row(sm100::smem_u32(sr_ring), logits + rn * cols, row_bytes, sm100::smem_u32(&s_full));
            }
        }
        // ---- scan over the blocks (warp 0) ---------------------------------------------------------------
        if (warp == 0) scan_blocks(nb, s_blk, &s_mfinal, lambda, lane);
        __syncthreads();
        const int jmine = chunk(lane / BPW) * BPW + lane % BPW;      // the block whose parameters I work out
        const unsigned slow = prepare_blocks<BPW, CODES>(s_blk, kNoGroup, jmine, lane < NV * BPW && (FULL || jmine < nb), lambda, s_mfinal,
                                                         CODES ? out.block_exp + row * nb : nullptr);
        constexpr bool kEarly = kScaledEarly<BK, CODES, FULL>;
        const float2 own = kEarly && lane < NV * BPW ? s_blk[jmine] : make_float2(0.f, 0.f);
        float dsum = 0.f;
        // ---- pass 2: weights against the block's own max (8-bit output: codes), their sum against the final max
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            if (!has(k)) break;
            const float2 bp = kEarly ? make_float2(__shfl_sync(0xffffffffu, own.x, k * BPW + lane / LPB),
                                                   __shfl_sync(0xffffffffu, own.y, k * BPW + lane / LPB))
                                     : s_blk[chunk(k) * BPW + lane / LPB];
            const bool any_pos = (slow >> (k * BPW)) & 1u;
            if constexpr (CODES) {
                uint32_t *c4 = reinterpret_cast<uint32_t *>(out.codes + row * cols);
                dsum = fmaf(emit_codes(c4 + chunk(k) * 32 + lane, table_words(v[k], bp.x, any_pos, rep, s_lut)), bp.y, dsum);
            } else {
                v[k] = vector_weights(v[k], bp.x, any_pos, k == 0 && warp == 0 && lane < LPB, rep, s_lut);
                if (kEarly) v[k] = make_float4(v[k].x * bp.y, v[k].y * bp.y, v[k].z * bp.y, v[k].w * bp.y);
                dsum = kEarly ? dsum + sum4(v[k]) : fmaf(sum4(v[k]), bp.y, dsum);
            }
        }
        dsum = warp_sum(dsum);
        if (lane == 0) s_red[warp] = dsum;
        __syncthreads();
        if constexpr (CODES) {
            if (warp == 0) {
                const float t = warp_sum(lane < nwarps ? s_red[lane] : 0.f);
                if (lane == 0) out.row_d[row] = t;
            }
        } else {
            // every warp adds the warps' partial sums itself, in the same order
            const float dinv = 1.f / warp_sum(lane < nwarps ? s_red[lane] : 0.f);
            // ---- pass 3 ---------------------------------------------------------------------------------
            float4 *p4 = reinterpret_cast<float4 *>(out.probs + row * cols);
#pragma unroll
            for (int k = 0; k < NV; ++k)
                if (has(k)) store_scaled(p4 + chunk(k) * 32 + lane, v[k], kEarly ? dinv : s_blk[chunk(k) * BPW + lane / LPB].y * dinv);
        }
        // (no barrier here: what the next row writes first, s_blk[].x, was last read before the third barrier
        // above; s_blk[].y, s_mfinal and s_red are written behind the next row's first and second barrier,
        // which every thread -- the one adding up s_red included -- joins only when it is done with this row)
    }
}

// Rows of more than 32K columns: one CTA of 1024 threads holds the whole row on chip, so HBM traffic stays one
// read and one write of the row and no barrier crosses SMs.  The row travels in four quarters of 16K columns
// (64 KB) through three shared-memory pieces.  Quarters 0 and 1 pass through the transit piece into registers
// (16 floats per thread each); quarters 2 and 3 stay in their pieces until the weights are formed.  The float
// output keeps the weights of the whole row in registers as packed bf16 (exact: an 8-bit value has at most
// four significant bits; block 0, in high precision, is formed again from its logits), so that the
// pieces of quarters 2 and 3 take the next row before the output is written.  The transit piece takes quarter 1
// once quarter 0 sits in registers and the next row's quarter 0 once quarter 1 does -- so of the next row only
// quarter 1 is waited for in the open.  Four barriers per row.
template <int BK, bool CODES, bool FULL = true>
__global__ void __launch_bounds__(1024, 1)
softmax_rows_quarters_kernel(const float *__restrict__ logits, RowsOut out, int64_t rows, int lambda, int cols_)
{
    constexpr int THREADS = 1024, NQ = 4, kWarps = THREADS / 32, kQuarter = NQ * THREADS * 4, kCols = 4 * kQuarter;
    constexpr int LPB = BK / 4, BPW = 32 / LPB, nbq = kQuarter / BK;
    const int cols = FULL ? kCols : cols_, nb = cols / BK;       // more than half of kCols
    // 128-column chunks of quarters 2 and 3 (the first two are whole)
    const int nch2 = FULL ? kQuarter / 128 : min(cols - 2 * kQuarter, kQuarter) / 128;
    const int nch3 = FULL ? kQuarter / 128 : max(cols - 3 * kQuarter, 0) / 128;
    constexpr uint32_t q_bytes = (uint32_t)kQuarter * 4u;
    static_assert(4 * NQ * BPW <= 32, "one block per lane");
    extern __shared__ __align__(128) uint8_t sr_ring[];          // three pieces of one quarter row each
    __shared__ __align__(8) uint64_t s_full[3];
    __shared__ int s_abort;
    __shared__ float2 s_blk[kCols / BK];
    __shared__ uint32_t s_lut[kLutN];
    __shared__ __align__(16) uint32_t s_rep[(16 + kLutNegN) * 32];
    __shared__ float s_red[kWarps];
    __shared__ float s_gmax[4 * kWarps], s_gm[4 * kWarps];       // group: a warp's blocks of one quarter
    __shared__ float s_mfinal;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rep = sm100::smem_u32(s_rep) + (uint32_t)lane * 4u;
    allow_next_kernel();
    fill_tables<CODES>(s_lut, s_rep, tid, THREADS);
    logits = await_previous_kernel(logits);
    if (tid == 0) {
        for (int i = 0; i < 3; ++i) sm100::mbar_init(sm100::smem_u32(&s_full[i]), 1);
        sm100::mbar_fence_init();
        s_abort = 0;
    }
    __syncthreads();
    // one thread: piece `pc` takes quarter `q` of row `r`
    auto request = [&](int pc, int64_t r, int q) {
        const uint32_t bytes = FULL || q < 2 ? q_bytes : (uint32_t)(q == 2 ? nch2 : nch3) * 512u;
        if (bytes == 0u) return;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        sm100::mbar_arrive_expect_tx(sm100::smem_u32(&s_full[pc]), bytes);
        bulk_load_row(sm100::smem_u32(sr_ring) + (uint32_t)pc * q_bytes, logits + r * cols + (int64_t)q * kQuarter, bytes,
                      sm100::smem_u32(&s_full[pc]));
    };
    if (tid == 0 && (int64_t)blockIdx.x < rows) {
        request(0, blockIdx.x, 0);
        request(1, blockIdx.x, 2);
        request(2, blockIdx.x, 3);
    }
    const float4 *piece[3] = {reinterpret_cast<const float4 *>(sr_ring), reinterpret_cast<const float4 *>(sr_ring + q_bytes),
                              reinterpret_cast<const float4 *>(sr_ring + 2 * q_bytes)};
    uint32_t ph0 = 0, ph1 = 0, ph2 = 0;         // phase parities of the three pieces (the same in every thread)
    // bounded waits; after a time-out the kernel runs on (on stale data) so that every thread keeps meeting
    // the same barriers, and the status word reports the failure
    auto wait_piece = [&](int pc, uint32_t &ph, int code) {
        sm100::mbar_wait(sm100::smem_u32(&s_full[pc]), ph & 1u, &s_abort, &g_async_status, code);
        ph ^= 1u;
    };
    // of every quarter a warp has NQ consecutive chunks of 128 columns (in quarters 2 and 3 perhaps fewer)
    auto has = [&](int q, int k) { return FULL || q < 2 || warp * NQ + k < (q == 2 ? nch2 : nch3); };
    const int vi0 = warp * NQ * 32 + lane;      // my vector k of a quarter is number vi0 + 32 k of it
    auto block_of = [&](int q, int k) { return q * nbq + (warp * NQ + k) * BPW + lane / LPB; };
    // the block whose parameters my lane works out: number lane % (NQ * BPW) of the warp's blocks of a quarter
    const int qmine = lane / (NQ * BPW) & 3, jmine = qmine * nbq + warp * NQ * BPW + lane % (NQ * BPW);
    auto quarter_max = [&](int q, auto vec) {
        float gmax = -INFINITY;
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            if (!has(q, k)) break;
            const float4 x = vec(k);
            const float mx = lanes_max<LPB>(fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)));
            if ((lane % LPB) == 0) s_blk[block_of(q, k)].x = mx;
            gmax = fmaxf(gmax, mx);
        }
        gmax = whole_warp_max<BPW>(gmax);
        if (lane == 0) s_gmax[q * kWarps + warp] = gmax;
    };

    for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
        const bool more = row + gridDim.x < rows;
        float4 v[2 * NQ];                       // quarters 0 and 1
        // ---- quarters 0 and 1: through the transit piece into registers, block maxima -----------------------
        wait_piece(0, ph0, 0x420);
#pragma unroll
        for (int k = 0; k < NQ; ++k) v[k] = piece[0][vi0 + k * 32];
        __syncthreads();
        if (tid == 0) request(0, row, 1);
        quarter_max(0, [&](int k) { return v[k]; });
        // ---- quarters 2 and 3: stay in their pieces; block maxima -------------------------------------------
        wait_piece(1, ph1, 0x422);
        quarter_max(2, [&](int k) { return piece[1][vi0 + k * 32]; });
        if (FULL || nch3 > 0) wait_piece(2, ph2, 0x423);
        quarter_max(3, [&](int k) { return piece[2][vi0 + k * 32]; });
        wait_piece(0, ph0, 0x421);
#pragma unroll
        for (int k = 0; k < NQ; ++k) v[NQ + k] = piece[0][vi0 + k * 32];
        quarter_max(1, [&](int k) { return v[NQ + k]; });
        __syncthreads();
        if (tid == 0 && more) request(0, row + gridDim.x, 0);
        if (warp == 0) scan_groups(4 * kWarps, NQ * BPW, nb, s_blk, s_gmax, s_gm, &s_mfinal, lambda, lane);
        __syncthreads();
        const unsigned slow = prepare_blocks<BPW, CODES>(s_blk, s_gm[qmine * kWarps + warp], jmine, lane < 4 * NQ * BPW && (FULL || jmine < nb), lambda, s_mfinal,
                                                         CODES ? out.block_exp + row * nb : nullptr);
        float dsum = 0.f;
        uint32_t pk[CODES ? 1 : 8 * NQ];        // float output: weights of the whole row, packed bf16
        float4 x0 = v[0];                       // the logits of block 0 (warp 0)
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) {
#pragma unroll
            for (int k = 0; k < NQ; ++k) {
                if (!has(qq, k)) break;
                const float2 bp = s_blk[block_of(qq, k)];
                const bool any_pos = (slow >> ((qq * NQ + k) * BPW)) & 1u;
                const float4 x = qq < 2 ? v[qq * NQ + k] : piece[qq - 1][vi0 + k * 32];
                if constexpr (CODES) {
                    uint32_t *c4 = reinterpret_cast<uint32_t *>(out.codes + row * cols);
                    dsum = fmaf(emit_codes(c4 + qq * (kQuarter / 4) + vi0 + k * 32, table_words(x, bp.x, any_pos, rep, s_lut)),
                                bp.y, dsum);
                } else {
                    const float4 w = vector_weights(x, bp.x, any_pos, qq == 0 && k == 0 && warp == 0 && lane < LPB, rep, s_lut);
                    dsum = fmaf(sum4(w), bp.y, dsum);
                    pk[2 * (qq * NQ + k)] = pack_bf16x2(w.x, w.y);
                    pk[2 * (qq * NQ + k) + 1] = pack_bf16x2(w.z, w.w);
                }
            }
        }
        dsum = warp_sum(dsum);
        if (lane == 0) s_red[warp] = dsum;
        __syncthreads();                        // nobody reads the pieces any more
        if (tid == 0 && more) { request(1, row + gridDim.x, 2); request(2, row + gridDim.x, 3); }
        if constexpr (CODES) {
            if (warp == 0) {
                const float t = warp_sum(s_red[lane]);
                if (lane == 0) out.row_d[row] = t;
            }
            // (s_blk[].x is written again behind the next row's waits; its readers are done, see the barrier above)
        } else {
            float4 *p4 = reinterpret_cast<float4 *>(out.probs + row * cols);
            const float dinv = 1.f / warp_sum(s_red[lane]);     // every warp adds the partial sums itself, in the same order
#pragma unroll
            for (int i = 0; i < 4 * NQ; ++i) {
                const int qq = i / NQ, k = i % NQ;
                if (!has(qq, k)) continue;
                const float2 bp = s_blk[block_of(qq, k)];
                float4 w = make_float4(__uint_as_float(pk[2 * i] << 16), __uint_as_float(pk[2 * i] & 0xFFFF0000u),
                                       __uint_as_float(pk[2 * i + 1] << 16), __uint_as_float(pk[2 * i + 1] & 0xFFFF0000u));
                if (i == 0 && warp == 0 && lane < LPB) w = vector_weights(x0, bp.x, false, true, rep, s_lut);
                store_scaled(p4 + qq * (kQuarter / 4) + vi0 + k * 32, w, bp.y * dinv);
            }
        }
        // (no barrier here: a warp writes s_blk[].x only for its own chunks, s_blk[].y, s_mfinal and s_red
        // are written behind the next row's second and third barrier)
    }
}

// Rows of up to 8K columns, several rows per CTA: GROUPS groups of THREADS threads each own one row
// at a time (register-resident, NV 16-byte vectors per thread; PF: the next row's loads always in flight,
// into a second set of registers) and share the CTA's tables; a group synchronises through its own
// hardware barrier (three per row), so the groups drift freely against each other.  With the tables
// shared, an SM holds as many rows in flight as its threads allow, where one-row CTAs stop at the six or
// seven copies of the 25 KB table that fit its shared memory.  CODES: 8-bit output.  FULL = false: groups of
// t_ <= THREADS threads, as few warps as hold the row, and as many of them as fit THREADS * GROUPS threads.
template <int BK, int THREADS, int NV, int GROUPS, bool CODES, bool PF = true, bool REDUX = true, bool FULL = true>
__global__ void __launch_bounds__(THREADS * GROUPS)
softmax_rows_group_kernel(const float *__restrict__ logits, RowsOut out, int64_t rows, int lambda, int cols_, int t_)
{
    constexpr int kMaxWarps = THREADS * GROUPS / 32;
    constexpr int LPB = BK / 4, BPW = 32 / LPB;
    const int cols = FULL ? NV * THREADS * 4 : cols_, nch = cols / 128, nb = cols / BK;
    const int nt = FULL ? THREADS : t_, nwarps = nt / 32, ngroups = FULL ? GROUPS : blockDim.x / nt;
    static_assert(GROUPS >= 1 && GROUPS <= 15 && NV * BPW <= 32, "barrier ids 1 .. 15; one block per lane");
    __shared__ float2 s_blk_all[kMaxWarps * NV * BPW];
    __shared__ uint32_t s_lut[kLutN];
    __shared__ __align__(16) uint32_t s_rep[(16 + kLutNegN) * 32];
    __shared__ float s_red_all[kMaxWarps];
    __shared__ float s_mfinal[15];
    allow_next_kernel();
    fill_tables<CODES>(s_lut, s_rep, threadIdx.x, nt * ngroups);
    logits = await_previous_kernel(logits);
    __syncthreads();
    const int grp = threadIdx.x / nt, tid = threadIdx.x % nt, lane = tid & 31, warp = tid >> 5;
    const uint32_t rep = sm100::smem_u32(s_rep) + (uint32_t)lane * 4u;
    float2 *const s_blk = s_blk_all + grp * nb;
    float *const s_red = s_red_all + grp * nwarps;
    auto gsync = [&] {
        asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "r"(nt) : "memory");
    };
    // my warp's k-th chunk of 128 columns: consecutive ones, so that every address is the warp's plus a constant
    // whatever the number of warps (dealt out round-robin, a run-time number of warps cost 20 %)
    auto chunk = [&](int k) { return warp * NV + k; };
    auto has = [&](int k) { return FULL || chunk(k) < nch; };
    const int64_t stride = (int64_t)gridDim.x * ngroups;
    int64_t row = (int64_t)blockIdx.x * ngroups + grp;
    float4 vn[PF ? NV : 1];
    if (PF && row < rows) {
        const float4 *x4 = reinterpret_cast<const float4 *>(logits + row * cols);
#pragma unroll
        for (int k = 0; k < (PF ? NV : 1); ++k)
            if (has(k)) vn[k] = __ldcs(x4 + chunk(k) * 32 + lane);
    }
    for (; row < rows; row += stride) {
        float4 v[NV];
        if constexpr (PF) {
#pragma unroll
            for (int k = 0; k < NV; ++k) v[k] = vn[k];
            if (row + stride < rows) {
                const float4 *xn = reinterpret_cast<const float4 *>(logits + (row + stride) * cols);
#pragma unroll
                for (int k = 0; k < NV; ++k)
                    if (has(k)) vn[k] = __ldcs(xn + chunk(k) * 32 + lane);
            }
        } else {
            const float4 *x4 = reinterpret_cast<const float4 *>(logits + row * cols);
#pragma unroll
            for (int k = 0; k < NV; ++k)
                if (has(k)) v[k] = __ldcs(x4 + chunk(k) * 32 + lane);
        }
        // ---- block maxima -------------------------------------------------------------------------
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            if (!has(k)) break;
            const float mx = lanes_max<LPB, REDUX>(fmaxf(fmaxf(v[k].x, v[k].y), fmaxf(v[k].z, v[k].w)));
            if ((lane % LPB) == 0) s_blk[chunk(k) * BPW + lane / LPB].x = mx;
        }
        gsync();
        // ---- scan over the blocks (the group's warp 0) ----------------------------------------------
        if (warp == 0) scan_blocks(nb, s_blk, &s_mfinal[grp], lambda, lane);
        gsync();
        const int jmine = warp * NV * BPW + lane;      // the block whose parameters I work out
        const unsigned slow = prepare_blocks<BPW, CODES>(s_blk, kNoGroup, jmine, lane < NV * BPW && (FULL || jmine < nb), lambda, s_mfinal[grp],
                                                         CODES ? out.block_exp + row * nb : nullptr);
        constexpr bool kEarly = kScaledEarly<BK, CODES, FULL>;
        const float2 own = kEarly && lane < NV * BPW ? s_blk[jmine] : make_float2(0.f, 0.f);
        float dsum = 0.f;
        // ---- weights against the block's own max (8-bit output: codes), their sum against the final max ----
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            if (!has(k)) break;
            const float2 bp = kEarly ? make_float2(__shfl_sync(0xffffffffu, own.x, k * BPW + lane / LPB),
                                                   __shfl_sync(0xffffffffu, own.y, k * BPW + lane / LPB))
                                     : s_blk[chunk(k) * BPW + lane / LPB];
            const bool any_pos = (slow >> (k * BPW)) & 1u;
            if constexpr (CODES) {
                uint32_t *c4 = reinterpret_cast<uint32_t *>(out.codes + row * cols);
                dsum = fmaf(emit_codes(c4 + chunk(k) * 32 + lane, table_words(v[k], bp.x, any_pos, rep, s_lut)), bp.y, dsum);
            } else {
                v[k] = vector_weights(v[k], bp.x, any_pos, k == 0 && warp == 0 && lane < LPB, rep, s_lut);
                if (kEarly) v[k] = make_float4(v[k].x * bp.y, v[k].y * bp.y, v[k].z * bp.y, v[k].w * bp.y);
                dsum = kEarly ? dsum + sum4(v[k]) : fmaf(sum4(v[k]), bp.y, dsum);
            }
        }
        dsum = warp_sum(dsum);
        if (lane == 0) s_red[warp] = dsum;
        gsync();
        // every thread adds the warps' partial sums itself, in the same order
        float t = 0.f;
        if constexpr (FULL) {
#pragma unroll
            for (int i = 0; i < THREADS / 32; ++i) t += s_red[i];
        } else {
            for (int i = 0; i < nwarps; ++i) t += s_red[i];
        }
        if constexpr (CODES) {
            if (tid == 0) out.row_d[row] = t;
        } else {
            const float dinv = 1.f / t;
            float4 *p4 = reinterpret_cast<float4 *>(out.probs + row * cols);
#pragma unroll
            for (int k = 0; k < NV; ++k)
                if (has(k)) store_scaled(p4 + chunk(k) * 32 + lane, v[k], kEarly ? dinv : s_blk[chunk(k) * BPW + lane / LPB].y * dinv);
        }
        // (no barrier here: what the next row writes first, s_blk[].x, was last read before the third barrier
        // above; s_blk[].y, s_mfinal and s_red are written behind the next row's first and second barrier,
        // which every thread -- the one adding up s_red included -- joins only when it is done with this row)
    }
}

// Short rows (up to 1152 columns; from ten chunks of 128 on the registers leave room for too few rows: 2^27
// logits at 1280 columns 200 us, 1152 columns 163): one warp per row, the row in registers, no block-wide barrier at all; ROWS
// consecutive rows per warp at a time so that short rows, too, keep enough loads in flight.
// Lane l holds the float4 number l of every 128-element chunk; a block of Algorithm 1 is a whole
// chunk (BK = 128) or half of one (BK = 64).  Block maxima by a warp reduction, the scan replicated in
// every lane (it is a handful of scalar steps per block), weights, warp-wide sum, write.  CODES: 8-bit output.
template <int BK, int NV, int ROWS, bool CODES>
__global__ void __launch_bounds__(512)
softmax_rows_warp_kernel(const float *__restrict__ logits, RowsOut out, int64_t rows, int lambda)
{
    constexpr int LPB = BK / 4, BPW = 32 / LPB;
    constexpr int cols = NV * 128, nb = cols / BK;
    static_assert(NV * BPW <= 32, "one block per lane");
    __shared__ uint32_t s_lut[kLutN];
    __shared__ __align__(16) uint32_t s_rep[(16 + kLutNegN) * 32];
    __shared__ float2 s_blk_all[16][NV * BPW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rep = sm100::smem_u32(s_rep) + (uint32_t)lane * 4u;
    float2 *const s_blk = s_blk_all[warp];
    allow_next_kernel();
    fill_tables<CODES>(s_lut, s_rep, tid, 512);
    logits = await_previous_kernel(logits);
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * 16 * ROWS;
    for (int64_t row0 = ((int64_t)blockIdx.x * 16 + warp) * ROWS; row0 < rows; row0 += step) {
        float4 vr[ROWS][NV];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            if (ROWS > 1 && row0 + r >= rows) break;
            const float4 *x4 = reinterpret_cast<const float4 *>(logits + (row0 + r) * cols);
#pragma unroll
            for (int k = 0; k < NV; ++k)
                vr[r][k] = __ldcs(x4 + k * 32 + lane);
        }
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int64_t row = row0 + r;
            if (ROWS > 1 && row >= rows) break;
            float4 (&v)[NV] = vr[r];
            float bmx[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                bmx[k] = lanes_max<LPB>(fmaxf(fmaxf(v[k].x, v[k].y), fmaxf(v[k].z, v[k].w)));    // of my block of chunk k
            }
            // scan over the blocks in order, identical in every lane; lane BPW * k + q keeps what block q of
            // vector k saw (its own maximum and the max before it)
            float m = -INFINITY;
            float2 mine = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
#pragma unroll
                for (int q = 0; q < BPW; ++q) {
                    const float bj = BPW == 1 ? bmx[k] : __shfl_sync(0xffffffffu, bmx[k], q * LPB);
                    if (lane == k * BPW + q) mine = make_float2(bj, m);
                    bool rs; float dl;
                    m = row_block_update(m, bj, k == 0 && q == 0, lambda, &rs, &dl);
                }
            }
            __syncwarp();                                        // the row before is done with s_blk
            if (lane < nb) s_blk[lane] = mine;
            const unsigned slow = prepare_blocks<BPW, CODES>(s_blk, kNoGroup, lane, lane < nb, lambda, m, CODES ? out.block_exp + row * nb : nullptr);
            float dsum = 0.f;
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const float2 bp = s_blk[k * BPW + lane / LPB];
                const bool any_pos = (slow >> (k * BPW)) & 1u;
                if constexpr (CODES) {
                    uint32_t *c4 = reinterpret_cast<uint32_t *>(out.codes + row * cols);
                    dsum = fmaf(emit_codes(c4 + k * 32 + lane, table_words(v[k], bp.x, any_pos, rep, s_lut)), bp.y, dsum);
                } else {
                    v[k] = vector_weights(v[k], bp.x, any_pos, k == 0 && lane < LPB, rep, s_lut);
                    dsum = fmaf(sum4(v[k]), bp.y, dsum);
                }
            }
            dsum = warp_sum(dsum);
            if constexpr (CODES) {
                if (lane == 0) out.row_d[row] = dsum;
            } else {
                float4 *p4 = reinterpret_cast<float4 *>(out.probs + row * cols);
                const float dinv = 1.f / dsum;
#pragma unroll
                for (int k = 0; k < NV; ++k)
                    store_scaled(p4 + k * 32 + lane, v[k], s_blk[k * BPW + lane / LPB].y * dinv);
            }
        }
    }
}

// Row softmax with 8-bit output: the weights leave as HiF8 codes (Algorithm 1's "P in 8-bit") with one
// integer exponent per block and one denominator per row,
//     probs[r, c] = value(codes[r, c]) * 2^(block_exp[r, c / BK]) / row_d[r],
// 5 bytes of HBM traffic per element (4 in, 1 out) instead of 8.  Same max bookkeeping as above; block 0
// is not kept in high precision here (its weights take the 8-bit exponential like all others: the
// output has 8 bits anyway).  block_exp = (max the block's T were taken against) - (final max) <= 0.
// The table entries carry value and code in one word: a HiF8 value has at most four significant mantissa
// bits, so the low byte of its fp32 pattern is free for the code.

// Launch the variant for the row length (see the head of this file).
// Grids: several times the CTAs that are resident at once (a few rows per CTA), so that the hardware
// scheduler evens out the SMs; measured on 2^28 logits, a grid of exactly the resident CTAs -- each
// with a fixed share of the rows -- loses 5 to 10 % to the slowest SM.  CTAs per SM, measured on 2^27 / 2^28 logits,
// float output: 4K columns 4 167 / 337 us, 6 170 / 332, 8 175 / 328 (64-column blocks: 4 168 / 332, 6 175 / 330);
// 16K columns 2 187 / 367, 4 176 / 351, 8 173 / 340, 12 179 / 338; 8-bit output 2 107 / 202, 8 114 / 209 and, at
// 4K columns, 4 115 / 215, 6 121 / 221.
// Up to 8K columns the rows are register-resident and several rows share a CTA and its tables
// (softmax_rows_group_kernel: 16 or 32 elements per thread); up to 1152 a warp per row needs no barrier at
// all.  At 16K and 32K only one or two CTAs fit an SM, and the ring lets the next row's read overlap
// the current row's passes.
template <int BK, bool CODES>
inline baps_status softmax_rows_dispatch(const float *logits, const RowsOut &out, int64_t rows, int cols, int lambda,
                                         int num_sms, cudaStream_t st)
{
    // a CTA per row.  The kernel's shared memory limit is state of the kernel, which other threads may be launching
    // with other row lengths: it is always set to the most the instance takes (kernel_most), the launch asks for `dyn`.
    auto ring = [&](auto kernel, int threads, int dyn, int kernel_most, int ctas_per_sm) -> baps_status {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kernel_most) != cudaSuccess)
            return BAPS_ERR_CUDA;
        const int64_t cap = (int64_t)num_sms * ctas_per_sm;
        return launch_kernel(kernel, (unsigned)(rows < cap ? rows : cap), threads, (size_t)dyn, st, logits, out, rows, lambda, cols);
    };
    // a group per row: `threads` of them (or, other lengths, as few warps as hold the row, NV chunks each)
    auto group = [&](auto kernel, int threads, int max_threads, int ctas) {
        const int groups = max_threads / threads < 15 ? max_threads / threads : 15;
        const int64_t want = (rows + groups - 1) / groups, cap = (int64_t)num_sms * ctas;
        return launch_kernel(kernel, (unsigned)(want < cap ? want : cap), threads * groups, 0, st, logits, out, rows, lambda, cols, threads);
    };
    auto warp_rows = [&](auto kernel, int rows_per_warp) {
        const int64_t want = (rows + 16 * rows_per_warp - 1) / (16 * rows_per_warp), cap = (int64_t)num_sms * 32;
        return launch_kernel(kernel, (unsigned)(want < cap ? want : cap), 512, 0, st, logits, out, rows, lambda);
    };
    const int nch = cols / 128, t4 = (nch + 3) / 4 * 32, t8 = (nch + 7) / 8 * 32;
    switch (cols) {
    case 128:   return warp_rows(softmax_rows_warp_kernel<BK, 1, 4, CODES>, 4);
    case 256:   return warp_rows(softmax_rows_warp_kernel<BK, 2, 4, CODES>, 4);
    case 384:   return warp_rows(softmax_rows_warp_kernel<BK, 3, 2, CODES>, 2);
    case 512:   return warp_rows(softmax_rows_warp_kernel<BK, 4, 2, CODES>, 2);
    case 640:   return warp_rows(softmax_rows_warp_kernel<BK, 5, 1, CODES>, 1);
    case 768:   return warp_rows(softmax_rows_warp_kernel<BK, 6, 1, CODES>, 1);
    case 896:   return warp_rows(softmax_rows_warp_kernel<BK, 7, 1, CODES>, 1);
    case 1024:  return warp_rows(softmax_rows_warp_kernel<BK, 8, 1, CODES>, 1);
    case 1152:  return warp_rows(softmax_rows_warp_kernel<BK, 9, 1, CODES>, 1);
    case 2048:  return group(softmax_rows_group_kernel<BK, 128, 4, 4, CODES, true>, 128, 512, 16);
    case 4096:  return group(softmax_rows_group_kernel<BK, 256, 4, 4, CODES, true, CODES>, 256, 1024, kScaledEarly<BK, CODES, true> ? 6 : 4);
    case 8192:  return group(softmax_rows_group_kernel<BK, 256, 8, 4, CODES, false>, 256, 1024, 4);
    case 16384: return ring(softmax_rows_ring_kernel<BK, 512, CODES, CODES>, 512, 65536, 65536, CODES ? 2 : 8);
    case 32768: return ring(softmax_rows_ring_kernel<BK, 1024, CODES>, 1024, 131072, 131072, 2);
    case 65536: return ring(softmax_rows_quarters_kernel<BK, CODES>, 1024, 196608, 196608, 2);
    }
    // Other lengths: as few warps per row as hold it, NV consecutive chunks of 128 columns each (every test
    // for the end of the row is the same for a whole warp).  Four chunks per warp and the next row's loads
    // in flight up to 1536 columns, eight from there on (2^27 logits, float / 8-bit output: 1536 columns 176 /
    // 161 us against 179 / 170, 1920 columns 183 / 183 against 176 / 144).
    if (cols <= 1536) return group(softmax_rows_group_kernel<BK, 256, 4, 4, CODES, true, true, false>, t4, 1024, 4);
    if (cols < 8192) return group(softmax_rows_group_kernel<BK, 256, 8, 4, CODES, false, true, false>, t8, 1024, 4);
    if (cols < 16384) return ring(softmax_rows_ring_kernel<BK, 512, CODES, true, false>, t8, cols * 4, 65536, 4);
    if (cols < 32768) return ring(softmax_rows_ring_kernel<BK, 1024, CODES, true, false>, t8, cols * 4, 131072, 2);
    return ring(softmax_rows_quarters_kernel<BK, CODES, false>, 1024, 196608, 196608, 2);
}

} // namespace baps
