// Fused BAPS attention forward on the 5th-generation tensor cores (tcgen05, sm_100a).
//
// (Algorithm 1 with two query tiles per CTA is paired_attention_tc_kernel's; this kernel serves small grids, B0 = {first,
// last} and the exact and Exp2 modes, and holds what all of them share.)
// One CTA owns two consecutive 128-row query tiles (t = 0, 1; small grids: one, see one_tile_per_cta) of one
// (batch, head) and walks the key tiles j in increasing order (Algorithm 1: tile 0 is the high-precision set B0, all later
// tiles are 8-bit tiles).  The unit of work is a task (t, j): S = Q_t K_j^T, softmax bookkeeping
// and weights P, O_t += P V_j.  Tasks run in the order (0,0) (1,0) (0,1) (1,1) ...; task k uses
// score buffer k % 2 of tensor memory, so the tensor core forms the scores of task k + 1 while
// the softmax warps work on task k, and no softmax warp ever waits for a product of its own
// previous task.  Roles, by warp (640 threads):
//   warps 0-15  softmax warps, all sixteen on the current task.  Warp w owns rows 32*(w%4) .. +31
//               (its TMEM lanes) and the 32 key columns of quarter w/4, i.e. a row is shared by
//               four threads.  Per task: read the 32 scores once into registers, quarter-row
//               maximum, exchange through shared memory; one reducing hardware barrier of the
//               sixteen warps orders the exchange and carries the tile-wide restart vote (B0 and
//               non-8-bit tiles: a plain barrier of the four warps of a lane quarter); decide
//               (B0 / restart / plain), form the weights
//               w = HiF8(2^HiF8(S*c - m~)) * 2^-delta through a bank-replicated table indexed by
//               the top bits of the fp32 pattern, and write them to TMEM as bf16 (exactly
//               representable) over score columns the thread itself has read.
//   warp 16     TMA producer: Q tiles once, then K_0, V_0, K_1, V_1, ... through a ring.
//   warp 17     MMA issuer: S = Q_t K_j^T (operands in shared memory, 128-byte swizzle) and
//               O_t += P V_j (P from TMEM, V as an MN-major shared operand), in bursts
//               PV(k), QK(k+2).  (Warps 18-19 idle: the fifth warpgroup exists so that its
//               registers can be handed to the softmax warps.)
// TMEM (512 columns): S buffer 0 | S buffer 1 | O_0 | O_1, 128 columns each (64 for O when
// D = 64).  The bf16 weights of column quarter q overwrite columns [32q, 32q + 16) of the buffer.
// Every wait on an mbarrier is bounded; on expiry the CTA raises an abort flag and records a code
// in the library's status word.  Every later wait then returns at once; the softmax warps still run
// through their task list so that the hardware barriers they share stay matched, and all roles
// meet at the common teardown.
#pragma once
#include <cuda_bf16.h>
#include "baps_common.cuh"
#include "baps_hif8.cuh"
#include "baps_register_split.cuh"
#include "baps_sm100.cuh"
#include "baps_tables.cuh"
#include "baps_tile_order.cuh"

namespace baps {

#ifdef BAPS_TEST_SKIP_LOAD
// Test build only (never defined for the product library): index of the K / V tile load that the
// TMA producer leaves out, so that the role waiting for that tile runs into its time limit.  -1: none.
__device__ int g_test_skip_load = -1;
#endif

struct AttnTcParams {
    __nv_bfloat16 *out;       // [B,H,S,D] or null
    float *out_f32;           // optional
    float *row_m, *row_d;     // optional [B,H,S]
    int32_t *restarts;        // optional [B,H,S/128]
    int B, H, Hkv, S, causal, lambda, mode;
    int b0_last;              // B0 = {first, last visible key tile}; one query tile per CTA
    const float *q_scale;     // 8-bit Q / K only: per query tile [B,H,S/128] and per key tile [B,Hkv,S/128]
    const float *k_scale;     // dequantisation scales (powers of two); null otherwise
    float c;                  // log2(e) * scale
    int nq, npairs;           // query tiles; work items per head (pairs of query tiles, or single tiles)
    KvChunks chunks;          // kv heads (of all batches) worked on together, see work_item
};

constexpr int kTcThreads = kTcSplit.threads;
constexpr int kTcSoftmaxWarps = kTcSplit.many_threads / 32;
constexpr int kLutRepEntries = 16 + kLutNegN;              // keys 0 .. 192, 32 copies each
constexpr int kLutRepBytes = kLutRepEntries * 128;

template <int D>
struct TcLayout {
    static constexpr int kTileBytes = 128 * D * 2;
    static constexpr int kStages = (D == 128) ? 4 : 8;
    static constexpr int kQOff = 0;
    static constexpr int kKvOff = 2 * kTileBytes;
    static constexpr int kLutRepOff = kKvOff + kStages * kTileBytes;
    static constexpr int kLutFullOff = kLutRepOff + kLutRepBytes;
    static constexpr int kBarOff = (kLutFullOff + kLutN * 4 + 15) & ~15;
    // barriers: q_full, s_full[2], p_full[2], pv_done[2], kv_full[stages], kv_empty[stages]
    static constexpr int kNumBars = 1 + 2 + 2 + 2 + 2 * kStages;
    static constexpr int kXchgOff = (kBarOff + kNumBars * 8 + 15) & ~15;   // float xchg[2][128][4]
    static constexpr int kMiscOff = kXchgOff + 2 * 128 * 4 * 4;            // tmem base, abort
    static constexpr int kTotal = kMiscOff + 16;
    static constexpr int kDynBytes = kTotal + 1024;                  // slack for 1024-byte alignment
};

__device__ __forceinline__ float lds_f32(uint32_t addr)
{
    float v;
    asm("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
// Global load that stays behind the wait for the kernel ahead (await_previous_kernel), as volatile statements do.
// (Not ld.global.nc, which asks for data that no kernel writes during this one's lifetime: that begins before the
// kernel ahead has ended.  And not for the compiler to move: 32 / 8 heads x 8192 with 8-bit Q / K 675 -> 712 us.)
__device__ __forceinline__ float ldg_f32(const float *p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// upper halves of two words as one: a's in the low half, b's in the high
__device__ __forceinline__ uint32_t upper_halves(float a, float b)
{
    return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}
__device__ __forceinline__ uint32_t min_u16x2(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
// low half of a * byte 0 of b + high half of a * byte 1 of b + c
__device__ __forceinline__ uint32_t dot_u16x2(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("dp2a.lo.u32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
// Hardware (named) barriers among the softmax warps: id 0 is __syncthreads.
__device__ __forceinline__ void named_bar_sync(uint32_t id, uint32_t nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
// Barrier that also ORs a predicate over all participating threads.
__device__ __forceinline__ bool named_bar_or(uint32_t id, uint32_t nthreads, bool pred)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.or.pred p, %2, %3, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)pred), "r"(id), "r"(nthreads)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ float4 lds_f32x4(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float2 lds_f32x2(uint32_t addr)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts_u32x4(uint32_t addr, uint4 v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint4 lds_u32x4(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts_f32(uint32_t addr, float v)
{
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
// 2^k for an integer-valued k (exact); 0 below the normal range, saturating far above it
__device__ __forceinline__ float pow2_int(float k)
{
    const int e = 127 + (int)k;
    return e > 0 ? __int_as_float(min(e, 254) << 23) : 0.f;
}

// ---- fast path -------------------------------------------------------------------------------
// Weights of 16 columns when every T = S*c - mref of the row is <= 0 (a plain 8-bit tile whose
// row maximum did not exceed the running max, or a restarted tile).
//   x   = -T * 2^-120, one packed FMA per two columns with flush-to-zero: x = +0 for
//         |T| < 2^-6 (weight 1), otherwise a normal number with biased exponent >= 1
//   key = min(bits(x) >> 19, 192): exponent and top four mantissa bits (what HiF8 rounding with
//         ties to the larger magnitude depends on); 192 stands for |T| >= 32 (weight 0) and is
//         also where a positive T lands (sign bit set) -- those entries are redone by the caller.
//         Two keys are cut out, limited and masked at once, as the halves of one word, each eight times
//         the key; the address of an entry's copy is then half * 16 + the lane's offset, one dot product
//         instruction.  (Shift, minimum and multiply-add per element took 749 cycles per 128 x 128 tile
//         with the rest of the weights and all warps busy; this form 676.)
//   w   = table[key], 32 copies per entry, one per bank: no conflicts
// The weights are exactly representable in bf16; the power-of-two factor 2^e (e >= 0) that
// expresses them against the accumulators' reference max is added to the packed exponents.
// Unscaled weights are summed pairwise (packed adds).
// kTwoStep (the Exp2 setup, whose running max is not an integer and may be smaller than 2^-6, too
// small to survive the 2^-120 scaling): T = S*c - m by a plain packed FMA (cn2 = c, mn2 = -m),
// then x = T * -2^-120 + 0 with flush-to-zero; the +0 addend turns a cancelled T into +0.
template <bool kTwoStep>
__device__ __forceinline__ void fast16(const uint32_t *r, uint32_t *pk, uint64_t cn2, uint64_t mn2,
                                       uint32_t escale, uint32_t tb, uint64_t &s01, uint64_t &s23)
{
    uint32_t a[16];
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
        float x0, x1;
        if constexpr (kTwoStep) {
            const uint64_t t2 = fma2(pack2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), cn2, mn2);
            unpack2(fma2_ftz(t2, pack2(-7.52316384526264e-37f, -7.52316384526264e-37f), 0ull), x0, x1);
        } else {
            unpack2(fma2_ftz(pack2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), cn2, mn2), x0, x1);
        }
        const uint32_t keys = min_u16x2(upper_halves(x0, x1), 0x06000600u) & 0xFFF8FFF8u;
        a[i] = dot_u16x2(keys, 0x0010u, tb);
        a[i + 1] = dot_u16x2(keys, 0x1000u, tb);
    }
    float w[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) w[i] = lds_f32(a[i]);
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
        s01 = add2(s01, pack2(w[i], w[i + 1]));
        s23 = add2(s23, pack2(w[i + 2], w[i + 3]));
        pk[i >> 1] = pack_bf16x2(w[i], w[i + 1]) + escale;
        pk[(i >> 1) + 1] = pack_bf16x2(w[i + 2], w[i + 3]) + escale;
    }
}

// Weight of a positive T (0 < T < 4 because the tile passed the restart test), from the positive window of the full
// table; 0 for any other T.
__device__ __forceinline__ float positive_weight(float u, uint32_t lut_pos)
{
    const uint32_t key = min(max(__float_as_uint(u) >> 19, (uint32_t)kLutPosLo), (uint32_t)kLutPosHi);
    float w;
    asm("{\n\t.reg .pred p;\n\t"
        "setp.gt.f32 p, %1, 0f00000000;\n\t"
        "mov.f32 %0, 0f00000000;\n\t"
        "@p ld.shared.f32 %0, [%2];\n\t}"
        : "=f"(w)
        : "f"(u), "r"(lut_pos + 4u * key));
    return w;
}
// Eight columns of a group that holds a positive T (rows whose maximum rose above the running max in a tile that was
// not restarted have a few of those; the fast path gave them weight 0, so theirs is added).  Returns the amount to
// add to the row sum.  Free of branches: with a divergent branch per element the eight lookups ran one after the
// other, and since a tile waits for its slowest warp, that, not the number of instructions, was what positive T
// cost (8 heads x 16384 tokens: 565 us, 470 with them left at weight 0).
__device__ __forceinline__ float fix8(const uint32_t *x, uint32_t *pk4, float c, float mref, uint32_t lut_full)
{
    const uint32_t lut_pos = lut_full + 4u * (uint32_t)(kLutNegN - kLutPosLo);
    float add = 0.f;
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
        const float w0 = positive_weight(fmaf(__uint_as_float(x[i]), c, -mref), lut_pos);
        const float w1 = positive_weight(fmaf(__uint_as_float(x[i + 1]), c, -mref), lut_pos);
        add += w0 + w1;
        pk4[i >> 1] += upper_halves(w0, w1);                 // exact in bf16
    }
    return add;
}
// Which of a warp's groups of eight columns hold a positive T in some row (bit g), from the groups' maxima.
template <int N>
__device__ __forceinline__ uint32_t positive_groups(const float (&g)[N], float c, float mref)
{
    uint32_t mask = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) mask |= fmaf(g[i], c, -mref) > 0.f ? 1u << i : 0u;
    return __reduce_or_sync(0xffffffffu, mask);
}

// High-precision tile (B0, or every tile in the exact mode): P = 2^(S*c - mref) in fp32, rounded
// to bf16 for the tensor core; the row sum uses the rounded values so that numerator and
// denominator see the same weights.  Masked entries arrive as -inf and give 0.
__device__ __forceinline__ float hp16(const uint32_t *r, uint32_t *pk, float c, float mref)
{
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
        const float u0 = fmaf(__uint_as_float(r[i]), c, -mref);
        const float u1 = fmaf(__uint_as_float(r[i + 1]), c, -mref);
        const uint32_t p = pack_bf16x2(ex2_approx(u0), ex2_approx(u1));
        s0 += __uint_as_float(p << 16);
        s1 += __uint_as_float(p & 0xFFFF0000u);
        pk[i >> 1] = p;
    }
    return s0 + s1;
}

// The restart test of a tile: HiF8(T) > lambda  <=>  T >= the midpoint between lambda and the next HiF8 value above it
// (rounding is monotone, ties go up): 2^-23 | 1.0625 | 2.125 | 3.125 for lambda 0 | 1 | 2 | 3.
__device__ __forceinline__ float restart_threshold(int lambda)
{
    return lambda == 0 ? 1.1920928955078125e-07f : (float)lambda + (lambda == 1 ? 0.0625f : 0.125f);
}
// ceil of the row maximum's score; the product was rounded: made sure that no T against it is positive.  Never -0, which
// ceilf gives for scores in (-1, 0): against that the key of a score of exactly 0 would be that of -0, a positive T's.
__device__ __forceinline__ float int_max(float mx, float c)
{
    const float smax = ceilf(mx * c);
    return smax + (fmaf(mx, c, -smax) > 0.f ? 1.f : 0.f);
}
// The thread's n columns of O~, n a multiple of 16, times f.
__device__ __forceinline__ void rescale_columns(uint32_t o_addr, int n, float f)
{
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 16) {
        uint32_t o[16];
        sm100::tmem_ld16(o_addr + i0, o);
        sm100::tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
        sm100::tmem_st16(o_addr + i0, o);
    }
}

// What a thread keeps of its row: m, the running max of Algorithm 1 (integer valued; real valued in the exact and
// Exp2 modes); m_ref, the max O~ and d are currently expressed against; d, the partial sum of the thread's columns.
// All rescale factors of Algorithm 1 are exact powers of two, so instead of multiplying O~ by 2^(m_old - m_new)
// whenever the max moves, a tile's weights are multiplied by 2^e, e = m - m_ref, held as what it adds to the
// exponents of a packed pair of weights.  O~ is touched only when the max moves and e has passed 61: a move without a
// restart adds 3 at most, so no weight is multiplied by more than 2^64.  The threads of a row take identical decisions.
// The max of a row moves a handful of times over all key tiles, so an 8-bit tile first asks whether it does in any
// row of the warp, and nothing below is worked out where it does not (attention_tc_kernel at D = 128 aside).
struct RowState {
    float m, m_ref, d;
    uint32_t escale;

    __device__ __forceinline__ void set_scale() { escale = (uint32_t)(int)(m - m_ref) * 0x00800080u; }
    // For a tile in which some row of the warp has a positive T (um: that of the row's maximum mx) or which is restarted (in
    // any other it does no more than a rebase that is due).  Moves m to the max that the tile's T are taken against and
    // returns the max after the tile.
    template <class Rebase>
    __device__ __forceinline__ float decide(float mx, float c, float um, bool restart_tile, Rebase rebase)
    {
        float m_next;
        if (restart_tile) {
            m_next = m = fmaxf(m, int_max(mx, c));
        } else {
            // delta = max(0, ceil(rowmax T8)); weights 2^T8 * 2^-delta = 2^T8 against the old max.
            // The tile passed the restart test, so T < 3.125, and ceil(HiF8(T)) only depends on which
            // rounding midpoints T has reached: 0 below 2^-23 (rounds to 0), else 1 below 1.0625,
            // else 2 below 2.125, else 3.
            m_next = m + ((um >= 1.1920928955078125e-07f ? 1.f : 0.f) + (um >= 1.0625f ? 1.f : 0.f) +
                          (um >= 2.125f ? 1.f : 0.f));
        }
        const float kk = m - m_ref;
        const bool need = kk > 61.f;
        if (__any_sync(0xffffffffu, need)) {
            const float f = need ? pow2_int(-kk) : 1.f;
            rebase(f);
            d *= f;
            if (need) m_ref = m;
        }
        set_scale();
        return m_next;
    }
    __device__ __forceinline__ void move(float m_next) { m = m_next; set_scale(); }
    __device__ __forceinline__ void add(float sum) { d += sum * __uint_as_float(0x3F800000u + (escale & 0x7F800000u)); }
};

// Tables of the softmax warps: the 32-way replicated fast-path table (one global load per entry, copies written with
// 16-byte stores) and the plain full table.
__device__ __forceinline__ void fill_attention_tables(uint8_t *rep_table, uint8_t *full_table, int t, int nthreads)
{
    float4 *rep = reinterpret_cast<float4 *>(rep_table);
    for (int e = t; e < kLutRepEntries; e += nthreads) {
        const float w = (e < 16) ? 1.f : g_w0.v[e - 16];
        const float4 w4 = make_float4(w, w, w, w);
#pragma unroll
        for (int i = 0; i < 8; ++i) rep[e * 8 + i] = w4;
    }
    float *full = reinterpret_cast<float *>(full_table);
    for (int i = t; i < kLutN; i += nthreads) full[i] = g_w0.v[i];
}

__device__ __forceinline__ float max8(const uint32_t *x)
{
    return max3(max3(__uint_as_float(x[0]), __uint_as_float(x[1]), __uint_as_float(x[2])),
                max3(__uint_as_float(x[3]), __uint_as_float(x[4]), __uint_as_float(x[5])),
                fmaxf(__uint_as_float(x[6]), __uint_as_float(x[7])));
}

// kQK8: Q and K arrive as E4M3 codes with one power-of-two scale per 128-row tile (the dequantisation
// the paper proposes to fuse, Section 3.4): Q K^T runs on the 8-bit tensor-core path and the two
// scales of a tile pair are folded into the score scale c, task by task.  D = 128 only.
// kB0Last: B0 = {first, last visible key tile} (compile-time, so that the usual order pays nothing).
// kMode (BAPS_MODE_*): Algorithm 1, the exact mode, or -- kExp2 below -- the "Exp2 HiF8" setup of Section 4.1 (Eq. (2) with a real-valued max, weights and
// rescale factor through the 8-bit exponent table); otherwise Algorithm 1 or the exact mode.
// kOne: a CTA owns one query tile instead of two (small grids, see one_tile_per_cta; always with kB0Last).
template <int D, int kMode, bool kQK8 = false, bool kB0Last = false, bool kOne = kB0Last>
__global__ void __launch_bounds__(kTcThreads, 1)
attention_tc_kernel(const __grid_constant__ CUtensorMap mq, const __grid_constant__ CUtensorMap mk,
                    const __grid_constant__ CUtensorMap mv, const AttnTcParams p)
{
    using namespace sm100;
    using L = TcLayout<D>;
    constexpr bool kExp2 = kMode == BAPS_MODE_EXP2_HIF8;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = sbase + L::kBarOff;
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    // q_full | s_full[buffer] | p_full[buffer] | pv_done[query tile] | kv_full[stage] | kv_empty[stage]
    constexpr int BQ = 0, BS = 1, BP = 3, BD = 5, BKF = 7, BKE = 7 + L::kStages;
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + L::kMiscOff);
    volatile int *s_abort = reinterpret_cast<volatile int *>(smem + L::kMiscOff + 4);

    allow_next_kernel();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    const WorkItem item = work_item(p.H, p.Hkv, p.npairs, p.chunks, blockIdx.x);
    const int pair = item.tile, hk = item.hk, b = item.b, h = item.h;
    const int nk = p.S / 128;
    // With B0 = {first, last} the key tiles are visited in the order 0, last, 1, ..., last - 1, and
    // "last" differs between neighbouring query tiles of a causal problem, so the two query tiles of
    // a pair could not share their K / V stream: the CTA then owns a single query tile (t = 0).
    const int qbase = kOne ? pair : 2 * pair;        // first query tile of this CTA
    int jm[2];                                   // number of key tiles of each query tile
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int qi = qbase + t;
        jm[t] = (qi < p.nq && !(kOne && t == 1)) ? (p.causal ? qi + 1 : nk) : 0;
    }
    const int J = jm[0] > jm[1] ? jm[0] : jm[1];
    const int nb0 = (kB0Last && J >= 2) ? 2 : 1;        // number of high-precision (B0) steps
    // key tile visited at step s
    auto key_tile = [&](int s) { return !kB0Last ? s : (s == 0 ? 0 : (s == 1 ? J - 1 : s - 1)); };
    const int q_row0 = (b * p.H + h) * p.S + qbase * 128;           // row in the [B*H*S, D] view
    const int kv_row0 = (b * p.Hkv + hk) * p.S;

    // built while the first Q / K tiles are on their way
    auto fill_tables = [&] {
        fill_attention_tables(smem + L::kLutRepOff, smem + L::kLutFullOff, tid, kTcSoftmaxWarps * 32);
    };

    // ---- setup --------------------------------------------------------------------------------
    // kEarly (D = 64 or one query tile, where a CTA lives for few tasks): the producer lane initialises the barriers itself and
    // starts the Q tiles and the first ring-full of K / V tiles before the CTA-wide barrier, so that the copies
    // are on their way while the rest of the CTA is still setting up.  (Two tiles at D = 128, by now the exact and Exp2
    // modes, keep the plain order: Algorithm 1's steady state was 2 % slower the other way while it ran in that form.)
    constexpr bool kEarly = (D == 64) || kOne;
    constexpr int kQkBoxes = kQK8 ? 1 : D / 64;
    constexpr uint32_t kQkTileBytes = kQK8 ? 128 * D : L::kTileBytes;
    const int n_early = kEarly ? (2 * J < L::kStages ? 2 * J : L::kStages) : 0;   // loads that need no free stage
    if constexpr (kEarly) {
        if (tid == 0) *s_abort = 0;
        if (warp == 16) {
            if (lane == 0) {
                mbar_init(bar(BQ), 1);
                for (int i = 0; i < 2; ++i) {
                    mbar_init(bar(BS + i), 1);
                    mbar_init(bar(BP + i), kTcSoftmaxWarps * 32);
                    mbar_init(bar(BD + i), 1);
                }
                for (int s = 0; s < L::kStages; ++s) { mbar_init(bar(BKF + s), 1); mbar_init(bar(BKE + s), 1); }
                mbar_fence_init();
                await_previous_kernel();
                const int nvalid = (jm[0] > 0) + (jm[1] > 0);
                mbar_arrive_expect_tx(bar(BQ), (uint32_t)nvalid * kQkTileBytes);
                for (int t = 0; t < 2; ++t)
                    if (jm[t] > 0)
                        for (int hh = 0; hh < kQkBoxes; ++hh)
                            tma_load_2d(sbase + L::kQOff + t * L::kTileBytes + hh * 16384, &mq, hh * 64,
                                        q_row0 + t * 128, bar(BQ));
                for (int l = 0; l < n_early; ++l) {
#ifdef BAPS_TEST_SKIP_LOAD
                    if (l == g_test_skip_load) continue;      // this tile never arrives
#endif
                    const int s = l % L::kStages;
                    mbar_arrive_expect_tx(bar(BKF + s), (l & 1) ? (uint32_t)L::kTileBytes : kQkTileBytes);
                    const CUtensorMap *m = (l & 1) ? &mv : &mk;
                    for (int hh = 0; hh < ((l & 1) ? D / 64 : kQkBoxes); ++hh)
                        tma_load_2d(sbase + L::kKvOff + s * L::kTileBytes + hh * 16384, m, hh * 64,
                                    kv_row0 + key_tile(l >> 1) * 128, bar(BKF + s));
                }
            }
            __syncwarp();
        }
        if (warp == 17) { tmem_alloc(smem_u32(s_tmem), 512); tmem_relinquish(); }
        if (warp < kTcSoftmaxWarps) fill_tables();
    } else {
        if (tid == 0) {
            mbar_init(bar(BQ), 1);
            for (int i = 0; i < 2; ++i) {
                mbar_init(bar(BS + i), 1);
                mbar_init(bar(BP + i), kTcSoftmaxWarps * 32);
                mbar_init(bar(BD + i), 1);
            }
            for (int s = 0; s < L::kStages; ++s) { mbar_init(bar(BKF + s), 1); mbar_init(bar(BKE + s), 1); }
            mbar_fence_init();
            *s_abort = 0;
        }
        if (warp == 16) { tmem_alloc(smem_u32(s_tmem), 512); tmem_relinquish(); }
    }
    if (warp == 17 && lane == 0) { tma_prefetch_desc(&mq); tma_prefetch_desc(&mk); tma_prefetch_desc(&mv); }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *s_tmem;

    // Register budget: the fifth warpgroup (producer, MMA issuer, two idle warps) needs few
    // registers and hands part of its share to the sixteen softmax warps (kTcSplit).
    if (warp >= kTcSoftmaxWarps) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kTcSplit.few));
      if (warp == 16) {
        // ======================= TMA producer ==================================================
        if (lane == 0) {
            if constexpr (!kEarly) {
                await_previous_kernel();
                const int nvalid = (jm[0] > 0) + (jm[1] > 0);
                mbar_arrive_expect_tx(bar(BQ), (uint32_t)nvalid * kQkTileBytes);
                for (int t = 0; t < 2; ++t)
                    if (jm[t] > 0)
                        for (int hh = 0; hh < kQkBoxes; ++hh)
                            tma_load_2d(sbase + L::kQOff + t * L::kTileBytes + hh * 16384, &mq, hh * 64,
                                        q_row0 + t * 128, bar(BQ));
            }
            int issued = n_early;
            for (int l = n_early; l < 2 * J; ++l) {
                const int s = l % L::kStages, n = l / L::kStages;
                if (n > 0 && !mbar_wait(bar(BKE + s), (uint32_t)((n - 1) & 1), s_abort, &g_async_status, 0x100 + s))
                    break;
#ifdef BAPS_TEST_SKIP_LOAD
                if (l == g_test_skip_load) continue;          // this tile never arrives
#endif
                mbar_arrive_expect_tx(bar(BKF + s), (l & 1) ? (uint32_t)L::kTileBytes : kQkTileBytes);
                const CUtensorMap *m = (l & 1) ? &mv : &mk;
                for (int hh = 0; hh < ((l & 1) ? D / 64 : kQkBoxes); ++hh)
                    tma_load_2d(sbase + L::kKvOff + s * L::kTileBytes + hh * 16384, m, hh * 64,
                                kv_row0 + key_tile(l >> 1) * 128, bar(BKF + s));
                issued = l + 1;
            }
            if (*s_abort) {
                // let copies already in flight land before the CTA's shared memory is released
                const int first = issued > L::kStages ? issued - L::kStages : 0;
                for (int l = first; l < issued; ++l) {
                    const int s = l % L::kStages, n = l / L::kStages;
                    const uint64_t t0 = globaltimer_ns();
                    while (!mbar_try_wait(bar(BKF + s), (uint32_t)(n & 1)) && globaltimer_ns() - t0 < 2000000ull) {}
                }
            }
        }
      } else if (warp == 17) {
        // ======================= MMA issuer ====================================================
        // The whole warp runs the loop (waits, task bookkeeping, descriptor arithmetic) so that the
        // compiler can keep it on the uniform datapath; one elected lane issues the MMAs and commits.
        {
            constexpr uint32_t idesc_qk = make_idesc_bf16(128, 128, false);
            constexpr uint32_t idesc_pv = make_idesc_bf16(128, D, true);
            auto kv_stage = [&](int l) { return l % L::kStages; };
            auto kv_parity = [&](int l) { return (uint32_t)((l / L::kStages) & 1); };
            // the last query tile that uses key tile j: its MMA releases the K / V stage
            auto last_user = [&](int j) { return (j < jm[1]) ? 1 : 0; };
            // task order (0,0) (1,0) (0,1) (1,1) ... restricted to j < jm[t]
            auto advance = [&](int &t, int &j) -> bool {
                if (t == 0 && j < jm[1]) { t = 1; return true; }
                ++j;
                if (j < jm[0]) { t = 0; return true; }
                if (j < jm[1]) { t = 1; return true; }
                return false;
            };
            auto wait_all = [&](uint32_t bar_addr, uint32_t parity, int code) -> bool {
                return __all_sync(0xffffffffu, mbar_wait(bar_addr, parity, s_abort, &g_async_status, code));
            };
            // (the limit of the first wait starts when the kernel ahead has ended, however long that takes; with kEarly
            // the producer has waited for it before the CTA-wide barrier)
            if constexpr (!kEarly) await_previous_kernel();
            bool ok = wait_all(bar(BQ), 0, 0x200);
            int k_ready = -1, v_ready = -1;      // key / value tiles whose arrival has been awaited
            auto await_k = [&](int j) -> bool {
                if (j <= k_ready) return true;
                if (!wait_all(bar(BKF + kv_stage(2 * j)), kv_parity(2 * j), 0x210)) return false;
                k_ready = j;
                return true;
            };
            auto await_v = [&](int j) -> bool {
                if (j <= v_ready) return true;
                if (!wait_all(bar(BKF + kv_stage(2 * j + 1)), kv_parity(2 * j + 1), 0x220)) return false;
                v_ready = j;
                return true;
            };
            // S buffer (k & 1) = Q_t K_j^T (issuing lane only)
            auto mma_qk = [&](int t, int j, int k) {
                const uint32_t qd = sdesc_lo(sbase + L::kQOff + t * L::kTileBytes, 16);
                const uint32_t kd = sdesc_lo(sbase + L::kKvOff + kv_stage(2 * j) * L::kTileBytes, 16);
                const uint32_t sd = tmem + (k & 1) * 128;
                if constexpr (kQK8) {
                    // rows of 128 E4M3 bytes: K = 32 per instruction, 32 bytes further along the row each
                    constexpr uint32_t idesc_qk8 = make_idesc_e4m3(128, 128);
#pragma unroll
                    for (int ks = 0; ks < D / 32; ++ks)
                        mma_ss_lo_f8(sd, qd + 2u * ks, kd + 2u * ks, idesc_qk8, ks > 0);
                } else {
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        const uint32_t off = (uint32_t)(((ks >> 2) * 16384 + (ks & 3) * 32) >> 4);
                        mma_ss_lo(sd, qd + off, kd + off, idesc_qk, ks > 0);
                    }
                }
                mma_commit(bar(BS + (k & 1)));
            };
            // O_t += P V_j with P in S buffer (k & 1): the weights of keys 16 ks .. 16 ks + 15 sit at
            // columns 32 (ks / 2) + 8 (ks % 2) of the buffer (issuing lane only; the keys in the order of
            // paired_attention_tc_kernel, so that both add up alike)
            auto mma_pv = [&](int t, int j, int k) {
                const uint32_t vd = sdesc_lo(sbase + L::kKvOff + kv_stage(2 * j + 1) * L::kTileBytes, 16384);
                const uint32_t od = tmem + 256 + t * D, pd = tmem + (k & 1) * 128;
                const uint32_t acc0 = j > 0 ? 1u : 0u;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int ks = (i >> 1 & 1) * 4 + (i < 4 ? 2 : 0) + (i & 1);    // column quarters 1, 3, 0, 2
                    mma_ts_lo(od, pd + (ks >> 1) * 32 + (ks & 1) * 8, vd + ks * 128, idesc_pv, i > 0 ? 1u : acc0);
                }
            };
            const bool leader = elect_one();
            if (ok && J > 0) {
                int t = 0, j = 0, k = 0;          // task whose P V comes next
                int tq = 0, jq = 0, kq = 0;       // task whose Q K^T comes next
                bool more_q = true;
                // scores of the first two tasks: both buffers are free
                for (int i = 0; i < 2 && ok && more_q; ++i) {
                    ok = await_k(jq);
                    if (!ok) break;
                    tc_fence_after_sync();
                    if (leader) {
                        mma_qk(tq, jq, kq);
                        if (tq == last_user(jq)) mma_commit(bar(BKE + kv_stage(2 * jq)));
                    }
                    __syncwarp();
                    more_q = advance(tq, jq);
                    ++kq;
                }
                while (ok) {
                    // One burst per task: P V of task k, then at once Q K^T of task k + 2 into the buffer
                    // P V reads (the tensor core runs them in order), so that the softmax warps find the
                    // scores of task k + 2 ready when they get there.  Everything the burst needs except P
                    // is awaited before P.
                    ok = await_v(j);
                    if (ok && more_q) ok = await_k(jq);
                    if (!ok) break;
                    ok = wait_all(bar(BP + (k & 1)), (uint32_t)((k >> 1) & 1), 0x230 + (k & 1));
                    if (!ok) break;
                    tc_fence_after_sync();
                    if (leader) {
                        mma_pv(t, j, k);
                        if (more_q) mma_qk(tq, jq, kq);
                        mma_commit(bar(BD + t));
                        if (t == last_user(j)) mma_commit(bar(BKE + kv_stage(2 * j + 1)));
                        if (more_q && tq == last_user(jq)) mma_commit(bar(BKE + kv_stage(2 * jq)));
                    }
                    __syncwarp();
                    if (more_q) { more_q = advance(tq, jq); ++kq; }
                    if (!advance(t, j)) break;
                    ++k;
                }
            }
        }
      }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kTcSplit.many));
        // ======================= softmax warps ==================================================
        // (kEarly: the tables were filled before the CTA-wide barrier, while a kernel ahead was still draining)
        if constexpr (!kEarly) {
            fill_tables();
            named_bar_sync(6, kTcSoftmaxWarps * 32);
        }
        await_previous_kernel();
        const int q4 = warp & 3;                 // TMEM lane quarter: rows 32 q4 .. 32 q4 + 31
        const int cq = warp >> 2;                // key column quarter: columns 32 cq .. 32 cq + 31
        const int row = q4 * 32 + lane;
        const uint32_t lane_sel = (uint32_t)(q4 * 32) << 16;
        const uint32_t s_col = tmem + lane_sel + cq * 32;                 // + 128 * buffer
        const uint32_t lut_full = sbase + L::kLutFullOff;
        const uint32_t tb = sbase + L::kLutRepOff + (uint32_t)lane * 4u;
        const uint32_t xrow = sbase + L::kXchgOff + (uint32_t)row * 16u;  // + 2048 * (k & 1); my slot + 4 cq
        const float c_base = p.c;
        constexpr bool exact = kMode == BAPS_MODE_EXACT;
        constexpr bool e2e = kMode == BAPS_MODE_E2E_HIF8;
        // With 128 columns of O~ the branch around the decisions costs more than it saves here, where every warp waits for
        // the slowest of sixteen (1 x 32768 425 -> 420 us without it, 8-bit Q / K 398 -> 384, B0 = {first, last}, 32 x 4096
        // bidirectional, 479 -> 474); at D = 64 it is the other way round (306 -> 294 with it).
        constexpr bool kAlwaysDecide = D == 128;
        const bool count_restarts = p.restarts != nullptr && warp == 0;
        const float over_thr = restart_threshold(p.lambda);
        // per query tile t; O~ and d are rebased past an exponent of 8 in the exact mode, whose factors are not exact
        RowState st[2] = {{-INFINITY, 0.f, 0.f, 0u}, {-INFINITY, 0.f, 0.f, 0u}};
        int n_restart[2] = {0, 0};
        int k = 0;                               // running task index
        uint32_t r[32];                          // scores of the current task (my quarter row)

        // One task.  T is a compile-time query tile so that the per-tile state stays in registers.
        // Scores of task k_ -> r (asynchronous; completed by tmem_wait_ld at the start of the task).
        auto load_scores = [&](int k_) {
            mbar_wait(bar(BS + (k_ & 1)), (uint32_t)((k_ >> 1) & 1), s_abort, &g_async_status, 0x300 + (k_ & 1));
            tc_fence_after_sync();
            tmem_ld32(s_col + (uint32_t)(k_ & 1) * 128u, r);
        };
        auto task = [&](auto tconst, const int j, const bool has_next) {
            constexpr int T = decltype(tconst)::value;
            const int qi = qbase + T;
            // score scale of this task: log2(e) * scale, times the dequantisation scales of the query tile
            // and of the key tile when Q and K are 8-bit (powers of two: the product is exact)
            float c = c_base;
            if constexpr (kQK8)
                c = c_base * ldg_f32(p.q_scale + (size_t)(b * p.H + h) * p.nq + qi) *
                    ldg_f32(p.k_scale + (size_t)(b * p.Hkv + hk) * nk + key_tile(j));
            const uint32_t s_addr = s_col + (uint32_t)(k & 1) * 128u;
            const uint32_t x_addr = xrow + (uint32_t)(k & 1) * 2048u;
            const bool diag = p.causal && (key_tile(j) == qi);
            // ---- scores of my quarter row, their maximum, exchange with the three partner threads ----
            tmem_wait_ld();
            if (diag) {
#pragma unroll
                for (int i = 0; i < 32; ++i) r[i] = (cq * 32 + i > row) ? 0xFF800000u : r[i];
            }
            const bool hp = !kExp2 && ((j < nb0) || exact);
            const float g[4] = {max8(&r[0]), max8(&r[8]), max8(&r[16]), max8(&r[24])};
            const float hm = fmaxf(fmaxf(g[0], g[1]), fmaxf(g[2], g[3]));
            sts_f32(x_addr + 4u * (uint32_t)cq, hm);
            auto row_max = [&] {
                const float4 pm = lds_f32x4(x_addr);
                return fmaxf(fmaxf(pm.x, pm.y), fmaxf(pm.z, pm.w));
            };
            auto rebase = [&](float f) {
                mbar_wait(bar(BD + T), (uint32_t)((j - 1) & 1), s_abort, &g_async_status, 0x330 + T);
                tc_fence_after_sync();
                rescale_columns(tmem + lane_sel + 256 + T * D + cq * (D / 4), D / 4, f);
            };
            // ---- decisions (Algorithm 1: B0 branch / restart test / max update) -----------------
            bool changed = false, restart_tile = false;
            float m_next, mref_w;                   // T of this tile is taken against mref_w
            if (e2e && !hp) {
                // The restart decision is tile-wide: does any row have HiF8(T of its maximum) >
                // lambda?  The test is monotone, so a row passes it iff one of its quarters does:
                // one reducing barrier over all softmax threads gives the verdict and also orders
                // the exchange of the quarter maxima.  T of the row maximum is formed exactly like every element's
                // T (one FMA).
                restart_tile = named_bar_or(5, kTcSoftmaxWarps * 32, fmaf(hm, c, -st[T].m) >= over_thr);
                const float mx = row_max();
                const float um = fmaf(mx, c, -st[T].m);
                changed = restart_tile || __any_sync(0xffffffffu, um > 0.f);
                m_next = st[T].m;
                if (kAlwaysDecide || changed) {
                    if (count_restarts && restart_tile) ++n_restart[T];
                    m_next = st[T].decide(mx, c, um, restart_tile, rebase);
                }
                mref_w = st[T].m;
            } else {
                named_bar_sync(1 + q4, 128);
                const float mx = row_max();
                if constexpr (kExp2) {
                    // Eq. (2): real-valued running max.  The product was rounded: step the max up by one
                    // unit in the last place if the row maximum's T would come out positive, so that every
                    // T of the tile is <= 0.
                    float smax = mx * c;
                    if (fmaf(mx, c, -smax) > 0.f)
                        smax = __uint_as_float(__float_as_uint(smax) + (smax >= 0.f ? 1u : 0xFFFFFFFFu));
                    m_next = mref_w = fmaxf(st[T].m, smax);
                    if (j > 0) {
                        // rescale factor 2^(m_old - m_new), 8-bit in and out (not a power of two): O~ and d
                        // are multiplied for real, once P V of this query tile's previous task is complete.
                        const float alpha = lds_f32(lut_full + 4u * (uint32_t)w0_index(st[T].m - m_next));
                        if (__any_sync(0xffffffffu, alpha != 1.f)) rebase(alpha);
                        st[T].d *= alpha;
                    }
                    st[T].m_ref = m_next;
                } else {
                    m_next = fmaxf(st[T].m, exact ? mx * c : int_max(mx, c));
                    if (j == 0) st[T].m_ref = m_next;
                    const float kk = m_next - st[T].m_ref;
                    const bool need = (j > 0) && (kk > (exact ? 8.f : 64.f));
                    if (__any_sync(0xffffffffu, need)) {
                        const float f = need ? (exact ? ex2_approx(-kk) : pow2_int(-kk)) : 1.f;
                        rebase(f);
                        st[T].d *= f;
                        if (need) st[T].m_ref = m_next;
                    }
                    mref_w = st[T].m_ref;
                }
                st[T].m = m_next;
                st[T].escale = 0u;                 // these weights are taken against m_ref (Exp2: against m, with e = 0)
            }
            const uint32_t escale = st[T].escale;
            // some row of this warp has T > 0 in a tile that was not restarted: the 8-column groups
            // holding those few entries are redone with the full table after the fast path
            const bool pos_tile = changed && !restart_tile;                    // warp-uniform
            // ---- weights -> bf16 P over score columns already read; row sum ---------------------------
            float sum = 0.f;
            uint32_t pk[16];
            if (hp) {
                sum = hp16(&r[0], &pk[0], c, mref_w) + hp16(&r[16], &pk[8], c, mref_w);
            } else {
                // (8-bit Q / K: c carries the dequantisation scales and may be far too small for the
                // combined constant c * 2^-120 to be a normal number, hence the two-step form there too)
                constexpr bool kTwo = kExp2 || kQK8;
                const float mnv = kTwo ? -mref_w : mref_w * 7.52316384526264e-37f;    // 2^-120
                const float cnv = kTwo ? c : -c * 7.52316384526264e-37f;
                const uint64_t cn2 = pack2(cnv, cnv), mn2 = pack2(mnv, mnv);
                uint64_t s01 = 0ull, s23 = 0ull;
                fast16<kTwo>(&r[0], &pk[0], cn2, mn2, escale, tb, s01, s23);
                fast16<kTwo>(&r[16], &pk[8], cn2, mn2, escale, tb, s01, s23);
                if (pos_tile) {
                    const uint32_t groups = positive_groups(g, c, mref_w);
#pragma unroll
                    for (int gg = 0; gg < 4; ++gg)
                        if (groups >> gg & 1u) sum += fix8(&r[gg * 8], &pk[gg * 4], c, mref_w, lut_full);
                }
                float a0, a1, a2, a3;
                unpack2(s01, a0, a1); unpack2(s23, a2, a3);
                sum += (a0 + a1) + (a2 + a3);
            }
            // 32 scores (columns 32 cq ..) become 16 packed columns 32 cq .. 32 cq + 15
            tmem_st16(s_addr, pk);
            tmem_wait_st();
            tc_fence_before_sync();
            mbar_arrive(bar(BP + (k & 1)));       // P is in place: the tensor core's burst may go
            st[T].add(sum);
            if ((e2e && kAlwaysDecide) || changed || (kB0Last && hp)) st[T].move(m_next);
            // the next task's scores travel into registers while the loop turns around
            if (has_next) load_scores(k + 1);
            ++k;
        };

        if (J > 0) load_scores(0);
        for (int j = 0; j < J; ++j) {
            if (j < jm[0]) task(std::integral_constant<int, 0>{}, j, (!kOne && j < jm[1]) || j + 1 < J);
            if constexpr (!kOne)
                if (j < jm[1]) task(std::integral_constant<int, 1>{}, j, j + 1 < J);
        }
        const bool ok = (*s_abort == 0);

        // ---- epilogue: O = O~ / d (each thread: its quarter of the output columns) ---------------------
        auto finish = [&](auto tconst) {
            constexpr int T = decltype(tconst)::value;
            const int jmax = jm[T];
            if (jmax == 0) return;                                   // uniform over the CTA
            const int qi = qbase + T;
            const bool done = mbar_wait(bar(BD + T), (uint32_t)((jmax - 1) & 1), s_abort, &g_async_status, 0x320 + T);
            tc_fence_after_sync();
            // total denominator of the row = the four quarter sums
            // the exchange buffer not used by the task before (that one may still be read by a partner)
            const uint32_t x_addr = xrow + (uint32_t)((k + T) & 1) * 2048u;
            sts_f32(x_addr + 4u * (uint32_t)cq, st[T].d);
            named_bar_sync(1 + q4, 128);
            const float4 pd = lds_f32x4(x_addr);
            const float dtot = (pd.x + pd.y) + (pd.z + pd.w);
            const bool good = ok && done;
            const float dinv = 1.f / dtot;
            const size_t grow = (size_t)q_row0 + (size_t)T * 128 + row;   // row in [B*H*S]
            const int ocol0 = cq * (D / 4);
            const uint32_t o_addr = tmem + lane_sel + 256 + T * D + ocol0;
            // The bf16 output goes through the (now idle) Q staging area of this tile so that the global
            // stores are whole rows: a thread owns 32 columns of one row, i.e. a warp's direct stores
            // would touch 32 rows with 16 bytes each.  Staged layout: row-major, the 16-byte chunks of a
            // row XOR-swizzled with the row number (conflict-free both ways).
            constexpr int kRowBytes = D * 2, kChunks = kRowBytes / 16;
            const uint32_t stage = sbase + L::kQOff + T * L::kTileBytes;
#pragma unroll 1
            for (int ch = 0; ch < D / 64; ++ch) {
                uint32_t rr[16];
                tmem_ld16(o_addr + ch * 16, rr);
                tmem_wait_ld();
                float o[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) o[i] = __uint_as_float(rr[i]) * dinv;
                if (p.out) {
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int chunk = (ocol0 + ch * 16) / 8 + i;
                        sts_u32x4(stage + (uint32_t)row * kRowBytes + (uint32_t)((chunk ^ (row & (kChunks - 1))) * 16),
                                  make_uint4(pack_bf16x2(o[8 * i], o[8 * i + 1]), pack_bf16x2(o[8 * i + 2], o[8 * i + 3]),
                                             pack_bf16x2(o[8 * i + 4], o[8 * i + 5]), pack_bf16x2(o[8 * i + 6], o[8 * i + 7])));
                    }
                }
                if (p.out_f32 && good) {
                    float4 *dst = reinterpret_cast<float4 *>(p.out_f32 + grow * D + ocol0 + ch * 16);
#pragma unroll
                    for (int i = 0; i < 4; ++i) dst[i] = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
                }
            }
            if (p.out) {
                // the four warps of a lane quarter staged the 32 rows of that quarter; each now writes eight
                // of them, 512 contiguous bytes per instruction
                named_bar_sync(1 + q4, 128);
                constexpr int kRowsPerInstr = 32 / kChunks;              // 2 (D = 128) or 4 (D = 64)
#pragma unroll
                for (int it = 0; it < 8 / kRowsPerInstr; ++it) {
                    const int rw = q4 * 32 + cq * 8 + it * kRowsPerInstr + lane / kChunks;
                    const int chunk = lane % kChunks;
                    const uint4 v = lds_u32x4(stage + (uint32_t)rw * kRowBytes + (uint32_t)((chunk ^ (rw & (kChunks - 1))) * 16));
                    if (good)
                        *reinterpret_cast<uint4 *>(reinterpret_cast<uint8_t *>(p.out) +
                                                   ((size_t)q_row0 + (size_t)T * 128 + rw) * kRowBytes + chunk * 16) = v;
                }
            }
            if (!good) return;
            if (cq == 0) {
                if (p.row_m) p.row_m[grow] = st[T].m;
                // d is held against m_ref; report it against the final max
                if (p.row_d) p.row_d[grow] = dtot * (exact ? ex2_approx(st[T].m_ref - st[T].m) : pow2_int(st[T].m_ref - st[T].m));
            }
            if (count_restarts && lane == 0)
                p.restarts[(size_t)(b * p.H + h) * p.nq + qi] = n_restart[T];
        };
        finish(std::integral_constant<int, 0>{});
        if constexpr (!kOne) finish(std::integral_constant<int, 1>{});
    }

    // ---- teardown ---------------------------------------------------------------------------------
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 16) { __syncwarp(); tmem_dealloc(tmem, 512); }
}

} // namespace baps
