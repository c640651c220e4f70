// Fused BAPS attention forward for heads of 128 (Algorithm 1, bf16 V, bf16 or 8-bit Q / K), two streams per CTA.
//
// One CTA owns two consecutive 128-row query tiles (t = 0, 1) of one (batch, head), which share the K / V stream, and
// eight softmax warps work on each.  The softmax warps of the two streams share no barrier: while one stream waits for its
// P V and its next Q K^T, or stands at the barrier of its tile-wide vote, the other issues.  They meet at the MMA warp, which
// serves them in a fixed order, tile by tile: it waits for stream 0's weights even if stream 1's are there first, so that
// neither gets more than a tile ahead of the other.  A row is shared by two threads (64 columns each), so that what is done
// once per row and tile -- maxima, vote, decisions, waits, stores -- costs half as many instructions per score as with four.
//   warps 0-15  softmax: stream t = w / 8; warp w owns rows 32 (w % 4) .. + 31 and the 64 key columns of half
//               (w / 4) % 2, in two chunks of 32.  Maxima of both chunks, exchange and vote, then the weights of the
//               second chunk (still in registers) and of the first (read again)
//   warp 16     TMA producer: Q tiles, then K_0, V_0, K_1, ... through a ring of four 32 KB stages
//   warp 17     MMA issuer, per tile and stream: P V of tile j for the keys of the second chunks as soon as their weights
//               are there, then for those of the first, and Q K^T of tile j + 1 into the same columns (the tensor
//               core runs them in order)
// (warps 18, 19 idle: they complete the warpgroup whose registers go to the softmax warps.)
// TMEM (512 columns): S_0 | S_1 | O_0 | O_1, 128 columns each; the bf16 weights of column quarter q overwrite columns
// [32 q, 32 q + 16) of S_t.
// The arithmetic, the bounded waits and the way every role ends after an expired wait are those of
// attention_tc_kernel; only the row sum is added up in another order (two partial sums per row, not four).
//
// What bounds it: the chain of a stream, not a pipe.  By clock64 stamps (8 / 2 heads x 16384, causal) a stream takes 3980
// cycles per tile, two tiles per SM in that time, of which the tensor core needs 1024 for each: from its scores to its last
// weights 2670, with two warps per scheduler and stream that do not cover the latency of the lookups, then P V and Q K^T.
// The weights of the second chunks are there 500 cycles before the MMA warp, which is still issuing for the other stream,
// gets to them.  Measured against sixteen warps on one tile after the other (attention_tc_kernel with two query tiles; causal,
// heads x tokens): 8 / 2 x 16384 614 -> 539 us, 64 / 16 x 8192 1250 -> 1092, 64 / 16 x 2048 116 -> 111; bidirectional 128 / 32 x 2048
// 354 -> 317.  Of that, at the first of these, P V in two halves 559 -> 540, both chunks requested at once 559 -> 538, the two
// together 539.  The lookups of 32 columns have to be in flight together: sixteen at a time in a rolled loop took 609 to 641.
// (tile() and the epilogue are attention_d64_kernel's with other offsets, and P in its score columns: a change to one is to
// be looked at in the other.)
#pragma once
#include "baps_attention_tc.cuh"

namespace baps {

struct PairLayout {
    static constexpr int kTileBytes = 128 * 128 * 2, kStages = 4;
    static constexpr int kQOff = 0;
    static constexpr int kKvOff = 2 * kTileBytes;
    static constexpr int kLutRepOff = kKvOff + kStages * kTileBytes;
    static constexpr int kLutFullOff = kLutRepOff + kLutRepBytes;
    static constexpr int kBarOff = (kLutFullOff + kLutN * 4 + 15) & ~15;
    // barriers: q_full, s_full[2], p_full[2][2], pv_done[2], kv_full[stages], kv_empty[stages]
    static constexpr int kXchgOff = (kBarOff + (9 + 2 * kStages) * 8 + 15) & ~15;      // float xchg[2 tiles][2][128][2]
    static constexpr int kMiscOff = kXchgOff + 2 * 2 * 128 * 2 * 4;                    // tmem base, abort
    static constexpr int kDynBytes = kMiscOff + 16 + 1024;                             // slack for 1024-byte alignment
};

template <bool kQK8>
__global__ void __launch_bounds__(kTcThreads, 1)
paired_attention_tc_kernel(const __grid_constant__ CUtensorMap mq, const __grid_constant__ CUtensorMap mk,
                           const __grid_constant__ CUtensorMap mv, const AttnTcParams p)
{
    using namespace sm100;
    using L = PairLayout;
    constexpr int D = 128;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    auto bar = [&](int i) { return sbase + L::kBarOff + 8u * (uint32_t)i; };
    // q_full | s_full[t] | p_full[2 t + half of the weights] | pv_done[t] | kv_full[stage] | kv_empty[stage]
    constexpr int BQ = 0, BS = 1, BP = 3, BD = 7, BKF = 9, BKE = 9 + L::kStages;
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + L::kMiscOff);
    volatile int *s_abort = reinterpret_cast<volatile int *>(smem + L::kMiscOff + 4);

    allow_next_kernel();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    const WorkItem item = work_item(p.H, p.Hkv, p.npairs, p.chunks, blockIdx.x);
    const int hk = item.hk, b = item.b, h = item.h;
    const int q0 = 2 * item.tile;                          // first query tile of this CTA
    // key tiles of the two query tiles; the second is absent where the number of query tiles is odd
    const int j0 = p.causal ? q0 + 1 : p.nq, j1 = q0 + 1 < p.nq ? (p.causal ? q0 + 2 : p.nq) : 0;
    const int J = j0 > j1 ? j0 : j1;
    const int q_row0 = (b * p.H + h) * p.S + q0 * 128;     // row in the [B*H*S, D] view
    const int kv_row0 = (b * p.Hkv + hk) * p.S;
    auto stage_of = [&](int l) { return l % L::kStages; };
    auto parity_of = [&](int l) { return (uint32_t)((l / L::kStages) & 1); };

    // ---- setup: the producer starts the first loads, the softmax warps fill their tables, then all meet
    constexpr int kQkBoxes = kQK8 ? 1 : 2;
    constexpr uint32_t kQkTileBytes = kQK8 ? 128 * D : L::kTileBytes;
    const int n_early = 2 * J < L::kStages ? 2 * J : L::kStages;     // loads that need no free stage
    auto load_kv = [&](int l) {                                      // l = 2 j: K_j, 2 j + 1: V_j
#ifdef BAPS_TEST_SKIP_LOAD
        if (l == g_test_skip_load) return;                           // this tile never arrives
#endif
        const int s = stage_of(l);
        mbar_arrive_expect_tx(bar(BKF + s), (l & 1) ? (uint32_t)L::kTileBytes : kQkTileBytes);
        const CUtensorMap *m = (l & 1) ? &mv : &mk;
        for (int hh = 0; hh < ((l & 1) ? 2 : kQkBoxes); ++hh)
            tma_load_2d(sbase + L::kKvOff + s * L::kTileBytes + hh * 16384, m, hh * 64, kv_row0 + (l >> 1) * 128, bar(BKF + s));
    };
    if (tid == 0) *s_abort = 0;
    if (warp == 16) {
        if (lane == 0) {
            mbar_init(bar(BQ), 1);
            for (int t = 0; t < 2; ++t) { mbar_init(bar(BS + t), 1); mbar_init(bar(BD + t), 1); }
            for (int i = 0; i < 4; ++i) mbar_init(bar(BP + i), 8);
            for (int s = 0; s < L::kStages; ++s) { mbar_init(bar(BKF + s), 1); mbar_init(bar(BKE + s), 1); }
            mbar_fence_init();
            await_previous_kernel();
            mbar_arrive_expect_tx(bar(BQ), (j1 ? 2u : 1u) * kQkTileBytes);
            for (int t = 0; t < (j1 ? 2 : 1); ++t)
                for (int hh = 0; hh < kQkBoxes; ++hh)
                    tma_load_2d(sbase + L::kQOff + t * L::kTileBytes + hh * 16384, &mq, hh * 64, q_row0 + t * 128, bar(BQ));
            for (int l = 0; l < n_early; ++l) load_kv(l);
        }
        __syncwarp();
    } else if (warp == 17) {
        tmem_alloc(smem_u32(s_tmem), 512); tmem_relinquish();
        if (lane == 0) { tma_prefetch_desc(&mq); tma_prefetch_desc(&mk); tma_prefetch_desc(&mv); }
    } else if (warp < kTcSoftmaxWarps) {
        fill_attention_tables(smem + L::kLutRepOff, smem + L::kLutFullOff, tid, kTcSoftmaxWarps * 32);
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *s_tmem;                        // S_0 | S_1 | O_0 | O_1

    if (warp >= kTcSoftmaxWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kTcSplit.few));
        if (warp == 16) {
            // ======================= TMA producer ==================================================
            if (lane == 0) {
                int issued = n_early;
                for (int l = n_early; l < 2 * J; ++l) {
                    if (!mbar_wait(bar(BKE + stage_of(l)), parity_of(l) ^ 1u, s_abort, &g_async_status, 0x100 + stage_of(l))) break;
                    load_kv(l);
                    issued = l + 1;
                }
                if (*s_abort) {
                    // let copies already in flight land before the CTA's shared memory is released
                    for (int l = issued > L::kStages ? issued - L::kStages : 0; l < issued; ++l) {
                        const uint64_t t0 = globaltimer_ns();
                        while (!mbar_try_wait(bar(BKF + stage_of(l)), parity_of(l)) && globaltimer_ns() - t0 < 2000000ull) {}
                    }
                }
            }
        } else if (warp == 17) {
            // ======================= MMA issuer ====================================================
            // (the whole warp runs the loop so that the compiler can keep it on the uniform datapath)
            constexpr uint32_t idesc_qk = make_idesc_bf16(128, 128, false);
            constexpr uint32_t idesc_pv = make_idesc_bf16(128, D, true);
            auto wait_all = [&](uint32_t bar_addr, uint32_t parity, int code) -> bool {
                return __all_sync(0xffffffffu, mbar_wait(bar_addr, parity, s_abort, &g_async_status, code));
            };
            auto mma_qk = [&](int t, int j) {
                const uint32_t qd = sdesc_lo(sbase + L::kQOff + t * L::kTileBytes, 16);
                const uint32_t kd = sdesc_lo(sbase + L::kKvOff + stage_of(2 * j) * L::kTileBytes, 16);
                const uint32_t sd = tmem + t * 128;
                if constexpr (kQK8) {
                    constexpr uint32_t idesc_qk8 = make_idesc_e4m3(128, 128);
#pragma unroll
                    for (int ks = 0; ks < D / 32; ++ks) mma_ss_lo_f8(sd, qd + 2u * ks, kd + 2u * ks, idesc_qk8, ks > 0);
                } else {
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        const uint32_t off = (uint32_t)(((ks >> 2) * 16384 + (ks & 3) * 32) >> 4);
                        mma_ss_lo(sd, qd + off, kd + off, idesc_qk, ks > 0);
                    }
                }
                mma_commit(bar(BS + t));
                if (t == (j < j1 ? 1 : 0)) mma_commit(bar(BKE + stage_of(2 * j)));         // the last that reads K_j
            };
            // O_t += P V_j over the keys of one half of the weights: 32-column quarters 1 and 3 (first), then 0 and 2
            auto mma_pv = [&](int t, int j, int half) {
                const uint32_t vd = sdesc_lo(sbase + L::kKvOff + stage_of(2 * j + 1) * L::kTileBytes, 16384);
                const uint32_t od = tmem + 256 + t * D, pd = tmem + t * 128;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int quarter = (i >> 1) * 2 + 1 - half, ks = 2 * quarter + (i & 1);
                    mma_ts_lo(od, pd + quarter * 32 + (i & 1) * 8, vd + ks * 128, idesc_pv, half || i || j > 0 ? 1u : 0u);
                }
            };
            const bool leader = elect_one();
            bool ok = wait_all(bar(BQ), 0, 0x200) && wait_all(bar(BKF), 0, 0x210);
            if (ok) {
                tc_fence_after_sync();
                if (leader) {
                    mma_qk(0, 0);
                    if (j1) mma_qk(1, 0);
                }
                __syncwarp();
            }
            for (int j = 0; ok && j < J; ++j) {
                // what both bursts of this step need besides the weights
                ok = wait_all(bar(BKF + stage_of(2 * j + 1)), parity_of(2 * j + 1), 0x220) &&
                     (j + 1 >= J || wait_all(bar(BKF + stage_of(2 * j + 2)), parity_of(2 * j + 2), 0x211));
                for (int t = 0; ok && t < 2; ++t) {
                    const int jt = t ? j1 : j0;
                    if (j >= jt) continue;
                    ok = wait_all(bar(BP + 2 * t), (uint32_t)(j & 1), 0x230 + t);
                    if (!ok) break;
                    tc_fence_after_sync();
                    if (leader) mma_pv(t, j, 0);
                    __syncwarp();
                    ok = wait_all(bar(BP + 2 * t + 1), (uint32_t)(j & 1), 0x232 + t);
                    if (!ok) break;
                    tc_fence_after_sync();
                    if (leader) {
                        mma_pv(t, j, 1);
                        if (j + 1 < jt) mma_qk(t, j + 1);
                        mma_commit(bar(BD + t));
                        if (t == (j < j1 ? 1 : 0)) mma_commit(bar(BKE + stage_of(2 * j + 1)));
                    }
                    __syncwarp();
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kTcSplit.many));
        // ======================= softmax warps ==================================================
        await_previous_kernel();
        const int t = warp >> 3;                 // query tile
        const int q4 = warp & 3;                 // TMEM lane quarter: rows 32 q4 .. 32 q4 + 31
        const int ch = (warp >> 2) & 1;          // key column half: columns 64 ch .. 64 ch + 63
        const int qi = q0 + t, jt = t ? j1 : j0;
        const int row = q4 * 32 + lane;
        const uint32_t lane_sel = (uint32_t)(q4 * 32) << 16;
        const uint32_t s_addr = tmem + lane_sel + t * 128 + ch * 64;
        const uint32_t o_addr = tmem + lane_sel + 256 + t * D + ch * 64;
        const uint32_t lut_full = sbase + L::kLutFullOff;
        const uint32_t tb = sbase + L::kLutRepOff + (uint32_t)lane * 4u;
        const uint32_t xrow = sbase + L::kXchgOff + (uint32_t)(t * 2048 + row * 8);   // + 1024 * (j & 1); my slot + 4 ch
        const uint32_t vote_bar = 1 + t, row_bar = 3 + t * 4 + q4;
        const bool count_restarts = p.restarts != nullptr && (warp & 7) == 0;
        const float over_thr = restart_threshold(p.lambda);
        RowState st{-INFINITY, 0.f, 0.f, 0u};
        int n_restart = 0;

        auto tile = [&](auto first, const int j) {
            constexpr bool hp = decltype(first)::value;          // B0: the high-precision tile
            float c = p.c;
            if constexpr (kQK8)
                c *= ldg_f32(p.q_scale + (size_t)(b * p.H + h) * p.nq + qi) * ldg_f32(p.k_scale + (size_t)(b * p.Hkv + hk) * p.nq + j);
            const uint32_t x_addr = xrow + (uint32_t)(j & 1) * 1024u;
            const bool diag = p.causal && j == qi;
            uint32_t r[32];
            float g[8];
            mbar_wait(bar(BS + t), (uint32_t)(j & 1), s_abort, &g_async_status, 0x300 + t);
            tc_fence_after_sync();
            // ---- maxima of my 64 columns, exchange with the partner thread, tile-wide vote ----------------
            auto mask_chunk = [&](uint32_t (&x)[32], int cc) {
                if (diag) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) x[i] = (ch * 64 + cc * 32 + i > row) ? 0xFF800000u : x[i];
                }
            };
            {
                // (both chunks on their way at once: nothing else is in registers yet)
                uint32_t x[32];
                tmem_ld32(s_addr, x);
                tmem_ld32(s_addr + 32, r);
                tmem_wait_ld();
                mask_chunk(x, 0);
                mask_chunk(r, 1);
#pragma unroll
                for (int i = 0; i < 4; ++i) g[i] = max8(&x[8 * i]);
#pragma unroll
                for (int i = 0; i < 4; ++i) g[4 + i] = max8(&r[8 * i]);
            }
            const float hm = max3(max3(g[0], g[1], g[2]), max3(g[3], g[4], g[5]), fmaxf(g[6], g[7]));
            sts_f32(x_addr + 4u * (uint32_t)ch, hm);
            bool restart_tile = false;
            if constexpr (hp) named_bar_sync(row_bar, 64);
            else restart_tile = named_bar_or(vote_bar, 256, fmaf(hm, c, -st.m) >= over_thr);
            const float2 pm = lds_f32x2(x_addr);
            const float mx = fmaxf(pm.x, pm.y);
            // ---- decisions (Algorithm 1) -------------------------------------------------------------------
            bool changed = false;                 // the max moves in some row of the warp (with or without a restart)
            float m_next = st.m;
            if constexpr (hp) {
                st.m = st.m_ref = m_next = fmaxf(st.m, int_max(mx, c));      // -inf for a row of NaN
            } else {
                const float um = fmaf(mx, c, -st.m);
                changed = restart_tile || __any_sync(0xffffffffu, um > 0.f);
                if (changed) {
                    if (count_restarts && restart_tile) ++n_restart;
                    m_next = st.decide(mx, c, um, restart_tile, [&](float f) {
                        mbar_wait(bar(BD + t), (uint32_t)((j - 1) & 1), s_abort, &g_async_status, 0x330 + t);
                        tc_fence_after_sync();
                        rescale_columns(o_addr, 64, f);
                    });
                }
            }
            // ---- weights -> bf16 P over score columns already read; row sum ---------------------------------
            float sum = 0.f;
            uint64_t s01 = 0ull, s23 = 0ull;
            const float mnv = kQK8 ? -st.m : st.m * 7.52316384526264e-37f;        // 2^-120
            const float cnv = kQK8 ? c : -c * 7.52316384526264e-37f;
            const uint64_t cn2 = pack2(cnv, cnv), mn2 = pack2(mnv, mnv);
            // the 8-column groups that hold a positive T are redone after the fast path
            const uint32_t pos = changed && !restart_tile ? positive_groups(g, c, st.m) : 0u;
            auto weights = [&](int cc) {
                uint32_t pk[16];
                if constexpr (hp) {
                    sum += hp16(&r[0], &pk[0], c, st.m) + hp16(&r[16], &pk[8], c, st.m);
                } else {
                    fast16<kQK8>(&r[0], &pk[0], cn2, mn2, st.escale, tb, s01, s23);
                    fast16<kQK8>(&r[16], &pk[8], cn2, mn2, st.escale, tb, s01, s23);
                    if (pos) {
#pragma unroll
                        for (int gg = 0; gg < 4; ++gg)
                            if (pos >> (4 * cc + gg) & 1u) sum += fix8(&r[gg * 8], &pk[gg * 4], c, st.m, lut_full);
                    }
                }
                tmem_st16(s_addr + cc * 32, pk);
            };
            auto arrive = [&](int half) {
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(BP + 2 * t + half));
            };
            weights(1);
            arrive(0);                                    // the tensor core starts on the keys of the second chunks
            tmem_ld32(s_addr, r);
            tmem_wait_ld();
            mask_chunk(r, 0);
            weights(0);
            arrive(1);                                    // all of P is in place
            if constexpr (!hp) {
                float a0, a1, a2, a3;
                unpack2(s01, a0, a1); unpack2(s23, a2, a3);
                sum += (a0 + a1) + (a2 + a3);
            }
            st.add(sum);
            if (changed) st.move(m_next);
        };
        if (jt > 0) tile(std::true_type{}, 0);
        for (int j = 1; j < jt; ++j) tile(std::false_type{}, j);
        const bool ok = (*s_abort == 0);

        // ---- epilogue: O = O~ / d (each thread: its half of the output columns) -------------------------
        if (jt > 0) {
            const bool good = mbar_wait(bar(BD + t), (uint32_t)((jt - 1) & 1), s_abort, &g_async_status, 0x320 + t) && ok;
            tc_fence_after_sync();
            // the exchange buffer not used by the tile before (that one may still be read by the partner)
            const uint32_t x_addr = xrow + (uint32_t)(jt & 1) * 1024u;
            sts_f32(x_addr + 4u * (uint32_t)ch, st.d);
            named_bar_sync(row_bar, 64);
            const float2 pd = lds_f32x2(x_addr);
            const float dtot = pd.x + pd.y, dinv = 1.f / dtot;
            const size_t grow = (size_t)q_row0 + (size_t)t * 128 + row;      // row in [B*H*S]
            // staged through the (now idle) Q tile, 16-byte chunks of a row XOR-swizzled with the row number, so
            // that the global stores are whole rows
            const uint32_t stage = sbase + L::kQOff + t * L::kTileBytes;
#pragma unroll 1
            for (int i0 = 0; i0 < 64; i0 += 16) {
                uint32_t rr[16];
                tmem_ld16(o_addr + i0, rr);
                tmem_wait_ld();
                float o[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) o[i] = __uint_as_float(rr[i]) * dinv;
                if (p.out) {
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int chunk = (ch * 64 + i0) / 8 + i;
                        sts_u32x4(stage + (uint32_t)row * 256u + (uint32_t)((chunk ^ (row & 15)) * 16),
                                  make_uint4(pack_bf16x2(o[8 * i], o[8 * i + 1]), pack_bf16x2(o[8 * i + 2], o[8 * i + 3]),
                                             pack_bf16x2(o[8 * i + 4], o[8 * i + 5]), pack_bf16x2(o[8 * i + 6], o[8 * i + 7])));
                    }
                }
                if (p.out_f32 && good) {
                    float4 *dst = reinterpret_cast<float4 *>(p.out_f32 + grow * D + ch * 64 + i0);
#pragma unroll
                    for (int i = 0; i < 4; ++i) dst[i] = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
                }
            }
            if (p.out) {
                named_bar_sync(row_bar, 64);
#pragma unroll
                for (int it = 0; it < 8; ++it) {
                    const int rw = q4 * 32 + ch * 16 + it * 2 + lane / 16, chunk = lane % 16;
                    const uint4 v = lds_u32x4(stage + (uint32_t)rw * 256u + (uint32_t)((chunk ^ (rw & 15)) * 16));
                    if (good)
                        *reinterpret_cast<uint4 *>(reinterpret_cast<uint8_t *>(p.out) +
                                                   ((size_t)q_row0 + (size_t)t * 128 + rw) * 256 + chunk * 16) = v;
                }
            }
            if (good) {
                if (ch == 0) {
                    if (p.row_m) p.row_m[grow] = st.m;
                    if (p.row_d) p.row_d[grow] = dtot * pow2_int(st.m_ref - st.m);
                }
                if (count_restarts && lane == 0) p.restarts[(size_t)(b * p.H + h) * p.nq + qi] = n_restart;
            }
        }
    }

    // ---- teardown ---------------------------------------------------------------------------------
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 17) { __syncwarp(); tmem_dealloc(tmem, 512); }
}

} // namespace baps
