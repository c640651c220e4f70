// Fused BAPS attention forward for heads of 64 (Algorithm 1, bf16 Q / K / V), two CTAs per SM.
//
// At D = 64 the tensor core needs 512 cycles for a 128 x 128 score tile and the softmax side several times that:
// the path is bound by the instructions the softmax warps issue and by how well their waits are covered.  Two
// things follow from the smaller accumulators.  A CTA with one query tile needs 256 columns of tensor memory --
// scores 128 | weights 64 | O~ 64 -- and 109 KB of shared memory, so two CTAs fit an SM, drift freely against each
// other, and one computes weights while the other is between tiles.  And the weights have columns of their own, so
// Q K^T of the next tile starts as soon as the scores of the current one have been read for the last time, while
// its weights are still being formed.  A row is shared by two threads (64 columns each) instead of four, which
// halves the bookkeeping per score.
//   warps 0-7   softmax: warp w owns rows 32 (w % 4) .. + 31 and the 64 key columns of half w / 4, in two chunks of
//               32.  Maxima of both chunks, exchange and tile-wide vote, then the weights of the second chunk
//               (still in registers) and of the first (read again)
//   warp 8      TMA producer: Q, then K_0, V_0, K_1, ... through a ring of four 16 KB stages
//   warp 9      MMA issuer: Q K^T of tile j + 1, then P V of tile j; also allocates the tensor memory
// (warps 10, 11 idle: they complete the warpgroup whose registers go to the softmax warps.)
// The arithmetic, the bounded waits and the way every role ends after an expired wait are those of
// attention_tc_kernel; only the row sum is added up in another order (two partial sums per row, not four).
// Measured against that kernel with two query tiles per CTA (heads x tokens): 512 x 1024 bidirectional 351 -> 330 us,
// 64 x 8192 causal 1233 -> 1101, 24 x 2048 causal 46.2 -> 42.8 on unit-Gaussian inputs; with a per-token key bias
// (more restarts and positive T) 512 x 1024 342 -> 313.  Small grids keep that kernel (two_ctas_per_sm).
// Since then: keys two at a time and decisions only where a max moves (RowState) 64 x 8192 1115 -> 1046 us, 512 x 1024 348
// -> 335; positive T without branches 1045 -> 1001, 335 -> 318; both chunks requested at once 1010 -> 1001, 321 -> 317.  P V in
// two halves, as in paired_attention_tc_kernel, is slower here (1030, 326): Q K^T of the next tile does not wait for it.
#pragma once
#include "baps_attention_tc.cuh"

namespace baps {

constexpr int kD64Threads = kD64Split.threads, kD64SoftmaxWarps = kD64Split.many_threads / 32;

struct D64Layout {
    static constexpr int kTileBytes = 128 * 64 * 2, kStages = 4;
    static constexpr int kQOff = 0;
    static constexpr int kKvOff = kTileBytes;
    static constexpr int kLutRepOff = kKvOff + kStages * kTileBytes;
    static constexpr int kLutFullOff = kLutRepOff + kLutRepBytes;
    static constexpr int kBarOff = (kLutFullOff + kLutN * 4 + 15) & ~15;
    // barriers: q_full, s_full, s_free, p_full, pv_done, kv_full[stages], kv_empty[stages]
    static constexpr int kXchgOff = (kBarOff + (5 + 2 * kStages) * 8 + 15) & ~15;      // float xchg[2][128][2]
    static constexpr int kMiscOff = kXchgOff + 2 * 128 * 2 * 4;                        // tmem base, abort
    static constexpr int kDynBytes = kMiscOff + 16 + 1024;                             // slack for 1024-byte alignment
};
static_assert(2 * (D64Layout::kDynBytes + 1024) <= 228 * 1024, "two CTAs per SM");

__global__ void __launch_bounds__(kD64Threads, 2)
attention_d64_kernel(const __grid_constant__ CUtensorMap mq, const __grid_constant__ CUtensorMap mk,
                     const __grid_constant__ CUtensorMap mv, const AttnTcParams p)
{
    using namespace sm100;
    using L = D64Layout;
    constexpr int D = 64;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    auto bar = [&](int i) { return sbase + L::kBarOff + 8u * (uint32_t)i; };
    constexpr int BQ = 0, BS = 1, BF = 2, BP = 3, BD = 4, BKF = 5, BKE = 5 + L::kStages;
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + L::kMiscOff);
    volatile int *s_abort = reinterpret_cast<volatile int *>(smem + L::kMiscOff + 4);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    const WorkItem item = work_item(p.H, p.Hkv, p.npairs, p.chunks, blockIdx.x);
    const int qi = item.tile, hk = item.hk, b = item.b, h = item.h;
    const int J = p.causal ? qi + 1 : p.nq;               // number of key tiles
    const int q_row0 = (b * p.H + h) * p.S + qi * 128;    // row in the [B*H*S, D] view
    const int kv_row0 = (b * p.Hkv + hk) * p.S;
    auto stage_of = [&](int l) { return l % L::kStages; };
    auto parity_of = [&](int l) { return (uint32_t)((l / L::kStages) & 1); };

    // ---- setup: the producer starts the first loads, the softmax warps fill their tables, then all meet
    const int n_early = 2 * J < L::kStages ? 2 * J : L::kStages;     // loads that need no free stage
    auto load_kv = [&](int l) {                                      // l = 2 j: K_j, 2 j + 1: V_j
#ifdef BAPS_TEST_SKIP_LOAD
        if (l == g_test_skip_load) return;                           // this tile never arrives
#endif
        const int s = stage_of(l);
        mbar_arrive_expect_tx(bar(BKF + s), (uint32_t)L::kTileBytes);
        tma_load_2d(sbase + L::kKvOff + s * L::kTileBytes, (l & 1) ? &mv : &mk, 0, kv_row0 + (l >> 1) * 128, bar(BKF + s));
    };
    if (tid == 0) *s_abort = 0;
    if (warp == 8) {
        if (lane == 0) {
            mbar_init(bar(BQ), 1);
            mbar_init(bar(BS), 1);
            mbar_init(bar(BF), kD64SoftmaxWarps);
            mbar_init(bar(BP), kD64SoftmaxWarps);
            mbar_init(bar(BD), 1);
            for (int s = 0; s < L::kStages; ++s) { mbar_init(bar(BKF + s), 1); mbar_init(bar(BKE + s), 1); }
            mbar_fence_init();
            await_previous_kernel();
            mbar_arrive_expect_tx(bar(BQ), (uint32_t)L::kTileBytes);
            tma_load_2d(sbase + L::kQOff, &mq, 0, q_row0, bar(BQ));
            for (int l = 0; l < n_early; ++l) load_kv(l);
        }
        __syncwarp();
    } else if (warp == 9) {
        // The allocation waits, without a limit, for tensor memory that another CTA on the SM holds.  So none is taken
        // while a kernel ahead may still have to take its own, and the next kernel starts only when every CTA of this
        // one has its share: no two can hold what the other waits for.  (attention_tc_kernel need not care: its CTA takes
        // 61440 of the SM's 65536 registers, and nothing that uses tensor memory fits beside it.)
        await_previous_kernel();
        tmem_alloc(smem_u32(s_tmem), 256); tmem_relinquish();
        allow_next_kernel();
        if (lane == 0) { tma_prefetch_desc(&mq); tma_prefetch_desc(&mk); tma_prefetch_desc(&mv); }
    } else if (warp < kD64SoftmaxWarps) {
        fill_attention_tables(smem + L::kLutRepOff, smem + L::kLutFullOff, tid, kD64SoftmaxWarps * 32);
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *s_tmem;                        // scores | weights (+ 128) | O~ (+ 192)

    if (warp >= kD64SoftmaxWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kD64Split.few));
        if (warp == 8) {
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
        } else if (warp == 9) {
            // ======================= MMA issuer ====================================================
            constexpr uint32_t idesc_qk = make_idesc_bf16(128, 128, false);
            constexpr uint32_t idesc_pv = make_idesc_bf16(128, D, true);
            auto wait_all = [&](uint32_t bar_addr, uint32_t parity, int code) -> bool {
                return __all_sync(0xffffffffu, mbar_wait(bar_addr, parity, s_abort, &g_async_status, code));
            };
            const bool leader = elect_one();
            auto mma_qk = [&](int j) {
                const uint32_t qd = sdesc_lo(sbase + L::kQOff, 16);
                const uint32_t kd = sdesc_lo(sbase + L::kKvOff + stage_of(2 * j) * L::kTileBytes, 16);
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) mma_ss_lo(tmem, qd + 2u * ks, kd + 2u * ks, idesc_qk, ks > 0);
                mma_commit(bar(BS));
                mma_commit(bar(BKE + stage_of(2 * j)));
            };
            bool ok = wait_all(bar(BQ), 0, 0x200) && wait_all(bar(BKF), 0, 0x210);
            if (ok) {
                tc_fence_after_sync();
                if (leader) mma_qk(0);
                __syncwarp();
            }
            for (int j = 0; ok && j < J; ++j) {
                if (j + 1 < J) {
                    // scores of the next tile as soon as the present ones have been read
                    ok = wait_all(bar(BKF + stage_of(2 * j + 2)), parity_of(2 * j + 2), 0x211) &&
                         wait_all(bar(BF), (uint32_t)(j & 1), 0x231);
                    if (!ok) break;
                    tc_fence_after_sync();
                    if (leader) mma_qk(j + 1);
                    __syncwarp();
                }
                ok = wait_all(bar(BKF + stage_of(2 * j + 1)), parity_of(2 * j + 1), 0x220) &&
                     wait_all(bar(BP), (uint32_t)(j & 1), 0x230);
                if (!ok) break;
                tc_fence_after_sync();
                if (leader) {
                    const uint32_t vd = sdesc_lo(sbase + L::kKvOff + stage_of(2 * j + 1) * L::kTileBytes, 16384);
                    const uint32_t acc0 = j > 0 ? 1u : 0u;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int ks = (i >> 1 & 1) * 4 + (i < 4 ? 2 : 0) + (i & 1);      // as in attention_tc_kernel
                        mma_ts_lo(tmem + 192, tmem + 128 + ks * 8, vd + ks * 128, idesc_pv, i > 0 ? 1u : acc0);
                    }
                    mma_commit(bar(BD));
                    mma_commit(bar(BKE + stage_of(2 * j + 1)));
                }
                __syncwarp();
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kD64Split.many));
        // ======================= softmax warps ==================================================
        await_previous_kernel();
        const int q4 = warp & 3;                 // TMEM lane quarter: rows 32 q4 .. 32 q4 + 31
        const int ch = warp >> 2;                // key column half: columns 64 ch .. 64 ch + 63
        const int row = q4 * 32 + lane;
        const uint32_t lane_sel = (uint32_t)(q4 * 32) << 16;
        const uint32_t s_addr = tmem + lane_sel + ch * 64, p_addr = tmem + lane_sel + 128 + ch * 32;
        const uint32_t o_addr = tmem + lane_sel + 192 + ch * 32;
        const uint32_t lut_full = sbase + L::kLutFullOff;
        const uint32_t tb = sbase + L::kLutRepOff + (uint32_t)lane * 4u;
        const uint32_t xrow = sbase + L::kXchgOff + (uint32_t)row * 8u;   // + 1024 * (j & 1); my slot + 4 ch
        const float c = p.c;
        const bool count_restarts = p.restarts != nullptr && warp == 0;
        const float over_thr = restart_threshold(p.lambda);
        RowState st{-INFINITY, 0.f, 0.f, 0u};
        int n_restart = 0;

        auto tile = [&](auto first, const int j) {
            constexpr bool hp = decltype(first)::value;          // B0: the high-precision tile
            const uint32_t x_addr = xrow + (uint32_t)(j & 1) * 1024u;
            const bool diag = p.causal && j == qi;
            uint32_t r[32];
            float g[8];
            mbar_wait(bar(BS), (uint32_t)(j & 1), s_abort, &g_async_status, 0x300);
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
            if constexpr (hp) named_bar_sync(2 + q4, 64);
            else restart_tile = named_bar_or(1, kD64SoftmaxWarps * 32, fmaf(hm, c, -st.m) >= over_thr);
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
                        mbar_wait(bar(BD), (uint32_t)((j - 1) & 1), s_abort, &g_async_status, 0x330);
                        tc_fence_after_sync();
                        rescale_columns(o_addr, 32, f);
                    });
                }
            }
            // ---- weights -> bf16 P; row sum ---------------------------------------------------------------
            float sum = 0.f;
            uint64_t s01 = 0ull, s23 = 0ull;
            const float mnv = st.m * 7.52316384526264e-37f, cnv = -c * 7.52316384526264e-37f;     // 2^-120
            const uint64_t cn2 = pack2(cnv, cnv), mn2 = pack2(mnv, mnv);
            // the 8-column groups that hold a positive T are redone after the fast path
            const uint32_t pos = changed && !restart_tile ? positive_groups(g, c, st.m) : 0u;
            auto weights = [&](int cc) {
                uint32_t pk[16];
                if constexpr (hp) {
                    sum += hp16(&r[0], &pk[0], c, st.m) + hp16(&r[16], &pk[8], c, st.m);
                } else {
                    fast16<false>(&r[0], &pk[0], cn2, mn2, st.escale, tb, s01, s23);
                    fast16<false>(&r[16], &pk[8], cn2, mn2, st.escale, tb, s01, s23);
                    if (pos) {
#pragma unroll
                        for (int gg = 0; gg < 4; ++gg)
                            if (pos >> (4 * cc + gg) & 1u) sum += fix8(&r[gg * 8], &pk[gg * 4], c, st.m, lut_full);
                    }
                }
                tmem_st16(p_addr + cc * 16, pk);
            };
            // P V of the tile before has read its weights (long done, as a rule)
            if constexpr (!hp) {
                mbar_wait(bar(BD), (uint32_t)((j - 1) & 1), s_abort, &g_async_status, 0x331);
                tc_fence_after_sync();
            }
            weights(1);
            tmem_ld32(s_addr, r);
            tmem_wait_ld();
            mask_chunk(r, 0);
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(BF));          // the scores have been read for the last time
            weights(0);
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(BP));          // P is in place
            if constexpr (!hp) {
                float a0, a1, a2, a3;
                unpack2(s01, a0, a1); unpack2(s23, a2, a3);
                sum += (a0 + a1) + (a2 + a3);
            }
            st.add(sum);
            if (changed) st.move(m_next);
        };
        tile(std::true_type{}, 0);
        for (int j = 1; j < J; ++j) tile(std::false_type{}, j);
        const bool ok = (*s_abort == 0);

        // ---- epilogue: O = O~ / d (each thread: its half of the output columns) -------------------------
        const bool good = mbar_wait(bar(BD), (uint32_t)((J - 1) & 1), s_abort, &g_async_status, 0x320) && ok;
        tc_fence_after_sync();
        // the exchange buffer not used by the tile before (that one may still be read by the partner)
        const uint32_t x_addr = xrow + (uint32_t)(J & 1) * 1024u;
        sts_f32(x_addr + 4u * (uint32_t)ch, st.d);
        named_bar_sync(2 + q4, 64);
        const float2 pd = lds_f32x2(x_addr);
        const float dtot = pd.x + pd.y, dinv = 1.f / dtot;
        const size_t grow = (size_t)q_row0 + row;                    // row in [B*H*S]
        // staged through the (now idle) Q tile, 16-byte chunks of a row XOR-swizzled with the row number, so
        // that the global stores are whole rows
        const uint32_t stage = sbase + L::kQOff;
#pragma unroll 1
        for (int i0 = 0; i0 < 32; i0 += 16) {
            uint32_t rr[16];
            tmem_ld16(o_addr + i0, rr);
            tmem_wait_ld();
            float o[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] = __uint_as_float(rr[i]) * dinv;
            if (p.out) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int chunk = (ch * 32 + i0) / 8 + i;
                    sts_u32x4(stage + (uint32_t)row * 128u + (uint32_t)((chunk ^ (row & 7)) * 16),
                              make_uint4(pack_bf16x2(o[8 * i], o[8 * i + 1]), pack_bf16x2(o[8 * i + 2], o[8 * i + 3]),
                                         pack_bf16x2(o[8 * i + 4], o[8 * i + 5]), pack_bf16x2(o[8 * i + 6], o[8 * i + 7])));
                }
            }
            if (p.out_f32 && good) {
                float4 *dst = reinterpret_cast<float4 *>(p.out_f32 + grow * D + ch * 32 + i0);
#pragma unroll
                for (int i = 0; i < 4; ++i) dst[i] = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
            }
        }
        if (p.out) {
            named_bar_sync(2 + q4, 64);
#pragma unroll
            for (int it = 0; it < 4; ++it) {
                const int rw = q4 * 32 + ch * 16 + it * 4 + lane / 8, chunk = lane % 8;
                const uint4 v = lds_u32x4(stage + (uint32_t)rw * 128u + (uint32_t)((chunk ^ (rw & 7)) * 16));
                if (good)
                    *reinterpret_cast<uint4 *>(reinterpret_cast<uint8_t *>(p.out) + ((size_t)q_row0 + rw) * 128 + chunk * 16) = v;
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

    // ---- teardown ---------------------------------------------------------------------------------
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 9) { __syncwarp(); tmem_dealloc(tmem, 256); }
}

} // namespace baps
