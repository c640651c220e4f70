// Host side of the bf16 / 8-bit fused attention: tensor maps, choice of kernel, launch.
#pragma once
#include "baps_attention_d64.cuh"
#include "baps_attention_tc.cuh"
#include "baps_tma_host.cuh"

namespace baps {

// One query tile per CTA or two?  Two share the K / V stream and the set-up of the CTA, and a task (one score
// tile, 1.35 us) waits less on the one before it; one halves the chain of tasks that the longest CTA walks
// through, which is what a grid that does not fill the SMs several times over takes.  Estimate of both in units
// of a two-tile task, SMs filled longest CTA first: the longest CTA or the average load of an SM, whichever is
// larger (all CTAs of a bidirectional problem are equally long: whole waves).  Besides its tasks a CTA costs
// kFixedTwo / kFixedOne (set-up, first scores, epilogues).  Measured, two tiles -> one (D = 128, causal, heads x
// tokens): 4 x 512 15.8 -> 11.4 us, 8 x 4096 90.8 -> 58.1, 32 x 1024 28.8 -> 23.7, 1 x 16384 326 -> 215; and
// where two stay: 16 x 4096 90.6 -> 111, 32 x 2048 53.7 -> 67, 4 x 32768 1190 -> 1501.
static inline bool one_tile_per_cta(long long heads, int nq, bool causal, int num_sms)
{
    constexpr double kFixedTwo = 4.5, kFixedOne = 3.5, kTaskOne = 1.25;
    const long long ctas2 = heads * ((nq + 1) / 2), ctas1 = heads * nq;
    const double longest1 = kTaskOne * nq + kFixedOne, longest2 = (causal || nq == 1 ? 2 * nq - 1 : 2 * nq) + kFixedTwo;
    double t1, t2;
    if (causal) {
        const double tasks = (double)heads * nq * (nq + 1) / 2;
        const double load1 = (kTaskOne * tasks + kFixedOne * ctas1) / num_sms, load2 = (tasks + kFixedTwo * ctas2) / num_sms;
        t1 = load1 > longest1 ? load1 : longest1;
        t2 = load2 > longest2 ? load2 : longest2;
    } else {
        t1 = (double)((ctas1 + num_sms - 1) / num_sms) * longest1;
        t2 = (double)((ctas2 + num_sms - 1) / num_sms) * longest2;
    }
    return t1 < t2;
}

// Heads of 64: attention_d64_kernel (two CTAs per SM) or attention_tc_kernel with one query tile per CTA, whose
// sixteen softmax warps are through with a lone tile sooner (1.25 us a task against 1.76 alone and 2.4 shared,
// but 1.22 per task and SM)?  The former when the SMs are full: more tiles than SMs (bidirectional: tiles 128
// 22.8 us against 15.4, 160 24.1 / 28.1, 512 47.8 / 57.4, 4096 330 / 403), or an average load of an SM of 1.3 times
// the longest causal tile (heads x tokens: 24 x 1024 21.5 / 15.6, 24 x 2048 42.8 / 44.2, 2 x 16384 265 / 162,
// 64 x 8192 1101 / 1269).
static inline bool two_ctas_per_sm(long long heads, int nq, bool causal, int num_sms)
{
    return causal ? 10 * heads * (nq + 1) >= 26LL * num_sms : heads * nq > num_sms;
}

// Host side: tensor maps, launch.
static inline baps_status attention_tc_launch(const void *q, const void *k, const void *v, void *out, int B, int H,
                                       int Hkv, int S, int D, int causal, int lambda, int mode, int b0_last, float c,
                                       const baps_stats &st, int num_sms, cudaStream_t stream,
                                       const float *q_scale = nullptr, const float *k_scale = nullptr)
{
    const bool qk8 = q_scale != nullptr;               // Q, K are E4M3 codes with per-tile scales
    CUtensorMap mq, mk, mv;
    if (qk8) {
        if (!make_tmap_u8_rows(&mq, q, (uint64_t)B * H * S, (uint64_t)D, 128) ||
            !make_tmap_u8_rows(&mk, k, (uint64_t)B * Hkv * S, (uint64_t)D, 128))
            return BAPS_ERR_CUDA;
    } else if (!make_tmap_bf16_rows(&mq, q, (uint64_t)B * H * S, (uint64_t)D, 128) ||
               !make_tmap_bf16_rows(&mk, k, (uint64_t)B * Hkv * S, (uint64_t)D, 128)) {
        return BAPS_ERR_CUDA;
    }
    if (!make_tmap_bf16_rows(&mv, v, (uint64_t)B * Hkv * S, (uint64_t)D, 128)) return BAPS_ERR_CUDA;
    AttnTcParams p;
    p.out = reinterpret_cast<__nv_bfloat16 *>(out);
    p.out_f32 = st.out_f32; p.row_m = st.row_m; p.row_d = st.row_d; p.restarts = st.restarts;
    p.B = B; p.H = H; p.Hkv = Hkv; p.S = S; p.causal = causal; p.lambda = lambda; p.mode = mode; p.c = c;
    p.b0_last = (b0_last && mode == BAPS_MODE_E2E_HIF8) ? 1 : 0;
    p.q_scale = q_scale; p.k_scale = k_scale;
    p.nq = S / 128;
    const bool usual = mode == BAPS_MODE_E2E_HIF8 && !p.b0_last;
    const bool d64 = D == 64 && usual && two_ctas_per_sm((long long)B * H, p.nq, causal != 0, num_sms);
    const bool one = p.b0_last || (usual && (D == 64 || one_tile_per_cta((long long)B * H, p.nq, causal != 0, num_sms)));
    p.npairs = one ? p.nq : (p.nq + 1) / 2;
    const long long nblocks = (long long)p.npairs * B * H;
    {
        // Chunks of kv heads whose K and V take 16 MB, but CTAs enough in each to keep the SMs evenly busy (causal:
        // three per SM, heavy and light ones mixed; with fewer 32 x 4096 tokens ran 2 % slower), and none at
        // all unless there are at least two.  Measured, inputs not in L2: 512 x 1024 of D = 64 344 -> 313 us,
        // 32 / 8 heads x 32768 9.89 -> 9.76 ms.
        const long long kv_heads = (long long)B * Hkv, per_kv = (long long)p.npairs * (H / Hkv);
        const long long least = ((causal ? 3LL : 2LL) * num_sms + per_kv - 1) / per_kv;
        long long chunk = (16LL << 20) / ((long long)S * D * (qk8 ? 3 : 4));
        if (chunk < least) chunk = least;
        p.chunk = (int)(2 * chunk > kv_heads ? kv_heads : chunk);
    }
    if (nblocks > 0x7fffffffLL) return BAPS_ERR_UNSUPPORTED;
    auto launch = [&](auto kernel, int sm, int threads = kTcThreads) -> baps_status {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sm) != cudaSuccess)
            return BAPS_ERR_CUDA;
        return launch_kernel(kernel, (unsigned)nblocks, threads, (size_t)sm, stream, mq, mk, mv, p);
    };
    constexpr int kE2E = BAPS_MODE_E2E_HIF8, kExact = BAPS_MODE_EXACT, kExp2m = BAPS_MODE_EXP2_HIF8;
    const bool b0l = p.b0_last != 0;
    if (qk8) {
        if (D != 128) return BAPS_ERR_UNSUPPORTED;
        if (mode == kExp2m) return launch(attention_tc_kernel<128, kExp2m, true, false>, TcLayout<128>::kDynBytes);
        if (mode == kExact) return launch(attention_tc_kernel<128, kExact, true, false>, TcLayout<128>::kDynBytes);
        return b0l ? launch(attention_tc_kernel<128, kE2E, true, true>, TcLayout<128>::kDynBytes)
                   : one ? launch(attention_tc_kernel<128, kE2E, true, false, true>, TcLayout<128>::kDynBytes)
                         : launch(attention_tc_kernel<128, kE2E, true, false, false>, TcLayout<128>::kDynBytes);
    }
    if (D == 128) {
        if (mode == kExp2m) return launch(attention_tc_kernel<128, kExp2m, false, false>, TcLayout<128>::kDynBytes);
        if (mode == kExact) return launch(attention_tc_kernel<128, kExact, false, false>, TcLayout<128>::kDynBytes);
        return b0l ? launch(attention_tc_kernel<128, kE2E, false, true>, TcLayout<128>::kDynBytes)
                   : one ? launch(attention_tc_kernel<128, kE2E, false, false, true>, TcLayout<128>::kDynBytes)
                         : launch(attention_tc_kernel<128, kE2E, false, false, false>, TcLayout<128>::kDynBytes);
    }
    if (mode == kExp2m) return launch(attention_tc_kernel<64, kExp2m, false, false>, TcLayout<64>::kDynBytes);
    if (mode == kExact) return launch(attention_tc_kernel<64, kExact, false, false>, TcLayout<64>::kDynBytes);
    if (d64) return launch(attention_d64_kernel, D64Layout::kDynBytes, kD64Threads);
    return b0l ? launch(attention_tc_kernel<64, kE2E, false, true>, TcLayout<64>::kDynBytes)
               : launch(attention_tc_kernel<64, kE2E, false, false, true>, TcLayout<64>::kDynBytes);
}

} // namespace baps
