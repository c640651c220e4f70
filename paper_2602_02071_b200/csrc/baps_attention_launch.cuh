// Host side of the bf16 / 8-bit fused attention: tensor maps, choice of kernel, launch.
#pragma once
#include "baps_attention_d64.cuh"
#include "baps_attention_pair.cuh"
#include "baps_attention_tc.cuh"
#include "baps_tma_host.cuh"

namespace baps {

// Whether the compiled kernel has the registers that its roles share out (see split_fits); asked once per kernel, the
// answer is part of the module image.
template <auto kernel>
static inline bool has_registers_for(const RegisterSplit &split)
{
    static std::atomic<bool> yes{false};
    if (yes.load(std::memory_order_relaxed)) return true;
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, kernel) != cudaSuccess) { (void)cudaGetLastError(); return false; }
    if (!split_fits(split, a.numRegs)) return false;
    yes.store(true, std::memory_order_relaxed);
    return true;
}

struct AttnLaunch { CUtensorMap mq, mk, mv; AttnTcParams p; long long nblocks; cudaStream_t stream; };
template <auto kernel, int kSmem>
static inline baps_status launch_attention(const AttnLaunch &a, const RegisterSplit &split = kTcSplit)
{
    if (!has_registers_for<kernel>(split) ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) != cudaSuccess)
        return BAPS_ERR_CUDA;
    return launch_kernel(kernel, (unsigned)a.nblocks, split.threads, (size_t)kSmem, a.stream, a.mq, a.mk, a.mv, a.p);
}

// Tensor maps, choice of kernel, launch.
static inline baps_status attention_tc_launch(const void *q, const void *k, const void *v, void *out, int B, int H,
                                       int Hkv, int S, int D, int causal, int lambda, int mode, int b0_last, float c,
                                       const baps_stats &st, int num_sms, cudaStream_t stream,
                                       const float *q_scale = nullptr, const float *k_scale = nullptr)
{
    const bool qk8 = q_scale != nullptr;               // Q, K are E4M3 codes with per-tile scales
    AttnLaunch a;
    if (qk8) {
        if (!make_tmap_u8_rows(&a.mq, q, (uint64_t)B * H * S, (uint64_t)D, 128) ||
            !make_tmap_u8_rows(&a.mk, k, (uint64_t)B * Hkv * S, (uint64_t)D, 128))
            return BAPS_ERR_CUDA;
    } else if (!make_tmap_bf16_rows(&a.mq, q, (uint64_t)B * H * S, (uint64_t)D, 128) ||
               !make_tmap_bf16_rows(&a.mk, k, (uint64_t)B * Hkv * S, (uint64_t)D, 128)) {
        return BAPS_ERR_CUDA;
    }
    if (!make_tmap_bf16_rows(&a.mv, v, (uint64_t)B * Hkv * S, (uint64_t)D, 128)) return BAPS_ERR_CUDA;
    AttnTcParams &p = a.p;
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
    a.nblocks = (long long)p.npairs * B * H;
    a.stream = stream;
    p.chunks = kv_chunks((long long)B * Hkv, (long long)S * D * (qk8 ? 3 : 4), (long long)p.npairs * (H / Hkv),
                         causal != 0, num_sms, d64 ? 2 : 1);
    if (a.nblocks > 0x7fffffffLL) return BAPS_ERR_UNSUPPORTED;
    constexpr int kE2E = BAPS_MODE_E2E_HIF8, kExact = BAPS_MODE_EXACT, kExp2m = BAPS_MODE_EXP2_HIF8;
    const bool b0l = p.b0_last != 0;
    if (qk8) {
        if (D != 128) return BAPS_ERR_UNSUPPORTED;
        if (mode == kExp2m) return launch_attention<attention_tc_kernel<128, kExp2m, true, false>, TcLayout<128>::kDynBytes>(a);
        if (mode == kExact) return launch_attention<attention_tc_kernel<128, kExact, true, false>, TcLayout<128>::kDynBytes>(a);
        return b0l ? launch_attention<attention_tc_kernel<128, kE2E, true, true>, TcLayout<128>::kDynBytes>(a)
                   : one ? launch_attention<attention_tc_kernel<128, kE2E, true, false, true>, TcLayout<128>::kDynBytes>(a)
                         : launch_attention<paired_attention_tc_kernel<true>, PairLayout::kDynBytes>(a);
    }
    if (D == 128) {
        if (mode == kExp2m) return launch_attention<attention_tc_kernel<128, kExp2m, false, false>, TcLayout<128>::kDynBytes>(a);
        if (mode == kExact) return launch_attention<attention_tc_kernel<128, kExact, false, false>, TcLayout<128>::kDynBytes>(a);
        return b0l ? launch_attention<attention_tc_kernel<128, kE2E, false, true>, TcLayout<128>::kDynBytes>(a)
                   : one ? launch_attention<attention_tc_kernel<128, kE2E, false, false, true>, TcLayout<128>::kDynBytes>(a)
                         : launch_attention<paired_attention_tc_kernel<false>, PairLayout::kDynBytes>(a);
    }
    if (mode == kExp2m) return launch_attention<attention_tc_kernel<64, kExp2m, false, false>, TcLayout<64>::kDynBytes>(a);
    if (mode == kExact) return launch_attention<attention_tc_kernel<64, kExact, false, false>, TcLayout<64>::kDynBytes>(a);
    if (d64) return launch_attention<attention_d64_kernel, D64Layout::kDynBytes>(a, kD64Split);
    return b0l ? launch_attention<attention_tc_kernel<64, kE2E, false, true>, TcLayout<64>::kDynBytes>(a)
               : launch_attention<attention_tc_kernel<64, kE2E, false, false, true>, TcLayout<64>::kDynBytes>(a);
}

} // namespace baps
