// Fused attention forward with float32 inputs: Algorithm 1 tile by tile, the scores accumulated in
// double precision.  This is the small-problem path (the single-head S = 128, D = 64 configuration) and
// the in-library cross-check of the tensor-core kernel.
//
// What bounds it is latency: a call has few query tiles, each walks its key tiles in order, and the
// double-precision products of one tile keep one SM busy for microseconds.  So a cluster of eight CTAs
// shares a query tile, BLK / 8 rows each (rows only meet in the tile-wide restart vote, one flag written to
// every CTA's shared memory before a cluster barrier), and in a CTA everything runs from shared memory:
//   A  S = Q_i K_j^T * log2(e) * scale: double-precision matrix instructions (mma m8n8k4), the K values
//      converted once, by the one warp that owns their 8 columns; K_j arrived by cp.async during tile j - 1
//   B  one warp per row: maximum, restart vote (restart condition), max update, weights (fp32 2^x in the B0
//      tile, HiF8 table else)                                            (lines m, P)
//   C  O~ = alpha O~ + W V_j in fp32: a thread owns 4 rows x 4 columns of O~ for a share of the keys
//      (one 16-byte load of V and one of W per 16 products); the shares are added up at the end; V_j
//      arrived by cp.async during A and B
// Measured on B200 (one head, S = 128, D = 64, 64 x 64 tiles): 182 us with one CTA of 256 threads per query
// tile reading K, V and Q from L2 for every product, 6.8 us now, back to back.
#pragma once
#include "baps_common.cuh"
#include "baps_hif8.cuh"
#include "baps_sm100.cuh"
#include "baps_tables.cuh"

namespace baps {

struct AttnF32Params {
    const float *q, *k, *v;
    float *out;                 // may be null
    float *row_m, *row_d, *out_f32;
    int32_t *restarts;
    int B, H, Hkv, S, D, causal, lambda, mode;
    int b0_last;                // B0 = {first, last visible key tile}: order 0, last, 1, ..., last - 1
    double c;                   // log2(e) * scale
};

// CTAs that share a query tile: the largest cluster every device configuration can place, and with it one
// 8-row matrix tile (64-row blocks) or two (128-row blocks) per CTA.
constexpr int kAfCluster = 8;

// Shared memory of one CTA, in floats unless said otherwise.  D is padded to a multiple of 16 with zeros
// (Dp) for the score products; the row strides keep the fragment loads free of bank conflicts: K rows
// 16 mod 32 words apart, Q rows (doubles) 4 mod 8 words, score rows 8 mod 32.
template <int BLK>
struct AfLayout {
    static constexpr int R = BLK / kAfCluster;             // query rows per CTA
    static constexpr int THREADS = BLK * 4;                // a warp per 8 score columns
    static constexpr int kSStride = BLK + 8, kWStride = R + 4;
    int Dp, ks, qs, v_off, q_off, s_off, w_off, total;     // strides; offsets in floats
    __host__ __device__ explicit AfLayout(int D)
    {
        Dp = (D + 15) & ~15;
        ks = Dp + ((Dp & 16) ? 0 : 16);
        qs = Dp + 2;
        v_off = BLK * ks;
        q_off = v_off + BLK * D;
        // (the partial outputs of the epilogue, at most 16 floats per thread, reuse the space of K and V)
        if (q_off < THREADS * 16) q_off = THREADS * 16;
        s_off = q_off + 2 * R * qs;
        w_off = s_off + R * kSStride;
        total = w_off + BLK * kWStride;
    }
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// c[8 x 8] += a[8 x 4] b[4 x 8]: lane l holds a(l / 4, l % 4), b(l % 4, l / 4), c(l / 4, 2 (l % 4) + {0, 1})
__device__ __forceinline__ void dmma(double (&c)[2], double a, double b)
{
    asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
        : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}

template <int BLK>
__global__ void __cluster_dims__(kAfCluster, 1, 1) __launch_bounds__(BLK * 4)
attention_f32_kernel(const AttnF32Params p)
{
    using L = AfLayout<BLK>;
    constexpr int R = L::R, MT = R / 8, THREADS = L::THREADS, EPL = BLK / 32;
    static_assert(THREADS / 32 == R, "one warp per query row");
    extern __shared__ __align__(16) float smem[];
    __shared__ float s_lut[kLutN];
    __shared__ float s_alpha[R], s_dinv[R];
    __shared__ int s_flag[3];

    allow_next_kernel();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = blockIdx.x % kAfCluster, tile = blockIdx.x / kAfCluster, h = blockIdx.y, b = blockIdx.z;
    const int D = p.D, S = p.S;
    const L lay(D);
    float *const s_K = smem, *const s_V = smem + lay.v_off, *const s_S = smem + lay.s_off, *const s_W = smem + lay.w_off;
    double *const s_Q = reinterpret_cast<double *>(smem + lay.q_off);
    const int i0 = tile * BLK + rank * R;                   // first query row of this CTA
    const int hk = h / (p.H / p.Hkv);
    const float *qh = p.q + ((size_t)b * p.H + h) * (size_t)S * D;
    const float *kh = p.k + ((size_t)b * p.Hkv + hk) * (size_t)S * D;
    const float *vh = p.v + ((size_t)b * p.Hkv + hk) * (size_t)S * D;

    const int jmax = p.causal ? tile + 1 : S / BLK;
    const bool e2e = p.mode == BAPS_MODE_E2E_HIF8;
    const bool order_last = p.b0_last && e2e;
    const int nb0 = (order_last && jmax >= 2) ? 2 : 1;      // number of high-precision tiles
    auto key_tile = [&](int step) { return !order_last ? step : (step == 0 ? 0 : (step == 1 ? jmax - 1 : step - 1)); };

    // rows of a [BLK, D] tile -> shared memory, 16 bytes per copy
    const int nc = D / 4, r_first = tid / nc, c_first = tid % nc, r_step = THREADS / nc, c_step = THREADS % nc;
    auto fetch = [&](float *dst, int stride, const float *src) {
        const uint32_t d0 = sm100::smem_u32(dst);
        for (int r = r_first, c = c_first; r < BLK;) {
            cp_async16(d0 + (uint32_t)(r * stride + 4 * c) * 4u, src + (size_t)r * D + 4 * c);
            r += r_step; c += c_step;
            if (c >= nc) { c -= nc; ++r; }
        }
        cp_async_commit();
    };
    for (int i = tid; i < kLutN; i += THREADS) s_lut[i] = g_w0.v[i];
    if (tid < 3) s_flag[tid] = 0;
    qh = await_previous_kernel(qh);
    fetch(s_K, lay.ks, kh);
    for (int i = tid; i < R * lay.Dp; i += THREADS) {
        const int r = i / lay.Dp, d = i % lay.Dp;
        s_Q[r * lay.qs + d] = d < D ? (double)qh[(size_t)(i0 + r) * D + d] : 0.0;
    }
    if (lay.Dp > D)                                          // the copies never touch the padding
        for (int i = tid; i < BLK * (lay.Dp - D); i += THREADS)
            s_K[(i / (lay.Dp - D)) * lay.ks + D + i % (lay.Dp - D)] = 0.f;
    // every CTA of the cluster has cleared its flags before another one may set them
    asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");

    // output accumulators: 4 rows x 4 columns per thread over every nkg-th key
    const int nrg = R / 4, nkg = THREADS / (nc * nrg);
    const int cg = tid % nc, rg = (tid / nc) % nrg, kg = tid / (nc * nrg);       // kg >= nkg: no share
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int t = 0; t < 4; ++t) acc[i][t] = 0.f;

    float m = -INFINITY, d = 0.f;                            // of row i0 + warp, the same in all lanes
    int n_restart = 0;
    for (int step = 0; step < jmax; ++step) {
        const int j = key_tile(step), c0 = j * BLK;
        cp_async_wait<0>();
        __syncthreads();                                     // K_j is here; nobody reads V_{j-1} any more
        fetch(s_V, D, vh + (size_t)c0 * D);
        // ---- A: scores of all rows, columns 8 warp .. 8 warp + 7 ----------------------------------------
        {
            constexpr int KS = MT == 1 ? 4 : 2;              // independent chains per 8 x 8 tile
            double c[MT][KS][2];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int s = 0; s < KS; ++s) c[mt][s][0] = c[mt][s][1] = 0.0;
            const float *kr = s_K + (warp * 8 + lane / 4) * lay.ks + 4 * (lane % 4);
            const double *qr = s_Q + (lane / 4) * lay.qs + 4 * (lane % 4);
#pragma unroll 2
            for (int d0 = 0; d0 < lay.Dp; d0 += 16) {
                // k index of the products: 4 consecutive columns per lane, one after the other
                const float4 kv = *reinterpret_cast<const float4 *>(kr + d0);
                const double kd[4] = {kv.x, kv.y, kv.z, kv.w};
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    const double2 q01 = *reinterpret_cast<const double2 *>(qr + mt * 8 * lay.qs + d0);
                    const double2 q23 = *reinterpret_cast<const double2 *>(qr + mt * 8 * lay.qs + d0 + 2);
                    dmma(c[mt][0], q01.x, kd[0]);
                    dmma(c[mt][1], q01.y, kd[1]);
                    dmma(c[mt][2 % KS], q23.x, kd[2]);
                    dmma(c[mt][3 % KS], q23.y, kd[3]);
                }
            }
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                const int r = mt * 8 + lane / 4, cc = warp * 8 + 2 * (lane % 4);
                float s[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    double a = c[mt][0][e] + c[mt][1][e];
                    if (KS == 4) a += c[mt][2 % KS][e] + c[mt][3 % KS][e];
                    s[e] = (float)(a * p.c);
                    if (p.causal && c0 + cc + e > i0 + r) s[e] = -INFINITY;
                }
                *reinterpret_cast<float2 *>(s_S + r * L::kSStride + cc) = make_float2(s[0], s[1]);
            }
        }
        __syncthreads();                                     // scores are written, K_j is free
        if (step + 1 < jmax) fetch(s_K, lay.ks, kh + (size_t)key_tile(step + 1) * BLK * D);
        else cp_async_commit();                              // keeps the count of outstanding groups
        // ---- B: row `warp`: restart test (one decision per tile), max update, weights -------------------
        const bool hp = (step < nb0 && p.mode != BAPS_MODE_EXP2_HIF8) || p.mode == BAPS_MODE_EXACT;
        {
            float s[EPL], mx = -INFINITY;
#pragma unroll
            for (int e = 0; e < EPL; ++e) {
                s[e] = s_S[warp * L::kSStride + lane + 32 * e];
                mx = fmaxf(mx, s[e]);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            bool restart = false;
            if (!hp && e2e) {
                // The vote: flag step % 3 of every CTA.  Its owner cleared it during step - 1: behind its own
                // readers (step - 3), before the cluster barrier that this step's writers have passed.
                const int f = step % 3;
                if (lane < kAfCluster && hif8_round(mx - m) > (float)p.lambda) {
                    uint32_t remote;
                    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(sm100::smem_u32(&s_flag[f])), "r"(lane));
                    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote), "r"(1) : "memory");
                }
                if (tid == 0) s_flag[(step + 1) % 3] = 0;
                __syncwarp();
                asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
                asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
                restart = *reinterpret_cast<volatile int *>(&s_flag[f]) != 0;
                if (restart) ++n_restart;
            }
            float mnew, alpha, sum = 0.f, w[EPL];
            if (p.mode == BAPS_MODE_EXACT) {
                mnew = fmaxf(m, mx);                                 // Eq. (2): real-valued max
                alpha = (m == -INFINITY) ? 0.f : exp2f(m - mnew);
#pragma unroll
                for (int e = 0; e < EPL; ++e) w[e] = (mnew == -INFINITY) ? 0.f : exp2f(s[e] - mnew);
            } else if (p.mode == BAPS_MODE_EXP2_HIF8) {
                // "Exp2 HiF8" setup (Section 4.1): Eq. (2) with every 2^x through Algorithm 2
                mnew = fmaxf(m, mx);
                alpha = (m == -INFINITY) ? 0.f : s_lut[w0_index(m - mnew)];
#pragma unroll
                for (int e = 0; e < EPL; ++e) w[e] = (mnew == -INFINITY) ? 0.f : s_lut[w0_index(s[e] - mnew)];
            } else if (hp || restart) {
                mnew = fmaxf(m, ceilf(mx));
                alpha = (m == -INFINITY) ? 0.f : exp2f(m - mnew);
#pragma unroll
                for (int e = 0; e < EPL; ++e) {
                    const float u = s[e] - mnew;
                    w[e] = hp ? ((mnew == -INFINITY) ? 0.f : exp2f(u)) : s_lut[w0_index(u)];
                }
            } else {
                const float t8 = hif8_round(mx - m);
                const float delta = fmaxf(0.f, ceilf(t8));           // 0 for an all-masked row
                mnew = m + delta;
                alpha = exp2f(-delta);
#pragma unroll
                for (int e = 0; e < EPL; ++e) w[e] = s_lut[w0_index(s[e] - m)] * alpha;
            }
#pragma unroll
            for (int e = 0; e < EPL; ++e) {
                s_W[(lane + 32 * e) * L::kWStride + warp] = w[e];
                sum += w[e];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            m = mnew;
            d = alpha * d + sum;
            if (lane == 0) s_alpha[warp] = alpha;
        }
        cp_async_wait<1>();                                  // V_j (K_{j+1} may still be on its way)
        __syncthreads();
        // ---- C: O~ = alpha O~ + W V_j --------------------------------------------------------------------
        if (kg < nkg) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float al = s_alpha[rg * 4 + i];
#pragma unroll
                for (int t = 0; t < 4; ++t) acc[i][t] *= al;
            }
#pragma unroll 4
            for (int cc = kg; cc < BLK; cc += nkg) {
                const float4 vv = *reinterpret_cast<const float4 *>(s_V + cc * D + 4 * cg);
                const float4 ww = *reinterpret_cast<const float4 *>(s_W + cc * L::kWStride + 4 * rg);
                const float wr[4] = {ww.x, ww.y, ww.z, ww.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (wr[i] != 0.f) {                      // a masked key takes no part, whatever its V holds
                        acc[i][0] = fmaf(wr[i], vv.x, acc[i][0]);
                        acc[i][1] = fmaf(wr[i], vv.y, acc[i][1]);
                        acc[i][2] = fmaf(wr[i], vv.z, acc[i][2]);
                        acc[i][3] = fmaf(wr[i], vv.w, acc[i][3]);
                    }
            }
        }
    }
    // ---- the shares of the key groups added up, normalisation and statistics ----------------------------
    if (lane == 0) s_dinv[warp] = 1.f / d;
    cp_async_wait<0>();
    __syncthreads();                                         // K and V make room for the partial outputs
    float *const s_part = smem;                              // [nkg][R][D]
    if (kg < nkg) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            *reinterpret_cast<float4 *>(s_part + (kg * R + rg * 4 + i) * D + 4 * cg) =
                make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    }
    __syncthreads();
    const size_t row0 = ((size_t)b * p.H + h) * S + i0;
    for (int i = tid; i < R * nc; i += THREADS) {
        const int r = i / nc, c = i % nc;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int g = 0; g < nkg; ++g) {
            const float4 x = *reinterpret_cast<const float4 *>(s_part + (g * R + r) * D + 4 * c);
            o.x += x.x; o.y += x.y; o.z += x.z; o.w += x.w;
        }
        const float dinv = s_dinv[r];
        o = make_float4(o.x * dinv, o.y * dinv, o.z * dinv, o.w * dinv);
        const size_t at = (row0 + r) * (size_t)D + 4 * c;
        if (p.out) *reinterpret_cast<float4 *>(p.out + at) = o;
        if (p.out_f32) *reinterpret_cast<float4 *>(p.out_f32 + at) = o;
    }
    if (lane == 0) {
        if (p.row_m) p.row_m[row0 + warp] = m;
        if (p.row_d) p.row_d[row0 + warp] = d;
    }
    if (tid == 0 && rank == 0 && p.restarts)
        p.restarts[((size_t)b * p.H + h) * (S / BLK) + tile] = n_restart;
}

} // namespace baps
