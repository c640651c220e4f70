// Which CTA of the fused attention works on which query tile of which head, and how many tiles a CTA takes.
// Integer arithmetic only: compiles for the device, and by itself as plain C++ (the CPU test does so).
#pragma once
#ifdef __CUDACC__
#define BAPS_HD __host__ __device__ __forceinline__
#else
#define BAPS_HD inline
#endif

namespace baps {

// One query tile per CTA or two (D = 128)?  Two share the K / V stream and the set-up of the CTA, and one of them works
// while the other waits: a task, one score tile, takes 1.06 us of a CTA with two against 1.65 of a CTA with one
// (kTaskOne, their ratio).  One halves the chain of tasks that the longest CTA walks through, which is what a grid that does
// not fill the SMs several times over takes; a single wave of them is always the faster.
//   All CTAs of a bidirectional problem are equally long: whole waves of them, with two tasks' time for set-up, first scores
// and epilogue beside the tasks.
//   Causal: by the load of an SM, all tasks spread evenly, in chains of the longest query tile.  Short chains change over
// earlier, since the set-up is a larger part of a CTA and one with two tiles pays it once; an odd number of tiles earlier
// still.  Up to five tiles whole waves show: two tiles a CTA in a second wave of a few CTAs lose to one tile in two full ones.
// Line and constants are fitted to which form was faster at 796 causal and as many bidirectional sizes of 1 to 385 heads x 128
// to 32768 tokens, half of them with 8-bit Q / K (one line serves both); the form chosen is at most 5 % behind the other.
// Measured, one tile / two tiles, causal (heads x tokens): 16 x 512 9.8 / 13.6 us, 32 x 1024 21.4 / 24.1, 16 x 2048 32.2 / 42.3,
// 8 x 4096 55.2 / 80.7, 1 x 16384 216 / 271, 75 x 384 14.6 / 18.2; and where two are taken: 48 x 640 17.2 / 14.3, 20 x 2048
// 44.2 / 42.5, 6 x 8192 164 / 146, 3 x 16384 315 / 282, 2 x 32768 776 / 527; bidirectional 8 x 2048 29.6 / 41.7, and 10 x 2048
// 58.9 / 45.6, 12 x 4096 168 / 153; 8-bit Q / K, causal: 8 x 4096 51.5 / 77.9, and 20 x 2048 42.2 / 41.7, 6 x 8192 153 / 142; the
// wrong side of the line: 36 x 1024 23.0 / 23.9.
inline bool one_tile_per_cta(long long heads, int nq, bool causal, int num_sms)
{
    constexpr double kFixed = 2.0, kTaskOne = 1.6;
    const long long ctas2 = heads * ((nq + 1) / 2), ctas1 = heads * nq;
    if (nq == 1) return false;                             // the same work; paired_attention_tc_kernel's set-up is 2 to 7 % shorter
    if (ctas1 <= num_sms) return true;
    if (causal) {
        const double load = (double)heads * (nq + 1) / (2.0 * num_sms);
        return load < 1.24 - (nq % 2 ? 2.4 : 1.6) / nq || (nq <= 5 && ctas2 > num_sms && ctas1 <= 2LL * num_sms);
    }
    const double t1 = (double)((ctas1 + num_sms - 1) / num_sms) * (kTaskOne * nq + kFixed);
    const double t2 = (double)((ctas2 + num_sms - 1) / num_sms) * (2 * nq + kFixed);
    return t1 < t2;
}

// Heads of 64: attention_d64_kernel (two CTAs per SM) or attention_tc_kernel with one query tile per CTA, whose sixteen
// softmax warps are through with a lone tile sooner?  The former when the SMs are full: more tiles than SMs, and causal by the
// load of an SM as above (short chains earlier, since there the set-up of one CTA runs beside the other).  The kernel chosen
// is at most 2 % behind the other at 398 causal and as many bidirectional sizes, nq = 1 with nearly as many heads as SMs aside
// (147 x 128: 5.5 / 4.9 us).  Measured, attention_tc_kernel / attention_d64_kernel, causal (heads x tokens): 24 x 1024 15.0 / 16.2
// us, 16 x 2048 27.5 / 28.4, 2 x 16384 153 / 173; and where the latter is taken: 64 x 512 14.8 / 12.0, 40 x 1024 25.3 / 19.7,
// 20 x 2048 36.8 / 33.3, 10 x 4096 58.9 / 55.4; bidirectional 8 x 2048 24.3 / 27.1, and 10 x 2048 47.4 / 41.0.
inline bool two_ctas_per_sm(long long heads, int nq, bool causal, int num_sms)
{
    return heads * nq > num_sms && (!causal || (double)heads * (nq + 1) / (2.0 * num_sms) >= 1.04 - 1.65 / nq);
}

// The kv heads (of all batches) are worked on in chunks: `wide` chunks of size + 1, then chunks of `size`.
struct KvChunks { int size, wide; };

// Chunks of kv heads whose K and V take 16 MB or a little more, with CTAs enough in each to keep the SMs evenly busy
// (causal: three for every one that is resident, heavy and light ones mixed), all of one size but for one head: the last
// chunk, too, starts with its longest CTAs, and with only a few heads left over these would run alone at the end.  Measured,
// all kv heads at once -> even chunks, calls back to back (causal, heads x tokens): 96 x 4096 521 -> 454 us, 16 x 16384
// 1138 -> 1100, 36 / 9 x 8192 664 -> 638, 64 / 16 x 8192 1187 -> 1173 (8-bit Q / K 1060 -> 1055), 32 x 4096 173 -> 170; D = 64:
// 9 x 16384 518 -> 518, 512 x 1024 bidirectional 305 -> 304.  A lone call that finds none of its inputs in L2 takes the same
// either way, to 0.5 %.  (With the kernels before these a ragged last chunk cost 10 to 20 % at 16 x 16384, 36 / 9 x 8192 and, D = 64,
// 9 x 16384; two CTAs for every one that is resident 2 % at 32 x 4096.)
// kv_bytes: of K and V of one head; per_kv: CTAs per kv head.
inline KvChunks kv_chunks(long long kv_heads, long long kv_bytes, long long per_kv, bool causal, int num_sms, int ctas_per_sm)
{
    const long long least = ((causal ? 3LL * ctas_per_sm : 2LL) * num_sms + per_kv - 1) / per_kv;
    long long size = (16LL << 20) / kv_bytes;
    if (size < least) size = least;
    const long long n = kv_heads / size > 1 ? kv_heads / size : 1;
    return {(int)(kv_heads / n), (int)(kv_heads % n)};
}

// Which tile of which head a CTA works on.  The kv heads are taken in chunks whose K and V together stay in L2 while
// their query tiles pass; within a chunk the heavy (late) query tiles come first and the query heads of one kv
// head are adjacent.
struct WorkItem { int tile, h, hk, b; };
BAPS_HD WorkItem work_item(int H, int Hkv, int npairs, KvChunks ch, int idx)
{
    const int gsz = H / Hkv, per_kv = gsz * npairs, in_wide = ch.wide * (ch.size + 1) * per_kv;
    int n = ch.size + 1, first = 0;
    if (idx >= in_wide) { idx -= in_wide; first = ch.wide * n; --n; }
    const int c = idx / (n * per_kv);
    idx -= c * n * per_kv;
    const int gi = idx % gsz;
    idx /= gsz;
    const int kv = first + c * n + idx % n;
    WorkItem w;
    w.tile = npairs - 1 - idx / n;
    w.hk = kv % Hkv;
    w.b = kv / Hkv;
    w.h = w.hk * gsz + gi;
    return w;
}

} // namespace baps
