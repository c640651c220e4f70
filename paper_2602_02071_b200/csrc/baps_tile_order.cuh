// Which CTA of the fused attention works on which query tile of which head, and how many tiles a CTA takes.
// Integer arithmetic only: compiles for the device, and by itself as plain C++ (the CPU test does so).
#pragma once
#ifdef __CUDACC__
#define BAPS_HD __host__ __device__ __forceinline__
#else
#define BAPS_HD inline
#endif

namespace baps {

// One query tile per CTA or two?  Two share the K / V stream and the set-up of the CTA, and one of them works while the
// other waits (a task, one score tile, takes 1.08 us of a CTA with two against 1.7 of a CTA with one); one halves the
// chain of tasks that the longest CTA walks through, which is what a grid that does not fill the SMs several times over
// takes.  Estimate of both in units of a two-tile task, SMs filled longest CTA first: the longest CTA or the average load of
// an SM, whichever is larger (all CTAs of a bidirectional problem are equally long: whole waves).  Besides its tasks a
// CTA costs kFixedTwo / kFixedOne (set-up, first scores, epilogues).  The constants are the middle of those that choose the
// faster form at all of 52 sizes from 4 x 512 to 4 x 32768 (heads x tokens, D = 128).  Measured, one tile / two tiles,
// causal: 16 x 512 10.0 / 13.8 us, 32 x 1024 22.6 / 24.7, 16 x 2048 33.6 / 43.3, 8 x 4096 57.0 / 79.1, 1 x 16384 219 / 274; and where
// two are taken: 64 x 512 17.5 / 15.4, 24 x 2048 51.8 / 44.0, 12 x 4096 89.8 / 78.4, 8 x 8192 206 / 145, 2 x 32768 788 / 523;
// bidirectional 16 x 512 10.8 / 14.8, 8 x 2048 31.3 / 42.4, and 24 x 2048 90.3 / 83.9, 12 x 4096 169 / 154.
inline bool one_tile_per_cta(long long heads, int nq, bool causal, int num_sms)
{
    constexpr double kFixedTwo = 4.5, kFixedOne = 4.0, kTaskOne = 1.35;
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
inline bool two_ctas_per_sm(long long heads, int nq, bool causal, int num_sms)
{
    return causal ? 10 * heads * (nq + 1) >= 26LL * num_sms : heads * nq > num_sms;
}

// The kv heads (of all batches) are worked on in chunks: `wide` chunks of size + 1, then chunks of `size`.
struct KvChunks { int size, wide; };

// Chunks of kv heads whose K and V take 16 MB or a little more, with CTAs enough in each to keep the SMs evenly busy
// (causal: three for every one that is resident, heavy and light ones mixed; with fewer 32 x 4096 tokens ran 2 %
// slower, with four the larger chunks cost 1 to 2 % in L2 misses), all of one size but for one head: the last chunk,
// too, starts with its longest CTAs, and with only a few heads left over these ran alone at the end.  Measured, all kv
// heads at once -> chunks of 16 MB and what is left -> even chunks (causal, heads x tokens, inputs not in L2): 16 x 16384
// 1198 -> 1348 -> 1200 us, 36 / 9 x 8192 717 -> 790 -> 719, 8-bit Q / K 64 / 16 x 8192 1341 -> 1430 -> 1340, D = 64
// 9 x 16384 632 -> 756 -> 611; and what the chunks are for: 96 x 4096 570 -> 535 -> 524, 512 x 1024 of D = 64,
// bidirectional, 350 -> 334 -> 334.
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
// head are adjacent.  (Taken all at once, 512 heads x 1024 tokens of D = 64 -- 134 MB of K and V -- were read from
// HBM again for every query tile.)
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
