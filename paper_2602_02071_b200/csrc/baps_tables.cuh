// The table of w0(u) = HiF8(2^HiF8(u)), worked out by the compiler (in double precision) and part of the
// module image: no kernel, wait or lock on a first call.  The kernels copy it into shared memory.
#pragma once
#include "baps_common.cuh"
#include "baps_hif8.cuh"

namespace baps {

constexpr double ct_pow2(int e)
{
    double r = 1.0;
    for (; e > 0; --e) r *= 2.0;
    for (; e < 0; ++e) r *= 0.5;
    return r;
}
// 2^t by the exponential series of the fractional part
constexpr double ct_exp2(double t)
{
    int n = (int)t;
    if (t < n) --n;
    const double x = (t - n) * 0.69314718055994530942;
    double term = 1.0, sum = 1.0;
    for (int k = 1; k < 28; ++k) { term *= x / k; sum += term; }
    return sum * ct_pow2(n);
}
// HiF8 rounding of |x| < 2^15 (see hif8_round)
constexpr double ct_hif8(double x)
{
    const double a = x < 0 ? -x : x;
    if (a < ct_pow2(-23)) return 0.0;
    if (a < ct_pow2(-22)) return x < 0 ? -ct_pow2(-22) : ct_pow2(-22);
    int e = 0;
    while (ct_pow2(e + 1) <= a) ++e;
    while (ct_pow2(e) > a) --e;
    const int ae = e < 0 ? -e : e;
    const double step = ct_pow2(e - (ae <= 3 ? 3 : ae <= 7 ? 2 : ae <= 15 ? 1 : 0));
    const double r = (double)(long long)(a / step + 0.5) * step;
    return x < 0 ? -r : r;
}

struct W0Table { float v[kLutN]; };
constexpr W0Table make_w0_table()
{
    W0Table t{};
    for (int i = 0; i < kLutN; ++i) {
        // the fp32 number whose top 13 bits (sign, exponent, four mantissa bits) are the entry's key
        const int key = i < kLutNegN ? kLutNegLo + i : kLutPosLo + (i - kLutNegN);
        const double mag = (1.0 + (key & 15) / 16.0) * ct_pow2(((key >> 4) & 0xFF) - 127);
        t.v[i] = (float)ct_hif8(ct_exp2(ct_hif8((key & 0x1000) ? -mag : mag)));
    }
    return t;
}
__device__ constexpr W0Table g_w0 = make_w0_table();

} // namespace baps
