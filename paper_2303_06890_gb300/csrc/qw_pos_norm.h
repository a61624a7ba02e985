/*
 * qw_pos_norm.h -- the norm of a positional step as fixed-point shares: how it
 * is packed, summed and read back.  Plain C++, shared by the kernels
 * (qw_pos.cuh) and the host-logic test.
 *
 * A share is a number of units, of which the renormalisation target holds 2^61
 * to 2^62, whatever its exponent: a lane's rounding is 2^-62 of the target, so
 * that the sum over 78 000 lanes is off by 2^-54 of it in the mean (2^-46 at
 * most), as an FP64 sum of them is.  Sums of shares are exact, so they do not
 * depend on the order of arrival.  A sum travels as two words that are both added
 * to:
 *   fine    the sum modulo 2^FIELD units,
 *   coarse  the sum of the shares' parts above 2^42 units (each cut down), and
 *           2^48 for every share that is kept out of the integer sums because it
 *           is not finite, or too large for them ("odd": it is added to an FP64
 *           number instead).
 * The coarse word says which multiple of 2^FIELD the fine one leaves out, for any
 * norm: nothing is assumed of how near the norm is to the target.  In the words
 * of the grid's barrier (FIELD = 56) the low 8 bits count arrivals; the sums lie
 * above them, so what they carry out of the word is lost, not counted.
 */
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define QW_HD __host__ __device__ __forceinline__
#else
#define QW_HD inline
#endif

constexpr int kUnitBits = 62;   /* the target has this many bits in units */
constexpr int kCoarseShift = 42;
constexpr int kCountBits = 8;   /* of a barrier word: up to 255 blocks */
constexpr int kGridField = 64 - kCountBits, kClusterField = 64;
constexpr uint64_t kCountMask = (1ull << kCountBits) - 1ull;
constexpr uint64_t kOddShare = 1ull << 48; /* in a coarse sum */
constexpr int kOddTarget = 4000; /* pos_unit_exp of a target without units: every non-zero share is odd */

/* Units are 2^-k: the target, a positive finite number, times 2^k is in [2^61,
 * 2^62); k = kOddTarget where it is not one. */
QW_HD int pos_unit_exp(double target)
{
    uint64_t u;
    memcpy(&u, &target, 8);
    const int e = (int)(u >> 52);
    if (u == 0 || e >= 0x7ff) return kOddTarget; /* 0, negative, not finite */
    if (e > 0) return kUnitBits - 1 + 1023 - e;
    int b = 0;
    while (u >> b > 1) ++b; /* subnormal: 2^b to 2^(b+1) times 2^-1074 */
    return kUnitBits - 1 + 1074 - b;
}

/* v times 2^k, v a finite number >= 0, rounded to a whole number below 2^63; odd where
 * it is 2^63 or more or v is not finite.  By integer operations on the
 * exponent (the FP64 pipe is slow). */
QW_HD uint64_t pos_units(double v, int k, bool &odd)
{
    uint64_t u;
    memcpy(&u, &v, 8);
    int e = (int)(u >> 52) & 0x7ff;
    odd = e == 0x7ff || (u != 0 && e + k >= 1023 + 63);
    e += k;
    if (odd || u >> 52 == 0 || e < 1023 - 1) return 0; /* 0, subnormal or below half a unit */
    const uint64_t m = (u & ((1ull << 52) - 1ull)) | (1ull << 52);
    const int s = e - 1023 - 52; /* m 2^s */
    return s >= 0 ? m << s : (m + (1ull << (-s - 1))) >> -s;
}

/* The multiple of 2^FIELD that the fine sum leaves out.  coarse: without the odd
 * shares; short by less than 2^13 (4096 shares) of the exact sum's part. */
template <int FIELD> QW_HD int64_t pos_wraps(uint64_t fine, uint64_t coarse)
{
    constexpr int up = FIELD - kCoarseShift;
    const int64_t d = (int64_t)coarse - (int64_t)(fine >> kCoarseShift);
    return (d + (1 << 13)) >> up;
}

/* Whether the sum is near the target -- it is where they differ by less than 2^53
 * units (2^-8 to 2^-9 of the target) -- by the coarse sum, which is short by at most
 * 4096 of its 2^42 units: the difference is then below 2^55 units, and the fine sum
 * tells it, left with a multiple of 2^56 or none. */
QW_HD bool pos_near(uint64_t target, uint64_t coarse)
{
    const int64_t d = (int64_t)(target >> kCoarseShift) - (int64_t)coarse;
    return d >= -2048 && d <= 2048 + 4096;
}
template <int FIELD> QW_HD int64_t pos_deviation(uint64_t target, uint64_t fine) /* target - sum */
{
    return (int64_t)((target - fine) << (64 - FIELD)) >> (64 - FIELD);
}

/* A factor as a float pair, 49 significant bits: h its rounding to FP32 (1 wherever it
 * is within 2^-25 of that, as a step's renormalisation mostly is), l the rest. */
QW_HD void factor_split(double v, float &h, float &l)
{
    h = (float)v;
    l = (float)(v - (double)h);
}

/* The factor sqrt(target / sum) = (1 - x)^(-1/2), x = dev / target, as a float pair h +
 * l, in FP32 alone (square root and division in FP64 take over a thousand cycles on
 * the device, between every two steps).  |x| < 2^-14 or false.  inv_h + inv_l:
 * 2^24 / target.  x = p + e within 2^-46 of itself; the series' terms beyond the
 * third are below 2^-57, its square and cube within 2^-50; h is 1 + p / 2 rounded,
 * with what that leaves out and the rest in l: within 2^-48 in all, what the
 * pair of a correctly rounded factor is. */
QW_HD bool pos_factor_pair(int64_t dev, float inv_h, float inv_l, float &h, float &l)
{
    const int64_t top = dev >> 24;
    if (top < -(1 << 23) || top >= 1 << 23) return false;
    const float d = (float)(int)top, low = (float)(int)(dev & 0xffffff) * (1.0f / 16777216.0f);
    const float p = d * inv_h;
    float e = fmaf(d, inv_h, -p);
    e = fmaf(d, inv_l, e);
    e = fmaf(low, inv_h, e);
    const float c = 0.5f * p;
    h = 1.0f + c;
    l = (c - (h - 1.0f)) + fmaf(p * p, fmaf(0.3125f, p, 0.375f), 0.5f * e);
    return true;
}

/* v 2^e, e of any size, v a finite number */
QW_HD double pos_scale2(double v, int e)
{
    for (; e > 1000; e -= 1000) v *= 0x1p1000;
    for (; e < -1000; e += 1000) v *= 0x1p-1000;
    const uint64_t u = (uint64_t)(1023 + e) << 52;
    double f;
    memcpy(&f, &u, 8);
    return v * f;
}

/* The norm: the sum in FP64, the odd shares (extra) included. */
template <int FIELD> QW_HD double pos_total(uint64_t fine, uint64_t coarse, double extra, int k)
{
    const bool odd = coarse >= kOddShare;
    coarse &= kOddShare - 1ull;
    const double sum = (double)fine + (double)pos_wraps<FIELD>(fine, coarse) * (FIELD == 64 ? 0x1p64 : 0x1p56);
    const double v = sum != 0.0 ? pos_scale2(sum, -k) : 0.0;
    return odd ? v + extra : v;
}
