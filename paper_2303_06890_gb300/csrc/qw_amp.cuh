/*
 * qw_amp.cuh -- amplitude arithmetic of the fused step kernels (qw_kernels.cu):
 * the conditional rotation, the zero-type group sum, pruning, the norm and
 * the renormalisation factor for complex128 (FP64) and complex64 (float
 * pairs), and the walk operator on one b2-pair of branches.
 * Everything is internal to each translation unit that includes it.
 */
#ifndef QW_AMP_CUH
#define QW_AMP_CUH

#include "qw_device.cuh"
#include "qw_pos_norm.h"

namespace {

/* sign flips as integer operations on the sign bit (keeps FP64 negations
 * and selects off GB300's slow FP64 pipe) */
/* sign flip of an FP64 value as an integer XOR on its high word, kept opaque
   (inline PTX) so that it stays on the integer pipe: an FP64 negation would
   take a slot of GB300's 1/64-rate FP64 pipe */
__device__ __forceinline__ double flip_if(double x, bool neg)
{
    const int m = (int)((unsigned)neg << 31);
    int hi = __double2hiint(x);
    asm("xor.b32 %0, %0, %1;" : "+r"(hi) : "r"(m));
    return __hiloint2double(hi, __double2loint(x));
}
__device__ __forceinline__ float flip_if(float x, bool neg)
{
    return __int_as_float(__float_as_int(x) ^ ((int)neg << 31));
}

template <typename AmpT> struct Amp;

/* complex128 path: FP64 arithmetic throughout */
__device__ __noinline__ double2 scale_c128(double2 a, double s) { return make_double2(a.x * s, a.y * s); }

/* the pruning decision inside the band around tau (rarely reached) */
__device__ __noinline__ bool keep_band(double x, double y, double tau2)
{
    return __dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)) > tau2;
}

template <> struct Amp<double2> {
    typedef double2 T;
    static constexpr bool kHeadLanes = true; /* rotate with one lane per pair head */
    struct Norm {
        double v = 0.0;
        __device__ void add(T a) { v = fma(a.x, a.x, fma(a.y, a.y, v)); }
        __device__ double get() const { return v; }
        __device__ double warp_total() const
        {
            double t = v;
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(FULL, t, o);
            return t;
        }
    };
    /* sum of a zero-type Hadamard group (FP64) */
    struct Sum {
        double x = 0.0, y = 0.0;
        __device__ void add(T a) { x += a.x; y += a.y; }
        __device__ void set(T a) { x = a.x; y = a.y; } /* add() to an empty sum */
        /* lane t < min(s, 32) holds the partial sums of the values t, t + 32, ...
           (s a power of two); with width < 32 each aligned group of width
           lanes reduces its own values.  Butterfly over the w = min(s, 32) lanes, x on
           lanes t < w/2 and y on lanes t >= w/2 after the first level, so one
           FP64 add serves both components; the same pairs and order as a
           butterfly over each component alone (FP64 addition commutes). */
        __device__ void reduce(int s, int width = 32)
        {
            const int w = s < 32 ? s : 32, h = w >> 1;
            if (h > 0) {
                const bool hy = (lane_id() & h) != 0;
                const double recv = __shfl_xor_sync(FULL, hy ? x : y, h);
                double v = (hy ? y : x) + recv;
                for (int o = h >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
                x = v;
                y = v;
            }
            x = __shfl_sync(FULL, x, 0, width);
            y = __shfl_sync(FULL, y, h, width);
        }
        __device__ void scale_pow2(double f) { x *= f; y *= f; }
        __device__ T minus(T a) const { return make_double2(x - a.x, y - a.y); }
        __device__ double2 value() const { return make_double2(x, y); }
    };
    __device__ static T zero() { return make_double2(0.0, 0.0); }
    __device__ static T neg(T a) { return make_double2(flip_if(a.x, true), flip_if(a.y, true)); }
    __device__ static double2 to_d(T a) { return a; }
    __device__ static T from_d(double2 a) { return a; }
    /* |a|^2 > tau^2 exactly as the un-fused FP64 formula, decided from the
       exponent bits except in a narrow band around tau; the band's FP64
       arithmetic sits in a call of its own, so that it is not if-converted
       into every call (a predicated-off FP64 instruction still takes its
       slot of the 1/64-rate FP64 pipe) */
    __device__ static bool keep(const QwSimDev &d, T a)
    {
        const uint64_t ux = (uint64_t)__double_as_longlong(a.x) & 0x7fffffffffffffffull;
        const uint64_t uy = (uint64_t)__double_as_longlong(a.y) & 0x7fffffffffffffffull;
        const uint64_t um = ux > uy ? ux : uy;
        if (um > d.tau_hi_bits) return true;
        if (um <= d.tau_lo_bits) return false;
        return keep_band(a.x, a.y, d.tau2);
    }
    struct Scale { /* the renormalisation (off by default for complex128): out of
                      line, so its FP64 products are not if-converted into the
                      loads that do not rescale */
        double s;
        __device__ explicit Scale(double v) : s(v) {}
        __device__ T apply(T a) const { return scale_c128(a, s); }
        /* staged once per block (the factor in 8 bytes of shared memory) */
        __device__ static void to_shared(double v, double *buf) { buf[0] = v; }
        __device__ void store(double *buf) const { buf[0] = s; }
        __device__ static Scale from_shared(const double *buf) { return Scale(buf[0]); }
    };
    typedef double2 RotVal; /* (sqrt|a|, sqrt(1-|a|)) */
    __device__ static RotVal rot_table(const QwSimDev &d, uint32_t A) { return __ldg(d.fg + A); }
    __device__ static RotVal rot_zero() { return make_double2(0.0, 1.0); }
    static constexpr bool kRotCode = false; /* FP64 square roots: read the table */
    __device__ static RotVal rot_code(uint32_t) { return rot_zero(); }
    __device__ static void rot(RotVal t, uint32_t A, bool dag, bool sneg, T a0, T a1, T &o0, T &o1);
    /* R^dag's b2 = 0 output, before any rounding beyond the FP64 merge's */
    typedef double2 Wide;
    __device__ static Wide rdag0(RotVal t, uint32_t A, bool sneg, T a0, T a1);
    __device__ static T narrow(Wide w) { return w; }
    __device__ static T sum_amp(const Sum &r) { return make_double2(r.x, r.y); }
    /* t times 2^-e, exactly, by integer operations (f and g are 0 or far
       above the subnormal range) */
    __device__ static RotVal prescale(RotVal t, int e)
    {
        const int fh = __double2hiint(t.x), gh = __double2hiint(t.y);
        return make_double2(__hiloint2double(fh ? fh - (e << 20) : 0, __double2loint(t.x)),
                            __hiloint2double(gh ? gh - (e << 20) : 0, __double2loint(t.y)));
    }
    __device__ static Wide wide_zero() { return make_double2(0.0, 0.0); }
    /* f r - a0 and g r - a1 (reflect_pair below) */
    __device__ static void reflect(const Sum &r, RotVal t, uint32_t A, bool sneg, T a0, T a1, T &o0, T &o1);
    /* |x| to within 2^-20 relative (a cut to 20 mantissa bits), 0 below
       2^-126 and at most 2^127, by integer operations: an FP64 conversion
       would take a slot of the 1/64-rate FP64 pipe; sign kept */
    __device__ static float approx(double x)
    {
        const uint32_t hi = (uint32_t)__double2hiint(x), m = hi & 0x7fffffffu;
        const uint32_t e = min(max(m, 896u << 20) - (896u << 20), 0x0fefffffu);
        return __uint_as_float((e << 3) | (hi & 0x80000000u));
    }
    __device__ static float2 approx2(T a) { return make_float2(approx(a.x), approx(a.y)); }
    /* the larger of |x|, |y| in FP32: cut by at most 2^-20 relative, raised to
       2^-126 where it is smaller, 0 for 0 */
    __device__ static float inf_norm(T a)
    {
        const uint32_t m = max((uint32_t)__double2hiint(a.x) & 0x7fffffffu, (uint32_t)__double2hiint(a.y) & 0x7fffffffu);
        const uint32_t e = min(max(m, 897u << 20) - (896u << 20), 0x0fefffffu);
        return m ? __uint_as_float(e << 3) : 0.0f;
    }
    __device__ static float rot_f(RotVal t) { return approx(t.x); }
    __device__ static float rot_g(RotVal t) { return approx(t.y); }
    static constexpr float kApproxErr = 1.0f / 131072.0f; /* 2^-17 of the terms' magnitudes */
};

/* complex64 path: amplitudes are float; each rotation output f a0 +- g a1 is
   formed from error-free products and an error-free sum on the FP32 pipe
   (f, g held as float pairs with ~48 significant bits) and rounded once. */
/* a * s with s = sh + sl, rounded once (a call of its own: rarely taken) */
__device__ __forceinline__ float mul_split(float a, float sh, float sl)
{
    const float p = __fmul_rn(sh, a);
    float e = __fmaf_rn(sh, a, -p);
    e = __fmaf_rn(sl, a, e);
    return __fadd_rn(p, e);
}
__device__ __noinline__ float2 scale_c64(float2 a, float sh, float sl)
{
    return make_float2(mul_split(a.x, sh, sl), mul_split(a.y, sh, sl));
}

/* a complex value as float pairs hi + lo, hi = the value rounded to FP32 */
struct WideF {
    float xh, xl, yh, yl;
};

template <> struct Amp<float2> {
    typedef float2 T;
    static constexpr bool kHeadLanes = false;
    struct Norm { /* |a|^2 rounded to FP32 once per branch (relative 2^-24), then
                     summed by TwoSum into a float pair, so the sum adds no
                     rounding error of note beyond those per-term roundings */
        float hi = 0.f, lo = 0.f;
        __device__ void add(T a)
        {
            const float v = __fadd_rn(__fmul_rn(a.x, a.x), __fmul_rn(a.y, a.y));
            const float s = __fadd_rn(hi, v);
            const float bp = __fsub_rn(s, hi);
            lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(v, bp)));
            hi = s;
        }
        __device__ double get() const { return (double)hi + (double)lo; }
        /* the warp's sum: a butterfly of float-pair additions, one conversion
           to FP64 on the lane that returns it (lane 0; the others return 0) */
        __device__ double warp_total() const;
    };
    /* float-pair (hi + lo) accumulator built from Knuth's TwoSum (the sum and
       its exact rounding error), ~48 significant bits */
    struct DF {
        float h = 0.f, l = 0.f;
        __device__ void add(float v)
        {
            const float s = __fadd_rn(h, v);
            const float bp = __fsub_rn(s, h);
            const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bp)), __fsub_rn(v, bp));
            h = s;
            l = __fadd_rn(l, e);
        }
        __device__ void add(float vh, float vl)
        {
            add(vh);
            l = __fadd_rn(l, vl);
            const float s = __fadd_rn(h, l); /* renormalise: |l| small */
            l = __fsub_rn(l, __fsub_rn(s, h));
            h = s;
        }

        /* round(h + l - v) */
        __device__ float minus(float v) const
        {
            const float s = __fsub_rn(h, v);
            const float bp = __fsub_rn(s, h);
            const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bp)), __fsub_rn(-v, bp));
            return __fadd_rn(s, __fadd_rn(e, l));
        }
    };
    /* sum of a zero-type Hadamard group of float-pair terms in a float pair:
       its error is of order 2^-46 times the sum of the terms' magnitudes */
    struct Sum {
        DF x, y;
        __device__ void add(const WideF &a) { x.add(a.xh, a.xl); y.add(a.yh, a.yl); }
        __device__ void set(const WideF &a) /* add() to an empty sum */
        {
            x.h = a.xh;
            x.l = a.xl;
            y.h = a.yh;
            y.l = a.yl;
        }
        /* lane t < min(s, 32) holds the partial sums of the values t, t + 32, ...
           (s a power of two); with width < 32 each aligned group of width
           lanes reduces its own values.  Butterfly over the w = min(s, 32) lanes, x on
           lanes t < w/2 and y on lanes t >= w/2 after the first level (where a
           y lane adds its own pair to its partner's, the order the partner
           would use), so one float-pair add serves both components. */
        __device__ void reduce(int s, int width = 32)
        {
            const int w = s < 32 ? s : 32, h = w >> 1;
            if (h > 0) {
                const bool hy = (lane_id() & h) != 0;
                const float rh = __shfl_xor_sync(FULL, hy ? x.h : y.h, h);
                const float rl = __shfl_xor_sync(FULL, hy ? x.l : y.l, h);
                DF v;
                if (hy) { /* partner's y, then own y */
                    v.h = rh;
                    v.l = rl;
                    v.add(y.h, y.l);
                } else {
                    v = x;
                    v.add(rh, rl);
                }
                for (int o = h >> 1; o > 0; o >>= 1) {
                    const float oh = __shfl_xor_sync(FULL, v.h, o), ol = __shfl_xor_sync(FULL, v.l, o);
                    v.add(oh, ol);
                }
                x = v;
                y = v;
            }
            x.h = __shfl_sync(FULL, x.h, 0, width);
            x.l = __shfl_sync(FULL, x.l, 0, width);
            y.h = __shfl_sync(FULL, y.h, h, width);
            y.l = __shfl_sync(FULL, y.l, h, width);
        }
        __device__ void scale_pow2(double f)
        {
            const float g = (float)f; /* 2/s: a power of two, exact */
            x.h *= g; x.l *= g; y.h *= g; y.l *= g;
        }
        __device__ T minus(T a) const { return make_float2(x.minus(a.x), y.minus(a.y)); }
        __device__ double2 value() const
        {
            return make_double2((double)x.h + (double)x.l, (double)y.h + (double)y.l);
        }
    };
    __device__ static T zero() { return make_float2(0.f, 0.f); }
    __device__ static T neg(T a) { return make_float2(-a.x, -a.y); }
    __device__ static double2 to_d(T a) { return make_double2((double)a.x, (double)a.y); }
    __device__ static T from_d(double2 a) { return make_float2((float)a.x, (float)a.y); }
    __device__ static bool keep(const QwSimDev &d, T a)
    {
        return __fadd_rn(__fmul_rn(a.x, a.x), __fmul_rn(a.y, a.y)) > d.tau2f;
    }
    struct Scale { /* the FP64 factor as a float pair, applied with one rounding;
                      where its high part is 1 that takes one FMA */
        float sh, sl;
        __device__ explicit Scale(double v) { factor_split(v, sh, sl); }
        __device__ Scale(float h, float l) : sh(h), sl(l) {}
        __device__ T apply(T a) const
        {
            if (sh == 1.0f) return make_float2(__fmaf_rn(a.x, sl, a.x), __fmaf_rn(a.y, sl, a.y));
            return scale_c64(a, sh, sl);
        }
        /* the split computed once per block (its FP64 conversions would
           otherwise take a slot of the 1/64-rate FP64 pipe in every thread) */
        __device__ static void to_shared(double v, double *buf)
        {
            float *f = reinterpret_cast<float *>(buf);
            factor_split(v, f[0], f[1]);
        }
        __device__ void store(double *buf) const
        {
            float *f = reinterpret_cast<float *>(buf);
            f[0] = sh;
            f[1] = sl;
        }
        __device__ static Scale from_shared(const double *buf)
        {
            const float *f = reinterpret_cast<const float *>(buf);
            return Scale(f[0], f[1]);
        }
    };
    /* A x + B y, A = ah + al, B = bh + bl, as a float pair: the products by the
       FMA-based TwoProduct (p = fl(a b), e = fma(a, b, -p) exact), their sum by
       Knuth's TwoSum, the low parts added to the error term; hi is the sum
       rounded once */
    __device__ static void dot2w(float ah, float al, float x, float bh, float bl, float y, float &hi, float &lo)
    {
        const float p1 = __fmul_rn(ah, x);
        float e1 = __fmaf_rn(ah, x, -p1);
        e1 = __fmaf_rn(al, x, e1);
        const float p2 = __fmul_rn(bh, y);
        float e2 = __fmaf_rn(bh, y, -p2);
        e2 = __fmaf_rn(bl, y, e2);
        const float s = __fadd_rn(p1, p2);
        const float bp = __fsub_rn(s, p1);
        const float t = __fadd_rn(__fsub_rn(p1, __fsub_rn(s, bp)), __fsub_rn(p2, bp));
        const float e = __fadd_rn(t, __fadd_rn(e1, e2));
        hi = __fadd_rn(s, e);
        lo = __fsub_rn(e, __fsub_rn(hi, s));
    }
    __device__ static float dot2(float ah, float al, float x, float bh, float bl, float y)
    {
        float hi, lo;
        dot2w(ah, al, x, bh, bl, y, hi, lo);
        return hi;
    }
    typedef float4 RotVal; /* (sqrt|a|, sqrt(1-|a|)) as float pairs */
    __device__ static RotVal rot_table(const QwSimDev &d, uint32_t A) { return __ldg(d.fg32 + A); }
    /* the table entry of code A (rot_bits = 0) computed in place: hi the
       correctly rounded square root, lo the Newton correction (x - hi^2) /
       (2 hi) with the residual exact by FMA -- the host builds the table the
       same way, so the bits agree */
    static constexpr bool kRotCode = true;
    __device__ static RotVal rot_code(uint32_t A)
    {
        const int q = (int)(int16_t)(uint16_t)A;
        const float x = (float)(q < 0 ? -q : q) * (1.0f / 32768.0f), y = 1.0f - x;
        const float fh = __fsqrt_rn(x), gh = __fsqrt_rn(y);
        const float fl = fh > 0.0f ? __fdiv_rn(__fmaf_rn(-fh, fh, x), 2.0f * fh) : 0.0f;
        const float gl = gh > 0.0f ? __fdiv_rn(__fmaf_rn(-gh, gh, y), 2.0f * gh) : 0.0f;
        return make_float4(fh, fl, gh, gl);
    }
    __device__ static RotVal rot_zero() { return make_float4(0.f, 0.f, 1.f, 0.f); }
    __device__ static void rot(RotVal t, uint32_t A, bool dag, bool sneg, T a0, T a1, T &o0, T &o1);
    /* R^dag's b2 = 0 output as float pairs (~48 bits), not rounded to FP32 */
    typedef WideF Wide;
    __device__ static Wide rdag0(RotVal t, uint32_t A, bool sneg, T a0, T a1);
    __device__ static T narrow(Wide w) { return make_float2(w.xh, w.yh); }
    __device__ static T sum_amp(const Sum &r) { return make_float2(r.x.h, r.y.h); }
    __device__ static RotVal prescale(RotVal t, int e)
    {
        const float c = __int_as_float((127 - e) << 23);
        return make_float4(t.x * c, t.y * c, t.z * c, t.w * c);
    }
    __device__ static Wide wide_zero() { return Wide{0.f, 0.f, 0.f, 0.f}; }
    __device__ static void reflect(const Sum &r, RotVal t, uint32_t A, bool sneg, T a0, T a1, T &o0, T &o1);
    /* round(F R - a), F = fh + fl, R = rh + rl */
    __device__ static float mul_sub(float fh, float fl, float rh, float rl, float a)
    {
        const float p = __fmul_rn(fh, rh);
        float e = __fmaf_rn(fh, rh, -p);
        e = __fmaf_rn(fh, rl, e);
        e = __fmaf_rn(fl, rh, e);
        const float s = __fsub_rn(p, a);
        const float bp = __fsub_rn(s, p);
        const float t = __fadd_rn(__fsub_rn(p, __fsub_rn(s, bp)), __fsub_rn(-a, bp));
        return __fadd_rn(s, __fadd_rn(t, e));
    }
    __device__ static float2 approx2(T a) { return a; }
    __device__ static float inf_norm(T a) { return fmaxf(fabsf(a.x), fabsf(a.y)); }
    __device__ static float rot_f(RotVal t) { return t.x; }
    __device__ static float rot_g(RotVal t) { return t.z; }
    static constexpr float kApproxErr = 1.0f / 524288.0f; /* 2^-19 of the terms' magnitudes */
};

__device__ double Amp<float2>::Norm::warp_total() const
{
    DF v;
    v.h = hi;
    v.l = lo;
    for (int o = 16; o > 0; o >>= 1) {
        const float oh = __shfl_xor_sync(FULL, v.h, o), ol = __shfl_xor_sync(FULL, v.l, o);
        v.add(oh, ol);
    }
    return lane_id() == 0 ? (double)v.h + (double)v.l : 0.0;
}

/* multiply by 1 (real f) or by i*sigma (imaginary f), sigma = sneg ? -1 : 1:
 * i sigma (x + i y) = -sigma y + i sigma x */
template <typename T>
__device__ __forceinline__ T rho(T a, bool imag, bool sneg)
{
    T r;
    r.x = imag ? flip_if(a.y, !sneg) : a.x;
    r.y = imag ? flip_if(a.x, sneg) : a.y;
    return r;
}

/* R:    o0 = f a0 - g a1,        o1 = g a0 + conj(f) a1
 * R^dag: o0 = conj(f) a0 + g a1, o1 = f a1 - g a0
 * with f = fm (a >= 0) or i sigma fm (a < 0): f x = fm rho(x, sigma),
 * conj(f) x = fm rho(x, -sigma). */
__device__ void Amp<double2>::rot(RotVal t, uint32_t A, bool dag, bool sneg, T a0, T a1, T &o0, T &o1)
{
    const double fm = t.x, g = t.y;
    const bool imag = (int16_t)(uint16_t)A < 0;
    const double2 x0 = rho(a0, imag, dag ? !sneg : sneg);
    const double2 x1 = rho(a1, imag, dag ? sneg : !sneg);
    if (!dag) {
        o0 = make_double2(fma(fm, x0.x, -g * a1.x), fma(fm, x0.y, -g * a1.y));
        o1 = make_double2(fma(g, a0.x, fm * x1.x), fma(g, a0.y, fm * x1.y));
    } else {
        o0 = make_double2(fma(fm, x0.x, g * a1.x), fma(fm, x0.y, g * a1.y));
        o1 = make_double2(fma(fm, x1.x, -g * a0.x), fma(fm, x1.y, -g * a0.y));
    }
}

__device__ double2 Amp<double2>::rdag0(RotVal t, uint32_t A, bool sneg, T a0, T a1)
{
    const bool imag = (int16_t)(uint16_t)A < 0;
    const double2 x0 = rho(a0, imag, !sneg);
    return make_double2(fma(t.x, x0.x, t.y * a1.x), fma(t.x, x0.y, t.y * a1.y));
}

__device__ void Amp<double2>::reflect(const Sum &r, RotVal t, uint32_t A, bool sneg, T a0, T a1, T &o0, T &o1)
{
    const bool imag = (int16_t)(uint16_t)A < 0;
    const double2 x = rho(make_double2(r.x, r.y), imag, sneg);
    o0 = make_double2(fma(t.x, x.x, -a0.x), fma(t.x, x.y, -a0.y));
    o1 = make_double2(fma(t.y, r.x, -a1.x), fma(t.y, r.y, -a1.y));
}

__device__ WideF Amp<float2>::rdag0(RotVal t, uint32_t A, bool sneg, T a0, T a1)
{
    const bool imag = (int16_t)(uint16_t)A < 0;
    const float2 x0 = rho(a0, imag, !sneg);
    WideF w;
    dot2w(t.x, t.y, x0.x, t.z, t.w, a1.x, w.xh, w.xl);
    dot2w(t.x, t.y, x0.y, t.z, t.w, a1.y, w.yh, w.yl);
    return w;
}

__device__ void Amp<float2>::reflect(const Sum &r, RotVal t, uint32_t A, bool sneg, T a0, T a1, T &o0, T &o1)
{
    /* f r = fm rho(r): i sigma (x + i y) = -sigma y + i sigma x */
    const bool imag = (int16_t)(uint16_t)A < 0;
    const float2 h = rho(make_float2(r.x.h, r.y.h), imag, sneg), l = rho(make_float2(r.x.l, r.y.l), imag, sneg);
    o0 = make_float2(mul_sub(t.x, t.y, h.x, l.x, a0.x), mul_sub(t.x, t.y, h.y, l.y, a0.y));
    o1 = make_float2(mul_sub(t.z, t.w, r.x.h, r.x.l, a1.x), mul_sub(t.z, t.w, r.y.h, r.y.l, a1.y));
}

__device__ void Amp<float2>::rot(RotVal t, uint32_t A, bool dag, bool sneg, T a0, T a1, T &o0, T &o1)
{
    /* t = (fh, fl, gh, gl) */
    const bool imag = (int16_t)(uint16_t)A < 0;
    const float2 x0 = rho(a0, imag, dag ? !sneg : sneg);
    const float2 x1 = rho(a1, imag, dag ? sneg : !sneg);
    if (!dag) {
        o0 = make_float2(dot2(t.x, t.y, x0.x, -t.z, -t.w, a1.x), dot2(t.x, t.y, x0.y, -t.z, -t.w, a1.y));
        o1 = make_float2(dot2(t.z, t.w, a0.x, t.x, t.y, x1.x), dot2(t.z, t.w, a0.y, t.x, t.y, x1.y));
    } else {
        o0 = make_float2(dot2(t.x, t.y, x0.x, t.z, t.w, a1.x), dot2(t.x, t.y, x0.y, t.z, t.w, a1.y));
        o1 = make_float2(dot2(t.x, t.y, x1.x, -t.z, -t.w, a0.x), dot2(t.x, t.y, x1.y, -t.z, -t.w, a0.y));
    }
}

/* 1 for a non-zero amplitude (+-0 is zero), tested on the bits: an FP64
   comparison would take a slot of the FP64 pipe */
__device__ __forceinline__ unsigned int nz(float2 a)
{
    return ((__float_as_uint(a.x) | __float_as_uint(a.y)) << 1) != 0u ? 1u : 0u;
}
__device__ __forceinline__ unsigned int nz(double2 a)
{
    return (((uint64_t)__double_as_longlong(a.x) | (uint64_t)__double_as_longlong(a.y)) << 1) != 0ull ? 1u : 0u;
}
__device__ __forceinline__ unsigned int nz_f(float4 t) { return t.x != 0.f ? 1u : 0u; } /* f of a RotVal */
__device__ __forceinline__ unsigned int nz_f(double2 t) { return (uint32_t)__double2hiint(t.x) != 0u ? 1u : 0u; }
__device__ __forceinline__ unsigned int nz_g(float4 t) { return t.z != 0.f ? 1u : 0u; } /* g of a RotVal */
__device__ __forceinline__ unsigned int nz_g(double2 t) { return (uint32_t)__double2hiint(t.y) != 0u ? 1u : 0u; }

/* ---- the walk operator on one b2-pair --------------------------------------- */
/*
 * T~^dag, P, T~ without S: R^dag, H P H, R on the pair (a0, a1) of one slot.
 * H P H = 2 Pi - 1 there (P keeps the sign of the zero-type group's uniform
 * superposition only), so with R R^dag = 1 a pair outside the zero-type
 * groups comes back as -(a0, a1), and the pair of slot l of a zero-type group
 * as (f_l r - a0, g_l r - a1), r = (2 / s) sum_v u_v, u_v = conj(f_v) a0_v +
 * g_v a1_v (R^dag's b2 = 0 outputs): one rotation instead of two, and one
 * rounding of the stored amplitude instead of three.
 * The intermediate branches still count and still prune as in the paper's
 * schedule: R^dag's outputs u, v and the reflected r - u with |.| <= tau are
 * dropped.  Where that drops a non-zero value, the pair takes the literal R
 * of what is left.  Which values are above tau is decided in FP32 (their
 * magnitudes to kApproxErr of the terms'); only the few that this leaves
 * open are formed exactly.
 */
template <typename AmpT> struct PairState {
    bool c0, c1; /* R^dag's outputs kept */
    bool lossy;  /* a non-zero intermediate was dropped: take the literal R */
};

__device__ __forceinline__ float max_abs(float x, float y) { return fmaxf(fabsf(x), fabsf(y)); }
__device__ __forceinline__ float sum_abs(float2 a) { return fabsf(a.x) + fabsf(a.y); }

/* kept / dropped of R^dag's outputs by their exact values */
template <typename AmpT>
__device__ __noinline__ unsigned pair_exact(const QwSimDev &d, typename Amp<AmpT>::RotVal t, uint32_t A, bool sneg,
                                            AmpT a0, AmpT a1)
{
    AmpT o0, o1;
    Amp<AmpT>::rot(t, A, true, sneg, a0, a1, o0, o1);
    const bool k0 = Amp<AmpT>::keep(d, o0), k1 = Amp<AmpT>::keep(d, o1);
    const bool lost = (!k0 && nz(o0)) || (!k1 && nz(o1));
    return (k0 ? 1u : 0u) | (k1 ? 2u : 0u) | (lost ? 4u : 0u);
}

/* R of what the pruning left of -R^dag (a0, a1) (outside the zero-type
   groups) or of (h0, -v) (h0: the reflected b2 = 0 member, hz given) */
template <typename AmpT>
__device__ __noinline__ void pair_literal(const QwSimDev &d, typename Amp<AmpT>::RotVal t, uint32_t A, bool sneg,
                                          AmpT a0, AmpT a1, bool c0, bool c1, bool zero_type, AmpT h0, AmpT &r0,
                                          AmpT &r1)
{
    AmpT o0, o1;
    Amp<AmpT>::rot(t, A, true, sneg, a0, a1, o0, o1);
    const AmpT b0 = zero_type ? h0 : (c0 ? Amp<AmpT>::neg(o0) : Amp<AmpT>::zero());
    const AmpT b1 = c1 ? Amp<AmpT>::neg(o1) : Amp<AmpT>::zero();
    Amp<AmpT>::rot(t, A, false, sneg, b0, b1, r0, r1);
}

/* R^dag on the pair: which outputs are kept (x0, x1: approx2 of a0, a1; u0:
   the b2 = 0 output, approximately) */
template <typename AmpT>
__device__ __forceinline__ PairState<AmpT> pair_state(const QwSimDev &d, typename Amp<AmpT>::RotVal t, uint32_t A,
                                                      bool sneg, AmpT a0, AmpT a1, float2 x0, float2 x1, float &m)
{
    const float f = Amp<AmpT>::rot_f(t), g = Amp<AmpT>::rot_g(t);
    const bool imag = (int16_t)(uint16_t)A < 0;
    m = sum_abs(x0) + sum_abs(x1);
    const float lim = fmaf(Amp<AmpT>::kApproxErr, m, d.thr32);
    const float2 y0 = rho(x0, imag, !sneg), y1 = rho(x1, imag, sneg);
    PairState<AmpT> p;
    p.c0 = max_abs(fmaf(f, y0.x, g * x1.x), fmaf(f, y0.y, g * x1.y)) > lim;
    p.c1 = max_abs(fmaf(f, y1.x, -g * x0.x), fmaf(f, y1.y, -g * x0.y)) > lim;
    p.lossy = false;
    /* products of which both are exactly 0 give an exact 0 */
    const bool n0 = nz(a0) != 0u, n1 = nz(a1) != 0u, nf = nz_f(t) != 0u, ng = nz_g(t) != 0u;
    const bool open = (!p.c0 && ((nf && n0) || (ng && n1))) || (!p.c1 && ((nf && n1) || (ng && n0)));
    if (open) {
        const unsigned e = pair_exact<AmpT>(d, t, A, sneg, a0, a1);
        p.c0 = (e & 1u) != 0u;
        p.c1 = (e & 2u) != 0u;
        p.lossy = (e & 4u) != 0u;
    }
    return p;
}

/* a pair outside the zero-type groups: (r0, r1) = -(a0, a1), and how many of
   R^dag's outputs are kept */
template <typename AmpT>
__device__ __forceinline__ unsigned pair_negate(const QwSimDev &d, typename Amp<AmpT>::RotVal t, uint32_t A, bool sneg,
                                                AmpT a0, AmpT a1, AmpT &r0, AmpT &r1)
{
    float m;
    const PairState<AmpT> p =
        pair_state<AmpT>(d, t, A, sneg, a0, a1, Amp<AmpT>::approx2(a0), Amp<AmpT>::approx2(a1), m);
    r0 = Amp<AmpT>::neg(a0);
    r1 = Amp<AmpT>::neg(a1);
    if (p.lossy) pair_literal<AmpT>(d, t, A, sneg, a0, a1, p.c0, p.c1, false, Amp<AmpT>::zero(), r0, r1);
    return (p.c0 ? 1u : 0u) + (p.c1 ? 1u : 0u);
}

/* R^dag on a pair of a zero-type group: its term u of the group's sum (0
   where dropped) */
template <typename AmpT>
__device__ __forceinline__ PairState<AmpT> pair_tdag(const QwSimDev &d, typename Amp<AmpT>::RotVal t, uint32_t A,
                                                     bool sneg, AmpT a0, AmpT a1, typename Amp<AmpT>::Wide &u, float &m)
{
    const PairState<AmpT> p =
        pair_state<AmpT>(d, t, A, sneg, a0, a1, Amp<AmpT>::approx2(a0), Amp<AmpT>::approx2(a1), m);
    u = p.c0 ? Amp<AmpT>::rdag0(t, A, sneg, a0, a1) : Amp<AmpT>::wide_zero();
    return p;
}

/* the pair after H P H and R where the FP32 decision left the reflected b2 = 0
   member open, or an intermediate was lost; returns whether it is kept */
template <typename AmpT>
__device__ __noinline__ bool pair_reflect_exact(const QwSimDev &d, typename Amp<AmpT>::Sum r,
                                                typename Amp<AmpT>::RotVal t, uint32_t A, bool sneg, AmpT a0, AmpT a1,
                                                PairState<AmpT> p, AmpT &r0, AmpT &r1)
{
    const AmpT u = p.c0 ? Amp<AmpT>::narrow(Amp<AmpT>::rdag0(t, A, sneg, a0, a1)) : Amp<AmpT>::zero();
    AmpT h0 = r.minus(u);
    const bool d0 = Amp<AmpT>::keep(d, h0);
    if (p.lossy || (!d0 && nz(h0)))
        pair_literal<AmpT>(d, t, A, sneg, a0, a1, p.c0, p.c1, true, d0 ? h0 : Amp<AmpT>::zero(), r0, r1);
    else
        Amp<AmpT>::reflect(r, t, A, sneg, a0, a1, r0, r1);
    return d0;
}

/* the pair after H P H and R, r: (2 / s) times the group's sum, ux: the
   pair's term of the sum, approximately; d0: the reflected b2 = 0 member is
   kept */
template <typename AmpT>
__device__ __forceinline__ void pair_reflect(const QwSimDev &d, const typename Amp<AmpT>::Sum &r,
                                             typename Amp<AmpT>::RotVal t, uint32_t A, bool sneg, AmpT a0, AmpT a1,
                                             float2 ux, float m, const PairState<AmpT> &p, AmpT &r0, AmpT &r1,
                                             bool &d0)
{
    const float2 rx = Amp<AmpT>::approx2(Amp<AmpT>::sum_amp(r));
    const float lim = fmaf(Amp<AmpT>::kApproxErr, m + sum_abs(rx), d.thr32);
    d0 = max_abs(rx.x - ux.x, rx.y - ux.y) > lim;
    Amp<AmpT>::reflect(r, t, A, sneg, a0, a1, r0, r1);
    if (!d0 || p.lossy) d0 = pair_reflect_exact<AmpT>(d, r, t, A, sneg, a0, a1, p, r0, r1);
}

} // namespace

#endif /* QW_AMP_CUH */
