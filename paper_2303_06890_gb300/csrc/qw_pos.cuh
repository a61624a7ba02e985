/*
 * qw_pos.cuh -- the positional layout (walk_variant 7): kernels and launchers,
 * instantiated for complex128 (qw_pos64.cu) and complex64 (qw_pos32.cu).
 */
#ifndef QW_POS_CUH
#define QW_POS_CUH

#include "qw_amp.cuh"
#include "qw_device.cuh"
#include "qw_internal.h"
#include "qw_pos_norm.h"

namespace {

/* ==== positional walk steps ==================================================== */
/*
 * The state of the walk held by position instead of by key.  At a step
 * boundary every branch that the walk reaches from T~|b~> sits in a row
 * (jc = 0, j < N, b1) with kc = A = 0, and its k is either a column of row j
 * (W = S (2 T~ Pi T~^dag - 1): the branches of T~ Pi's range are those of
 * T~'s rows, the swapped ones have k = a row whose padded column list holds j)
 * -- entry g s + l for the column in slot l of row g -- or one of the rows x
 * whose slot l_x holds column j while row j holds no column x (a padded, so
 * unpaired, entry): an extra, entry N s + e in a list of all rows' extras in
 * row order.  An entry holds four amplitudes: A0, A1 of row (j, b1 = 0), b2 = 0
 * and 1, and B0, B1 of row (j, b1 = 1).  An absent branch is 0, so the place is
 * the key.
 *
 * B1 stays empty: S gives a b1 = b2 = 1 branch only from one of the same kind,
 * and T~|b~> has none.  The arithmetic takes it as 0 unless an imported state
 * put something there (FULLST).
 *
 * Layout (PosMem): S scatters a slot's outputs to one entry, and what a step
 * costs at large N is the 32-byte sectors it writes (each counted twice in L2,
 * which has a part on either die).  complex64: an entry is one sector {A0, A1,
 * B0, B1}, read and written by one 32-byte access -- one full sector a slot
 * instead of two partial ones with A and B apart.  complex128: A0, A1 are one
 * sector, B0 and B1 planes of their own, B1 not touched (48 bytes a slot: with
 * B0, B1 as a second sector the state of Table 1's E would be 134 MB a step in
 * and out, more than L2 holds).
 *
 * The lane of slot (j, l) runs the walk operator on the slot's two pairs
 * (T~^dag's maps take them to (l, 0), T~'s back to k = col): b1 = 0 reflected
 * in the zero-type group (the unit's lanes), b1 = 1 negated; S sends the
 * outputs to entry dst(j, l) -- that of k = j in row col(j, l) -- A from the two
 * b2 = 0 outputs, B0 and B1 from the b2 = 1 ones.  An extra is outside every
 * zero-type group and its maps leave A = 0 (kc = x ^ col(j, 0) != 0 after
 * O_s'^dag, so O_A' does not fire): R(0) (-1) R(0)^dag = -1 on its pair
 * (each output the negated input, kept where the input is), sent to slot
 * (x, l_x); extras run 32 to a warp on their own.  Every entry of the output has
 * exactly one writer and pruned outputs are written as 0: no counts, atomics,
 * searches or keys, and nothing to clear between steps.
 *
 * Several steps run in one launch: a grid of at most one block per SM,
 * launched cooperatively, with a barrier over the grid between steps that
 * also carries the norm.  What a step needs of the matrix --
 * each slot's rotation, destination and flags -- is laid out once per launch
 * in shared memory (TAB) in the order the block's lanes use it, so that a
 * step reads the state and nothing else.
 *
 * Bounds: a step at small N is a chain of latencies -- state load, rotation,
 * group sum, store, barrier -- and one launch per step added the launch and
 * the last block's reduction to it.  At large N: the sectors written, and the
 * FP64 pipe for complex128 (12 FP64 instructions a slot, 16 cycles each on an
 * SM).
 */
constexpr int kPosMaxWarps = 16; /* 512 threads: up to 128 registers a thread */

/* An entry's four amplitudes; state accesses go to L2 (another SM wrote what
   this one reads). */
template <typename AmpT> struct Entry {
    AmpT a0, a1, b0, b1;
};
template <typename AmpT> struct PosMem;
template <> struct PosMem<float2> {
    /* index of one amplitude of entry i (T entries in all) */
    __device__ static size_t at(size_t, size_t i, int b1, int b2) { return 4 * i + 2 * b1 + b2; }
    template <bool FULLST> __device__ static void load(const float2 *p, uint32_t, uint32_t i, Entry<float2> &e)
    {
        asm volatile("ld.global.cg.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(e.a0.x), "=f"(e.a0.y), "=f"(e.a1.x), "=f"(e.a1.y), "=f"(e.b0.x), "=f"(e.b0.y),
                       "=f"(e.b1.x), "=f"(e.b1.y)
                     : "l"(p + 4 * (size_t)i));
    }
    template <bool FULLST> __device__ static void store(float2 *p, uint32_t, uint32_t i, const Entry<float2> &e)
    {
        asm volatile("st.global.cg.v8.f32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"f"(e.a0.x), "f"(e.a0.y),
                     "f"(e.a1.x), "f"(e.a1.y), "f"(e.b0.x), "f"(e.b0.y), "f"(e.b1.x), "f"(e.b1.y), "l"(p + 4 * (size_t)i)
                     : "memory");
    }
};
template <> struct PosMem<double2> {
    __device__ static size_t at(size_t T, size_t i, int b1, int b2) { return b1 ? (2 + b2) * T + i : 2 * i + b2; }
    template <bool FULLST> __device__ static void load(const double2 *p, uint32_t T, uint32_t i, Entry<double2> &e)
    {
        asm volatile("ld.global.cg.v4.f64 {%0, %1, %2, %3}, [%4];"
                     : "=d"(e.a0.x), "=d"(e.a0.y), "=d"(e.a1.x), "=d"(e.a1.y) : "l"(p + 2 * (size_t)i));
        e.b0 = __ldcg(p + 2 * (size_t)T + i);
        if (FULLST) e.b1 = __ldcg(p + 3 * (size_t)T + i);
    }
    template <bool FULLST> __device__ static void store(double2 *p, uint32_t T, uint32_t i, const Entry<double2> &e)
    {
        asm volatile("st.global.cg.v4.f64 [%4], {%0, %1, %2, %3};" ::"d"(e.a0.x), "d"(e.a0.y), "d"(e.a1.x), "d"(e.a1.y),
                     "l"(p + 2 * (size_t)i) : "memory");
        __stcg(p + 2 * (size_t)T + i, e.b0);
        if (FULLST) __stcg(p + 3 * (size_t)T + i, e.b1);
    }
};

/* ---- barrier over the grid, with the norm ---------------------------------- */
/*
 * Two 64-bit words per step (qw_pos_norm.h): every block adds 1 to the count in
 * their low 8 bits and its share of the norm above it, to one the share modulo
 * 2^56 units, to the other its high part, so an atomic on each is both the
 * block's arrival and its term of a sum that does not depend on the order of
 * arrival, and that no norm carries into the count.  Without renormalisation
 * only the first is used.  They lie side by side and are polled by one load; the
 * second's add goes before the first's, which releases the block's stores.  A
 * block that holds a share out of the units' range (or not finite) adds all of its
 * own to the step's FP64 number and says so.  Four sets take turns; passing step t,
 * block 0 clears that of step t + 2, which every block has left (it was step t - 2's).
 * Beside one word with a lane's share rounded to 2^-54 of the target (QLS, N = 1024
 * complex64: 4.44 us a step) the second word costs 0.05 us a step.
 */
struct PosNorm { /* per launch, in shared memory */
    int k;                     /* units are 2^-k */
    float s1, s2;              /* s1 s2 = 2^k */
    unsigned long long target; /* the renormalisation target in units */
    float inv_h, inv_l;        /* 2^24 / target */
};

__device__ __forceinline__ void pos_norm_setup(const QwStepArgs &a, PosNorm &pn)
{
    const double t = *a.renorm_target;
    bool odd;
    pn.k = pos_unit_exp(t);
    pn.target = pos_units(t, pn.k, odd);
    const double inv = pn.target ? 16777216.0 / (double)pn.target : 0.0;
    pn.inv_h = (float)inv;
    pn.inv_l = (float)(inv - (double)pn.inv_h);
    /* (FP32 shares: 2^k in two factors; beyond 2^252 every non-zero share is odd) */
    const int k = pn.k > 252 ? 252 : (pn.k < -252 ? -252 : pn.k), h = k >> 1;
    pn.s1 = __int_as_float((127 + h) << 23);
    pn.s2 = __int_as_float((127 + k - h) << 23);
}

/* a lane's norm share in units */
__device__ __forceinline__ unsigned long long to_units(const Amp<double2>::Norm &n, const PosNorm &pn, bool &odd)
{
    return pos_units(n.get(), pn.k, odd);
}
__device__ __forceinline__ unsigned long long to_units(const Amp<float2>::Norm &n, const PosNorm &pn, bool &odd)
{
    /* the scaling by powers of two is exact; hi has 24 bits, lo is rounded to a unit */
    const float h = n.hi * pn.s1 * pn.s2, l = n.lo * pn.s1 * pn.s2;
    odd = !(h >= 0.0f && h < 0x1p63f);
    return odd ? 0ull : (unsigned long long)(__float2ll_rn(h) + __float2ll_rn(l));
}
/* Sums of shares below 2^63, exact through the integer reduction of three limbs,
   of 22 bits and the rest: up to 512 lanes' fit 32 bits each */
struct PosLimbs {
    unsigned int a, b, c;
    __device__ __forceinline__ void reduce()
    {
        a = __reduce_add_sync(FULL, a);
        b = __reduce_add_sync(FULL, b);
        c = __reduce_add_sync(FULL, c);
    }
    __device__ __forceinline__ unsigned long long low() const { return (unsigned long long)a + ((unsigned long long)b << 22); }
    __device__ __forceinline__ unsigned long long fine() const { return low() + ((unsigned long long)c << 44); }
    __device__ __forceinline__ unsigned long long coarse() const
    {
        return ((unsigned long long)c << (44 - kCoarseShift)) + (low() >> kCoarseShift);
    }
};
__device__ __forceinline__ PosLimbs warp_sum_units(unsigned long long v)
{
    PosLimbs l{(unsigned)(v & 0x3fffffull), (unsigned)((v >> 22) & 0x3fffffull), (unsigned)(v >> 44)};
    l.reduce();
    return l;
}

__device__ __forceinline__ void word_add(unsigned long long *p, unsigned long long v)
{
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void word_add_relaxed(unsigned long long *p, unsigned long long v)
{
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ ulonglong2 words_load(const unsigned long long *p) /* each word of its own moment */
{
    ulonglong2 v;
    asm volatile("ld.acquire.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long word_load(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

/* The renormalisation factor sqrt(target / sum) between two steps of a run, from a sum
 * near the target, where FP32 arithmetic gives it as well as FP64's does: complex64,
 * which applies it as a float pair, within 2^-14 (pos_factor_pair); complex128 where
 * x = (target - sum) / target is below 2^-30 (what rounding alone leaves is 2^-50),
 * as 1 + x / 2, off by 2^-54 at most before it is rounded to FP64.  Otherwise false,
 * and pos_scale_exact; that too for the factor a launch leaves behind. */
__device__ __noinline__ double pos_scale_exact(double target, double norm)
{
    return norm > 0.0 ? sqrt(target / norm) : 1.0;
}
__device__ __forceinline__ bool pos_scale(const PosNorm &pn, int64_t dev, Amp<float2>::Scale &s)
{
    return pos_factor_pair(dev, pn.inv_h, pn.inv_l, s.sh, s.sl);
}
__device__ __forceinline__ bool pos_scale(const PosNorm &pn, int64_t dev, Amp<double2>::Scale &s)
{
    const float x = (float)dev * (pn.inv_h * 0x1p-24f);
    s.s = 1.0 + (double)(0.5f * x);
    return fabsf(x) < 0x1p-30f;
}
template <int FIELD>
__device__ __noinline__ double pos_norm(const PosNorm &pn, unsigned long long fine, unsigned long long coarse, double extra)
{
    return pos_total<FIELD>(fine, coarse, extra, pn.k);
}

/* FP64 work of the read-out and of a complex128 norm, out of line: a
   predicated-off FP64 instruction takes its slot of the 1/64-rate pipe */
__device__ __noinline__ double pos_readout(double2 *y, double unit, double sx, double sy)
{
    double2 acc = __ldcg(y);
    acc.x += unit * sx;
    acc.y += unit * sy;
    __stcg(y, acc);
    return fma(acc.x, acc.x, acc.y * acc.y);
}
__device__ __noinline__ double norm_c128(double v, double2 a) { return fma(a.x, a.x, fma(a.y, a.y, v)); }
__device__ __forceinline__ void norm_add(Amp<double2>::Norm &n, double2 a) { n.v = norm_c128(n.v, a); }
__device__ __forceinline__ void norm_add(Amp<float2>::Norm &n, float2 a) { n.add(a); }

/* The pruning rule on a value of which m = inf_norm: above thr32 kept, the
   rest exactly (0 is the common case there) */
template <typename AmpT> __device__ __noinline__ bool keep_exact(const QwSimDev &d, AmpT a)
{
    return Amp<AmpT>::keep(d, a);
}
__device__ __forceinline__ bool pos_keep(const QwSimDev &d, double2 a)
{
    const float m = Amp<double2>::inf_norm(a);
    bool k = m > d.thr32;
    if (!k && m > 0.0f) k = keep_exact<double2>(d, a);
    return k;
}
__device__ __forceinline__ bool pos_keep(const QwSimDev &d, float2 a) { return Amp<float2>::keep(d, a); }

/* both rows of a slot where the FP32 bounds leave a decision open: the kept
   flags by the exact values (bits 0, 1: u, v; bit 2: a non-zero one dropped) */
template <typename AmpT>
__device__ __noinline__ void negate_exact(const QwSimDev &d, typename Amp<AmpT>::RotVal t, uint32_t A, bool sneg,
                                          AmpT q0, AmpT q1, AmpT &r0, AmpT &r1, unsigned &kept)
{
    const unsigned e = pair_exact<AmpT>(d, t, A, sneg, q0, q1);
    kept = (e & 1u) + ((e >> 1) & 1u);
    if (e & 4u) pair_literal<AmpT>(d, t, A, sneg, q0, q1, (e & 1u) != 0u, (e & 2u) != 0u, false, Amp<AmpT>::zero(), r0, r1);
}

/* branch counters of a lane, packed 8 bits each (in, rdag, hph, out) so that
   one predicated addition counts a branch in several; unpacked before a field
   can overflow */
constexpr uint32_t kCntIn = 1u, kCntRdag = 1u << 8, kCntHph = 1u << 16, kCntOut = 1u << 24;
struct PosStats {
    unsigned int rows = 0, in = 0, rdag = 0, hph = 0, out = 0;
    __device__ __forceinline__ void take(uint32_t &c)
    {
        in += c & 0xffu;
        rdag += (c >> 8) & 0xffu;
        hph += (c >> 16) & 0xffu;
        out += c >> 24;
        c = 0;
    }
    __device__ void flush(const QwStepArgs &a)
    {
        unsigned int v[5] = {rows, in, rdag, hph, out};
#pragma unroll
        for (int i = 0; i < 5; ++i) v[i] = __reduce_add_sync(FULL, v[i]);
        if (a.stats && lane_id() == 0 && v[1]) {
            atomicAdd(a.stats + QW_STAT_ROWS, (unsigned long long)v[0]);
            atomicAdd(a.stats + QW_STAT_IN, (unsigned long long)v[1]);
            atomicAdd(a.stats + QW_STAT_RDAG, (unsigned long long)v[2]);
            atomicAdd(a.stats + QW_STAT_HPH, (unsigned long long)v[3]);
            atomicAdd(a.stats + QW_STAT_OUT, (unsigned long long)v[4]);
        }
    }
};

/* The walk operator on a group's slots (both rows' pairs of each): the lane's
 * SPL slots, rotations rv and flags dst (bit 31 sigma = -1, bit 30 a negative
 * element) in, on_sum(the group sum, scaled by 2 / s) for the read-out, on_out(q,
 * the entry that slot q sends to its destination). */
template <typename AmpT, int S, bool FULLST, int SPL, typename OnSum, typename OnOut>
__device__ __forceinline__ void pos_group(const QwSimDev &d, const typename Amp<AmpT>::RotVal (&rv)[SPL],
                                          const uint32_t (&dst)[SPL], const Entry<AmpT> (&in)[SPL], bool rescale,
                                          const typename Amp<AmpT>::Scale &scale, bool valid, bool renorm,
                                          typename Amp<AmpT>::Norm &nrm, uint32_t &cnt, PosStats &st, OnSum on_sum,
                                          OnOut on_out)
{
    constexpr int SW = S > 32 ? 32 : S;
    constexpr int LOG2S = S == 4 ? 2 : S == 8 ? 3 : S == 16 ? 4 : S == 32 ? 5 : 6;
    constexpr float kHalfS = 0.5f * S, kErr = Amp<AmpT>::kApproxErr;
    const AmpT zero = Amp<AmpT>::zero();
    const int lane = threadIdx.x & 31, ul = lane / SW, lb = lane % SW;
    AmpT a0[SPL], a1[SPL], q0[SPL], q1[SPL];
    float A0[SPL], A1[SPL], Q0[SPL];
    bool any = false;
#pragma unroll
    for (int q = 0; q < SPL; ++q) {
        a0[q] = in[q].a0;
        a1[q] = in[q].a1;
        q0[q] = in[q].b0;
        q1[q] = FULLST ? in[q].b1 : zero;
        if (rescale) {
            a0[q] = scale.apply(a0[q]);
            a1[q] = scale.apply(a1[q]);
            q0[q] = scale.apply(q0[q]);
            if (FULLST) q1[q] = scale.apply(q1[q]);
        }
        A0[q] = Amp<AmpT>::inf_norm(a0[q]);
        A1[q] = Amp<AmpT>::inf_norm(a1[q]);
        Q0[q] = Amp<AmpT>::inf_norm(q0[q]);
        const bool n0 = A0[q] != 0.0f, n1 = A1[q] != 0.0f, m0 = Q0[q] != 0.0f, m1 = FULLST && nz(q1[q]) != 0u;
        if (n0) cnt += kCntIn;
        if (n1) cnt += kCntIn;
        if (m0) cnt += kCntIn;
        if (m1) cnt += kCntIn;
        any = any || n0 || n1 || m0 || m1;
    }
    {
        const unsigned m = __ballot_sync(FULL, any);
        const unsigned um = SW == 32 ? m : (m >> (ul * SW)) & ((1u << (SW & 31)) - 1u);
        if (lb == 0 && um != 0) st.rows += 1; /* units holding branches */
    }
    /* b1 = 0: R^dag's b2 = 0 output u (its exact value, scaled by 2 / s),
       and whether u and v are kept: |v| >= | f |a1| - g |a0| | in the
       maximum norm, which the phases leave alone, so the norms decide
       unless they nearly cancel */
    typename Amp<AmpT>::Wide u[SPL];
    PairState<AmpT> ps[SPL];
    float f[SPL], g_[SPL], U[SPL];
#pragma unroll
    for (int q = 0; q < SPL; ++q) {
        const uint32_t sgn = (dst[q] & 0x40000000u) >> 15; /* the value's sign bit (bit 15) */
        const bool sneg = (dst[q] >> 31) != 0u;
        f[q] = Amp<AmpT>::rot_f(rv[q]);
        g_[q] = Amp<AmpT>::rot_g(rv[q]);
        u[q] = Amp<AmpT>::rdag0(Amp<AmpT>::prescale(rv[q], LOG2S - 1), sgn, sneg, a0[q], a1[q]);
        U[q] = kHalfS * Amp<AmpT>::inf_norm(Amp<AmpT>::narrow(u[q]));
        const float fa = f[q] * A1[q], ga = g_[q] * A0[q];
        ps[q].c0 = U[q] > d.thr32;
        ps[q].c1 = fabsf(fa - ga) > fmaf(kErr, fa + ga, d.thr32);
        ps[q].lossy = false;
        if ((!ps[q].c0 && U[q] > 0.0f) || (!ps[q].c1 && fa + ga > 0.0f)) {
            const unsigned e = pair_exact<AmpT>(d, rv[q], sgn, sneg, a0[q], a1[q]);
            ps[q].c0 = (e & 1u) != 0u;
            ps[q].c1 = (e & 2u) != 0u;
            ps[q].lossy = (e & 4u) != 0u;
            if (!ps[q].c0) {
                u[q] = Amp<AmpT>::wide_zero();
                U[q] = 0.0f;
            }
        }
        if (ps[q].c0) cnt += kCntRdag;
        if (ps[q].c1) cnt += kCntRdag + kCntHph;
    }
    __syncwarp();
    typename Amp<AmpT>::Sum sum;
    sum.set(u[0]);
#pragma unroll
    for (int q = 1; q < SPL; ++q) sum.add(u[q]);
    sum.reduce(SW, SW);
    on_sum(sum);
    const float Rn = Amp<AmpT>::inf_norm(Amp<AmpT>::sum_amp(sum));
#pragma unroll
    for (int q = 0; q < SPL; ++q) {
        const uint32_t sgn = (dst[q] & 0x40000000u) >> 15;
        const bool sneg = (dst[q] >> 31) != 0u;
        /* the reflected r - u, then R: (f r - a0, g r - a1) */
        AmpT rA0, rA1;
        bool d0 = fabsf(Rn - U[q]) > fmaf(kErr, Rn + U[q], d.thr32);
        Amp<AmpT>::reflect(sum, rv[q], sgn, sneg, a0[q], a1[q], rA0, rA1);
        if (ps[q].lossy || (!d0 && Rn + U[q] > 0.0f))
            d0 = pair_reflect_exact<AmpT>(d, sum, rv[q], sgn, sneg, a0[q], a1[q], ps[q], rA0, rA1);
        if (d0) cnt += kCntHph;
        /* b1 = 1: R^dag, -1, R */
        AmpT rB0 = Amp<AmpT>::neg(q0[q]), rB1 = Amp<AmpT>::neg(q1[q]);
        if (FULLST) {
            const unsigned kept = pair_negate<AmpT>(d, rv[q], sgn, sneg, q0[q], q1[q], rB0, rB1);
            cnt += kept * (kCntRdag + kCntHph);
        } else { /* q1 = 0: |u| = f |q0|, |v| = g |q0| */
            const float fq = f[q] * Q0[q], gq = g_[q] * Q0[q], lim = fmaf(kErr, Q0[q], d.thr32);
            const bool c0 = fq > lim, c1 = gq > lim;
            unsigned kept = (c0 ? 1u : 0u) + (c1 ? 1u : 0u);
            if ((!c0 && fq > 0.0f) || (!c1 && gq > 0.0f))
                negate_exact<AmpT>(d, rv[q], sgn, sneg, q0[q], zero, rB0, rB1, kept);
            cnt += kept * (kCntRdag + kCntHph);
        }
        const bool eA0 = pos_keep(d, rA0), eA1 = pos_keep(d, rA1);
        const bool eB0 = pos_keep(d, rB0), eB1 = FULLST && pos_keep(d, rB1);
        if (valid) {
            if (renorm) {
                if (eA0) norm_add(nrm, rA0);
                if (eB0) norm_add(nrm, rB0);
                if (eA1) norm_add(nrm, rA1);
                if (FULLST && eB1) norm_add(nrm, rB1);
            }
            /* S: (k, b2) <-> (j, b1) */
            const Entry<AmpT> o = {eA0 ? rA0 : zero, eB0 ? rB0 : zero, eA1 ? rA1 : zero, eB1 ? rB1 : zero};
            on_out(q, o);
        }
        if (eA0) cnt += kCntOut;
        if (eB0) cnt += kCntOut;
        if (eA1) cnt += kCntOut;
        if (eB1) cnt += kCntOut;
    }
}

template <typename AmpT, int S, bool FULLST, bool TAB>
__global__ void __launch_bounds__(kPosMaxWarps * 32, 1) k_walk_pos(QwSimDev d, QwPosArgs p, QwStepArgs a)
{
    typedef typename Amp<AmpT>::RotVal RotVal;
    /* a unit (one j) on SW lanes, each lane holding SPL of its slots (l = lb
       + 32 k); RPP units per warp (a group) */
    constexpr int SW = S > 32 ? 32 : S, SPL = S / SW, RPP = 32 / SW;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ PosLimbs part_u[kPosMaxWarps]; /* the warps' shares of the norm */
    __shared__ double part_n[kPosMaxWarps]; /* the same in FP64: of a single step, and with odd ones */
    __shared__ double part_d[kPosMaxWarps]; /* ... of ||Y||^2 */
    __shared__ double scale_sm;
    __shared__ PosNorm pn;
    __shared__ int flag_sm, odd_sm;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, PW = blockDim.x >> 5;
    const bool rot_in_place = Amp<AmpT>::kRotCode && d.rot_calc;
    const AmpT zero = Amp<AmpT>::zero();
    const uint32_t n = (uint32_t)d.pos_rows, T = (uint32_t)d.pos_T; /* rows, entries; 4 T < 2^31 */
    const uint32_t X = T - n * S;                                     /* extras */
    const uint32_t ngroups = (n + RPP - 1) / RPP, xgroups = (X + 31) / 32, nwarps = gridDim.x * PW;
    const uint32_t g0 = blockIdx.x * PW + warp, x0 = nwarps - 1 - g0; /* extras from the last warp down */
    const int ul = lane / SW, lb = lane % SW;

    /* per-launch tables of the block's groups, [turn][warp] */
    const uint32_t turns = (ngroups + nwarps - 1) / nwarps, xturns = (xgroups + nwarps - 1) / nwarps;
    RotVal *t_rot = reinterpret_cast<RotVal *>(smem);
    uint32_t *t_dst = reinterpret_cast<uint32_t *>(t_rot + (size_t)turns * PW * 32 * SPL);
    uint32_t *t_x = t_dst + (size_t)turns * PW * 32 * SPL;
    /* what a slot needs of the matrix, as it lies in memory; its rotation, its
       destination entry with flags: bit 31 sigma = -1, bit 30 a negative element */
    struct Slot {
        uint32_t w, dst;
        RotVal rot;
    };
    auto slot_load = [&](uint32_t at, Slot &x) {
        x.w = __ldg(d.img + at);
        x.dst = __ldg(d.pos_dst + at);
        if (!rot_in_place) x.rot = __ldg(static_cast<const RotVal *>(d.slot_rot) + at);
    };
    auto slot_use = [&](const Slot &x, RotVal &t, uint32_t &dst) {
        const uint32_t val = x.w & 0xffffu;
        /* a 0 element rotates by R(0) */
        t = val == 0 ? Amp<AmpT>::rot_zero() : (rot_in_place ? Amp<AmpT>::rot_code(val) : x.rot);
        dst = x.dst | ((val & 0x8000u) << 15);
    };
    /* a group's state, loaded one group ahead, and without the tables the words of
       the matrix too: a single step meets them in DRAM (29.0 -> 25.3 us a flushed step at N = 16384
       complex64, 28.5 -> 24.6 complex128; not where they
       would spill: two complex128 slots a lane) */
    constexpr bool kSlotAhead = SPL == 1 || sizeof(AmpT) == 8;
    struct In {
        Entry<AmpT> e[SPL];
        Slot x[TAB ? 1 : SPL];
    };
    auto fetch = [&](const AmpT *A, uint32_t gg, In &x) {
        const uint32_t jj = gg * RPP + ul;
        const bool have = gg < ngroups && jj < n;
        const uint32_t i0 = jj * S + lb;
#pragma unroll
        for (int q = 0; q < SPL; ++q) {
            x.e[q].a0 = x.e[q].a1 = x.e[q].b0 = x.e[q].b1 = zero;
            if (have) PosMem<AmpT>::template load<FULLST>(A, T, i0 + 32 * q, x.e[q]);
            if (!TAB && kSlotAhead) {
                x.x[TAB ? 0 : q].w = x.x[TAB ? 0 : q].dst = 0;
                if (have) slot_load(i0 + 32 * q, x.x[TAB ? 0 : q]);
            }
        }
    };

    /* a single step issues its first loads before anything that waits for one (the
       status, the norm's target: DRAM latencies too when the L2 is cold; 25.3 -> 25.0 us a flushed
       step complex64, 24.6 -> 23.7 complex128) */
    const AmpT *A = static_cast<const AmpT *>(p.in);
    constexpr bool kFirst = !TAB && SPL == 1, kXAhead = kFirst && sizeof(AmpT) == 8;
    In first;
    Entry<AmpT> xe = {zero, zero, zero, zero};
    uint32_t xto = 0;
    if (kFirst) fetch(A, g0, first);
    if (kXAhead && x0 * 32 + lane < X) {
        PosMem<AmpT>::template load<FULLST>(A, T, n * S + x0 * 32 + lane, xe);
        xto = __ldg(d.pos_xdst + x0 * 32 + lane);
    }
    if (*(volatile int32_t *)a.status != 0) return; /* after a failed step: nothing (the whole grid alike) */
    if (TAB) {
        for (uint32_t k = 0; k < turns; ++k) {
            const uint32_t g = g0 + k * nwarps, jj = g * RPP + ul;
#pragma unroll
            for (int q = 0; q < SPL; ++q) {
                RotVal t = Amp<AmpT>::rot_zero();
                uint32_t dst = 0;
                if (g < ngroups && jj < n) {
                    Slot x;
                    slot_load(jj * S + lb + 32 * q, x);
                    slot_use(x, t, dst);
                }
                const uint32_t at = ((k * PW + warp) * SPL + q) * 32 + lane;
                t_rot[at] = t;
                t_dst[at] = dst;
            }
        }
        for (uint32_t k = 0; k < xturns; ++k) {
            const uint32_t x = (x0 + k * nwarps) * 32 + lane;
            t_x[(k * PW + warp) * 32 + lane] = x < X ? __ldg(d.pos_xdst + x) : 0u;
        }
        __syncwarp(); /* a warp reads only what it wrote */
    }

    PosStats st;
    uint32_t cnt = 0;
    bool rescale = a.scale_in != nullptr;
    if (threadIdx.x == 0) {
        Amp<AmpT>::Scale::to_shared(rescale ? *a.scale_in : 1.0, &scale_sm);
        if (a.renorm && p.words != nullptr) pos_norm_setup(a, pn);
        odd_sm = 0;
    }
    __syncthreads();
    for (int step = 0; step < p.nsteps; ++step) {
        AmpT *O = static_cast<AmpT *>((step & 1) ? p.out1 : p.out0);
        const bool readout = p.qls ? (step & 1) != 0 : a.qls_readout != 0;
        double unit = 0.0, pshare = 0.0;
        if (readout) /* u here is scaled by 2 / s */
            unit = (p.qls ? a.qls_coefs[p.qls_term + (step >> 1)] : a.qls_coefs[*a.qls_j]) * (d.inv_sqrt_s * (0.5 * S));
        const typename Amp<AmpT>::Scale scale = Amp<AmpT>::Scale::from_shared(&scale_sm);
        typename Amp<AmpT>::Norm nrm;
        In nxt;
        if (!kFirst || step > 0) fetch(A, g0, nxt);
        else nxt = first;
        for (uint32_t k = 0, g = g0; g < ngroups; ++k, g += nwarps) {
            const In cur = nxt;
            fetch(A, g + nwarps, nxt);
            const uint32_t j = g * RPP + ul;
            const bool valid = j < n;
            RotVal rv[SPL];
            uint32_t dst[SPL];
#pragma unroll
            for (int q = 0; q < SPL; ++q) {
                if (TAB) {
                    const uint32_t at = ((k * PW + warp) * SPL + q) * 32 + lane;
                    rv[q] = t_rot[at];
                    dst[q] = t_dst[at];
                } else {
                    Slot x = cur.x[TAB ? 0 : q];
                    if (!kSlotAhead) {
                        x.w = x.dst = 0;
                        if (valid) slot_load(j * S + lb + 32 * q, x);
                    }
                    slot_use(x, rv[q], dst[q]);
                }
            }
            pos_group<AmpT, S, FULLST>(
                d, rv, dst, cur.e, rescale, scale, valid, a.renorm != 0, nrm, cnt, st,
                [&](const typename Amp<AmpT>::Sum &sum) {
                    if (readout && valid && lb == 0) { /* flag-0 amplitude (1/sqrt s) sum u: the QLS accumulator */
                        const double2 sv = sum.value();
                        pshare += pos_readout(a.qls_y + j, unit, sv.x, sv.y);
                    }
                },
                [&](int q, const Entry<AmpT> &o) { PosMem<AmpT>::template store<FULLST>(O, T, dst[q] & 0x3fffffffu, o); });
            if ((k & 7u) == 7u) st.take(cnt);
        }
        st.take(cnt);
        /* the extras, 32 at a time */
        for (uint32_t k = 0, x = x0 * 32 + lane; k < xturns; ++k, x += nwarps * 32) {
            if (x >= X) break;
            const uint32_t i = n * S + x;
            uint32_t to = xto;
            Entry<AmpT> e = xe;
            if (!kXAhead || k > 0 || step > 0) {
                to = TAB ? t_x[(k * PW + warp) * 32 + lane] : __ldg(d.pos_xdst + x);
                PosMem<AmpT>::template load<FULLST>(A, T, i, e);
            }
            AmpT a0 = e.a0, a1 = e.a1, q0 = e.b0, q1 = FULLST ? e.b1 : zero;
            if (rescale) {
                a0 = scale.apply(a0);
                a1 = scale.apply(a1);
                q0 = scale.apply(q0);
                if (FULLST) q1 = scale.apply(q1);
            }
            const bool k0 = pos_keep(d, a0), k1 = pos_keep(d, a1), h0 = pos_keep(d, q0), h1 = FULLST && pos_keep(d, q1);
            const uint32_t kept = (k0 ? 1u : 0u) + (k1 ? 1u : 0u) + (h0 ? 1u : 0u) + (h1 ? 1u : 0u);
            cnt += (nz(a0) + nz(a1) + nz(q0) + (FULLST ? nz(q1) : 0u)) * kCntIn + kept * (kCntRdag + kCntHph + kCntOut);
            if (a.renorm) {
                if (k0) norm_add(nrm, a0);
                if (k1) norm_add(nrm, a1);
                if (h0) norm_add(nrm, q0);
                if (FULLST && h1) norm_add(nrm, q1);
            }
            const Entry<AmpT> o = {k0 ? Amp<AmpT>::neg(a0) : zero, h0 ? Amp<AmpT>::neg(q0) : zero,
                                   k1 ? Amp<AmpT>::neg(a1) : zero, h1 ? Amp<AmpT>::neg(q1) : zero};
            PosMem<AmpT>::template store<FULLST>(O, T, to, o);
            if ((k & 15u) == 15u) st.take(cnt);
        }
        st.take(cnt);
        __syncwarp();
        /* the warp's shares of the norm and of ||Y||^2 */
        if (a.renorm && p.words == nullptr) {
            const double v = nrm.warp_total();
            if (lane == 0) part_n[warp] = v;
        } else if (a.renorm) {
            bool odd;
            const PosLimbs v = warp_sum_units(to_units(nrm, pn, odd));
            if (lane == 0) part_u[warp] = v;
            if (odd) odd_sm = 1;
        }
        if (p.qls && readout) {
            const double pv = warp_sum(pshare);
            if (lane == 0) part_d[warp] = pv;
        }
        __syncthreads();
        A = O;
        const bool last = step == p.nsteps - 1;
        if (p.words == nullptr) break; /* one step: finished below by the last block */
        const bool odd = a.renorm && odd_sm != 0;
        if (odd) { /* (the whole block alike) */
            const double v = nrm.warp_total();
            if (lane == 0) part_n[warp] = v;
            __syncthreads();
            if (threadIdx.x == 0) odd_sm = 0;
        }
        const unsigned at = (unsigned)(p.epoch + (unsigned long long)step) & 3u, at2 = (at + 2u) & 3u;
        double *pshares = p.pshare + ((unsigned)(step >> 1) & 1u) * gridDim.x;
        if (warp == 0) {
            PosLimbs share{0u, 0u, 0u};
            if (a.renorm) {
                if (lane < PW) share = part_u[lane];
                share.reduce();
            }
            double odd_share = 0.0;
            if (odd) odd_share = warp_sum(lane < PW ? part_n[lane] : 0.0);
            if (p.qls && readout) {
                const double ps = warp_sum(lane < PW ? part_d[lane] : 0.0);
                if (lane == 0) __stcg(pshares + blockIdx.x, ps);
            }
            if (lane == 0) {
                unsigned long long *const word = p.words + 2 * at, *const clear = p.words + 2 * at2;
                if (odd) atomicAdd(p.extra + at, odd_share);
                if (a.renorm) word_add_relaxed(word + 1, ((odd ? kOddShare : share.coarse()) << kCountBits) + 1ull);
                word_add(word, ((odd ? 0ull : share.fine()) << kCountBits) + 1ull);
                bool ok = true;
                if (!last || blockIdx.x == 0) {
                    ulonglong2 w = {0ull, 0ull};
                    ok = false;
                    for (int polls = 0; polls < (1 << 22) && !ok; ++polls) {
                        if (a.renorm) w = words_load(word);
                        else w.x = w.y = word_load(word);
                        ok = (w.x & kCountMask) == gridDim.x && (w.y & kCountMask) == gridDim.x;
                    }
                    if (!ok) atomicOr(a.status, QW_ST_GRID_WAIT);
                    if (ok && blockIdx.x == 0) {
                        clear[0] = clear[1] = 0ull;
                        if (a.renorm) p.extra[at2] = 0.0;
                    }
                    double fac = 1.0, norm = 0.0;
                    if (a.renorm) {
                        const unsigned long long fine = w.x >> kCountBits, coarse = w.y >> kCountBits;
                        typename Amp<AmpT>::Scale f(1.0);
                        if (!last && pos_near(pn.target, coarse) && pos_scale(pn, pos_deviation<kGridField>(pn.target, fine), f)) {
                            f.store(&scale_sm);
                        } else {
                            norm = pos_norm<kGridField>(pn, fine, coarse, coarse >= kOddShare ? __ldcg(p.extra + at) : 0.0);
                            fac = pos_scale_exact(*a.renorm_target, norm);
                            Amp<AmpT>::Scale::to_shared(fac, &scale_sm);
                        }
                    }
                    if (last && ok) {
                        *a.norm_out = norm;
                        if (a.scale_out) *a.scale_out = fac;
                        if (a.steps_done) *a.steps_done += p.nsteps;
                        if (a.stats) a.stats[QW_STAT_STEPS] += p.nsteps;
                    }
                }
                flag_sm = ok ? 1 : 0;
            }
        }
        __syncthreads();
        if (flag_sm == 0) break;
        rescale = a.renorm != 0;
        /* p_j = ||Y||^2 of the term: the shares of all blocks, by one warp of a
           block that changes from term to term, while the others go on */
        if (p.qls && readout && warp == PW - 1) {
            const unsigned who = last ? 0u : (unsigned)(step >> 1) % gridDim.x;
            if (blockIdx.x == who) {
                double v = 0.0;
                for (unsigned b = lane; b < gridDim.x; b += 32) v += __ldcg(pshares + b);
                v = warp_sum(v);
                if (lane == 0) a.qls_p[p.qls_term + (step >> 1)] = v;
            }
        }
    }
    st.flush(a);
    if (p.words != nullptr) return;

    /* one step: the block's share of the norm, the last block reduces (FP64) */
    if (warp == 0) {
        double share = 0.0;
        if (a.renorm) share = warp_sum(lane < PW ? part_n[lane] : 0.0);
        if (lane == 0) {
            a.partials[blockIdx.x] = share;
            __threadfence();
            const unsigned prev = atomicAdd(a.done_ctr, 1u);
            flag_sm = prev == gridDim.x - 1;
        }
        __syncwarp();
        if (!flag_sm) return;
        __threadfence();
        double norm = 0.0;
        if (a.renorm) {
            for (unsigned bb = lane; bb < gridDim.x; bb += 32) norm += __ldcg(a.partials + bb);
            norm = warp_sum(norm);
        }
        if (lane == 0) {
            if (*(volatile int32_t *)a.status == 0) {
                *a.norm_out = norm;
                if (a.scale_out) *a.scale_out = a.renorm ? pos_scale_exact(*a.renorm_target, norm) : 1.0;
                if (a.steps_done) *a.steps_done += 1;
                if (a.stats) a.stats[QW_STAT_STEPS] += 1;
            }
            *a.done_ctr = 0u;
        }
    }
}

/* ==== small states: several steps on one cluster, the state in shared memory ==== */
/*
 * A step of a small state is a chain of latencies, and over the grid most of it is
 * L2: the state's load and store, the norm's atomic, the barrier word's polls --
 * 3.5 us at N = 1000, whatever the arithmetic.  Up to a few hundred groups the
 * blocks of one cluster hold the state instead, each its own warps' entries in
 * shared memory (two buffers); S writes to the destination block's shared
 * memory, each warp adds its share of the norm to all blocks' sums there, and the
 * cluster's hardware barrier ends the step.  The QLS accumulator Y stays in
 * shared memory too.  200 steps with T~ and two marginals, grid -> cluster: N = 256, s = 8
 * complex128 776 -> 479 us, complex64 702 -> 492; N = 700 768 -> 634, 694 -> 539.  What
 * is left is still latency: the arithmetic's chain and the barrier, 2.1 us a step at
 * 64 groups, whatever the number of blocks they are on.
 *
 * Entry (k, warp, q, lane) of a block -- the order in which its lanes use them --
 * is number ((k warps + warp) SPL + q) 32 + lane of its buffers, extras behind the
 * slots; a destination is its block (bits 20 .. 23) and that
 * index (bits 0 .. 19), with the flags of k_walk_pos above.  A buffer written in step
 * t was last read in step t - 1, before the barrier that every block passed to
 * start t; the norm's sums (qw_pos_norm.h, both words as wide as they are) take
 * turns three by three, cleared two steps ahead.
 */
constexpr int kPosCluster = 16; /* blocks of a cluster, at most (more than 8: opt-in) */

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t peer_addr(uint32_t a, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void peer_store(uint32_t a, float2 v)
{
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t a, double2 v)
{
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void peer_store_pair(uint32_t a, float2 u, float2 v)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(u.x), "f"(u.y), "f"(v.x), "f"(v.y)
                 : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t a, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void peer_add(uint32_t a, unsigned long long v)
{
    asm volatile("red.relaxed.cluster.shared::cluster.add.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void peer_add(uint32_t a, double v)
{
    asm volatile("red.relaxed.cluster.shared::cluster.add.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
/* One buffer of E entries in shared memory.  complex64: (A0, A1) one 16-byte
   access, B0 behind; complex128: three planes (16-byte accesses either way). */
template <typename AmpT> struct ClusterBuf;
template <> struct ClusterBuf<float2> {
    static constexpr int kBytes = 24;
    __device__ static void load(const unsigned char *b, uint32_t E, uint32_t at, Entry<float2> &e)
    {
        const float4 v = reinterpret_cast<const float4 *>(b)[at];
        e.a0 = make_float2(v.x, v.y);
        e.a1 = make_float2(v.z, v.w);
        e.b0 = reinterpret_cast<const float2 *>(b + 16 * (size_t)E)[at];
        e.b1 = make_float2(0.0f, 0.0f);
    }
    __device__ static void store(unsigned char *b, uint32_t E, uint32_t at, const Entry<float2> &e)
    {
        reinterpret_cast<float4 *>(b)[at] = make_float4(e.a0.x, e.a0.y, e.a1.x, e.a1.y);
        reinterpret_cast<float2 *>(b + 16 * (size_t)E)[at] = e.b0;
    }
    __device__ static void send(uint32_t b, uint32_t E, uint32_t at, const Entry<float2> &e)
    {
        peer_store_pair(b + 16u * at, e.a0, e.a1);
        peer_store(b + 16u * E + 8u * at, e.b0);
    }
};
template <> struct ClusterBuf<double2> {
    static constexpr int kBytes = 48;
    __device__ static void load(const unsigned char *b, uint32_t E, uint32_t at, Entry<double2> &e)
    {
        const double2 *p = reinterpret_cast<const double2 *>(b);
        e.a0 = p[at];
        e.a1 = p[E + at];
        e.b0 = p[2 * (size_t)E + at];
        e.b1 = make_double2(0.0, 0.0);
    }
    __device__ static void store(unsigned char *b, uint32_t E, uint32_t at, const Entry<double2> &e)
    {
        double2 *p = reinterpret_cast<double2 *>(b);
        p[at] = e.a0;
        p[E + at] = e.a1;
        p[2 * (size_t)E + at] = e.b0;
    }
    __device__ static void send(uint32_t b, uint32_t E, uint32_t at, const Entry<double2> &e)
    {
        peer_store(b + 16u * at, e.a0);
        peer_store(b + 16u * (E + at), e.a1);
        peer_store(b + 16u * (2u * E + at), e.b0);
    }
};
/* FP64 out of line, as pos_readout; Y in shared memory */
__device__ __noinline__ double pos_readout_sm(double2 *y, double unit, double sx, double sy)
{
    double2 acc = *y;
    acc.x += unit * sx;
    acc.y += unit * sy;
    *y = acc;
    return fma(acc.x, acc.x, acc.y * acc.y);
}

template <typename AmpT, int S>
__global__ void __launch_bounds__(kPosMaxWarps * 32, 1) k_walk_cluster(QwSimDev d, QwPosArgs p, QwStepArgs a)
{
    typedef typename Amp<AmpT>::RotVal RotVal;
    constexpr int SW = S > 32 ? 32 : S, SPL = S / SW, RPP = 32 / SW;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long nsum[2][3]; /* fine, coarse */
    __shared__ double nodd[3];                /* the odd shares */
    __shared__ double pshares[2][kPosCluster * kPosMaxWarps];
    __shared__ PosNorm pn;
    if (*(volatile int32_t *)a.status != 0) return; /* after a failed step: nothing (every block alike) */
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, PW = blockDim.x >> 5;
    const bool rot_in_place = Amp<AmpT>::kRotCode && d.rot_calc;
    const AmpT zero = Amp<AmpT>::zero();
    const uint32_t n = (uint32_t)d.pos_rows, T = (uint32_t)d.pos_T, X = T - n * S;
    const uint32_t ngroups = (n + RPP - 1) / RPP, xgroups = (X + 31) / 32;
    const uint32_t CL = gridDim.x, rank = blockIdx.x, nwarps = CL * PW; /* the grid is one cluster */
    const uint32_t g0 = rank * PW + warp, x0 = nwarps - 1 - g0; /* extras from the last warp down */
    const int ul = lane / SW, lb = lane % SW;
    const uint32_t turns = (ngroups + nwarps - 1) / nwarps, xturns = (xgroups + nwarps - 1) / nwarps;
    const uint32_t slots = turns * PW * 32 * SPL, E = slots + xturns * PW * 32;

    typedef ClusterBuf<AmpT> Buf;
    const uint32_t buf_bytes = E * (uint32_t)Buf::kBytes; /* (a multiple of 16: E is one of 32) */
    RotVal *t_rot = reinterpret_cast<RotVal *>(smem + 2 * (size_t)buf_bytes);
    double2 *y_sm = reinterpret_cast<double2 *>(t_rot + slots);
    uint32_t *t_dst = reinterpret_cast<uint32_t *>(y_sm + (p.qls ? turns * PW * RPP : 0u));
    uint32_t *t_x = t_dst + slots;
    /* where entry e of the state lies */
    auto place = [&](uint32_t e) {
        uint32_t g, in;
        if (e < n * S) {
            const uint32_t j = e / S, l = e % S, gr = j / RPP, k = gr / nwarps;
            g = gr % nwarps;
            in = ((k * PW + g % PW) * SPL + l / SW) * 32 + (j % RPP) * SW + l % SW;
        } else {
            const uint32_t x = e - n * S, xg = x / 32, k = xg / nwarps;
            g = nwarps - 1 - xg % nwarps;
            in = slots + (k * PW + g % PW) * 32 + x % 32;
        }
        return (g / PW) << 20 | in;
    };
    auto load = [&](uint32_t at, uint32_t e, bool have) {
        Entry<AmpT> v = {zero, zero, zero, zero};
        if (have) PosMem<AmpT>::template load<false>(static_cast<const AmpT *>(p.in), T, e, v);
        Buf::store(smem, E, at, v);
    };
    for (uint32_t k = 0; k < turns; ++k) {
        const uint32_t jj = (g0 + k * nwarps) * RPP + ul;
        const bool have = jj < n;
#pragma unroll
        for (int q = 0; q < SPL; ++q) {
            const uint32_t at = ((k * PW + warp) * SPL + q) * 32 + lane, e = jj * S + lb + 32 * q;
            RotVal t = Amp<AmpT>::rot_zero();
            uint32_t dst = 0;
            if (have) {
                const uint32_t val = __ldg(d.img + e) & 0xffffu, to = __ldg(d.pos_dst + e);
                if (val != 0)
                    t = rot_in_place ? Amp<AmpT>::rot_code(val) : __ldg(static_cast<const RotVal *>(d.slot_rot) + e);
                dst = place(to & 0x3fffffffu) | (to & 0x80000000u) | ((val & 0x8000u) << 15);
            }
            t_rot[at] = t;
            t_dst[at] = dst;
            load(at, e, have);
        }
        if (p.qls && lb == 0) y_sm[(k * PW + warp) * RPP + ul] = have ? __ldcg(a.qls_y + jj) : make_double2(0.0, 0.0);
    }
    for (uint32_t k = 0; k < xturns; ++k) {
        const uint32_t x = (x0 + k * nwarps) * 32 + lane, at = (k * PW + warp) * 32 + lane;
        t_x[at] = x < X ? place(__ldg(d.pos_xdst + x)) : 0u;
        load(slots + at, n * S + x, x < X);
    }
    if (threadIdx.x == 0) {
        for (int t = 0; t < 3; ++t) {
            nsum[0][t] = nsum[1][t] = 0ull;
            nodd[t] = 0.0;
        }
        if (a.renorm) pos_norm_setup(a, pn);
    }
    const uint32_t buf_addr = smem_addr(smem);
    const uint32_t peer = lane < CL ? lane : 0u; /* the block this lane adds the warp's norm to */
    const uint32_t sum_peer = peer_addr(smem_addr(nsum), peer), odd_peer = peer_addr(smem_addr(nodd), peer);
    auto send = [&](uint32_t out, uint32_t to, const Entry<AmpT> &o) { /* out: the buffer's own address */
        Buf::send(peer_addr(out, (to >> 20) & 15u), E, to & 0xfffffu, o);
    };

    PosStats st;
    uint32_t cnt = 0;
    bool rescale = a.scale_in != nullptr;
    typename Amp<AmpT>::Scale scale(rescale ? *a.scale_in : 1.0);
    double coef = p.qls ? __ldg(a.qls_coefs + p.qls_term) : 0.0, coef_next = 0.0;
    const double unit_of = d.inv_sqrt_s * (0.5 * S); /* u is scaled by 2 / s */
    cluster_sync(); /* every block's state, tables and sums are there */
    for (int step = 0; step < p.nsteps; ++step) {
        const unsigned char *A = smem + (size_t)(step & 1) * buf_bytes;
        const uint32_t out = buf_addr + ((step & 1) ^ 1) * buf_bytes;
        const bool readout = p.qls && (step & 1) != 0, last = step == p.nsteps - 1;
        const int64_t term = p.qls_term + (step >> 1);
        double unit = 0.0, pshare = 0.0;
        if (readout) {
            unit = coef * unit_of;
            if (!last) coef_next = __ldg(a.qls_coefs + term + 1);
        }
        typename Amp<AmpT>::Norm nrm;
        for (uint32_t k = 0, g = g0; g < ngroups; ++k, g += nwarps) {
            const bool valid = g * RPP + ul < n;
            RotVal rv[SPL];
            uint32_t dst[SPL];
            Entry<AmpT> in[SPL];
#pragma unroll
            for (int q = 0; q < SPL; ++q) {
                const uint32_t at = ((k * PW + warp) * SPL + q) * 32 + lane;
                rv[q] = t_rot[at];
                dst[q] = t_dst[at];
                Buf::load(A, E, at, in[q]);
            }
            pos_group<AmpT, S, false>(
                d, rv, dst, in, rescale, scale, valid, a.renorm != 0, nrm, cnt, st,
                [&](const typename Amp<AmpT>::Sum &sum) {
                    if (readout && valid && lb == 0) {
                        const double2 sv = sum.value();
                        pshare += pos_readout_sm(y_sm + (k * PW + warp) * RPP + ul, unit, sv.x, sv.y);
                    }
                },
                [&](int q, const Entry<AmpT> &o) { send(out, dst[q], o); });
            if ((k & 7u) == 7u) st.take(cnt);
        }
        st.take(cnt);
        for (uint32_t k = 0, x = x0 * 32 + lane; k < xturns; ++k, x += nwarps * 32) {
            if (x >= X) break;
            const uint32_t at = (k * PW + warp) * 32 + lane;
            Entry<AmpT> e;
            Buf::load(A, E, slots + at, e);
            AmpT a0 = e.a0, a1 = e.a1, q0 = e.b0;
            if (rescale) {
                a0 = scale.apply(a0);
                a1 = scale.apply(a1);
                q0 = scale.apply(q0);
            }
            const bool k0 = pos_keep(d, a0), k1 = pos_keep(d, a1), h0 = pos_keep(d, q0);
            const uint32_t kept = (k0 ? 1u : 0u) + (k1 ? 1u : 0u) + (h0 ? 1u : 0u);
            cnt += (nz(a0) + nz(a1) + nz(q0)) * kCntIn + kept * (kCntRdag + kCntHph + kCntOut);
            if (a.renorm) {
                if (k0) norm_add(nrm, a0);
                if (k1) norm_add(nrm, a1);
                if (h0) norm_add(nrm, q0);
            }
            const Entry<AmpT> o = {k0 ? Amp<AmpT>::neg(a0) : zero, h0 ? Amp<AmpT>::neg(q0) : zero,
                                   k1 ? Amp<AmpT>::neg(a1) : zero, zero};
            send(out, t_x[at], o);
            if ((k & 15u) == 15u) st.take(cnt);
        }
        st.take(cnt);
        __syncwarp();
        /* the warp's shares of the norm, to every block, and of ||Y||^2, to the
           term's */
        const uint32_t turn = (uint32_t)step % 3u;
        const uint32_t who = last ? 0u : (uint32_t)(step >> 1) % CL;
        if (a.renorm) {
            bool odd;
            const PosLimbs v = warp_sum_units(to_units(nrm, pn, odd));
            odd = __any_sync(FULL, odd);
            double total = 0.0;
            if (odd) total = __shfl_sync(FULL, nrm.warp_total(), 0);
            if (lane < CL) {
                peer_add(sum_peer + 8u * turn, odd ? 0ull : v.fine());
                peer_add(sum_peer + 24u + 8u * turn, odd ? kOddShare : v.coarse());
                if (odd) peer_add(odd_peer + 8u * turn, total);
            }
        }
        double *const ps = pshares[(step >> 1) & 1];
        if (readout) {
            const double pv = warp_sum(pshare);
            if (lane == 0) peer_store(peer_addr(smem_addr(ps + rank * PW + warp), who), pv);
        }
        cluster_sync();
        if (a.renorm) {
            if (threadIdx.x == 0) {
                const uint32_t next = (turn + 2u) % 3u;
                nsum[0][next] = nsum[1][next] = 0ull;
                nodd[next] = 0.0;
            }
            const unsigned long long fine = nsum[0][turn], coarse = nsum[1][turn];
            if (!pos_near(pn.target, coarse) || !pos_scale(pn, pos_deviation<kClusterField>(pn.target, fine), scale))
                scale = typename Amp<AmpT>::Scale(
                    pos_scale_exact(*a.renorm_target, pos_norm<kClusterField>(pn, fine, coarse, nodd[turn])));
        }
        rescale = a.renorm != 0;
        if (readout) coef = coef_next;
        /* p_j = ||Y||^2 of the term, by one warp of a block that changes from term to
           term, while the others go on */
        if (readout && warp == PW - 1 && rank == who) {
            double v = 0.0;
            for (uint32_t b = lane; b < nwarps; b += 32) v += ps[b];
            v = warp_sum(v);
            if (lane == 0) a.qls_p[term] = v;
        }
    }
    st.flush(a);

    /* the last barrier is passed: the other blocks' shared memory is left alone */
    AmpT *O = static_cast<AmpT *>((p.nsteps & 1) ? p.out0 : p.out1);
    const unsigned char *A = smem + (size_t)(p.nsteps & 1) * buf_bytes;
    auto store = [&](uint32_t at, uint32_t e) {
        Entry<AmpT> v;
        Buf::load(A, E, at, v);
        PosMem<AmpT>::template store<false>(O, T, e, v);
    };
    for (uint32_t k = 0; k < turns; ++k) {
        const uint32_t jj = (g0 + k * nwarps) * RPP + ul;
        if (jj >= n) continue;
#pragma unroll
        for (int q = 0; q < SPL; ++q) store(((k * PW + warp) * SPL + q) * 32 + lane, jj * S + lb + 32 * q);
        if (p.qls && lb == 0) __stcg(a.qls_y + jj, y_sm[(k * PW + warp) * RPP + ul]);
    }
    for (uint32_t k = 0; k < xturns; ++k) {
        const uint32_t x = (x0 + k * nwarps) * 32 + lane;
        if (x < X) store(slots + (k * PW + warp) * 32 + lane, n * S + x);
    }
    if (rank == 0 && threadIdx.x == 0) {
        double fac = 1.0, norm = 0.0;
        if (a.renorm) {
            const uint32_t turn = (uint32_t)(p.nsteps - 1) % 3u;
            norm = pos_norm<kClusterField>(pn, nsum[0][turn], nsum[1][turn], nodd[turn]);
            fac = pos_scale_exact(*a.renorm_target, norm);
        }
        *a.norm_out = norm;
        if (a.scale_out) *a.scale_out = fac;
        if (a.steps_done) *a.steps_done += p.nsteps;
        if (a.stats) a.stats[QW_STAT_STEPS] += p.nsteps;
    }
}

/* T~|b~> written straight into rows g0 .. g0 + n (one instance): |b~> holds one
 * branch per row, a = b_j (divided by the pending renormalisation factor when
 * other instances share the state); T~'s Hadamard gives (l, z = 0) with
 * a / sqrt(s) for every slot l, its maps take slot l to k = col(j, l), and
 * R(A_jl) on (a / sqrt(s), 0) gives A0, A1 of the slot's entry -- the
 * arithmetic of k_tinit.  The rest, the rows' extras (x0 .. x0 + nx) included,
 * is written 0.  b lies in the simulator's pinned host memory and is read from
 * there: S lanes share a value, so its bytes cross the link once, without a
 * copy before the launch.  words: 8-byte words of the simulator's scalars to
 * set (all of them for a single instance), so that no copy is needed for those
 * either.  One thread per entry: bound by the writes. */
template <typename AmpT>
__global__ void k_tinit_pos(QwSimDev d, AmpT *pbuf, int full, uint32_t g0, uint32_t n, uint32_t x0, uint32_t nx,
                            const double *b_re, const double *b_im, const double *scale, QwScalarWords words)
{
    typedef typename Amp<AmpT>::RotVal RotVal;
    if (blockIdx.x == 0 && (int)threadIdx.x < words.n) words.dst[threadIdx.x] = words.w[threadIdx.x];
    const uint32_t S = (uint32_t)d.s, T = (uint32_t)d.pos_T, ns = n * S, total = ns + nx;
    const AmpT zero = Amp<AmpT>::zero();
    const bool rot_in_place = Amp<AmpT>::kRotCode && d.rot_calc;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        AmpT o0 = zero, o1 = zero;
        uint32_t at = (uint32_t)d.pos_rows * S + x0 + (i - ns);
        if (i < ns) {
            const uint32_t j = i / S;
            at = g0 * S + i;
            double2 v = make_double2(b_re[j], b_im ? b_im[j] : 0.0);
            if (scale) v = make_double2(v.x / *scale, v.y / *scale);
            const double2 a = Amp<AmpT>::to_d(Amp<AmpT>::from_d(v)); /* as stored by |b~> */
            const AmpT h = Amp<AmpT>::from_d(make_double2(d.inv_sqrt_s * a.x, d.inv_sqrt_s * a.y));
            if ((v.x != 0.0 || v.y != 0.0) && Amp<AmpT>::keep(d, h)) {
                const uint32_t w = __ldg(d.img + at), val = w & 0xffffu;
                const RotVal rv = val == 0 ? Amp<AmpT>::rot_zero()
                                           : (rot_in_place ? Amp<AmpT>::rot_code(val)
                                                           : __ldg(static_cast<const RotVal *>(d.slot_rot) + at));
                Amp<AmpT>::rot(rv, val, false, j > (w >> 16), h, zero, o0, o1); /* R */
                if (!Amp<AmpT>::keep(d, o0)) o0 = zero;
                if (!Amp<AmpT>::keep(d, o1)) o1 = zero;
            }
        }
        const Entry<AmpT> e = {o0, o1, zero, zero};
        if (full) PosMem<AmpT>::template store<true>(pbuf, T, at, e);
        else PosMem<AmpT>::template store<false>(pbuf, T, at, e);
    }
}

/* |a|^2 in FP64 */
template <typename AmpT> __device__ __forceinline__ double amp_norm2(AmpT a)
{
    if (nz(a) == 0u) return 0.0;
    const double2 v = Amp<AmpT>::to_d(a);
    return fma(v.x, v.x, v.y * v.y);
}

/* Marginal of one register over rows g0 .. g0 + n (the key of an entry: jc =
 * kc = 0, j = its row, b1 and b2 by member, k = the slot's column or the
 * extra's row), LPR lanes a row.  j: the row's own entries.  k: a gather
 * instead of an atomic per branch -- the branches with k = v sit at dst(v, l)
 * for every slot l of row v (the entry of k = v in row col(v, l)) and at slot
 * (x, l_x) for every extra x of row v.  Both write every bin of probs (which may
 * be host memory: a block's rows as one run of 8-byte words).  The other
 * registers: sums by (b1, b2), one atomic per block into zeroed bins.
 * stat_dst (host memory, nullable): the two words of the status head. */
template <typename AmpT>
__global__ void __launch_bounds__(256) k_measure_pos(QwSimDev d, const AmpT *pbuf, int full, int64_t g0, int64_t n,
                                                     const double *scale, int reg, double *probs, int64_t len,
                                                     const unsigned long long *stat_src, unsigned long long *stat_dst)
{
    __shared__ double acc_sm[4][8];
    __shared__ double row_sm[256];
    const uint32_t S = (uint32_t)d.s, T = (uint32_t)d.pos_T, N = (uint32_t)d.pos_rows;
    const int lpr = S >= 32 ? 32 : (int)S, rpb = 256 / lpr; /* lanes a row, rows a block */
    const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5, rl = threadIdx.x / lpr, lr = threadIdx.x % lpr;
    const double sc = scale ? *scale * *scale : 1.0;
    const bool rows = reg == 1 || reg == 4;
    if (stat_dst && blockIdx.x == 0 && threadIdx.x < 2) stat_dst[threadIdx.x] = __ldcg(stat_src + threadIdx.x);
    double acc[4] = {0.0, 0.0, 0.0, 0.0}; /* by (b1, b2) */
    const int64_t end = rows && len > n ? len : n;
    for (int64_t j0 = (int64_t)blockIdx.x * rpb; j0 < end; j0 += (int64_t)gridDim.x * rpb) {
        const int64_t j = j0 + rl;
        double row = 0.0;
        if (j < n) {
            const uint32_t g = (uint32_t)(g0 + j), x0 = __ldg(d.pos_xptr + g), P = S + __ldg(d.pos_xptr + g + 1) - x0;
            for (uint32_t i = lr; i < P; i += lpr) {
                uint32_t at = i < S ? g * S + i : N * S + x0 + (i - S);
                if (reg == 4) at = i < S ? (__ldg(d.pos_dst + at) & 0x3fffffffu) : __ldg(d.pos_xdst + x0 + (i - S));
                Entry<AmpT> e;
                if (full) PosMem<AmpT>::template load<true>(pbuf, T, at, e);
                else PosMem<AmpT>::template load<false>(pbuf, T, at, e);
                const double p[4] = {amp_norm2(e.a0), amp_norm2(e.a1), amp_norm2(e.b0), full ? amp_norm2(e.b1) : 0.0};
                if (rows) {
                    row += (p[0] + p[1]) + (p[2] + p[3]);
                } else {
#pragma unroll
                    for (int t = 0; t < 4; ++t) acc[t] += p[t];
                }
            }
        }
        if (rows) {
            for (int o = lpr >> 1; o > 0; o >>= 1) row += __shfl_xor_sync(FULL, row, o);
            if (lr == 0) row_sm[rl] = sc * row;
            __syncthreads();
            const int64_t v = j0 + threadIdx.x;
            if ((int)threadIdx.x < rpb && v < len) probs[v] = row_sm[threadIdx.x];
            __syncthreads();
        }
    }
    if (reg == 1 || reg == 4) return;
    for (int t = 0; t < 4; ++t) {
        acc[t] = warp_sum(acc[t]);
        if (lane == 0) acc_sm[t][wb] = acc[t];
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        double v = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += acc_sm[threadIdx.x][w];
        const int b1 = threadIdx.x >> 1, b2 = threadIdx.x & 1;
        const int64_t bin = reg == 2 ? b1 : reg == 5 ? b2 : 0; /* jc = kc = 0 */
        if (bin < len && v != 0.0) atomicAdd(probs + bin, sc * v);
    }
}

/* the row buckets into the positional layout (pbuf zeroed by the caller):
   one thread per bucket slot; a branch with b1 = b2 = 1 sets QW_ST_POS_FULL */
template <typename AmpT>
__global__ void k_pos_pack(QwSimDev d, QwBufDev buf, AmpT *pbuf, int32_t *status)
{
    const int S = d.s;
    const int64_t total = d.total_buckets * (int64_t)d.cap_row;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = i / d.cap_row;
        const int p = (int)(i - b * d.cap_row);
        if (p >= buf.count[b]) continue;
        if (b >= d.dense_buckets) { /* a row with jc != 0 */
            atomicOr(status, QW_ST_POS_UNREP);
            continue;
        }
        int64_t j = b >> 1, n = d.n_single, g0 = 0;
        if (d.ninst > 1) {
            const int inst = d.unit_inst[b >> 1];
            j = (b - d.inst_bkt[inst]) >> 1;
            n = d.inst_n[inst];
            g0 = d.inst_img[inst] / S;
        }
        if (j >= n) { /* a row j >= N */
            atomicOr(status, QW_ST_POS_UNREP);
            continue;
        }
        const int64_t gr = g0 + j; /* the row among all instances' rows */
        const Regs x = decode_r(buf.key[i], d.nb);
        int64_t at = -1;
        if (x.kc == 0 && x.A == 0) {
            const uint32_t *row = d.img + gr * S;
            int lo = 0, hi = S; /* lower bound of k among the row's sorted columns */
            while (lo < hi) {
                const int m = (lo + hi) >> 1;
                if ((row[m] >> 16) < x.k) lo = m + 1;
                else hi = m;
            }
            if (lo < S && (row[lo] >> 16) == x.k) {
                at = gr * S + lo;
            } else {
                for (uint32_t e = d.pos_xptr[gr]; e < d.pos_xptr[gr + 1]; ++e)
                    if (d.pos_xdst[e] / (uint32_t)S - g0 == x.k) {
                        at = d.pos_rows * S + e;
                        break;
                    }
            }
        }
        if (at < 0) {
            atomicOr(status, QW_ST_POS_UNREP);
            continue;
        }
        const AmpT v = static_cast<const AmpT *>(buf.amp)[i];
        pbuf[PosMem<AmpT>::at((size_t)d.pos_T, (size_t)at, (int)(b & 1), (int)x.b2)] = v;
        if ((b & 1) != 0 && x.b2 != 0 && nz(v)) atomicOr(status, QW_ST_POS_FULL);
    }
}

/* the positional layout into the row buckets (cleared by the caller): one
   thread per amplitude, non-zero ones appended to their row */
template <typename AmpT>
__global__ void k_pos_unpack(QwSimDev d, const AmpT *pbuf, int full, QwBufDev buf, int32_t *status)
{
    const int64_t S = d.s, T = d.pos_T, total = 4 * T;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t at = i >> 2;
        const int b1 = (int)(i >> 1) & 1, b2 = (int)i & 1;
        if (b1 && b2 && !full) continue;
        const AmpT v = pbuf[PosMem<AmpT>::at((size_t)T, (size_t)at, b1, b2)];
        if (v.x == 0 && v.y == 0) continue;
        int64_t gr = at / S; /* the row among all instances' rows */
        uint32_t k;          /* the branch's k, a row among all instances' for an extra */
        if (gr < d.pos_rows) {
            k = d.img[at] >> 16;
        } else { /* the extra's row: the last one whose extras start at or before it */
            const uint32_t e = (uint32_t)(at - d.pos_rows * S);
            int64_t lo = 0, hi = d.pos_rows - 1;
            while (lo < hi) {
                const int64_t m = (lo + hi + 1) >> 1;
                if (d.pos_xptr[m] <= e) lo = m;
                else hi = m - 1;
            }
            gr = lo;
            k = d.pos_xdst[e] / (uint32_t)S;
        }
        int64_t g0 = 0, b = 2 * gr + b1; /* the instance's first row; the bucket */
        if (d.ninst > 1) {
            const int inst = d.pos_rowinst[gr];
            g0 = d.inst_img[inst] / S;
            b = d.inst_bkt[inst] + 2 * (gr - g0) + b1;
        }
        Regs x;
        x.kc = 0;
        x.A = 0;
        x.b2 = (uint32_t)b2;
        x.k = at < d.pos_rows * S ? k : k - (uint32_t)g0;
        const int p = atomicAdd(buf.count + b, 1);
        if (p >= d.cap_row) {
            atomicOr(status, QW_ST_ROW_OVERFLOW);
            continue;
        }
        const int64_t sl = b * d.cap_row + p;
        buf.key[sl] = encode_r(x, d.nb);
        static_cast<AmpT *>(buf.amp)[sl] = v;
    }
}

/* ---- launch shapes ------------------------------------------------------------- */

template <typename AmpT, bool FULLST, bool TAB>
void *pos_kernel(int s)
{
    if (s == 4) return (void *)k_walk_pos<AmpT, 4, FULLST, TAB>;
    if (s == 8) return (void *)k_walk_pos<AmpT, 8, FULLST, TAB>;
    if (s == 16) return (void *)k_walk_pos<AmpT, 16, FULLST, TAB>;
    if (s == 32) return (void *)k_walk_pos<AmpT, 32, FULLST, TAB>;
    return (void *)k_walk_pos<AmpT, 64, FULLST, TAB>;
}

/* Slots up to which a run goes to one cluster, either precision: 16 SMs then issue the
   arithmetic of more than 12 warps each, and the grid's 152 make up for its
   barrier -- 200 steps of 175 groups of 32 slots (N = 700, s = 8) 694 us on the
   grid, 539 on the cluster (complex64), 768 and 634 (complex128); 100 steps of 256
   groups (N = 1024) 378 and 386, 250 (N = 1000) 430 and 437. */
constexpr int64_t kClusterSlots = 6144;
constexpr int kClusterStatic = 8192; /* more than the kernel's static shared memory and what the system takes */

inline void cluster_config(const QwPosPlan &pl, cudaLaunchConfig_t &c, cudaLaunchAttribute &at, cudaStream_t st)
{
    c = cudaLaunchConfig_t{};
    at = cudaLaunchAttribute{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)pl.cl;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    c.gridDim = dim3((unsigned)pl.cl);
    c.blockDim = dim3((unsigned)pl.cl_warps * 32);
    c.dynamicSmemBytes = pl.cl_smem;
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = 1;
}

template <typename AmpT>
void *cluster_kernel(int s)
{
    if (s == 4) return (void *)k_walk_cluster<AmpT, 4>;
    if (s == 8) return (void *)k_walk_cluster<AmpT, 8>;
    if (s == 16) return (void *)k_walk_cluster<AmpT, 16>;
    if (s == 32) return (void *)k_walk_cluster<AmpT, 32>;
    return (void *)k_walk_cluster<AmpT, 64>;
}

/* The launch of a run on one cluster, or cl = 0 where the grid is faster or the
 * state does not fit.  Without the opt-in size of 16 blocks: 8. */
template <typename AmpT>
void cluster_plan(const QwSimDev &d, int64_t groups, int64_t xgroups, int spl, int rpp, int optin, QwPosPlan &pl)
{
    constexpr bool c128 = sizeof(AmpT) == 16;
    const int64_t few = c128 ? 4 : 8; /* groups a block: fewer blocks, not slower (measured) */
    pl.cl = 0;
    if (groups * 32 * spl > kClusterSlots) return;
    int cl = 1;
    while (cl < kPosCluster && groups * spl > cl * few) cl *= 2;
    for (; cl >= 1; cl /= 2) {
        const int64_t per = (groups + cl - 1) / cl, t0 = (per + kPosMaxWarps - 1) / kPosMaxWarps;
        int64_t pw = (per + t0 - 1) / t0;
        if (pw < 4) pw = 4;
        const int64_t turns = (groups + cl * pw - 1) / (cl * pw), xturns = (xgroups + cl * pw - 1) / (cl * pw);
        const int64_t slots = turns * pw * 32 * spl, E = slots + xturns * pw * 32;
        const int64_t smem = 2 * E * (int64_t)ClusterBuf<AmpT>::kBytes + slots * (int64_t)(sizeof(typename Amp<AmpT>::RotVal) + 4) +
                             turns * pw * rpp * 16 + xturns * pw * 32 * 4;
        if (E >= 1 << 20 || smem + kClusterStatic > optin) return; /* (fewer blocks would need more) */
        void *k = cluster_kernel<AmpT>(d.s);
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - kClusterStatic) != cudaSuccess ||
            (cl > 8 && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
            cudaGetLastError();
            continue;
        }
        pl.cl = cl;
        pl.cl_warps = (int)pw;
        pl.cl_smem = (size_t)smem;
        cudaLaunchConfig_t c;
        cudaLaunchAttribute at;
        cluster_config(pl, c, at, nullptr);
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, k, &c) == cudaSuccess && fit >= 1) return;
        cudaGetLastError();
        pl.cl = 0;
    }
}

/* One block per SM: every group of rows has a warp within a few turns, with
 * as many groups for each warp as for the others (54 groups an SM at N =
 * 16384, s = 16: 4 turns of 14 warps instead of 16, 16, 16, 6); the tables
 * fit shared memory up to about 300 groups a block (46 000 in all).  At least
 * 4 warps a block, one per scheduler. */
template <typename AmpT>
QwPosPlan pos_plan(const QwSimDev &d)
{
    QwPosPlan pl{};
    const int s = d.s, rpp = s >= 32 ? 1 : 32 / s, spl = s > 32 ? s / 32 : 1;
    const int64_t xgroups = (d.pos_T - d.pos_rows * s + 31) / 32;
    const int64_t groups = (d.pos_rows + rpp - 1) / rpp, sms = qw_sm_count();
    const int64_t per_sm = (groups + sms - 1) / sms;
    const int64_t turns = (per_sm + kPosMaxWarps - 1) / kPosMaxWarps;
    int64_t pw = (per_sm + turns - 1) / turns;
    if (pw < 4) pw = 4;
    int64_t grid = (groups + pw * turns - 1) / (pw * turns);
    if (grid > sms) grid = sms;
    pl.warps = (int)pw;
    pl.grid = (int)(grid < 1 ? 1 : grid);
    const int64_t t = (groups + pl.grid * pw - 1) / (pl.grid * pw);
    const int64_t xt = (xgroups + pl.grid * pw - 1) / (pl.grid * pw);
    pl.smem = (size_t)(t * pw * 32) * (size_t)(spl * 20) + (size_t)(xt * pw * 32) * 4;
    int dev = 0, optin = 0, coop = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    pl.tab = pl.smem + 1024 <= (size_t)optin; /* beside the kernel's static arrays */
    if (!pl.tab) pl.smem = 0;
    pl.coop = coop != 0 && pl.grid < 256; /* the barrier word's count has 8 bits */
    cluster_plan<AmpT>(d, groups, xgroups, spl, rpp, optin, pl);
    if (pl.tab) /* the limit belongs to the process, not to this simulator: always the largest */
        cudaFuncSetAttribute(pos_kernel<AmpT, false, true>(s), cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024);
    return pl;
}

template <typename AmpT>
cudaError_t launch_pos_t(const QwSimDev &d, const QwPosPlan &pl, const QwPosArgs &p, const QwStepArgs &a, int full,
                         cudaStream_t st)
{
    if (p.words && pl.cl && !full) {
        QwSimDev dc = d;
        QwPosArgs pc = p;
        QwStepArgs ac = a;
        void *cargs[] = {&dc, &pc, &ac};
        cudaLaunchConfig_t c;
        cudaLaunchAttribute at;
        cluster_config(pl, c, at, st);
        return cudaLaunchKernelExC(&c, cluster_kernel<AmpT>(d.s), cargs);
    }
    /* one step reads each table entry once: straight from memory */
    const bool tab = pl.tab && p.nsteps > 1 && !full;
    void *k = full ? pos_kernel<AmpT, true, false>(d.s)
                   : (tab ? pos_kernel<AmpT, false, true>(d.s) : pos_kernel<AmpT, false, false>(d.s));
    QwSimDev dd = d;
    QwPosArgs pp = p;
    QwStepArgs aa = a;
    void *args[] = {&dd, &pp, &aa};
    const dim3 grid((unsigned)pl.grid), block((unsigned)pl.warps * 32);
    if (p.words) return cudaLaunchCooperativeKernel(k, grid, block, args, tab ? pl.smem : 0, st);
    return cudaLaunchKernel(k, grid, block, args, 0, st);
}

template <typename AmpT>
cudaError_t launch_tinit_pos_t(const QwSimDev &d, void *pbuf, int full, int64_t g0, int64_t n, int64_t x0, int64_t nx,
                               const double *b_re, const double *b_im, const double *scale, const QwScalarWords &words,
                               cudaStream_t st)
{
    const int64_t want = (n * d.s + nx + 255) / 256, cap = 16 * (int64_t)qw_sm_count();
    k_tinit_pos<AmpT><<<(unsigned)(want < cap ? want : cap), 256, 0, st>>>(
        d, static_cast<AmpT *>(pbuf), full, (uint32_t)g0, (uint32_t)n, (uint32_t)x0, (uint32_t)nx, b_re, b_im, scale, words);
    return cudaGetLastError();
}

template <typename AmpT>
cudaError_t launch_measure_pos_t(const QwSimDev &d, const void *pbuf, int full, int64_t g0, int64_t n,
                                 const double *scale, int reg, double *probs, int64_t len,
                                 const unsigned long long *stat_src, unsigned long long *stat_dst, cudaStream_t st)
{
    /* j, k: enough blocks that every row's loads are in flight at once; the
       other registers, with one atomic per block: fewer */
    const bool rows = reg == 1 || reg == 4;
    const int64_t rpb = 256 / (d.s >= 32 ? 32 : d.s), end = rows && len > n ? len : n;
    const int64_t want = (end + rpb - 1) / rpb, cap = (rows ? 64 : 4) * (int64_t)qw_sm_count();
    k_measure_pos<AmpT><<<(unsigned)(want < cap ? want : cap), 256, 0, st>>>(
        d, static_cast<const AmpT *>(pbuf), full, g0, n, scale, reg, probs, len, stat_src, stat_dst);
    return cudaGetLastError();
}

template <typename AmpT>
cudaError_t launch_pos_pack_t(const QwSimDev &d, const QwBufDev &buf, void *pbuf, int32_t *status, cudaStream_t st)
{
    k_pos_pack<AmpT><<<4 * qw_sm_count(), 256, 0, st>>>(d, buf, static_cast<AmpT *>(pbuf), status);
    return cudaGetLastError();
}

template <typename AmpT>
cudaError_t launch_pos_unpack_t(const QwSimDev &d, const void *pbuf, int full, const QwBufDev &buf, int32_t *status,
                                cudaStream_t st)
{
    k_pos_unpack<AmpT><<<4 * qw_sm_count(), 256, 0, st>>>(d, static_cast<const AmpT *>(pbuf), full, buf, status);
    return cudaGetLastError();
}

} // namespace

/* the launchers of one precision (declared in qw_internal.h) */
#define QW_POS_INSTANTIATE(SUFFIX, AmpT)                                                                              \
    QwPosPlan qw_pos_plan##SUFFIX(const QwSimDev &d) { return pos_plan<AmpT>(d); }                                    \
    cudaError_t qw_launch_walk_pos##SUFFIX(const QwSimDev &d, const QwPosPlan &pl, const QwPosArgs &p,                \
                                           const QwStepArgs &a, int full, cudaStream_t st)                            \
    {                                                                                                                 \
        return launch_pos_t<AmpT>(d, pl, p, a, full, st);                                                             \
    }                                                                                                                 \
    cudaError_t qw_launch_tinit_pos##SUFFIX(const QwSimDev &d, void *pbuf, int full, int64_t g0, int64_t n,           \
                                            int64_t x0, int64_t nx, const double *b_re, const double *b_im,           \
                                            const double *scale, const QwScalarWords &words, cudaStream_t st)         \
    {                                                                                                                 \
        return launch_tinit_pos_t<AmpT>(d, pbuf, full, g0, n, x0, nx, b_re, b_im, scale, words, st);                  \
    }                                                                                                                 \
    cudaError_t qw_launch_measure_pos##SUFFIX(const QwSimDev &d, const void *pbuf, int full, int64_t g0, int64_t n,   \
                                              const double *scale, int reg, double *probs, int64_t len,               \
                                              const unsigned long long *stat_src, unsigned long long *stat_dst,       \
                                              cudaStream_t st)                                                        \
    {                                                                                                                 \
        return launch_measure_pos_t<AmpT>(d, pbuf, full, g0, n, scale, reg, probs, len, stat_src, stat_dst, st);      \
    }                                                                                                                 \
    cudaError_t qw_launch_pos_pack##SUFFIX(const QwSimDev &d, const QwBufDev &buf, void *pbuf, int32_t *status,       \
                                           cudaStream_t st)                                                           \
    {                                                                                                                 \
        return launch_pos_pack_t<AmpT>(d, buf, pbuf, status, st);                                                     \
    }                                                                                                                 \
    cudaError_t qw_launch_pos_unpack##SUFFIX(const QwSimDev &d, const void *pbuf, int full, const QwBufDev &buf,      \
                                             int32_t *status, cudaStream_t st)                                        \
    {                                                                                                                 \
        return launch_pos_unpack_t<AmpT>(d, pbuf, full, buf, status, st);                                             \
    }

#endif /* QW_POS_CUH */
