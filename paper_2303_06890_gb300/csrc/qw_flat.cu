/*
 * qw_flat.cu -- the walk step as the paper's simulator runs it, on one flat
 * list of branches in global memory (Sec. V-A): every register map applied to
 * every branch, and every interference operation as
 *   (1) grouping: a stable LSD radix sort of the whole list by the registers
 *       that make the groups, so that the branches equal on every idle
 *       register are contiguous (8-bit digits over the bits that vary between
 *       keys, one single-pass kernel per digit carrying a permutation, the
 *       entries moved once);
 *   (2) computing: the small dense operator on each group's zero-filled
 *       vector (for H the groups are found first, so that s outputs are
 *       formed per group, not per list entry);
 *   (3) clearing: outputs with |a| <= tau dropped as they are written, at places
 *       from a single-pass prefix sum over the tiles of (2).
 * T~^dag, H, P, H, T~ and S run in the order of Alg. "Quantum walk operator",
 * with the element register A allocated for the whole step.  Nothing here is
 * bounded by the row buckets or the on-chip buffers of the step kernels, only
 * by device memory: this is the path of a step whose rows outgrow them, and a
 * schedule that can be selected on its own.  Amplitudes are complex FP64
 * whatever the storage precision (converted when the state is gathered and
 * rounded when it is stored back).
 *
 * Packed key of a branch (two 64-bit words, bit 0 first), the layout of
 * qw_state_export:  b2 | k (nb) | kc (nb) | b1 | j (nb) | jc (nb) | A (16) |
 * inst (16), 4 nb + 34 bits.
 */
#include <vector>

#include "qw_device.cuh"
#include "qw_sort_chunks.h"

namespace {

/* a packed register key of NW 64-bit words (2: the qw_state_export layout;
   10: the register-faithful layout, the working registers above bit 128) */
template <int NW> struct FKeyN {
    uint64_t w[NW];
};
typedef FKeyN<2> FKey;
constexpr int NW_FAITH = 10;
typedef FKeyN<NW_FAITH> FKeyW;

struct FLayout {
    int nb, pk, pkc, pb1, pj, pjc, pA, pinst;
};

__host__ __device__ inline FLayout flayout(int nb)
{
    FLayout f;
    f.nb = nb;
    f.pk = 1;
    f.pkc = 1 + nb;
    f.pb1 = 1 + 2 * nb;
    f.pj = 2 + 2 * nb;
    f.pjc = 2 + 3 * nb;
    f.pA = 2 + 4 * nb;
    f.pinst = 18 + 4 * nb;
    return f;
}

/* word i of a key by selection over its words, so that the key stays in
   registers whatever i is (an indexed access moves it to local memory) */
template <int NW>
__device__ __forceinline__ uint64_t fword(const FKeyN<NW> &k, int i)
{
    uint64_t v = k.w[0];
#pragma unroll
    for (int t = 1; t < NW; ++t) v = t == i ? k.w[t] : v;
    return v;
}

template <int NW>
__device__ __forceinline__ uint64_t fget(const FKeyN<NW> &k, int pos, int w)
{
    const int i = pos >> 6, o = pos & 63;
    uint64_t v = fword(k, i) >> o;
    if (o + w > 64 && i + 1 < NW) v |= fword(k, i + 1) << (64 - o);
    return v & (w >= 64 ? ~0ull : ((1ull << w) - 1ull));
}

/* OR v into a field (the field must be 0) */
template <int NW>
__device__ __forceinline__ void fput(FKeyN<NW> &k, int pos, int w, uint64_t v)
{
    v &= (w >= 64 ? ~0ull : ((1ull << w) - 1ull));
    const int i = pos >> 6, o = pos & 63;
#pragma unroll
    for (int t = 0; t < NW; ++t) {
        if (t == i) k.w[t] |= v << o;
        if (t == i + 1 && o + w > 64) k.w[t] |= v >> (64 - o);
    }
}

struct FRegs {
    uint32_t inst, jc, j, b1;
    Regs x; /* k, kc, A, b2 */
};

/* the base registers (4 nb + 34 bits) lie in words 0 and 1 of any key
   width: they are decoded from and encoded into those two words */
template <int NW>
__device__ __forceinline__ FKeyN<2> fbase(const FKeyN<NW> &k)
{
    FKeyN<2> b;
    b.w[0] = k.w[0];
    b.w[1] = k.w[1];
    return b;
}

/* words 0 and 1 of a key in global memory, as one 16-byte load */
template <int NW>
__device__ __forceinline__ FKeyN<2> fbase_load(const FKeyN<NW> *k)
{
    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(k);
    FKeyN<2> b;
    b.w[0] = v.x;
    b.w[1] = v.y;
    return b;
}

template <int NW>
__device__ __forceinline__ FRegs fdecode(const FKeyN<NW> &key, const FLayout &L)
{
    const FKeyN<2> k = fbase(key);
    FRegs r;
    r.x.b2 = fget(k, 0, 1);
    r.x.k = fget(k, L.pk, L.nb);
    r.x.kc = fget(k, L.pkc, L.nb);
    r.b1 = fget(k, L.pb1, 1);
    r.j = fget(k, L.pj, L.nb);
    r.jc = fget(k, L.pjc, L.nb);
    r.x.A = fget(k, L.pA, 16);
    r.inst = fget(k, L.pinst, 16);
    return r;
}

/* the base registers into k (their fields must be 0) */
template <int NW>
__device__ __forceinline__ void fencode_into(FKeyN<NW> &key, const FRegs &r, const FLayout &L)
{
    FKeyN<2> k = fbase(key);
    fput(k, 0, 1, r.x.b2);
    fput(k, L.pk, L.nb, r.x.k);
    fput(k, L.pkc, L.nb, r.x.kc);
    fput(k, L.pb1, 1, r.b1);
    fput(k, L.pj, L.nb, r.j);
    fput(k, L.pjc, L.nb, r.jc);
    fput(k, L.pA, 16, r.x.A);
    fput(k, L.pinst, 16, r.inst);
    key.w[0] = k.w[0];
    key.w[1] = k.w[1];
}

/* the base registers of a wider key rewritten, its other bits kept */
template <int NW>
__device__ __forceinline__ void frewrite(FKeyN<NW> &k, const FRegs &r, const FLayout &L)
{
    const int bits = L.pinst + 16;
    k.w[0] &= bits >= 64 ? 0ull : ~((1ull << bits) - 1ull);
    if (bits > 64) k.w[1] &= bits >= 128 ? 0ull : ~((1ull << (bits - 64)) - 1ull);
    fencode_into(k, r, L);
}

/* The row descriptor of a branch, reading its QRAM row straight from the
 * image in global memory. */
__device__ __forceinline__ Row frow(const QwSimDev &d, const FRegs &f)
{
    Row r;
    r.inst = f.inst;
    r.jc = f.jc;
    r.j = f.j;
    r.b1 = f.b1;
    r.n_inst = d.ninst == 1 ? (uint32_t)d.n_single : (uint32_t)d.inst_n[f.inst];
    r.img_base = d.ninst == 1 ? 0 : d.inst_img[f.inst];
    r.valid = f.j < r.n_inst;
    r.simg = r.valid ? d.img + r.img_base + (int64_t)f.j * d.s : nullptr;
    r.sfg = nullptr;
    return r;
}

/* grouping orders: ORDER_R groups b2-pairs (b2 is bit 0 already); ORDER_H
 * groups the Hadamard's 2^L values of the low L bits of k, which move below
 * b2 (the low L + 1 bits rotate by one) */
constexpr int ORDER_R = 0, ORDER_H = 1;

/* word 0 of the key with the target's bits moved below the others */
template <int ORDER>
__device__ __forceinline__ uint64_t permuted0(uint64_t w0, int L)
{
    if (ORDER == ORDER_H && L > 0) {
        const uint64_t m = (1ull << L) - 1ull;
        w0 = (w0 & ~((m << 1) | 1ull)) | ((w0 >> 1) & m) | ((w0 & 1ull) << L);
    }
    return w0;
}

template <int ORDER, int NW>
__device__ __forceinline__ bool same_group(const FKeyN<NW> &a, const FKeyN<NW> &b, int L)
{
    const uint64_t m = ORDER == ORDER_R ? 1ull : (((1ull << L) - 1ull) << 1);
    bool eq = (a.w[0] & ~m) == (b.w[0] & ~m);
#pragma unroll
    for (int i = 1; i < NW; ++i) eq = eq && a.w[i] == b.w[i];
    return eq;
}

/* ---- gather, maps, phase ------------------------------------------------------ */

template <typename AmpT, int NW>
__global__ void k_f_gather(QwSimDev d, QwBufDev buf, int inst, const double *scale, FKeyN<NW> *keys, double2 *amps,
                           unsigned long long *counter, int64_t cap)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    const int lane = threadIdx.x & 31;
    const double sc = scale ? *scale : 1.0;
    const FLayout L = flayout(d.nb);
    for (int64_t b = warp; b < d.total_buckets; b += nw) {
        int n = buf.count[b];
        if (n <= 0) continue;
        if (n > d.cap_row) n = d.cap_row;
        Row r;
        if (!row_of(d, buf, b, r)) continue;
        if (inst >= 0 && r.inst != (uint32_t)inst) continue;
        unsigned long long p0 = 0; /* a row's branches take adjacent places: one atomic a row */
        if (lane == 0) p0 = atomicAdd(counter, (unsigned long long)n);
        p0 = __shfl_sync(FULL, p0, 0);
        for (int i = lane; i < n; i += 32) {
            const int64_t slot = b * (int64_t)d.cap_row + i;
            const unsigned long long p = p0 + (unsigned long long)i;
            if ((int64_t)p >= cap) continue;
            FRegs f;
            f.inst = r.inst;
            f.jc = r.jc;
            f.j = r.j;
            f.b1 = r.b1;
            f.x = decode_r(buf.key[slot], d.nb);
            FKeyN<NW> k;
#pragma unroll
            for (int t = 0; t < NW; ++t) k.w[t] = 0ull;
            fencode_into(k, f, L);
            keys[p] = k;
            amps[p] = cscale(sc, load_amp<AmpT>(buf.amp, slot));
        }
    }
}

/* op codes of k_f_map, applied from the lowest 4 bits up */
constexpr int F_OSDAG = 1, F_OA = 2, F_OS = 3, F_S = 4, F_A0 = 5;

template <int NW>
__global__ void k_f_map(QwSimDev d, FKeyN<NW> *keys, int64_t M, uint32_t ops, int32_t *status)
{
    const FLayout L = flayout(d.nb);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        /* the base registers are words 0 and 1 of any key width: only they
           are read and written */
        ulonglong2 *base = reinterpret_cast<ulonglong2 *>(keys + i);
        const ulonglong2 b01 = *base;
        FKey k;
        k.w[0] = b01.x;
        k.w[1] = b01.y;
        FRegs f = fdecode(k, L);
        for (uint32_t o = ops; o != 0; o >>= 4) {
            const uint32_t op = o & 15u;
            const Row r = frow(d, f);
            if (op == F_OSDAG) op_osdag(d, r, f.x);
            else if (op == F_OA) op_oa(d, r, f.x);
            else if (op == F_OS) op_os(d, r, f.x);
            else if (op == F_A0) {
                if (f.x.A != 0) atomicOr(status, QW_ST_ANCILLA);
            } else if (op == F_S) { /* (jc, j, b1) <-> (kc, k, b2) */
                const uint32_t jc = f.jc, j = f.j, b1 = f.b1;
                f.jc = f.x.kc;
                f.j = f.x.k;
                f.b1 = f.x.b2;
                f.x.kc = jc;
                f.x.k = j;
                f.x.b2 = b1;
            }
        }
        frewrite(k, f, L);
        *base = make_ulonglong2(k.w[0], k.w[1]);
    }
}

/* P = 2 Pi - 1 (Eq. (impl)): the sign flips unless b1, k, b2, jc, kc are 0 */
template <int NW>
__global__ void k_f_phase(QwSimDev d, const FKeyN<NW> *keys, double2 *amps, int64_t M)
{
    const FLayout L = flayout(d.nb);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const FRegs f = fdecode(fbase_load(keys + i), L);
        const bool zero = f.b1 == 0 && f.x.k == 0 && f.x.b2 == 0 && f.jc == 0 && f.x.kc == 0;
        if (!zero) amps[i] = cneg(amps[i]);
    }
}

/* ---- register-faithful sub-operations (10-word keys) -------------------------- */
/*
 * The working registers of O_s' (its QRAM address, computed out of place:
 * Eq. "Newprocess"), of O_A' and of the quantum binary search (Alg. 1: left,
 * right, mid, midval, the flag and the two comparison bits, and the push/pop
 * garbage stack of (mid, midval, cl, ce) frames, one per probe) held in each
 * branch's key between the sub-operations, above bit 128:
 *   addr, left, right, mid (aw bits each), midval (16), flag, cl, ce (1 each),
 *   then L + 1 frames of mid (aw), midval (16), cl, ce.
 * Addresses follow the QRAM of Fig. 1: the value segment [0, N s), the column
 * segment [N s, 2 N s), row j's slot l at j s + l; a read outside its segment
 * gives 0.
 */
struct FaithLayout {
    int aw;
    int p_addr, p_left, p_right, p_mid, p_midval, p_flag, p_cl, p_ce, p_stk, frame;
};

/* field access on a key held in shared memory (k_fq: word i of the thread's
   key at w[256 i], so that a warp's accesses to one word are conflict-free) */
constexpr int FQ_THREADS = 256;
__device__ __forceinline__ uint64_t sget(const uint64_t *w, int pos, int n)
{
    const int i = pos >> 6, o = pos & 63;
    uint64_t v = w[i * FQ_THREADS] >> o;
    if (o + n > 64 && i + 1 < NW_FAITH) v |= w[(i + 1) * FQ_THREADS] << (64 - o);
    return v & (n >= 64 ? ~0ull : ((1ull << n) - 1ull));
}

__device__ __forceinline__ void sput(uint64_t *w, int pos, int n, uint64_t v)
{
    v &= (n >= 64 ? ~0ull : ((1ull << n) - 1ull));
    const int i = pos >> 6, o = pos & 63;
    w[i * FQ_THREADS] |= v << o;
    if (o + n > 64 && i + 1 < NW_FAITH) w[(i + 1) * FQ_THREADS] |= v >> (64 - o);
}

__device__ __forceinline__ void sclear(uint64_t *w, int pos, int n)
{
    const uint64_t m = (n >= 64 ? ~0ull : ((1ull << n) - 1ull));
    const int i = pos >> 6, o = pos & 63;
    w[i * FQ_THREADS] &= ~(m << o);
    if (o + n > 64 && i + 1 < NW_FAITH) w[(i + 1) * FQ_THREADS] &= ~(m >> (64 - o));
}

/* sub-operation codes (the same numbering as the oracle's) */
constexpr int FQ_ADDR_COL = 1, FQ_QRAM_COL = 2, FQ_QBS_FWD = 3, FQ_QBS_BWD = 4, FQ_SWAP = 5, FQ_ADDR_VAL = 6,
              FQ_QRAM_VAL = 7;

__device__ __forceinline__ uint64_t fq_qram(const QwSimDev &d, uint64_t addr, bool col_segment)
{
    const uint64_t ns = (uint64_t)d.n_single * (uint64_t)d.s;
    if (col_segment) {
        if (addr < ns || addr >= 2 * ns) return 0;
        return (uint64_t)(__ldg(d.img + (addr - ns)) >> 16);
    }
    if (addr >= ns) return 0;
    return (uint64_t)(__ldg(d.img + addr) & 0xffffu);
}

/* A run of sub-operations (their codes in `ops`, 4 bits each, from the lowest
 * up) on every branch, its working registers held on chip from one to the
 * next: the key is read once and written once a run instead of once per
 * sub-operation.  QBS: the run holds Alg. 1 (or its uncomputation), whose
 * frames live in the key's upper words -- the whole key goes to shared memory
 * -- otherwise the address register (bits 128 .. 128 + aw - 1, in word 2) is
 * the only working register touched and words 0..2 are read.  idle: the
 * working registers must be 0 after the run (an interference op, P or S
 * follows); words 2..9 are then written only where they changed from or to
 * something else than 0.
 * Bound: one launch per sub-operation moved 6 x 80 to 15 x 112 bytes a branch
 * between two interference ops; now 80 to 96, and the time is the QRAM
 * reads of Alg. 1's probes, L + 1 dependent ones each way.  A step at N = 8192, s = 32
 * (with T~ and two marginals): 2097 -> 1458 us. */
template <bool QBS>
__global__ void __launch_bounds__(FQ_THREADS) k_fq(QwSimDev d, FKeyW *keys, int64_t M, uint64_t ops, FaithLayout F,
                                                   int idle, int32_t *status)
{
    const FLayout L = flayout(d.nb);
    const int aw = F.aw;
    const uint64_t am = aw >= 64 ? ~0ull : (1ull << aw) - 1ull;
    const uint64_t ns = (uint64_t)d.n_single * (uint64_t)d.s;
    __shared__ uint64_t sk[QBS ? NW_FAITH * FQ_THREADS : 1];
    uint64_t *kw = sk + (QBS ? threadIdx.x : 0);
    const bool whole = QBS || idle;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        ulonglong2 *g = reinterpret_cast<ulonglong2 *>(keys + i);
        const ulonglong2 b01 = g[0];
        FKey b;
        b.w[0] = b01.x;
        b.w[1] = b01.y;
        uint64_t w2, upper = 0ull; /* upper: words 3..9 */
        if (whole) {
            ulonglong2 v = g[1];
            w2 = v.x;
            upper = v.y;
            if (QBS) kw[3 * FQ_THREADS] = v.y;
#pragma unroll
            for (int t = 2; t < NW_FAITH / 2; ++t) {
                v = g[t];
                upper |= v.x | v.y;
                if (QBS) {
                    kw[2 * t * FQ_THREADS] = v.x;
                    kw[(2 * t + 1) * FQ_THREADS] = v.y;
                }
            }
            if (QBS) kw[2 * FQ_THREADS] = w2;
        } else {
            w2 = keys[i].w[2];
        }
        const uint64_t w2_in = w2;
        FRegs f = fdecode(b, L);
        uint64_t addr = w2 & am;
        const uint64_t offset = ns + (uint64_t)f.j * (uint64_t)d.s;
        for (uint64_t o = ops; o != 0; o >>= 4) {
            const int op = (int)(o & 15u);
            if (op == FQ_ADDR_COL) {
                addr ^= offset + f.x.k;
            } else if (op == FQ_QRAM_COL) {
                f.x.kc ^= (uint32_t)fq_qram(d, addr, true);
            } else if (op == FQ_ADDR_VAL) {
                if (f.jc == 0 && f.x.kc == 0) addr ^= (uint64_t)f.j * (uint64_t)d.s + f.x.k;
            } else if (op == FQ_QRAM_VAL) {
                if (f.jc == 0 && f.x.kc == 0) f.x.A ^= (uint32_t)fq_qram(d, addr, false);
            } else if (op == FQ_SWAP) {
                const uint32_t t = f.x.k;
                f.x.k = f.x.kc;
                f.x.kc = t;
            } else if (QBS) { /* FQ_QBS_FWD, FQ_QBS_BWD */
                uint64_t left = sget(kw, F.p_left, aw), right = sget(kw, F.p_right, aw);
                uint64_t mid = sget(kw, F.p_mid, aw), midval = sget(kw, F.p_midval, 16);
                uint32_t flag = (uint32_t)sget(kw, F.p_flag, 1), cl = (uint32_t)sget(kw, F.p_cl, 1);
                uint32_t ce = (uint32_t)sget(kw, F.p_ce, 1);
                const uint64_t target = f.x.kc;
                if (op == FQ_QBS_FWD) { /* Alg. 1's loop, every probe's registers pushed */
                    left ^= offset;
                    right ^= left + (uint64_t)d.s;
                    flag ^= 1u;
                    for (int it = 0; it <= d.L; ++it) {
                        if (flag) mid ^= (left + right) / 2;
                        if (flag) midval ^= fq_qram(d, mid, true);
                        if (flag) {
                            cl ^= (midval < target) ? 1u : 0u;
                            ce ^= (midval == target) ? 1u : 0u;
                        }
                        if (ce) f.x.k ^= (uint32_t)(mid - offset);
                        if (ce) flag ^= 1u;
                        if (flag && cl) {
                            const uint64_t t = mid;
                            mid = left;
                            left = t;
                        }
                        if (flag) cl ^= 1u;
                        if (flag && cl) {
                            const uint64_t t = mid;
                            mid = right;
                            right = t;
                        }
                        const int pf = F.p_stk + it * F.frame; /* push: the frame takes them, zeros stay */
                        sput(kw, pf, aw, mid);
                        sput(kw, pf + aw, 16, midval);
                        sput(kw, pf + aw + 16, 1, cl);
                        sput(kw, pf + aw + 17, 1, ce);
                        mid = midval = 0;
                        cl = ce = 0u;
                    }
                } else { /* the loop undone in reverse: pop, then every step inverted */
                    for (int it = d.L; it >= 0; --it) {
                        const int pf = F.p_stk + it * F.frame;
                        mid = sget(kw, pf, aw);
                        midval = sget(kw, pf + aw, 16);
                        cl = (uint32_t)sget(kw, pf + aw + 16, 1);
                        ce = (uint32_t)sget(kw, pf + aw + 17, 1);
                        sclear(kw, pf, F.frame);
                        if (flag && cl) {
                            const uint64_t t = mid;
                            mid = right;
                            right = t;
                        }
                        if (flag) cl ^= 1u;
                        if (flag && cl) {
                            const uint64_t t = mid;
                            mid = left;
                            left = t;
                        }
                        if (ce) flag ^= 1u;
                        if (flag) {
                            cl ^= (midval < target) ? 1u : 0u;
                            ce ^= (midval == target) ? 1u : 0u;
                        }
                        if (flag) midval ^= fq_qram(d, mid, true);
                        if (flag) mid ^= (left + right) / 2;
                        if (mid != 0 || midval != 0 || cl != 0 || ce != 0) atomicOr(status, QW_ST_ANCILLA);
                        mid = midval = 0;
                        cl = ce = 0u;
                    }
                    flag ^= 1u;
                    right ^= left + (uint64_t)d.s;
                    left ^= offset;
                    if (left != 0 || right != 0 || flag != 0) atomicOr(status, QW_ST_ANCILLA);
                    left = right = 0;
                    flag = 0u;
                }
                sclear(kw, F.p_left, aw);
                sclear(kw, F.p_right, aw);
                sclear(kw, F.p_mid, aw);
                sclear(kw, F.p_midval, 16);
                sclear(kw, F.p_flag, 3);
                sput(kw, F.p_left, aw, left);
                sput(kw, F.p_right, aw, right);
                sput(kw, F.p_mid, aw, mid);
                sput(kw, F.p_midval, 16, midval);
                sput(kw, F.p_flag, 1, flag);
                sput(kw, F.p_cl, 1, cl);
                sput(kw, F.p_ce, 1, ce);
            }
            /* a register holds what its field has room for */
            addr &= am;
            f.x.k &= (1u << L.nb) - 1u;
            f.x.kc &= (1u << L.nb) - 1u;
        }
        uint64_t upper_out = upper;
        if (QBS) {
            w2 = kw[2 * FQ_THREADS];
            upper_out = 0ull;
#pragma unroll
            for (int t = 3; t < NW_FAITH; ++t) upper_out |= kw[t * FQ_THREADS];
        }
        w2 = (w2 & ~am) | addr;
        if (idle && (w2 | upper_out) != 0ull) atomicOr(status, QW_ST_ANCILLA);
        if (QBS && (upper | upper_out) != 0ull) {
            g[1] = make_ulonglong2(w2, kw[3 * FQ_THREADS]);
#pragma unroll
            for (int t = 2; t < NW_FAITH / 2; ++t)
                g[t] = make_ulonglong2(kw[2 * t * FQ_THREADS], kw[(2 * t + 1) * FQ_THREADS]);
        } else if (w2 != w2_in) {
            keys[i].w[2] = w2;
        }
        frewrite(b, f, L);
        if (b.w[0] != b01.x || b.w[1] != b01.y) g[0] = make_ulonglong2(b.w[0], b.w[1]);
    }
}

/* the working registers must be 0 (an interference op, P, S or the store) */
__global__ void k_fq_check_idle(const FKeyW *keys, int64_t M, int from_bit, int32_t *status)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const FKeyW k = keys[i];
        bool any = false;
        for (int t = from_bit >> 6; t < NW_FAITH; ++t) {
            uint64_t v = k.w[t];
            if (t == (from_bit >> 6)) v &= ~((1ull << (from_bit & 63)) - 1ull);
            any = any || v != 0ull;
        }
        if (any) atomicOr(status, QW_ST_ANCILLA);
    }
}

/* a list as a table of registers: QW_FQ_COLS values per branch in the order
   inst, jc, j, b1, kc, k, b2, A, addr, left, right, mid, midval, flag, cl,
   ce, then QW_FQ_FRAMES frames of (mid, midval, cl, ce) */
__global__ void k_fq_export(QwSimDev d, const FKeyW *keys, int64_t M, FaithLayout F, uint64_t *table)
{
    const FLayout L = flayout(d.nb);
    const int aw = F.aw;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const FKeyW k = keys[i];
        const FRegs f = fdecode(k, L);
        uint64_t *t = table + i * QW_FQ_COLS;
        t[0] = f.inst;
        t[1] = f.jc;
        t[2] = f.j;
        t[3] = f.b1;
        t[4] = f.x.kc;
        t[5] = f.x.k;
        t[6] = f.x.b2;
        t[7] = f.x.A;
        t[8] = fget(k, F.p_addr, aw);
        t[9] = fget(k, F.p_left, aw);
        t[10] = fget(k, F.p_right, aw);
        t[11] = fget(k, F.p_mid, aw);
        t[12] = fget(k, F.p_midval, 16);
        t[13] = fget(k, F.p_flag, 1);
        t[14] = fget(k, F.p_cl, 1);
        t[15] = fget(k, F.p_ce, 1);
        for (int it = 0; it < QW_FQ_FRAMES; ++it) {
            uint64_t *fr = t + 16 + 4 * it;
            if (it <= d.L) {
                const int pf = F.p_stk + it * F.frame;
                fr[0] = fget(k, pf, aw);
                fr[1] = fget(k, pf + aw, 16);
                fr[2] = fget(k, pf + aw + 16, 1);
                fr[3] = fget(k, pf + aw + 17, 1);
            } else {
                fr[0] = fr[1] = fr[2] = fr[3] = 0ull;
            }
        }
    }
}

/* ---- single-pass compaction ------------------------------------------------------ */
/*
 * Kernels that write a varying number of outputs per input take tiles of their
 * input in the order blocks start (a counter), hold a tile's outputs in
 * registers, and learn where they go from the counts of the tiles before, summed
 * by looking back 32 tiles at a time (the single-pass prefix sum of the sort,
 * one count a tile): the outputs are formed once and written once.  With flags, a
 * three-kernel scan and a copy (R, R^dag) or a counting pass before the
 * writing one (H) they were formed or moved twice.  Two flat steps at N = 16384,
 * s = 16: 2495 -> 2224 us; one faithful step at N = 8192, s = 32: 1365 -> 1284.
 */
struct TileSum {            /* zeroed before the launch */
    unsigned int next, pad; /* the next tile */
    unsigned long long total;
    unsigned long long tile[1]; /* per tile: 1 << 62 its count, 2 << 62 with the tiles before */
};
constexpr unsigned long long TS_AGG = 1ull << 62, TS_INC = 2ull << 62, TS_CNT = TS_AGG - 1ull;
constexpr int TS_SPIN_LIMIT = 1 << 22;

/* the counts of the tiles before vb (called by one warp); count: this tile's.  A
   wait that outlasts the limit sets the status and the host's word; the outputs'
   places are then wrong (and checked against the array's end), and the host drops
   them all: what it would find between them are not keys. */
__device__ unsigned long long tile_before(TileSum *ts, int64_t vb, unsigned int count, int32_t *status,
                                          unsigned long long *host)
{
    const int lane = threadIdx.x & 31;
    volatile unsigned long long *t = ts->tile;
    if (vb == 0) {
        if (lane == 0) t[0] = TS_INC | count;
        return 0ull;
    }
    if (lane == 0) t[vb] = TS_AGG | count;
    unsigned long long before = 0ull;
    int64_t p = vb - 1;
    for (int spins = 0;;) {
        unsigned long long v = TS_INC; /* before tile 0: an end of count 0 */
        if (p >= lane) v = t[p - lane];
        const unsigned empty = __ballot_sync(FULL, (v >> 62) == 0ull), inc = __ballot_sync(FULL, (v >> 62) == 2ull);
        /* the tiles up to the nearest one that includes those before it */
        const int end = inc ? __ffs(inc) - 1 : 31;
        const unsigned need = end == 31 ? FULL : (2u << end) - 1u;
        if (empty & need) {
            if (++spins > TS_SPIN_LIMIT) {
                if (lane == 0) {
                    atomicOr(status, QW_ST_SORT_WAIT);
                    *(volatile unsigned long long *)(host + QW_TOTAL_WAIT) = 1ull;
                }
                break;
            }
            if (spins > 32) __nanosleep(64);
            continue;
        }
        unsigned long long c = lane <= end ? v & TS_CNT : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
        before += c;
        if (inc) break;
        p -= 32;
    }
    if (lane == 0) t[vb] = TS_INC | (before + count);
    return before;
}

/* A block's share of it: n outputs of this thread, the number of those of the
   threads before it in the block and all before the tile; the last tile writes the
   total, to the host's pinned memory too. */
template <int THREADS>
__device__ __forceinline__ unsigned long long tile_place(TileSum *ts, int64_t vb, int64_t ntiles, unsigned int n,
                                                         int32_t *status, unsigned long long *host)
{
    constexpr int W = THREADS / 32;
    __shared__ unsigned int ws[W];
    __shared__ unsigned long long base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned int x = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned int y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    unsigned int pre = 0, all = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        if (w < warp) pre += ws[w];
        all += ws[w];
    }
    if (warp == 0) {
        const unsigned long long b = tile_before(ts, vb, all, status, host);
        if (lane == 0) {
            base = b;
            if (vb == ntiles - 1) ts->total = *host = b + all;
        }
    }
    __syncthreads();
    return base + pre + x - n;
}

/* the block's tile */
__device__ __forceinline__ int64_t tile_take(TileSum *ts)
{
    __shared__ unsigned int vb;
    if (threadIdx.x == 0) vb = atomicAdd(&ts->next, 1u);
    __syncthreads();
    return vb;
}

/* ---- radix sort ------------------------------------------------------------------ */

/* OR of every permuted key and of its complement, word by word: a bit set in
   both differs between keys.  acc and *done zeroed by the caller; the last block
   writes the result to the host's pinned memory.  The key array is read as a flat array of 64-bit words; the
   grid's stride is a multiple of NW, so each thread always sees one word
   index. */
template <int ORDER, int NW>
__global__ void k_f_orand(const uint64_t *words, int64_t nwords, int L, unsigned long long *acc, unsigned int *done,
                          unsigned long long *host)
{
    __shared__ unsigned long long s_or[NW], s_nor[NW];
    __shared__ bool last;
    if (threadIdx.x < NW) s_or[threadIdx.x] = s_nor[threadIdx.x] = 0ull;
    __syncthreads();
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int wi = (int)(g % NW);
    uint64_t ov = 0ull, nv = 0ull;
    for (int64_t q = g; q < nwords; q += stride) {
        uint64_t v = words[q];
        if (wi == 0) v = permuted0<ORDER>(v, L);
        ov |= v;
        nv |= ~v;
    }
    atomicOr(&s_or[wi], (unsigned long long)ov);
    atomicOr(&s_nor[wi], (unsigned long long)nv);
    __syncthreads();
    if (threadIdx.x < NW) {
        atomicOr(acc + threadIdx.x, s_or[threadIdx.x]);
        atomicOr(acc + NW + threadIdx.x, s_nor[threadIdx.x]);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x < 2 * NW) host[threadIdx.x] = __ldcg(acc + threadIdx.x);
}

/* The sort runs on a compacted key (the chunks of qw_sort_chunks.h).  LSD
 * order carries over chunks: chunk 0 is sorted first, chunk c + 1 is formed
 * from the keys in the order chunk c left. */
constexpr int OS_THREADS = 256, OS_IPT = 8, OS_TILE = OS_THREADS * OS_IPT;
constexpr int OS_SPIN_LIMIT = 1 << 22;

/* The chunk's compacted key of every entry -- the entry at position i of the
   current order, i.e. keys[perm[i]] (perm == nullptr: i) -- and the global
   count of every 8-bit digit of it for each of the chunk's passes
   (ghist[pass * 256 + digit], zeroed by the caller). */
template <int ORDER, int NW>
__global__ void __launch_bounds__(256) k_f_ckey(const FKeyN<NW> *keys, const uint32_t *perm, int64_t M, int L,
                                                CkRuns runs, uint64_t *ck, uint32_t *ghist)
{
    __shared__ uint32_t h[CK_MAXPASS * 256];
    for (int t = threadIdx.x; t < CK_MAXPASS * 256; t += blockDim.x) h[t] = 0u;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t j = perm ? (int64_t)perm[i] : i;
        if (j >= M) j = 0; /* only after a sort wait gave up */
        const FKeyN<NW> *k = keys + j;
        uint64_t c = 0ull, v = 0ull;
        int dst = 0, cw = -1;
        for (int r = 0; r < runs.n; ++r) {
            const int w = runs.word[r];
            if (w != cw) {
                v = k->w[w];
                if (w == 0) v = permuted0<ORDER>(v, L);
                cw = w;
            }
            const int ln = runs.len[r];
            const uint64_t m = ln >= 64 ? ~0ull : (1ull << ln) - 1ull;
            c |= ((v >> runs.shift[r]) & m) << dst;
            dst += ln;
        }
        ck[i] = c;
        for (int p = 0; p < runs.npass; ++p) atomicAdd(&h[p * 256 + (int)((c >> (8 * p)) & 255ull)], 1u);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < runs.npass * 256; t += blockDim.x)
        if (h[t]) atomicAdd(ghist + t, h[t]);
}

/* status of a tile in one pass, one 64-bit word per (tile, digit): the pass
   tag (bits 40..63; a word of another pass reads as not ready), 1 = the
   tile's own count / 2 = the inclusive prefix over tiles 0..vb (bits 38, 39),
   the count (bits 0..37) */
constexpr uint64_t OS_AGG = 1ull << 38, OS_INC = 2ull << 38, OS_CNT = (1ull << 38) - 1ull;

__device__ __forceinline__ uint64_t os_load(const uint64_t *p)
{
    return *reinterpret_cast<const volatile uint64_t *>(p);
}

__device__ __forceinline__ void os_store(uint64_t *p, uint64_t v)
{
    *reinterpret_cast<volatile uint64_t *>(p) = v;
}

/* One stable pass on the 8-bit digit at `shift` of the compacted key.  A
 * block takes tile vb in the order blocks start (a counter), so every tile
 * before it belongs to a block already running.  Warp w ranks items vb T +
 * 256 w + 32 r + lane (r = 0..7) by their digit in that order; the tile's
 * digit counts are published, then the counts of the tiles before it are
 * summed by looking back until a tile with its inclusive prefix (single-pass
 * "decoupled look-back" prefix sum); an item goes to the digit's global
 * start (the exclusive scan of ghist) + the tiles before + the warps before
 * + its rank.  A wait that outlasts OS_SPIN_LIMIT polls sets
 * QW_ST_SORT_WAIT and the block carries on (the sort's result is then
 * wrong, and the host reports the status). */
template <bool FIRST, bool WRITE_CK>
__global__ void __launch_bounds__(OS_THREADS, 4) k_f_onesweep(const uint64_t *ckin, const uint32_t *ixin, uint64_t *ckout,
                                                           uint32_t *ixout, int64_t M, int shift,
                                                           const uint32_t *ghist, uint64_t *stat, uint64_t tag,
                                                           unsigned int *ctr, int32_t *status)
{
    __shared__ uint32_t hw[8][256];
    __shared__ uint32_t sbase[256];
    __shared__ uint32_t wsum[8];
    __shared__ unsigned int svb;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) svb = atomicAdd(ctr, 1u);
#pragma unroll
    for (int w = 0; w < 8; ++w) hw[w][t] = 0u;
    __syncthreads();
    const int64_t vb = svb;
    const int64_t base = vb * OS_TILE + warp * (32 * OS_IPT) + lane;
    uint64_t c[OS_IPT];
    uint32_t ix[OS_IPT], rk[OS_IPT];
#pragma unroll
    for (int r = 0; r < OS_IPT; ++r) {
        const int64_t i = base + 32 * r;
        c[r] = 0ull;
        ix[r] = 0u;
        if (i < M) {
            c[r] = ckin[i];
            ix[r] = FIRST ? (uint32_t)i : ixin[i];
        }
    }
    auto digit = [&](int r) { return base + 32 * r < M ? (int)((c[r] >> shift) & 255ull) : 256; };
    const unsigned below = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < OS_IPT; ++r) {
        const int d = digit(r);
        /* the lanes of the same digit (9 bits: 256 = none), by ballots: the
           match instruction runs once per distinct value */
        unsigned m = FULL;
#pragma unroll
        for (int b = 0; b < 9; ++b) {
            const unsigned bal = __ballot_sync(FULL, (d >> b) & 1);
            m &= (d >> b) & 1 ? bal : ~bal;
        }
        const uint32_t cnt = d < 256 ? hw[warp][d] : 0u;
        rk[r] = cnt + (uint32_t)__popc(m & below);
        __syncwarp();
        if (d < 256 && (m & below) == 0u) hw[warp][d] = cnt + (uint32_t)__popc(m);
        __syncwarp();
    }
    __syncthreads();
    /* thread t owns digit t: the warps' exclusive prefix, the tile's count */
    uint32_t run = 0u;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const uint32_t v = hw[w][t];
        hw[w][t] = run;
        run += v;
    }
    uint64_t *my = stat + vb * 256 + t;
    os_store(my, (tag << 40) | (vb == 0 ? OS_INC : OS_AGG) | run);
    /* global start of digit t: exclusive scan of this pass's digit counts */
    const uint32_t g = ghist[t];
    uint32_t x = g;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    /* look back over the tiles before */
    uint64_t excl = 0ull;
    if (vb > 0) {
        int64_t p = vb - 1;
        int spins = 0;
        while (p >= 0) {
            const uint64_t v = os_load(stat + p * 256 + t);
            if ((v >> 40) != tag) {
                if (++spins > OS_SPIN_LIMIT) {
                    atomicOr(status, QW_ST_SORT_WAIT);
                    break;
                }
                if (spins > 32) __nanosleep(64);
                continue;
            }
            excl += v & OS_CNT;
            if (v & OS_INC) break;
            --p;
        }
        os_store(my, (tag << 40) | OS_INC | (excl + run));
    }
    __syncthreads();
    uint32_t pre = 0u;
    for (int w = 0; w < warp; ++w) pre += wsum[w];
    sbase[t] = pre + x - g + (uint32_t)excl;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < OS_IPT; ++r) {
        const int d = digit(r);
        const uint32_t dest = d < 256 ? sbase[d] + hw[warp][d] + rk[r] : 0u;
        if (d < 256 && (int64_t)dest < M) { /* always, unless a wait gave up */
            if (WRITE_CK) ckout[dest] = c[r];
            ixout[dest] = ix[r];
        }
    }
}

/* the sorted list: entry i is the entry perm[i] of the input */
template <int NW>
__global__ void k_f_permute(const FKeyN<NW> *kin, const double2 *ain, const uint32_t *perm, FKeyN<NW> *kout,
                            double2 *aout, int64_t M)
{
    static_assert(NW % 2 == 0, "keys are copied as 16-byte words");
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t j = perm[i];
        if (j >= M) j = 0; /* only after a sort wait gave up */
        const ulonglong2 *s = reinterpret_cast<const ulonglong2 *>(kin + j);
        ulonglong2 *o = reinterpret_cast<ulonglong2 *>(kout + i);
#pragma unroll
        for (int q = 0; q < NW / 2; ++q) o[q] = s[q];
        aout[i] = ain[j];
    }
}

/* ---- per-group transforms (the "computing" step) -------------------------------- */

/* R (DAG = false) or R^dag on b2-pairs (the list sorted in ORDER_R, a pair in
 * either order): the first member of each pair forms both outputs, R = [[f, -g],
 * [g, conj f]] (Alg. T~ and the footnote of Sec. IV); the kept ones are written in
 * the order of the pairs, b2 = 0 first, at most cap.  Bound by the keys read and
 * written (a thread per entry, the neighbours' keys from L1). */
constexpr int RT_THREADS = 256;
template <bool DAG, int NW>
__global__ void __launch_bounds__(RT_THREADS) k_f_rot(QwSimDev d, const FKeyN<NW> *keys, const double2 *amps, int64_t M,
                                                      FKeyN<NW> *okeys, double2 *oamps, int64_t cap, TileSum *ts,
                                                      int32_t *status, unsigned long long *host)
{
    const FLayout L = flayout(d.nb);
    const int64_t vb = tile_take(ts), i = vb * RT_THREADS + threadIdx.x;
    FKeyN<NW> k;
    double2 o0 = make_double2(0, 0), o1 = o0;
    bool k0 = false, k1 = false;
    if (i < M) {
        k = keys[i];
        const bool head = i == 0 || !same_group<ORDER_R>(keys[i - 1], k, 0);
        if (head) {
            double2 a0 = amps[i], a1 = make_double2(0, 0);
            if (i + 1 < M && same_group<ORDER_R>(k, keys[i + 1], 0)) a1 = amps[i + 1];
            if ((k.w[0] & 1ull) != 0) {
                const double2 t = a0;
                a0 = a1;
                a1 = t;
            }
            const FRegs f = fdecode(k, L);
            double2 fv;
            double g;
            rot_fg(d, f.x.A, f.j, f.x.k, fv, g);
            if (!DAG) {
                o0 = csub(cmul(fv, a0), cscale(g, a1));
                o1 = cadd(cscale(g, a0), cmul(cconj(fv), a1));
            } else {
                o0 = cadd(cmul(cconj(fv), a0), cscale(g, a1));
                o1 = csub(cmul(fv, a1), cscale(g, a0));
            }
            k0 = keep(o0, d.tau2);
            k1 = keep(o1, d.tau2);
        }
    }
    int64_t at = (int64_t)tile_place<RT_THREADS>(ts, vb, gridDim.x, (k0 ? 1u : 0u) + (k1 ? 1u : 0u), status, host);
    if (k0 && at < cap) {
        k.w[0] &= ~1ull;
        okeys[at] = k;
        oamps[at] = o0;
        ++at;
    }
    if (k1 && at < cap) {
        k.w[0] |= 1ull;
        okeys[at] = k;
        oamps[at] = o1;
    }
}

/* The groups of H on the low L bits of k (the list sorted in ORDER_H): starts[g]
 * = the first member of group g, starts[G] = M.  8 entries a thread. */
constexpr int ST_THREADS = 256, ST_IPT = 8;
template <int NW>
__global__ void __launch_bounds__(ST_THREADS) k_f_starts(QwSimDev d, const FKeyN<NW> *keys, int64_t M, int64_t *starts,
                                                         TileSum *ts, int32_t *status, unsigned long long *host)
{
    const int64_t vb = tile_take(ts), i0 = vb * (ST_THREADS * ST_IPT) + (threadIdx.x >> 5) * (32 * ST_IPT);
    const int lane = threadIdx.x & 31;
    /* a warp takes 256 entries in a row, 32 at a time */
    unsigned heads[ST_IPT];
    unsigned n = 0;
#pragma unroll
    for (int r = 0; r < ST_IPT; ++r) {
        const int64_t i = i0 + 32 * r + lane;
        const bool head = i < M && (i == 0 || !same_group<ORDER_H>(keys[i - 1], keys[i], d.L));
        heads[r] = __ballot_sync(FULL, head);
        n += __popc(heads[r]);
    }
    /* the warp's count on its first lane: every lane's place is its warp's */
    unsigned long long at = tile_place<ST_THREADS>(ts, vb, gridDim.x, lane == 0 ? n : 0u, status, host);
    at = __shfl_sync(FULL, at, 0);
#pragma unroll
    for (int r = 0; r < ST_IPT; ++r) {
        const unsigned long long g = at + __popc(heads[r] & ((1u << lane) - 1u));
        if ((heads[r] >> lane) & 1u) {
            if (g < (unsigned long long)M) starts[g] = i0 + 32 * r + lane;
        }
        at += __popc(heads[r]);
    }
    /* the end of the last group */
    if (vb == gridDim.x - 1 && threadIdx.x == 0) {
        const unsigned long long G = *(volatile unsigned long long *)&ts->total;
        if (G <= (unsigned long long)M) starts[G] = M;
    }
}

/* H on each group's zero-filled vector of 2^L = s entries (the groups of
 * the list sorted in ORDER_H, starts[g] .. starts[g + 1]): output u of a group
 * is s^-1/2 sum_m (-1)^{|u & v_m|} a_m over its members m (v_m: their low L
 * bits of k).  A warp runs 32 / s groups (s < 32) or one group (s >= 32).
 * For s <= 128 lane t of a group holds entries t, t + 32, ... of the
 * zero-filled vector, and the L butterfly stages of the fast Walsh-Hadamard
 * transform (Sylvester order, (x, y) -> (x + y, x - y) on index bit h) run
 * over shuffles (bits below 32) and between the lane's registers (bits
 * above): s L additions per group instead of s^2; the FP64 pipe is the
 * limit.  Larger s: s / 32 rounds of 32 outputs, each the direct sum over
 * the members in list order (a lane loads one member per round and the
 * warp's shuffles hand them to every output).
 * The kept outputs are written in the order of the groups and of u, at most cap
 * (the fast transform: tiles of HG_ITERS x 8 warps' groups, the outputs held in
 * registers until the counts of the tiles before are known).  The direct sums
 * go over the groups twice -- their outputs, s / 32 a lane, do not fit registers. */
constexpr int HG_WARPS = 8;
template <int R> struct HgIters { static constexpr int n = R == 1 ? 4 : (R == 2 ? 2 : 1); }; /* R x n outputs a lane */
template <int NW, int FWHT_ROUNDS>
__global__ void __launch_bounds__(32 * HG_WARPS) k_f_hgroups(QwSimDev d, const FKeyN<NW> *keys, const double2 *amps,
                                                             int64_t M, const int64_t *starts, int64_t G,
                                                             FKeyN<NW> *okeys, double2 *oamps, int64_t cap, TileSum *ts, int32_t *status,
                                                             unsigned long long *host)
{
    const int s = d.s;
    const int sw = s < 32 ? s : 32, gpw = 32 / sw, rounds = s / sw;
    const int lane = threadIdx.x & 31, sub = lane / sw, ul = lane - sub * sw, first = sub * sw;
    const unsigned below = (1u << lane) - 1u;
    const uint64_t lowm = ((uint64_t)s - 1ull) << 1;
    constexpr int ZR = FWHT_ROUNDS > 0 ? FWHT_ROUNDS : 1;
    constexpr bool fwht = FWHT_ROUNDS > 0;
    constexpr int ITERS = HgIters<FWHT_ROUNDS>::n;
    const int64_t vb = tile_take(ts), wg0 = (vb * HG_WARPS + (threadIdx.x >> 5)) * ITERS; /* the warp's first set of groups */
    const int ns = rounds;
    /* group g's first member and their number (in bounds whatever starts holds) */
    auto group_at = [&](bool act, int64_t g, int64_t &b, int64_t &nm) {
        b = act ? starts[g] : 0;
        if (b < 0 || b >= M) b = 0;
        const int64_t e = act ? starts[g + 1] : 0;
        nm = e > b ? (e < M ? e : M) - b : 0;
    };
    if (fwht) {
        __shared__ double2 zv[HG_WARPS][32 * ZR];
        double2 *vec = zv[threadIdx.x >> 5];
        /* entry q sw + ul of the group's zero-filled vector in x[it][q], the
           butterflies of index bits below sw over shuffles, the ones above between
           the lane's registers; x[it][q] is then output u = q sw + ul */
        double2 x[ITERS][ZR];
        unsigned kept[ITERS][ZR]; /* the warp's lanes whose output is kept */
        int64_t b[ITERS];
        unsigned n = 0;
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            const int64_t g = (wg0 + it) * gpw + sub;
            const bool act = g < G;
            int64_t nm;
            group_at(act, g, b[it], nm);
#pragma unroll
            for (int q = 0; q < ZR; ++q)
                if (q < ns) vec[first + q * sw + ul] = make_double2(0, 0);
            __syncwarp();
#pragma unroll
            for (int q = 0; q < ZR; ++q) {
                const int64_t mi = (int64_t)q * sw + ul;
                if (q < ns && mi < nm)
                    vec[first + (int)((keys[b[it] + mi].w[0] >> 1) & (uint64_t)(s - 1))] = amps[b[it] + mi];
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < ZR; ++q) x[it][q] = q < ns ? vec[first + q * sw + ul] : make_double2(0, 0);
            __syncwarp();
            for (int h = 1; h < sw; h <<= 1) {
#pragma unroll
                for (int q = 0; q < ZR; ++q) {
                    if (q >= ns) continue;
                    const double yx = __shfl_xor_sync(FULL, x[it][q].x, h), yy = __shfl_xor_sync(FULL, x[it][q].y, h);
                    x[it][q] = (ul & h) ? make_double2(yx - x[it][q].x, yy - x[it][q].y)
                                        : make_double2(x[it][q].x + yx, x[it][q].y + yy);
                }
            }
#pragma unroll
            for (int hq = 1; hq < ZR; hq <<= 1) {
#pragma unroll
                for (int q = 0; q < ZR; ++q) {
                    if ((q & hq) || (q | hq) >= ns) continue;
                    const double2 lo = x[it][q], hi = x[it][q | hq];
                    x[it][q] = make_double2(lo.x + hi.x, lo.y + hi.y);
                    x[it][q | hq] = make_double2(lo.x - hi.x, lo.y - hi.y);
                }
            }
#pragma unroll
            for (int q = 0; q < ZR; ++q) {
                x[it][q] = cscale(d.inv_sqrt_s, x[it][q]);
                kept[it][q] = __ballot_sync(FULL, act && q < ns && keep(x[it][q], d.tau2));
                n += __popc(kept[it][q]);
            }
        }
        unsigned long long at = tile_place<32 * HG_WARPS>(ts, vb, gridDim.x, lane == 0 ? n : 0u, status, host);
        at = __shfl_sync(FULL, at, 0);
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            /* s < 32: one round, the warp's groups one after another; s >= 32: one group */
#pragma unroll
            for (int q = 0; q < ZR; ++q) {
                const int64_t dst = (int64_t)at + __popc(kept[it][q] & below);
                if (((kept[it][q] >> lane) & 1u) && dst < cap) {
                    FKeyN<NW> ko = keys[b[it]];
                    ko.w[0] = (ko.w[0] & ~lowm) | ((uint64_t)(q * sw + ul) << 1);
                    okeys[dst] = ko;
                    oamps[dst] = x[it][q];
                }
                at += __popc(kept[it][q]);
            }
        }
        return;
    }
    /* s > 128: one group a warp */
    const bool act = wg0 < G;
    int64_t b, nm;
    group_at(act, wg0, b, nm);
    unsigned long long at = 0;
    for (int pass = 0; pass < 2; ++pass) { /* counted, then written */
        unsigned run = 0;
        for (int q = 0; q < rounds; ++q) {
            const uint32_t u = (uint32_t)(q * sw + ul);
            double2 o = make_double2(0, 0);
            for (int q2 = 0; q2 < rounds; ++q2) {
                const int64_t mi = (int64_t)q2 * sw + ul;
                uint32_t mv = 0u;
                double2 ma = make_double2(0, 0);
                if (mi < nm) {
                    mv = (uint32_t)((keys[b + mi].w[0] >> 1) & (uint64_t)(s - 1));
                    ma = amps[b + mi];
                }
                for (int j = 0; j < sw; ++j) {
                    const uint32_t v = __shfl_sync(FULL, mv, first + j);
                    const double ax = __shfl_sync(FULL, ma.x, first + j);
                    const double ay = __shfl_sync(FULL, ma.y, first + j);
                    if ((int64_t)q2 * sw + j < nm) {
                        const double2 a = make_double2(ax, ay);
                        o = (__popc(u & v) & 1) ? csub(o, a) : cadd(o, a);
                    }
                }
            }
            o = cscale(d.inv_sqrt_s, o);
            const unsigned bal = __ballot_sync(FULL, act && keep(o, d.tau2));
            const int64_t dst = (int64_t)at + run + __popc(bal & below);
            if (pass == 1 && ((bal >> lane) & 1u) && dst < cap) {
                FKeyN<NW> ko = keys[b];
                ko.w[0] = (ko.w[0] & ~lowm) | ((uint64_t)u << 1);
                okeys[dst] = ko;
                oamps[dst] = o;
            }
            run += (unsigned)__popc(bal);
        }
        if (pass == 0) {
            at = tile_place<32 * HG_WARPS>(ts, vb, gridDim.x, lane == 0 ? run : 0u, status, host);
            at = __shfl_sync(FULL, at, 0);
        }
    }
}

/* QLS read-out after T~^dag's H: Y[j] += a_j * (the flag-0 amplitude of row j) */
template <int NW>
__global__ void k_f_readout(QwSimDev d, const FKeyN<NW> *keys, const double2 *amps, int64_t M, QwStepArgs a)
{
    const FLayout L = flayout(d.nb);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const FRegs f = fdecode(fbase_load(keys + i), L);
        if (f.jc != 0 || f.b1 != 0 || f.x.kc != 0 || f.x.k != 0 || f.x.b2 != 0 || f.x.A != 0) continue;
        if (f.j >= (uint32_t)d.n_single) continue;
        const double coef = a.qls_coefs[*a.qls_j];
        const double2 v = amps[i];
        atomicAdd(&a.qls_y[f.j].x, coef * v.x);
        atomicAdd(&a.qls_y[f.j].y, coef * v.y);
    }
}

/* the output into the row buckets, |stored a|^2 summed per block into *norm */
template <typename AmpT, int NW>
__global__ void k_f_scatter(QwSimDev d, QwBufDev out, const FKeyN<NW> *keys, const double2 *amps, int64_t M,
                            int32_t *status, unsigned int *maxrow, double *norm)
{
    __shared__ double ws[8];
    const FLayout L = flayout(d.nb);
    double acc = 0.0;
    unsigned int longest = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const FRegs f = fdecode(fbase_load(keys + i), L);
        if (f.x.A != 0) {
            atomicOr(status, QW_ST_ANCILLA);
            continue;
        }
        const int64_t b = bucket_of(d, out, f.inst, f.jc, f.j, f.b1, status);
        if (b < 0) continue;
        const int p = atomicAdd(out.count + b, 1);
        longest = max(longest, (unsigned int)(p + 1));
        if (p >= d.cap_row) {
            atomicOr(status, QW_ST_ROW_OVERFLOW);
            continue;
        }
        const int64_t slot = b * (int64_t)d.cap_row + p;
        out.key[slot] = encode_r(f.x, d.nb);
        acc += store_amp<AmpT>(out.amp, slot, amps[i]);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
    longest = __reduce_max_sync(FULL, longest);
    if ((threadIdx.x & 31) == 0) {
        ws[threadIdx.x >> 5] = acc;
        if (longest) atomicMax(maxrow, longest);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += ws[w];
        atomicAdd(norm, t);
    }
}

/* the step's bookkeeping, as the step kernels' last block does it */
__global__ void k_f_finish(QwStepArgs a, const double *norm, unsigned long long in, unsigned long long rdag,
                           unsigned long long h1, unsigned long long hph, unsigned long long out)
{
    const bool clean = *(volatile int32_t *)a.status == 0;
    if (!clean) return;
    const double tot = *norm;
    *a.norm_out = tot;
    if (a.scale_out) *a.scale_out = (a.renorm && tot > 0.0) ? sqrt(*a.renorm_target / tot) : 1.0;
    if (a.steps_done) *a.steps_done += 1;
    if (a.stats) {
        a.stats[QW_STAT_IN] += in;
        a.stats[QW_STAT_RDAG] += rdag;
        a.stats[QW_STAT_H1] += h1;
        a.stats[QW_STAT_HPH] += hph;
        a.stats[QW_STAT_OUT] += out;
        a.stats[QW_STAT_STEPS] += 1;
    }
}

/* ---- state import and export ------------------------------------------------------ */
/*
 * A list of branches as the caller holds it: W 64-bit words a key, of which
 * the layout takes the low 4 nb + 34 bits.  All passes are streams over 32 to
 * 100 bytes a branch.  N = 2047, s = 8 (49 000 branches), an import, ten steps and
 * an export: 12.30 ms with the keys packed bit by bit and sorted by comparison on
 * the host, 0.74 ms so (what is left: launches, synchronisations and the copies
 * from and to the caller's pageable arrays).
 */

/* keys of W words to the two-word layout, *bad set by one that the layout
   does not hold: a bit above it, a non-zero A, an instance beyond the last */
__global__ void k_io_load(const uint64_t *in, int W, int64_t M, FLayout L, uint32_t ninst, FKey *keys, QwIoFlags *f)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        FKey k;
        k.w[0] = in[i * W];
        k.w[1] = W > 1 ? in[i * W + 1] : 0ull;
        uint64_t above = L.pinst + 16 < 64 ? k.w[1] | (k.w[0] >> (L.pinst + 16))
                                           : (L.pinst + 16 == 64 ? k.w[1] : k.w[1] >> (L.pinst + 16 - 64));
        for (int t = 2; t < W; ++t) above |= in[i * W + t];
        if (above != 0ull || fget(k, L.pA, 16) != 0ull || fget(k, L.pinst, 16) >= ninst) f->bad = 1;
        keys[i] = k;
    }
}

/* the order of the list: *unsorted unless ascending, *dup if two neighbours
   are equal, and the longest run of one row (inst, A, jc, j, b1: the bits from
   b1 up), found from its first member by doubling and bisection -- a row's
   length where the list is sorted */
__global__ void k_io_order(const FKey *keys, int64_t M, FLayout L, QwIoFlags *f)
{
    unsigned int longest = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const FKey k = keys[i];
        auto same_row = [&](const FKey &o) { return o.w[1] == k.w[1] && (o.w[0] >> L.pb1) == (k.w[0] >> L.pb1); };
        if (i > 0) {
            const FKey q = keys[i - 1];
            if (q.w[1] == k.w[1] && q.w[0] == k.w[0]) f->dup = 1;
            if (q.w[1] > k.w[1] || (q.w[1] == k.w[1] && q.w[0] > k.w[0])) f->unsorted = 1;
            if (same_row(q)) continue;
        }
        int64_t in = i, step = 1; /* in: in the run */
        while (in + step < M && same_row(keys[in + step])) {
            in += step;
            step <<= 1;
        }
        int64_t out = in + step < M ? in + step : M; /* beyond it */
        while (out - in > 1) {
            const int64_t m = (in + out) >> 1;
            if (same_row(keys[m])) in = m;
            else out = m;
        }
        const int64_t len = out - i;
        longest = max(longest, (unsigned int)(len < 0x7fffffff ? len : 0x7fffffff));
    }
    longest = __reduce_max_sync(FULL, longest);
    if ((threadIdx.x & 31) == 0 && longest) atomicMax(&f->longest, longest);
}

/* two-word keys to W words */
__global__ void k_io_store(const FKey *keys, int W, int64_t M, uint64_t *out)
{
    const int64_t n = M * W;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = i % W;
        out[i] = t < 2 ? keys[i / W].w[t] : 0ull;
    }
}

int grid_for(int64_t n, int threads)
{
    int64_t g = (n + threads - 1) / threads;
    const int cap = 16 * qw_sm_count();
    if (g > cap) g = cap;
    return (int)(g < 1 ? 1 : g);
}

} // namespace

/* ---- launchers ------------------------------------------------------------------------ */
/* kw: the key words (2, the export layout; 10, the register-faithful layout) */

cudaError_t qw_flat_gather(const QwSimDev &d, const QwBufDev &buf, int inst, int fp32, const double *scale,
                           void *keys, double2 *amps, unsigned long long *counter, int64_t cap, cudaStream_t st, int kw)
{
    const int grid = 4 * qw_sm_count();
    if (kw == NW_FAITH) {
        if (fp32)
            k_f_gather<float2, NW_FAITH><<<grid, 256, 0, st>>>(d, buf, inst, scale, static_cast<FKeyW *>(keys), amps,
                                                               counter, cap);
        else
            k_f_gather<double2, NW_FAITH><<<grid, 256, 0, st>>>(d, buf, inst, scale, static_cast<FKeyW *>(keys), amps,
                                                                counter, cap);
    } else if (fp32) {
        k_f_gather<float2, 2><<<grid, 256, 0, st>>>(d, buf, inst, scale, static_cast<FKey *>(keys), amps, counter, cap);
    } else {
        k_f_gather<double2, 2><<<grid, 256, 0, st>>>(d, buf, inst, scale, static_cast<FKey *>(keys), amps, counter, cap);
    }
    return cudaGetLastError();
}

cudaError_t qw_flat_map(const QwSimDev &d, void *keys, int64_t M, uint32_t ops, int32_t *status, cudaStream_t st,
                        int kw)
{
    if (M <= 0) return cudaSuccess;
    if (kw == NW_FAITH) k_f_map<NW_FAITH><<<grid_for(M, 256), 256, 0, st>>>(d, static_cast<FKeyW *>(keys), M, ops, status);
    else k_f_map<2><<<grid_for(M, 256), 256, 0, st>>>(d, static_cast<FKey *>(keys), M, ops, status);
    return cudaGetLastError();
}

cudaError_t qw_flat_phase(const QwSimDev &d, const void *keys, double2 *amps, int64_t M, cudaStream_t st, int kw)
{
    if (M <= 0) return cudaSuccess;
    if (kw == NW_FAITH)
        k_f_phase<NW_FAITH><<<grid_for(M, 256), 256, 0, st>>>(d, static_cast<const FKeyW *>(keys), amps, M);
    else k_f_phase<2><<<grid_for(M, 256), 256, 0, st>>>(d, static_cast<const FKey *>(keys), amps, M);
    return cudaGetLastError();
}

namespace {
/* work layout of qw_flat_sort, in bytes: the tiles' status words, the
   digit counts of every chunk, the block counters of every pass, two
   compacted-key and two permutation arrays */
struct SortWork {
    uint64_t *stat;
    uint32_t *ghist;
    unsigned int *ctr;
    unsigned long long *acc;
    uint64_t *ck[2];
    uint32_t *ix[2];
    size_t zero_bytes, total;
};

constexpr int SORT_MAXPASSES = 64 * NW_FAITH / 8; /* counters: one a pass, the last for k_f_orand */

size_t align256(size_t b)
{
    return (b + 255) & ~(size_t)255;
}

SortWork sort_work(void *base, int64_t M)
{
    const int64_t n = M < 1 ? 1 : M;
    const int64_t nblk = (n + OS_TILE - 1) / OS_TILE;
    char *p = static_cast<char *>(base);
    SortWork w;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *q = p ? p + off : nullptr;
        off += align256(bytes);
        return q;
    };
    w.stat = reinterpret_cast<uint64_t *>(take((size_t)nblk * 256 * 8));
    w.ghist = reinterpret_cast<uint32_t *>(take((size_t)NW_FAITH * CK_MAXPASS * 256 * 4));
    w.ctr = reinterpret_cast<unsigned int *>(take((size_t)(SORT_MAXPASSES + 1) * 4));
    w.acc = reinterpret_cast<unsigned long long *>(take(2 * NW_FAITH * 8));
    w.zero_bytes = off;
    w.ck[0] = reinterpret_cast<uint64_t *>(take((size_t)n * 8));
    w.ck[1] = reinterpret_cast<uint64_t *>(take((size_t)n * 8));
    w.ix[0] = reinterpret_cast<uint32_t *>(take((size_t)n * 4));
    w.ix[1] = reinterpret_cast<uint32_t *>(take((size_t)n * 4));
    w.total = off;
    return w;
}

/* Stable sort of (keys, amps) by the permuted key of `order` (0: R, 1: H);
 * group: only so far that the groups are contiguous, without the target's bits
 * (the transforms take a group's members in any order; the direct sums of s >
 * 128 in that of the list, so not there) and, where A is known to follow from
 * the other idle registers, without A's -- 30 bits for 46 at N = 16384's R^dag. Two
 * steps there, with T~ and two marginals: 2765 -> 2495 us, the sort's ranks by
 * ballots included.
 * One synchronisation reads which bits vary; they are sorted in chunks of
 * 64, each by 8-bit passes carrying a permutation; the entries are moved
 * once at the end, into tmpk / tmpa (*in_tmp = 1).  A list whose keys are
 * all equal is already sorted (*in_tmp = 0). */
template <int NW>
cudaError_t flat_sort_t(const QwSimDev &d, void *keys, double2 *amps, void *tmpk, double2 *tmpa, int64_t M, int order,
                        int group, void *work, unsigned long long *h, int32_t *status, cudaStream_t st, int *in_tmp)
{
    *in_tmp = 0;
    if (M <= 1) return cudaSuccess;
    if (M > (int64_t)UINT32_MAX) return cudaErrorInvalidValue; /* 32-bit positions */
    const int L = d.L;
    const SortWork w = sort_work(work, M);
    cudaError_t e = cudaMemsetAsync(w.stat, 0, w.zero_bytes, st);
    if (e != cudaSuccess) return e;
    const int othreads = 32 * NW;
    const int ogrid = grid_for(M * NW, othreads);
    const uint64_t *kwords = static_cast<const uint64_t *>(keys);
    unsigned int *done = w.ctr + SORT_MAXPASSES;
    if (order == ORDER_R) k_f_orand<ORDER_R, NW><<<ogrid, othreads, 0, st>>>(kwords, M * NW, L, w.acc, done, h);
    else k_f_orand<ORDER_H, NW><<<ogrid, othreads, 0, st>>>(kwords, M * NW, L, w.acc, done, h);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    /* the varying bits as runs, split into chunks of 64 */
    uint64_t var[NW];
    for (int wi = 0; wi < NW; ++wi) var[wi] = h[wi] & h[NW + wi];
    if (group != QW_SORT_FULL) {
        if (order == ORDER_R) var[0] &= ~1ull;
        else if (d.s <= 128) var[0] &= ~((1ull << L) - 1ull);
    }
    if (group == QW_SORT_GROUP_NO_A) {
        const int pA = flayout(d.nb).pA; /* bits pA .. pA + 15 */
        for (int b = pA; b < pA + 16; ++b) var[b >> 6] &= ~(1ull << (b & 63));
    }
    std::vector<CkRuns> chunks(NW);
    chunks.resize((size_t)qw_sort_chunks(var, NW, chunks.data()));
    if (chunks.empty()) return cudaSuccess;
    const int64_t nblk = (M + OS_TILE - 1) / OS_TILE;
    const int kgrid = grid_for(M, 256);
    const FKeyN<NW> *kin = static_cast<const FKeyN<NW> *>(keys);
    int curix = -1, curck = 0;
    uint64_t tag = 0;
    for (size_t c = 0; c < chunks.size(); ++c) {
        const CkRuns &r = chunks[c];
        uint32_t *gh = w.ghist + c * CK_MAXPASS * 256;
        const uint32_t *perm = curix < 0 ? nullptr : w.ix[curix];
        if (order == ORDER_R) k_f_ckey<ORDER_R, NW><<<kgrid, 256, 0, st>>>(kin, perm, M, L, r, w.ck[curck], gh);
        else k_f_ckey<ORDER_H, NW><<<kgrid, 256, 0, st>>>(kin, perm, M, L, r, w.ck[curck], gh);
        for (int p = 0; p < r.npass; ++p) {
            ++tag;
            const bool wck = p + 1 < r.npass;
            const int outix = curix == 0 ? 1 : 0;
            const uint64_t *ci = w.ck[curck];
            uint64_t *co = w.ck[curck ^ 1];
            uint32_t *xo = w.ix[outix];
            unsigned int *ctr = w.ctr + (tag - 1);
            const uint32_t *ghp = gh + p * 256;
            const unsigned grid = (unsigned)nblk;
            if (curix < 0) {
                if (wck) k_f_onesweep<true, true><<<grid, OS_THREADS, 0, st>>>(ci, nullptr, co, xo, M, 8 * p, ghp, w.stat, tag, ctr, status);
                else k_f_onesweep<true, false><<<grid, OS_THREADS, 0, st>>>(ci, nullptr, co, xo, M, 8 * p, ghp, w.stat, tag, ctr, status);
            } else {
                const uint32_t *xi = w.ix[curix];
                if (wck) k_f_onesweep<false, true><<<grid, OS_THREADS, 0, st>>>(ci, xi, co, xo, M, 8 * p, ghp, w.stat, tag, ctr, status);
                else k_f_onesweep<false, false><<<grid, OS_THREADS, 0, st>>>(ci, xi, co, xo, M, 8 * p, ghp, w.stat, tag, ctr, status);
            }
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            curix = outix;
            if (wck) curck ^= 1;
        }
    }
    k_f_permute<NW><<<kgrid, 256, 0, st>>>(kin, amps, w.ix[curix], static_cast<FKeyN<NW> *>(tmpk), tmpa, M);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    *in_tmp = 1;
    return cudaSuccess;
}
} // namespace

size_t qw_flat_sort_bytes(int64_t M)
{
    return sort_work(nullptr, M).total;
}

cudaError_t qw_flat_sort(const QwSimDev &d, void *keys, double2 *amps, void *tmpk, double2 *tmpa, int64_t M,
                         int order, int group, void *work, unsigned long long *host, int32_t *status, cudaStream_t st,
                         int kw, int *in_tmp)
{
    if (kw == NW_FAITH)
        return flat_sort_t<NW_FAITH>(d, keys, amps, tmpk, tmpa, M, order, group, work, host, status, st, in_tmp);
    return flat_sort_t<2>(d, keys, amps, tmpk, tmpa, M, order, group, work, host, status, st, in_tmp);
}

/* The single-pass kernels' tile sums, zeroed: tiles of `per` inputs */
size_t qw_flat_tiles_bytes(int64_t n)
{
    /* one word per tile; the smallest tiles are the direct sums', 8 groups */
    return sizeof(TileSum) + (size_t)((n + HG_WARPS - 1) / HG_WARPS) * 8;
}

namespace {
cudaError_t tiles_clear(void *ts, int64_t ntiles, cudaStream_t st)
{
    return cudaMemsetAsync(ts, 0, sizeof(TileSum) + (size_t)ntiles * 8, st);
}
} // namespace

cudaError_t qw_flat_rot(const QwSimDev &d, int op, const void *keys, const double2 *amps, int64_t M, void *okeys,
                        double2 *oamps, int64_t cap, void *tiles, unsigned long long *host, int32_t *status,
                        cudaStream_t st, int kw)
{
    if (M <= 0) return cudaSuccess;
    const int64_t nt = (M + RT_THREADS - 1) / RT_THREADS;
    const cudaError_t e = tiles_clear(tiles, nt, st);
    if (e != cudaSuccess) return e;
    TileSum *ts = static_cast<TileSum *>(tiles);
    const unsigned grid = (unsigned)nt;
    if (kw == NW_FAITH) {
        const FKeyW *k = static_cast<const FKeyW *>(keys);
        FKeyW *ok = static_cast<FKeyW *>(okeys);
        if (op == 0) k_f_rot<true, NW_FAITH><<<grid, RT_THREADS, 0, st>>>(d, k, amps, M, ok, oamps, cap, ts, status, host);
        else k_f_rot<false, NW_FAITH><<<grid, RT_THREADS, 0, st>>>(d, k, amps, M, ok, oamps, cap, ts, status, host);
    } else {
        const FKey *k = static_cast<const FKey *>(keys);
        FKey *ok = static_cast<FKey *>(okeys);
        if (op == 0) k_f_rot<true, 2><<<grid, RT_THREADS, 0, st>>>(d, k, amps, M, ok, oamps, cap, ts, status, host);
        else k_f_rot<false, 2><<<grid, RT_THREADS, 0, st>>>(d, k, amps, M, ok, oamps, cap, ts, status, host);
    }
    return cudaGetLastError();
}

cudaError_t qw_flat_starts(const QwSimDev &d, const void *keys, int64_t M, int64_t *starts, void *tiles,
                           unsigned long long *host, int32_t *status, cudaStream_t st, int kw)
{
    if (M <= 0) return cudaSuccess;
    const int64_t nt = (M + ST_THREADS * ST_IPT - 1) / (ST_THREADS * ST_IPT);
    const cudaError_t e = tiles_clear(tiles, nt, st);
    if (e != cudaSuccess) return e;
    TileSum *ts = static_cast<TileSum *>(tiles);
    const unsigned grid = (unsigned)nt;
    if (kw == NW_FAITH)
        k_f_starts<NW_FAITH><<<grid, ST_THREADS, 0, st>>>(d, static_cast<const FKeyW *>(keys), M, starts, ts, status, host);
    else k_f_starts<2><<<grid, ST_THREADS, 0, st>>>(d, static_cast<const FKey *>(keys), M, starts, ts, status, host);
    return cudaGetLastError();
}

namespace {
template <int NW, int R>
cudaError_t launch_hgroups(const QwSimDev &d, const void *keys, const double2 *amps, int64_t M, const int64_t *starts,
                           int64_t G, void *okeys, double2 *oamps, int64_t cap, void *tiles, unsigned long long *host, int32_t *status, cudaStream_t st)
{
    const int64_t per = (int64_t)HG_WARPS * HgIters<R>::n * (d.s < 32 ? 32 / d.s : 1), nt = (G + per - 1) / per;
    const cudaError_t e = tiles_clear(tiles, nt, st);
    if (e != cudaSuccess) return e;
    k_f_hgroups<NW, R><<<(unsigned)nt, 32 * HG_WARPS, 0, st>>>(d, static_cast<const FKeyN<NW> *>(keys), amps, M, starts, G,
                                                             static_cast<FKeyN<NW> *>(okeys), oamps, cap,
                                                             static_cast<TileSum *>(tiles), status, host);
    return cudaGetLastError();
}

/* the fast transform's vector entries a lane: 1 (s <= 32), 2 (64), 4 (128);
   0: the direct sums (s > 128) */
template <int NW>
cudaError_t launch_hgroups_s(const QwSimDev &d, const void *keys, const double2 *amps, int64_t M, const int64_t *starts, int64_t G,
                             void *okeys, double2 *oamps, int64_t cap, void *tiles, unsigned long long *host, int32_t *status, cudaStream_t st)
{
    if (d.s <= 32) return launch_hgroups<NW, 1>(d, keys, amps, M, starts, G, okeys, oamps, cap, tiles, host, status, st);
    if (d.s == 64) return launch_hgroups<NW, 2>(d, keys, amps, M, starts, G, okeys, oamps, cap, tiles, host, status, st);
    if (d.s == 128) return launch_hgroups<NW, 4>(d, keys, amps, M, starts, G, okeys, oamps, cap, tiles, host, status, st);
    return launch_hgroups<NW, 0>(d, keys, amps, M, starts, G, okeys, oamps, cap, tiles, host, status, st);
}
} // namespace

cudaError_t qw_flat_hgroups(const QwSimDev &d, const void *keys, const double2 *amps, int64_t M, const int64_t *starts, int64_t G,
                            void *okeys, double2 *oamps, int64_t cap, void *tiles, unsigned long long *host,
                            int32_t *status, cudaStream_t st, int kw)
{
    if (G <= 0) return cudaSuccess;
    if (kw == NW_FAITH)
        return launch_hgroups_s<NW_FAITH>(d, keys, amps, M, starts, G, okeys, oamps, cap, tiles, host, status, st);
    return launch_hgroups_s<2>(d, keys, amps, M, starts, G, okeys, oamps, cap, tiles, host, status, st);
}

cudaError_t qw_flat_readout(const QwSimDev &d, const void *keys, const double2 *amps, int64_t M, const QwStepArgs &a,
                            cudaStream_t st, int kw)
{
    if (M <= 0) return cudaSuccess;
    if (kw == NW_FAITH)
        k_f_readout<NW_FAITH><<<grid_for(M, 256), 256, 0, st>>>(d, static_cast<const FKeyW *>(keys), amps, M, a);
    else k_f_readout<2><<<grid_for(M, 256), 256, 0, st>>>(d, static_cast<const FKey *>(keys), amps, M, a);
    return cudaGetLastError();
}

cudaError_t qw_flat_scatter(const QwSimDev &d, const QwBufDev &out, int fp32, const void *keys, const double2 *amps,
                            int64_t M, int32_t *status, unsigned int *maxrow, double *norm, cudaStream_t st, int kw)
{
    if (M <= 0) return cudaSuccess;
    if (kw == NW_FAITH) {
        const FKeyW *k = static_cast<const FKeyW *>(keys);
        if (fp32)
            k_f_scatter<float2, NW_FAITH><<<grid_for(M, 256), 256, 0, st>>>(d, out, k, amps, M, status, maxrow, norm);
        else
            k_f_scatter<double2, NW_FAITH><<<grid_for(M, 256), 256, 0, st>>>(d, out, k, amps, M, status, maxrow, norm);
    } else {
        const FKey *k = static_cast<const FKey *>(keys);
        if (fp32) k_f_scatter<float2, 2><<<grid_for(M, 256), 256, 0, st>>>(d, out, k, amps, M, status, maxrow, norm);
        else k_f_scatter<double2, 2><<<grid_for(M, 256), 256, 0, st>>>(d, out, k, amps, M, status, maxrow, norm);
    }
    return cudaGetLastError();
}

cudaError_t qw_flat_finish(const QwStepArgs &a, const double *norm, const int64_t *counts, cudaStream_t st)
{
    k_f_finish<<<1, 1, 0, st>>>(a, norm, (unsigned long long)counts[0], (unsigned long long)counts[1],
                                (unsigned long long)counts[2], (unsigned long long)counts[3],
                                (unsigned long long)counts[4]);
    return cudaGetLastError();
}

cudaError_t qw_io_load(const QwSimDev &d, const uint64_t *in, int words, int64_t M, void *keys, QwIoFlags *f,
                       cudaStream_t st)
{
    if (M <= 0) return cudaSuccess;
    k_io_load<<<grid_for(M, 256), 256, 0, st>>>(in, words, M, flayout(d.nb), (uint32_t)d.ninst, static_cast<FKey *>(keys), f);
    return cudaGetLastError();
}

cudaError_t qw_io_order(const QwSimDev &d, const void *keys, int64_t M, QwIoFlags *f, cudaStream_t st)
{
    if (M <= 0) return cudaSuccess;
    k_io_order<<<grid_for(M, 256), 256, 0, st>>>(static_cast<const FKey *>(keys), M, flayout(d.nb), f);
    return cudaGetLastError();
}

cudaError_t qw_io_store(const void *keys, int words, int64_t M, uint64_t *out, cudaStream_t st)
{
    if (M <= 0) return cudaSuccess;
    k_io_store<<<grid_for(M * words, 256), 256, 0, st>>>(static_cast<const FKey *>(keys), words, M, out);
    return cudaGetLastError();
}

/* register-faithful layout of a simulator: address width and field positions */
static FaithLayout faith_layout(const QwSimDev &d)
{
    FaithLayout F;
    const uint64_t ns = (uint64_t)d.n_single * (uint64_t)d.s;
    const uint64_t top = ns + (((uint64_t)1 << d.nb) * (uint64_t)d.s) + ((uint64_t)1 << d.nb) + 1;
    int b = 0;
    while (((uint64_t)1 << b) < top) b++;
    F.aw = b;
    F.p_addr = 128;
    F.p_left = F.p_addr + b;
    F.p_right = F.p_left + b;
    F.p_mid = F.p_right + b;
    F.p_midval = F.p_mid + b;
    F.p_flag = F.p_midval + 16;
    F.p_cl = F.p_flag + 1;
    F.p_ce = F.p_cl + 1;
    F.p_stk = F.p_ce + 1;
    F.frame = b + 18;
    return F;
}

int qw_faithful_layout(const QwSimDev &d, int *addr_bits, int *layout_bits)
{
    const FaithLayout F = faith_layout(d);
    if (addr_bits) *addr_bits = F.aw;
    const int bits = F.p_stk + (d.L + 1) * F.frame;
    if (layout_bits) *layout_bits = bits;
    return bits <= 64 * NW_FAITH && d.L + 1 <= QW_FQ_FRAMES;
}

cudaError_t qw_faithful_run(const QwSimDev &d, void *keys, int64_t M, const int32_t *ops, int n, int idle,
                            int32_t *status, cudaStream_t st)
{
    if (M <= 0 || n <= 0) return cudaSuccess;
    if (n > QW_FQ_RUN) return cudaErrorInvalidValue;
    uint64_t packed = 0;
    bool qbs = false;
    for (int i = 0; i < n; ++i) {
        packed |= (uint64_t)ops[i] << (4 * i);
        qbs = qbs || ops[i] == FQ_QBS_FWD || ops[i] == FQ_QBS_BWD;
    }
    FKeyW *k = static_cast<FKeyW *>(keys);
    const int grid = grid_for(M, FQ_THREADS);
    if (qbs) k_fq<true><<<grid, FQ_THREADS, 0, st>>>(d, k, M, packed, faith_layout(d), idle, status);
    else k_fq<false><<<grid, FQ_THREADS, 0, st>>>(d, k, M, packed, faith_layout(d), idle, status);
    return cudaGetLastError();
}

cudaError_t qw_faithful_export(const QwSimDev &d, const void *keys, int64_t M, uint64_t *table, cudaStream_t st)
{
    if (M <= 0) return cudaSuccess;
    k_fq_export<<<grid_for(M, 256), 256, 0, st>>>(d, static_cast<const FKeyW *>(keys), M, faith_layout(d), table);
    return cudaGetLastError();
}

cudaError_t qw_faithful_check_idle(const QwSimDev &d, const void *keys, int64_t M, int32_t *status, cudaStream_t st)
{
    if (M <= 0) return cudaSuccess;
    k_fq_check_idle<<<grid_for(M, 256), 256, 0, st>>>(static_cast<const FKeyW *>(keys), M, faith_layout(d).p_addr,
                                                       status);
    return cudaGetLastError();
}
