/*
 * qw_internal.h -- device data layout shared by the kernels (qw_kernels.cu)
 * and the host side of the C ABI (qw_api.cpp).
 *
 * Layout in HBM.  The state is bucketed by row: one bucket per (inst, jc, j, b1)
 * value, i.e. per value of the registers that T~, P and T~^dag never change
 * and that every QRAM access of those operators indexes (row j).  A bucket
 * holds up to cap_row branches as
 *   key[b * cap_row + i]  uint64, the "local" registers (k, kc, A, b2) packed
 *                         in the R layout below,
 *   amp[b * cap_row + i]  double2 or float2,
 *   count[b]              int32 branches present.
 * Rows with jc = 0 have dense buckets: inst_bkt[inst] + (j << 1 | b1).  Rows
 * with jc != 0 (garbage subspace) go to spill buckets dense_buckets + slot,
 * slot found by open addressing on the packed row key in spill[].
 * Three such buffers rotate: a step reads X_t, writes X_{t+1} and clears
 * X_{t+2}; X_t stays intact until the step after next.
 *
 * Local-key layouts (bit 0 first):
 *   R layout: b2 | k (nb) | kc (nb) | A (16)            -- b2-pairs adjacent
 *   H layout: k_low (L) | b2 | k_high (nb-L) | kc | A   -- Hadamard groups adjacent
 * Both keep kc and A at bits 1+nb and above.
 */
#ifndef QW_INTERNAL_H
#define QW_INTERNAL_H

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/qwalk.h"

#define QW_SPILL_EMPTY (~0ull)

/* device status word bits */
#define QW_ST_ROW_OVERFLOW 1   /* a bucket received more than cap_row branches */
#define QW_ST_WARP_OVERFLOW 2  /* a row outgrew the on-chip row buffer */
#define QW_ST_SPILL_FULL 4     /* no free spill slot for a jc != 0 row */
#define QW_ST_ANCILLA 8        /* register A not zero where it must be */
#define QW_ST_NOT_BTILDE 16    /* T~ at initialisation met a row that was not |b~> */
#define QW_ST_OUTBOX_FULL 32   /* a partition's outbox toward another overflowed */
#define QW_ST_POS_UNREP 64     /* a branch the positional layout has no position for */
#define QW_ST_SORT_WAIT 128    /* the flat path's radix sort gave up waiting for a tile's count */
#define QW_ST_POS_FULL 256     /* a packed state has branches with b1 = b2 = 1 (pos_pack) */
#define QW_ST_GRID_WAIT 512    /* a positional step gave up waiting for the other blocks */

/* A branch sent by S to a row another partition owns: its row key
   (qw_rowkey), its local registers (R layout) and its amplitude in FP64. */
struct QwPartEntry {
    uint64_t rowkey, local;
    double re, im;
};

/* per-step branch counters (index into QwStepArgs.stats) */
#define QW_STAT_ROWS 0      /* rows processed */
#define QW_STAT_IN 1        /* branches entering the step (input of R^dag) */
#define QW_STAT_RDAG 2      /* after R^dag (input of the H P H stage) */
#define QW_STAT_H1 3        /* after the first H (literal mode only) */
#define QW_STAT_HPH 4       /* after H P H (input of R) */
#define QW_STAT_OUT 5       /* after R (branches written) */
#define QW_STAT_STEPS 6     /* clean steps counted */
#define QW_NSTAT 8

/* step kernel modes */
#define QW_MODE_WALK_FUSED 0   /* T~^dag, (H P H as one reflection), T~, S */
#define QW_MODE_WALK_LITERAL 1 /* T~^dag, H, P, H, T~, S */
#define QW_MODE_T 2            /* T~ only, in place on a bucket range */
#define QW_MODE_WALK_FUSED_PF 3 /* fused step, row loop software-pipelined */
#define QW_MODE_WALK_SEG 4      /* fused step, both rows of a j as one segment */
#define QW_MODE_WALK_SEG_PF 5   /* segments, software-pipelined */
#define QW_MODE_WALK_SLOT 6     /* fused step, one lane per QRAM slot (s = 8, 16, 32) */
#define QW_MODE_WALK_FLAT 7     /* the literal step on one globally sorted branch list (qw_flat.cu) */
#define QW_MODE_WALK_FAITHFUL 8 /* the flat step with every working register in a 10-word key */
#define QW_MODE_WALK_POS 9      /* the state held by position, one lane per QRAM slot (s = 4 .. 64) */

struct QwSimDev {
    int nb, s, L, ninst;
    int n_single;  /* N of the instance when ninst == 1 (tables not read then) */
    int cap_row;   /* branches per bucket */
    int warp_cap;  /* on-chip branches per warp */
    int spill_slots;          /* power of two */
    int64_t dense_buckets;    /* sum over instances */
    int64_t total_buckets;    /* dense + spill */
    double tau2;              /* prune threshold squared */
    uint64_t tau_hi_bits;     /* bits of tau (1 + 2^-30): |x| above it => kept */
    uint64_t tau_lo_bits;     /* bits of tau sqrt(1/2) (1 - 2^-30): |x|,|y| at most it => pruned */
    float tau2f;              /* tau^2 as float (complex64 path) */
    float thr32;              /* at least tau and 2^-100 (2^-60 for complex64, whose squares it keeps normal): above it (plus the approximation's error) => kept */
    int rot_calc;             /* rot_bits == 0: the FP32 rotation pairs follow from the code alone */
    double inv_sqrt_s;        /* 1 / sqrt(s) */
    double two_over_s;        /* 2 / s */
    const uint32_t *img;      /* QRAM words: column << 16 | Q1.15 value */
    const double2 *fg;        /* per Q1.15 code: (sqrt|a|, sqrt(1-|a|)) */
    const float4 *fg32;       /* the same as float pairs: (hi, lo) of each, hi + lo ~ 48 bits */
    const void *slot_rot;     /* per QRAM slot: its code's entry of fg (FP64) or fg32 (FP32) */
    const int32_t *inst_n;    /* N per instance */
    const int64_t *inst_img;  /* image offset per instance */
    const int64_t *inst_bkt;  /* first dense bucket per instance, ninst + 1 entries */
    const uint16_t *unit_inst; /* instance of dense bucket pair u (buckets 2u, 2u + 1); ninst > 1 */
    /* row-partitioned walk (single instance): rows (jc = 0, j < N) in blocks of
       part_rows per partition, the others by a hash of (jc, j); S sends a
       branch whose new row another partition owns to that partition's
       outbox segment (outbox_cap entries each) */
    int nparts, part;
    int64_t part_rows;
    QwPartEntry *outbox;
    unsigned long long *outbox_count;
    int64_t outbox_cap;
    /* positional layout (qw_pos.cuh): the rows j < N of all instances in order,
       row g (instance i, g = inst_img[i] / s + j) of pos_rows; entries g s + l
       (slot l of row g), then the extras of row g at pos_rows s + pos_xptr[g] ..
       pos_xptr[g + 1], pos_T entries in all; pos_dst[g s + l]: the entry of the
       branch k = j in row col(j, l) of the instance, bit 31: j > col(j, l);
       pos_xdst[e]: the slot (x, l_x) of extra e of row j, whose column is j
       while row j holds no column x; pos_rowinst[g]: the instance of row g
       (null with one) */
    int64_t pos_rows, pos_T;
    const uint32_t *pos_dst;
    const uint32_t *pos_xptr;
    const uint32_t *pos_xdst;
    const uint16_t *pos_rowinst;
};

struct QwBufDev {
    uint64_t *key;
    void *amp;
    int32_t *count;
    uint64_t *spill;
};

struct QwStepArgs {
    int mode;
    int renorm;
    int64_t bucket_lo, bucket_hi; /* bucket range processed (MODE_T) */
    const double *scale_in;  /* amplitude scale of the input (renormalisation), nullable */
    double *partials;        /* per-block norm partial sums */
    unsigned int *done_ctr;  /* blocks finished (last block reduces partials) */
    double *norm_out;        /* ||output||^2 */
    double *scale_out;       /* sqrt(target / norm_out) when renorm, else 1 */
    const double *renorm_target; /* sum of the instances' initial ||b||^2 */
    int64_t *steps_done;     /* incremented by each step that completes cleanly */
    int32_t *status;
    unsigned long long *stats; /* QW_STAT_* counters, accumulated (nullable) */
    double2 *qls_y;          /* flag-0 accumulator (nullable) */
    const double *qls_coefs; /* Y += qls_coefs[*qls_j] * Pi_0 tau at this step's midpoint */
    const int64_t *qls_j;    /* index of the current QLS term (advanced by k_qls_norm) */
    double *qls_p;           /* p_j (written by the positional kernel's own terms) */
    int qls_readout;
    int32_t *deferred;          /* slot kernel: units left to the row pipeline (dense unit u,
                                   or 0x80000000 | garbage-row slot), run by the last block */
    unsigned int *deferred_ctr; /* entries in deferred (reset by the last block) */
    unsigned int *work_ctr;     /* slot kernel: groups claimed beyond each warp's first
                                   (reset by the last block) */
};

/* positional steps: one launch runs nsteps of them, in -> out0 -> out1 -> out0
   ...; with words, blocks wait for one another between steps (a cooperative
   launch), otherwise nsteps is 1 */
struct QwPosArgs {
    const void *in;
    void *out0, *out1;
    int nsteps;
    int qls;                  /* QLS terms of two steps, read out on the second */
    int64_t qls_term;         /* index of the first */
    unsigned long long epoch; /* of the first step: its barrier's turn is epoch & 3 */
    unsigned long long *words; /* [4][2]: the barrier's words; or null */
    double *extra;            /* [4]: norm shares no word takes */
    double *pshare;           /* [2][grid]: the blocks' shares of p_j */
};
/* 8-byte words of the barrier's memory: words, extra (on a line of its own), then pshare */
#define QW_POS_EXTRA 16
#define QW_POS_WORDS 32
struct QwScalarWords { /* 8-byte words of the simulator's scalars a kernel sets */
    unsigned long long *dst;
    int n;
    unsigned long long w[20];
};
struct QwPosPlan {
    int grid, warps; /* blocks, warps a block */
    int tab;         /* the matrix's tables fit shared memory */
    int coop;        /* the device takes cooperative launches */
    size_t smem;
    int cl, cl_warps; /* runs go to one cluster of cl blocks (0: to the grid) */
    size_t cl_smem;
};

/* launchers (qw_kernels.cu); all return cudaGetLastError() of the launch */
int qw_sm_count(void);
cudaError_t qw_launch_step(const QwSimDev &d, const QwBufDev &in, const QwBufDev &out,
                           const QwBufDev &clear, const QwStepArgs &a, int fp32, int grid,
                           cudaStream_t st);
/* whether the slot kernel (QW_MODE_WALK_SLOT) covers this sparsity */
int qw_slot_supported(const QwSimDev &d);
/* whether the positional layout (QW_MODE_WALK_POS) covers this s (4 .. 64) */
int qw_pos_supported(const QwSimDev &d);
/* dynamic shared memory per block of the step kernel of `mode` */
size_t qw_step_smem_bytes(const QwSimDev &d, int fp32, int mode);
/* positional layout (qw_pos.cuh; 32: complex64, 64: complex128): the launch
   shape, walk steps, T~|b~> written into rows g0 .. g0 + n (x0, nx: their
   extras), a register marginal of those rows (j and k write every bin, the
   others add to zeroed ones; probs and stat_dst may be pinned host memory),
   and the conversions
   from and to the row buckets (pack: pbuf zeroed by the caller, a branch
   without a place sets QW_ST_POS_UNREP; unpack: the buckets cleared by the
   caller); full: the state has b1 = b2 = 1
   branches */
#define QW_POS_DECLARE(SUFFIX)                                                                                        \
    QwPosPlan qw_pos_plan##SUFFIX(const QwSimDev &d);                                                                 \
    cudaError_t qw_launch_walk_pos##SUFFIX(const QwSimDev &d, const QwPosPlan &pl, const QwPosArgs &p,                \
                                           const QwStepArgs &a, int full, cudaStream_t st);                           \
    cudaError_t qw_launch_tinit_pos##SUFFIX(const QwSimDev &d, void *pbuf, int full, int64_t g0, int64_t n,           \
                                            int64_t x0, int64_t nx, const double *b_re, const double *b_im,           \
                                            const double *scale, const QwScalarWords &words, cudaStream_t st);        \
    cudaError_t qw_launch_measure_pos##SUFFIX(const QwSimDev &d, const void *pbuf, int full, int64_t g0, int64_t n,   \
                                              const double *scale, int reg, double *probs, int64_t len,               \
                                              const unsigned long long *stat_src, unsigned long long *stat_dst,       \
                                              cudaStream_t st);                                                       \
    cudaError_t qw_launch_pos_pack##SUFFIX(const QwSimDev &d, const QwBufDev &buf, void *pbuf, int32_t *status,       \
                                           cudaStream_t st);                                                          \
    cudaError_t qw_launch_pos_unpack##SUFFIX(const QwSimDev &d, const void *pbuf, int full, const QwBufDev &buf,      \
                                             int32_t *status, cudaStream_t st);
QW_POS_DECLARE(32)
QW_POS_DECLARE(64)
#undef QW_POS_DECLARE
static inline QwPosPlan qw_pos_plan(const QwSimDev &d, int fp32) { return fp32 ? qw_pos_plan32(d) : qw_pos_plan64(d); }
static inline cudaError_t qw_launch_walk_pos(const QwSimDev &d, const QwPosPlan &pl, const QwPosArgs &p,
                                             const QwStepArgs &a, int fp32, int full, cudaStream_t st)
{
    return fp32 ? qw_launch_walk_pos32(d, pl, p, a, full, st) : qw_launch_walk_pos64(d, pl, p, a, full, st);
}
static inline cudaError_t qw_launch_tinit_pos(const QwSimDev &d, void *pbuf, int full, int64_t g0, int64_t n,
                                              int64_t x0, int64_t nx, const double *b_re, const double *b_im,
                                              const double *scale, const QwScalarWords &words, int fp32,
                                              cudaStream_t st)
{
    return fp32 ? qw_launch_tinit_pos32(d, pbuf, full, g0, n, x0, nx, b_re, b_im, scale, words, st)
                : qw_launch_tinit_pos64(d, pbuf, full, g0, n, x0, nx, b_re, b_im, scale, words, st);
}
static inline cudaError_t qw_launch_measure_pos(const QwSimDev &d, const void *pbuf, int full, int64_t g0, int64_t n,
                                                int fp32, const double *scale, int reg, double *probs, int64_t len,
                                                const unsigned long long *stat_src, unsigned long long *stat_dst,
                                                cudaStream_t st)
{
    return fp32 ? qw_launch_measure_pos32(d, pbuf, full, g0, n, scale, reg, probs, len, stat_src, stat_dst, st)
                : qw_launch_measure_pos64(d, pbuf, full, g0, n, scale, reg, probs, len, stat_src, stat_dst, st);
}
static inline cudaError_t qw_launch_pos_pack(const QwSimDev &d, const QwBufDev &buf, void *pbuf, int fp32,
                                             int32_t *status, cudaStream_t st)
{
    return fp32 ? qw_launch_pos_pack32(d, buf, pbuf, status, st) : qw_launch_pos_pack64(d, buf, pbuf, status, st);
}
static inline cudaError_t qw_launch_pos_unpack(const QwSimDev &d, const void *pbuf, int full, const QwBufDev &buf,
                                               int fp32, int32_t *status, cudaStream_t st)
{
    return fp32 ? qw_launch_pos_unpack32(d, pbuf, full, buf, status, st)
                : qw_launch_pos_unpack64(d, pbuf, full, buf, status, st);
}
int qw_step_grid(const QwSimDev &d, int fp32, int mode);
cudaError_t qw_launch_clear(const QwSimDev &d, const QwBufDev &buf, int64_t lo, int64_t hi,
                            int clear_spill, cudaStream_t st);
cudaError_t qw_launch_init_b(const QwSimDev &d, const QwBufDev &buf, int inst, const double *b_re,
                             const double *b_im, int n, int fp32, const double *scale, cudaStream_t st);
cudaError_t qw_launch_tinit(const QwSimDev &d, const QwBufDev &buf, int64_t lo, int64_t hi, int fp32,
                            int32_t *status, cudaStream_t st);
cudaError_t qw_launch_measure(const QwSimDev &d, const QwBufDev &buf, int inst, int fp32,
                              const double *scale, int reg, double *probs, int64_t len,
                              cudaStream_t st);
/* pbuf (nullable): read rows g0 .. g0 + pn of the positional layout (pfull:
   b1 = b2 = 1 branches too) instead of buf */
cudaError_t qw_launch_measure_noalloc(const QwSimDev &d, const QwBufDev &buf, int inst, int fp32,
                                      const double *scale, int reg, double *host_probs,
                                      int64_t len, int device, cudaStream_t st, const void *pbuf = nullptr,
                                      int pfull = 0, int64_t g0 = 0, int64_t pn = 0);
cudaError_t qw_launch_count(const QwSimDev &d, const QwBufDev &buf, int inst,
                            unsigned long long *counter, cudaStream_t st);
cudaError_t qw_launch_qls_norm(const double2 *y, int n, double *p, int64_t *jctr, cudaStream_t st);
/* copy buffer `from` (row capacity cap_old) into new key/amp arrays laid out
   with d.cap_row entries per bucket */
cudaError_t qw_launch_regrow(const QwSimDev &d, const QwBufDev &from, int cap_old, uint64_t *key_new, void *amp_new,
                             int fp32, cudaStream_t st);

/* flat, globally sorted step (qw_flat.cu): keys are packed register keys of
   kw 64-bit words (2: the qw_state_export layout; 10: the register-faithful
   layout with the working registers above bit 128), amplitudes complex FP64;
   see qw_flat.cu for each stage */
#define QW_FLAT_OSDAG 1u
#define QW_FLAT_OA 2u
#define QW_FLAT_OS 3u
#define QW_FLAT_S 4u
#define QW_FLAT_A0 5u /* check A = 0 */
#define QW_FAITH_WORDS 10
/* inst >= 0: that instance's branches only */
cudaError_t qw_flat_gather(const QwSimDev &d, const QwBufDev &buf, int inst, int fp32, const double *scale,
                           void *keys, double2 *amps, unsigned long long *counter, int64_t cap, cudaStream_t st, int kw);
cudaError_t qw_flat_map(const QwSimDev &d, void *keys, int64_t M, uint32_t ops, int32_t *status, cudaStream_t st,
                        int kw);
cudaError_t qw_flat_phase(const QwSimDev &d, const void *keys, double2 *amps, int64_t M, cudaStream_t st, int kw);
/* stable sort by the permuted key (order 0: R, 1: H); work holds
   qw_flat_sort_bytes(M); host: 2 kw words of pinned memory for which bits vary
   (synchronises to read them); the result is left in tmpk / tmpa when *in_tmp */
size_t qw_flat_sort_bytes(int64_t M);
#define QW_SORT_FULL 0       /* by every register */
#define QW_SORT_GROUP 1      /* the target's bits left out: groups contiguous */
#define QW_SORT_GROUP_NO_A 2 /* A's too: it follows from the other idle registers */
cudaError_t qw_flat_sort(const QwSimDev &d, void *keys, double2 *amps, void *tmpk, double2 *tmpa, int64_t M,
                         int order, int group, void *work, unsigned long long *host, int32_t *status, cudaStream_t st,
                         int kw, int *in_tmp);
/* Scratch of a single-pass kernel over n entries or groups; it leaves the number
   of its outputs in *host (pinned), and a 1 in host[QW_TOTAL_WAIT] where one of its
   waits gave up: its outputs then have holes, which hold no keys. */
#define QW_TOTAL_WAIT 3
size_t qw_flat_tiles_bytes(int64_t n);
/* op 0 (R^dag) and 1 (R) on the sorted list: the kept outputs (up to 2 M; cap
   is the room in okeys / oamps) */
cudaError_t qw_flat_rot(const QwSimDev &d, int op, const void *keys, const double2 *amps, int64_t M, void *okeys,
                        double2 *oamps, int64_t cap, void *tiles, unsigned long long *host, int32_t *status,
                        cudaStream_t st, int kw);
/* the Hadamard stage's groups: the first member of each (their number G is the
   kernel's total), starts[G] = M; starts has room for M + 1 */
cudaError_t qw_flat_starts(const QwSimDev &d, const void *keys, int64_t M, int64_t *starts, void *tiles,
                           unsigned long long *host, int32_t *status, cudaStream_t st, int kw);
/* H on the G groups: the kept outputs (up to G s) */
cudaError_t qw_flat_hgroups(const QwSimDev &d, const void *keys, const double2 *amps, int64_t M, const int64_t *starts, int64_t G,
                            void *okeys, double2 *oamps, int64_t cap, void *tiles, unsigned long long *host,
                            int32_t *status, cudaStream_t st, int kw);
cudaError_t qw_flat_readout(const QwSimDev &d, const void *keys, const double2 *amps, int64_t M, const QwStepArgs &a,
                            cudaStream_t st, int kw);
cudaError_t qw_flat_scatter(const QwSimDev &d, const QwBufDev &out, int fp32, const void *keys, const double2 *amps,
                            int64_t M, int32_t *status, unsigned int *maxrow, double *norm, cudaStream_t st, int kw);
/* state import and export: the caller's keys of `words` 64-bit words to the
   two-word layout and back, and what an import has to know of its list */
struct QwIoFlags {
    double norm;                  /* (the scatter's, unused) */
    unsigned int maxrow, longest; /* longest: branches of the longest row (sorted list) */
    int32_t status;               /* the sort's */
    int32_t bad, unsorted, dup;
};
cudaError_t qw_io_load(const QwSimDev &d, const uint64_t *in, int words, int64_t M, void *keys, QwIoFlags *f,
                       cudaStream_t st);
cudaError_t qw_io_order(const QwSimDev &d, const void *keys, int64_t M, QwIoFlags *f, cudaStream_t st);
cudaError_t qw_io_store(const void *keys, int words, int64_t M, uint64_t *out, cudaStream_t st);
cudaError_t qw_flat_finish(const QwStepArgs &a, const double *norm, const int64_t *counts, cudaStream_t st);
/* register-faithful sub-operations on 10-word keys (op codes QW_FQ_* of qwalk.h) */
int qw_faithful_layout(const QwSimDev &d, int *addr_bits, int *layout_bits);
#define QW_FQ_RUN 16 /* sub-operations of one launch */
cudaError_t qw_faithful_run(const QwSimDev &d, void *keys, int64_t M, const int32_t *ops, int n, int idle,
                            int32_t *status, cudaStream_t st);
cudaError_t qw_faithful_check_idle(const QwSimDev &d, const void *keys, int64_t M, int32_t *status, cudaStream_t st);
cudaError_t qw_faithful_export(const QwSimDev &d, const void *keys, int64_t M, uint64_t *table, cudaStream_t st);
/* the other partitions' outbox segments toward this one (entries and device
   counts, cap entries each) and the norm slots of all parts' last step */
struct QwPartSources {
    const QwPartEntry *e[64];
    const unsigned long long *count[64];
    int n;
    int64_t cap;
};
struct QwPartNorms {
    const double *norm[64];
    int n;
};
cudaError_t qw_launch_part_gather(const QwSimDev &d, const QwBufDev &buf, const QwPartSources &src, int fp32,
                                  int32_t *status, cudaStream_t st);
cudaError_t qw_launch_part_scale(const QwPartNorms &nm, const double *target, double *scale_out, int renorm,
                                 cudaStream_t st);
cudaError_t qw_launch_part_inbox(const QwSimDev &d, const QwBufDev &buf, const QwPartEntry *e, int64_t count, int fp32,
                                 int32_t *status, cudaStream_t st);

/* Partition owning row (jc, j) of a row-partitioned walk: blocks of
 * part_rows rows for jc = 0, j < N; a hash of (jc, j) otherwise (the rows
 * only states outside the walk's subspace reach). */
__host__ __device__ static inline int qw_part_owner_of(const QwSimDev &d, uint32_t jc, uint32_t j)
{
    if (jc == 0 && j < (uint32_t)d.n_single) return (int)((int64_t)j / d.part_rows);
    uint64_t x = ((uint64_t)jc << 20) | (uint64_t)j;
    x ^= x >> 33;
    x *= 0xff51afd7ed558ccdull;
    x ^= x >> 33;
    return (int)(x % (uint64_t)d.nparts);
}

/* packed row key: inst << 40 | jc << 20 | j << 1 | b1  (nb <= 19) */
__host__ __device__ static inline uint64_t qw_rowkey(uint32_t inst, uint32_t jc, uint32_t j,
                                                     uint32_t b1)
{
    return ((uint64_t)inst << 40) | ((uint64_t)jc << 20) | ((uint64_t)j << 1) | (uint64_t)b1;
}

#endif /* QW_INTERNAL_H */
