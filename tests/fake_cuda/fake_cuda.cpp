/*
 * The CUDA runtime and the kernel launchers as qw_api.cpp sees them, on the
 * host: device memory is host memory, every call completes at once, and a
 * device clock advances by what the tests say a launch costs.  The launchers
 * compute no walk; they keep the simulator's scalars (steps done, status) as
 * the kernels do, so that the host side's decisions can be tested without a
 * GPU, the ones after a failure on the device included.
 */
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <vector>

#include "qw_internal.h"

namespace {

struct Fake {
    double clock_us = 0.0;
    double step_us[16] = {0};   /* one bucket step, by mode */
    double run_us = 0.0;        /* one step of a positional run */
    double single_us = 0.0;     /* a positional step launched alone */
    double launch_us = 0.0;     /* what a run's launch takes beside its steps */
    double first_us = 0.0;      /* what the first launch of each kind takes on top */
    std::map<int, int> launched; /* launches by mode (a positional run: 100) */
    int fail_malloc = -1;       /* device allocations until one fails; -1: none does */
    int64_t bytes = 0, room = -1; /* of the device allocations; at most (-1: no limit) */
    std::vector<uint64_t> list; /* keys, then amplitudes' real parts, of the last two-word scatter */
    cudaError_t last = cudaSuccess;
    int give_up = 0;            /* the next positional launch gives up its wait */
    int status_bits = 0;        /* the next bucket step or scatter sets these */
    int flat_wait = 0;          /* the next single-pass launch of the flat path gives up */
    int64_t map_most = 0;       /* entries of the longest list given to qw_flat_map */
    size_t pinned_most = 0;     /* the largest pinned allocation */
    int64_t live = 0;           /* device allocations not yet freed */
    int64_t sync_copies = 0;    /* cudaMemcpy: ordered on the default stream alone */
    bool pending = false;       /* default-stream work that need not be done when its call returns */
    int64_t unordered = 0;      /* kernels launched meanwhile (on another stream, as the tests read it) */
    int capturing = 0;
    unsigned long long words[8] = {0}; /* the barrier words a positional run started on */
    int64_t tinits = 0;
    std::map<void *, size_t> sizes; /* of the device allocations */
    int64_t overruns = 0;           /* row buckets shorter than cap_row says, as a clear of them finds */
    int refuse = 0;                 /* the next positional launch is refused */
    unsigned long long epoch = 0;   /* of the last one that was not */
    int64_t run_steps = 0;          /* steps of the runs since the last reset */
    unsigned int longest = 0;       /* an imported list's longest row */
    double target = 0.0; /* the renormalisation target of the last step */
} F;

template <typename T> T *handle() { return reinterpret_cast<T *>(std::malloc(16)); }

cudaError_t done(cudaError_t e = cudaSuccess)
{
    if (e != cudaSuccess) F.last = e;
    return e;
}

cudaError_t take(void **p, size_t n)
{
    *p = nullptr;
    if (F.fail_malloc == 0 || (F.room >= 0 && F.bytes + (int64_t)n > F.room)) return done(cudaErrorMemoryAllocation);
    if (F.fail_malloc > 0) --F.fail_malloc;
    *p = std::calloc(n ? n : 1, 1);
    F.sizes[*p] = n;
    F.bytes += (int64_t)n;
    ++F.live;
    return cudaSuccess;
}

cudaError_t give(void *p)
{
    if (p) {
        --F.live;
        F.bytes -= (int64_t)F.sizes[p];
    }
    std::free(p);
    return cudaSuccess;
}

/* what every launcher ends with: an error of an earlier call not yet taken shows here */
cudaError_t launch(int kind, double us)
{
    F.unordered += F.pending;
    F.clock_us += us + (F.launched[kind]++ == 0 ? F.first_us : 0.0);
    const cudaError_t e = F.last;
    F.last = cudaSuccess;
    return e;
}

} // namespace

extern "C" {

Fake *fake_state() { return &F; }
void fake_reset() { F = Fake{}; }
void fake_set_step(int mode, double us) { F.step_us[mode] = us; }
void fake_set_times(double run, double single, double launch_, double first)
{
    F.run_us = run;
    F.single_us = single;
    F.launch_us = launch_;
    F.first_us = first;
}
void fake_fail_malloc(int after) { F.fail_malloc = after; }
void fake_room(int64_t more) { F.room = more < 0 ? -1 : F.bytes + more; }
void fake_longest(int n) { F.longest = (unsigned int)n; }
uint64_t fake_listed(int64_t i) { return F.list.at((size_t)i); }
void fake_give_up(int n) { F.give_up = n; }
void fake_status(int bits) { F.status_bits = bits; }
void fake_flat_wait(int n) { F.flat_wait = n; }
void fake_capture(int on) { F.capturing = on; }
int64_t fake_live() { return F.live; }
int64_t fake_unordered() { return F.unordered; }
int64_t fake_pinned_most() { return (int64_t)F.pinned_most; }
int64_t fake_sync_copies() { return F.sync_copies; }
int64_t fake_map_most() { return F.map_most; }
int64_t fake_tinits() { return F.tinits; }
void fake_refuse(int n) { F.refuse = n; }
unsigned long long fake_epoch() { return F.epoch; }
int64_t fake_run_steps() { return F.run_steps; }
int64_t fake_overruns() { return F.overruns; }
double fake_target() { return F.target; }
int fake_launched(int kind) { return F.launched.count(kind) ? F.launched[kind] : 0; }
unsigned long long fake_word(int i) { return F.words[i]; }
int fake_last_error() { return (int)F.last; }

/* ---- the runtime ------------------------------------------------------------- */
cudaError_t cudaMalloc(void **p, size_t n) { return take(p, n); }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return take(p, n); }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) { return take(p, n); }
cudaError_t cudaFree(void *p) { return give(p); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return give(p); }
cudaError_t cudaMallocHost(void **p, size_t n)
{
    F.pinned_most = n > F.pinned_most ? n : F.pinned_most;
    *p = std::calloc(n ? n : 1, 1);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p)
{
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind kind)
{
    ++F.sync_copies;
    F.pending = kind == cudaMemcpyHostToDevice; /* (one to the host is waited for) */
    std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    if (F.capturing) return cudaSuccess; /* a node of the graph: nothing runs */
    std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n)
{
    F.pending = true;
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t)
{
    if (!F.capturing) std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d)
{
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 1;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void)
{
    F.pending = false;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t st)
{
    if (!st) F.pending = false;
    return F.capturing ? done(cudaErrorStreamCaptureUnsupported) : cudaSuccess;
}
cudaError_t cudaGetLastError(void)
{
    const cudaError_t e = F.last;
    F.last = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t)
{
    *f = *t = (size_t)1 << 40;
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *)
{
    *p = handle<std::remove_pointer<cudaMemPool_t>::type>();
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p)
{
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e)
{
    *e = handle<std::remove_pointer<cudaEvent_t>::type>();
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned int) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e)
{
    std::free(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t)
{
    std::memcpy(e, &F.clock_us, sizeof F.clock_us);
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b)
{
    double x, y;
    std::memcpy(&x, a, 8);
    std::memcpy(&y, b, 8);
    *ms = (float)((y - x) / 1000.0);
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned int)
{
    *s = handle<std::remove_pointer<cudaStream_t>::type>();
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s)
{
    std::free(s);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned int) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *c)
{
    *c = F.capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
/* (no graphs: the tests that take steps create their simulators without) */
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

} // extern "C"

/* ---- the launchers ----------------------------------------------------------- */

int qw_sm_count(void) { return 152; }
int qw_slot_supported(const QwSimDev &d) { return d.s == 8 || d.s == 16 || d.s == 32; }
int qw_pos_supported(const QwSimDev &d) { return d.s >= 4 && d.s <= 64; }
size_t qw_step_smem_bytes(const QwSimDev &, int, int) { return 1024; }
int qw_step_grid(const QwSimDev &, int, int) { return 152; }

cudaError_t qw_launch_step(const QwSimDev &, const QwBufDev &, const QwBufDev &, const QwBufDev &, const QwStepArgs &a,
                           int, int, cudaStream_t)
{
    F.target = *a.renorm_target;
    if (!F.capturing && *a.status == 0) {
        *a.status |= F.status_bits;
        F.status_bits = 0;
        if (*a.status == 0) *a.steps_done += 1;
    }
    return launch(a.mode, F.step_us[a.mode]);
}

static cudaError_t walk_pos(const QwPosArgs &p, const QwStepArgs &a)
{
    if (F.refuse > 0) {
        --F.refuse;
        return done(cudaErrorLaunchOutOfResources);
    }
    F.target = *a.renorm_target;
    if (p.words) {
        F.epoch = p.epoch;
        F.run_steps += p.nsteps;
    }
    if (p.words) std::memcpy(F.words, p.words, 8 * sizeof(unsigned long long));
    if (!F.capturing && *a.status == 0) {
        if (F.give_up > 0) {
            --F.give_up;
            *a.status |= QW_ST_GRID_WAIT;
            if (p.words) p.words[2 * (p.epoch & 3)] = 7ull; /* some blocks had arrived */
        } else {
            *a.steps_done += p.nsteps;
            a.stats[QW_STAT_STEPS] += (unsigned long long)p.nsteps;
            *a.norm_out = 1.0;
        }
    }
    return p.words ? launch(100, F.launch_us + F.run_us * p.nsteps) : launch(QW_MODE_WALK_POS, F.single_us);
}

static QwPosPlan plan()
{
    QwPosPlan pl{};
    pl.grid = 152;
    pl.warps = 4;
    pl.tab = pl.coop = 1;
    return pl;
}

static cudaError_t tinit_pos(const QwScalarWords &w)
{
    if (!F.capturing) std::memcpy(w.dst, w.w, 8 * (size_t)w.n);
    ++F.tinits;
    return launch(101, 0.0);
}

static cudaError_t measure_pos(double *probs, int64_t len, const unsigned long long *src, unsigned long long *dst)
{
    if (dst) std::memcpy(dst, src, 16);
    for (int64_t i = 0; i < len; ++i) probs[i] = 1.0;
    return launch(102, 0.0);
}

#define POS(SUFFIX)                                                                                                   \
    QwPosPlan qw_pos_plan##SUFFIX(const QwSimDev &) { return plan(); }                                                \
    cudaError_t qw_launch_walk_pos##SUFFIX(const QwSimDev &, const QwPosPlan &, const QwPosArgs &p,                   \
                                           const QwStepArgs &a, int, cudaStream_t)                                    \
    {                                                                                                                 \
        return walk_pos(p, a);                                                                                        \
    }                                                                                                                 \
    cudaError_t qw_launch_tinit_pos##SUFFIX(const QwSimDev &, void *, int, int64_t, int64_t, int64_t, int64_t,        \
                                            const double *, const double *, const double *, const QwScalarWords &w,   \
                                            cudaStream_t)                                                             \
    {                                                                                                                 \
        return tinit_pos(w);                                                                                          \
    }                                                                                                                 \
    cudaError_t qw_launch_measure_pos##SUFFIX(const QwSimDev &, const void *, int, int64_t, int64_t, const double *,  \
                                              int, double *probs, int64_t len, const unsigned long long *src,         \
                                              unsigned long long *dst, cudaStream_t)                                  \
    {                                                                                                                 \
        return measure_pos(probs, len, src, dst);                                                                     \
    }                                                                                                                 \
    cudaError_t qw_launch_pos_pack##SUFFIX(const QwSimDev &, const QwBufDev &, void *, int32_t *status, cudaStream_t) \
    {                                                                                                                 \
        *status |= F.status_bits;                                                                                     \
        F.status_bits = 0;                                                                                            \
        return launch(103, 0.0);                                                                                      \
    }                                                                                                                 \
    cudaError_t qw_launch_pos_unpack##SUFFIX(const QwSimDev &, const void *, int, const QwBufDev &, int32_t *,        \
                                             cudaStream_t)                                                            \
    {                                                                                                                 \
        return launch(104, 0.0);                                                                                      \
    }
POS(32)
POS(64)
#undef POS

cudaError_t qw_launch_clear(const QwSimDev &d, const QwBufDev &buf, int64_t, int64_t, int, cudaStream_t)
{
    if (F.sizes[buf.key] < (size_t)d.total_buckets * (size_t)d.cap_row * 8) ++F.overruns;
    return launch(105, 0.0);
}
cudaError_t qw_launch_init_b(const QwSimDev &, const QwBufDev &, int, const double *, const double *, int, int, const double *,
                             cudaStream_t)
{
    return launch(106, 0.0);
}
cudaError_t qw_launch_tinit(const QwSimDev &, const QwBufDev &, int64_t, int64_t, int, int32_t *, cudaStream_t) { return launch(107, 0.0); }
cudaError_t qw_launch_measure(const QwSimDev &, const QwBufDev &, int, int, const double *, int, double *, int64_t, cudaStream_t)
{
    return launch(108, 0.0);
}
cudaError_t qw_launch_measure_noalloc(const QwSimDev &, const QwBufDev &, int, int, const double *, int, double *, int64_t, int,
                                      cudaStream_t, const void *, int, int64_t, int64_t)
{
    return launch(109, 0.0);
}
/* a state of 1000 branches wherever one is counted */
cudaError_t qw_launch_count(const QwSimDev &, const QwBufDev &, int, unsigned long long *counter, cudaStream_t)
{
    *counter = 1000;
    return launch(110, 0.0);
}
cudaError_t qw_launch_qls_norm(const double2 *, int, double *, int64_t *, cudaStream_t) { return launch(111, 0.0); }
cudaError_t qw_launch_regrow(const QwSimDev &, const QwBufDev &, int, uint64_t *, void *, int, cudaStream_t) { return launch(112, 0.0); }
/* (two-word keys: from the highest down, key i's amplitude i + 2 i times i) */
cudaError_t qw_flat_gather(const QwSimDev &, const QwBufDev &, int, int, const double *, void *keys, double2 *amps,
                           unsigned long long *, int64_t cap, cudaStream_t, int kw)
{
    uint64_t *k = static_cast<uint64_t *>(keys);
    for (int64_t i = 0; kw == 2 && i < cap; ++i) {
        const int64_t v = cap - 1 - i;
        k[2 * i] = (uint64_t)(v % 7);
        k[2 * i + 1] = (uint64_t)(v / 7);
        amps[i] = make_double2((double)v, 2.0 * (double)v);
    }
    return launch(113, 0.0);
}
cudaError_t qw_flat_map(const QwSimDev &, void *, int64_t M, uint32_t, int32_t *, cudaStream_t, int)
{
    F.map_most = M > F.map_most ? M : F.map_most;
    return launch(114, 0.0);
}
cudaError_t qw_flat_phase(const QwSimDev &, const void *, double2 *, int64_t, cudaStream_t, int) { return launch(115, 0.0); }
size_t qw_flat_sort_bytes(int64_t M) { return (size_t)M * 25; }
cudaError_t qw_flat_sort(const QwSimDev &, void *, double2 *, void *, double2 *, int64_t, int, int, void *, unsigned long long *,
                         int32_t *, cudaStream_t, int, int *in_tmp)
{
    *in_tmp = 0;
    return launch(116, 0.0);
}
size_t qw_flat_tiles_bytes(int64_t n) { return 64 + (size_t)n; }

/* a single-pass kernel: as many outputs as inputs; one that gives up its wait
   sets the status, says so beside the total, and counts what it did not write */
static cudaError_t single_pass(int64_t n, unsigned long long *host, int32_t *status)
{
    host[0] = (unsigned long long)n;
    if (F.flat_wait > 0 && --F.flat_wait == 0) {
        *status |= QW_ST_SORT_WAIT;
        host[0] = 2ull * (unsigned long long)n;
        host[QW_TOTAL_WAIT] = 1ull;
    }
    return launch(117, 0.0);
}
cudaError_t qw_flat_rot(const QwSimDev &, int, const void *, const double2 *, int64_t M, void *, double2 *, int64_t, void *,
                        unsigned long long *host, int32_t *status, cudaStream_t, int)
{
    return single_pass(M, host, status);
}
cudaError_t qw_flat_starts(const QwSimDev &, const void *, int64_t M, int64_t *, void *, unsigned long long *host, int32_t *status,
                           cudaStream_t, int)
{
    return single_pass(M, host, status);
}
cudaError_t qw_flat_hgroups(const QwSimDev &, const void *, const double2 *, int64_t M, const int64_t *, int64_t, void *, double2 *,
                            int64_t, void *, unsigned long long *host, int32_t *status, cudaStream_t, int)
{
    return single_pass(M, host, status);
}
cudaError_t qw_flat_readout(const QwSimDev &, const void *, const double2 *, int64_t, const QwStepArgs &, cudaStream_t, int)
{
    return launch(118, 0.0);
}
cudaError_t qw_flat_scatter(const QwSimDev &, const QwBufDev &, int, const void *keys, const double2 *amps, int64_t M,
                            int32_t *status, unsigned int *, double *, cudaStream_t, int kw)
{
    if (kw == 2) {
        const uint64_t *k = static_cast<const uint64_t *>(keys);
        F.list.assign(k, k + 2 * M);
        for (int64_t i = 0; i < M; ++i) F.list.push_back((uint64_t)amps[i].x);
    }
    *status |= F.status_bits;
    F.status_bits = 0;
    return launch(119, 0.0);
}
cudaError_t qw_io_load(const QwSimDev &, const uint64_t *, int, int64_t, void *, QwIoFlags *, cudaStream_t) { return launch(120, 0.0); }
cudaError_t qw_io_order(const QwSimDev &, const void *, int64_t, QwIoFlags *f, cudaStream_t)
{
    f->longest = F.longest;
    return launch(121, 0.0);
}
cudaError_t qw_io_store(const void *, int, int64_t, uint64_t *, cudaStream_t) { return launch(122, 0.0); }
cudaError_t qw_flat_finish(const QwStepArgs &a, const double *, const int64_t *, cudaStream_t)
{
    if (*a.status == 0) *a.steps_done += 1;
    return launch(123, 0.0);
}
int qw_faithful_layout(const QwSimDev &, int *, int *) { return 1; }
cudaError_t qw_faithful_run(const QwSimDev &, void *, int64_t, const int32_t *, int, int, int32_t *, cudaStream_t) { return launch(124, 0.0); }
cudaError_t qw_faithful_check_idle(const QwSimDev &, const void *, int64_t, int32_t *, cudaStream_t) { return launch(125, 0.0); }
cudaError_t qw_faithful_export(const QwSimDev &, const void *, int64_t, uint64_t *, cudaStream_t) { return launch(126, 0.0); }
cudaError_t qw_launch_part_gather(const QwSimDev &, const QwBufDev &, const QwPartSources &, int, int32_t *, cudaStream_t)
{
    return launch(127, 0.0);
}
cudaError_t qw_launch_part_scale(const QwPartNorms &, const double *, double *, int, cudaStream_t) { return launch(128, 0.0); }
cudaError_t qw_launch_part_inbox(const QwSimDev &, const QwBufDev &, const QwPartEntry *, int64_t, int, int32_t *, cudaStream_t)
{
    return launch(129, 0.0);
}
