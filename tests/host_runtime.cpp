// The library's host code (csrc/fdtd_capi.cu) over a CUDA runtime of its own:
// device memory is host memory, and what is queued on a stream runs only when
// the stream is waited for, as a runtime may do it.  The kernels are replaced
// by launches that advance the step counters and note which path they belong
// to.  Host memory that is freed is overwritten and kept, so that a copy
// queued from it shows.  One scenario per run, named by the first argument.
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <malloc.h>
#include <new>

void *operator new(size_t n) { return std::malloc(n ? n : 1); }
void operator delete(void *p) noexcept { if (p) __builtin_memset(p, 0xA5, malloc_usable_size(p)); }
void operator delete(void *p, size_t) noexcept { operator delete(p); }

#include "fdtd_capi.cu"

typedef std::vector<std::function<void()>> Ops;
static Ops queued, *recording = nullptr;
static void later(std::function<void()> f) { (recording ? *recording : queued).push_back(std::move(f)); }
static void drain()
{
    for (size_t i = 0; i < queued.size(); ++i) queued[i]();
    queued.clear();
}

extern "C" {
static int mallocs_left = -1;   // then none succeeds
cudaError_t cudaMalloc(void **p, size_t n)
{
    if (!mallocs_left) return cudaErrorMemoryAllocation;
    --mallocs_left;
    *p = std::aligned_alloc(256, (n + 255) / 256 * 256);
    return cudaSuccess;
}
cudaError_t cudaFree(void *) { drain(); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    later([=] { std::memcpy(d, s, n); });
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { drain(); std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { later([=] { std::memset(p, v, n); }); return cudaSuccess; }
static void copy2d(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h)
{
    for (size_t r = 0; r < h; ++r) std::memcpy((char *)d + r * dp, (const char *)s + r * sp, w);
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t)
{
    later([=] { copy2d(d, dp, s, sp, w, h); });
    return cudaSuccess;
}
cudaError_t cudaMemcpy2D(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind)
{
    drain();
    copy2d(d, dp, s, sp, w, h);
    return cudaSuccess;
}
cudaError_t cudaMemcpy3DPeerAsync(const cudaMemcpy3DPeerParms *q, cudaStream_t)
{
    const cudaMemcpy3DPeerParms p = *q;
    later([=] { copy2d(p.dstPtr.ptr, p.dstPtr.pitch, p.srcPtr.ptr, p.srcPtr.pitch, p.extent.width, p.extent.height); });
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { drain(); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { recording = new Ops; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g)
{
    *g = (cudaGraph_t)recording;
    recording = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long) { *e = (cudaGraphExec_t)g; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t)
{
    for (auto &f : *(Ops *)e) queued.push_back(f);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *, unsigned) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaHostRegister(void *, size_t, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaHostUnregister(void *) { return cudaSuccess; }
static int device;
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *q)
{
    static auto encode = [](CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                            const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                            CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; };
    *p = (void *)(PFN_cuTensorMapEncodeTiled_v12000)encode;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
}

static int bad = 0;
static void expect(bool ok, const char *what)
{
    if (!ok) {
        std::printf("not so: %s\n", what);
        ++bad;
    }
}

// The kernels: which path advanced a board by how many steps.
static long long tiled_steps, resident_steps;
static bool refuse_cooperative;   // the device takes no resident launch
static void advance(Board *const *boards, int b, int n, long long &count)
{
    Board *const B = boards[b];
    const long long did = std::max(0LL, std::min<long long>(n, *B->stop - *B->step));
    *B->step += did;
    count += did;
}
namespace fdtd {
cudaError_t launch_step(const Plan &p, int, int, cudaStream_t, const SideStream &)
{
    later([p] { for (int b = 0; b < p.nb; ++b) advance(p.boards, b, 1, tiled_steps); });
    return cudaSuccess;
}
cudaError_t launch_phase(const Plan &p, int prec, int phase, int cap, cudaStream_t st)
{
    return phase == kPhasePost ? launch_step(p, prec, cap, st, SideStream{}) : cudaSuccess;
}
cudaError_t launch_pair(const Plan &p, int, int, cudaStream_t)
{
    later([p] { advance(p.boards, 0, 2, tiled_steps); });
    return cudaSuccess;
}
cudaError_t launch_pair_part(const Plan &p, int prec, int i, int cap, cudaStream_t st) { return launch_phase(p, prec, kPairPhase[i], cap, st); }
bool resident_fits(const ResPlan &) { return !refuse_cooperative; }
cudaError_t launch_resident(const ResPlan &p, int n, cudaStream_t)
{
    if (refuse_cooperative) return cudaErrorCooperativeLaunchTooLarge;
    later([p, n] {
        for (int b = 0; b < p.n_blocks; ++b)
            if (p.blocks[b].first) advance(p.boards, p.teams[p.blocks[b].team].board, n, resident_steps);
    });
    return cudaSuccess;
}
size_t resident_smem(const ResPlan &) { return 0; }
size_t resident_arrive_bytes(int n) { return (size_t)n * 128; }
cudaError_t resident_set_smem_limit() { return cudaSuccess; }
cudaError_t launch_dft(const Plan &, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_set_i64(long long *p, long long v, cudaStream_t) { later([=] { *p = v; }); return cudaSuccess; }
cudaError_t launch_energy(const Board *, const Board &, double *, int, double *, cudaStream_t) { return cudaSuccess; }
int energy_partials(const Board &) { return 1; }
cudaError_t fused_set_smem_limits() { return cudaSuccess; }
bool fused_tile_supported(int tx, int ty) { return (tx == 62 || tx == 124) && (ty == 4 || ty == 8); }
static int mbarrier_gives_up = kStatusTmaWait, team_gives_up = kStatusBarrier;
cudaError_t launch_wait_selftest(int *s, unsigned, cudaStream_t) { later([=] { *s |= mbarrier_gives_up; }); return cudaSuccess; }
cudaError_t launch_barrier_selftest(int *s, unsigned *n, unsigned, cudaStream_t)
{
    later([=] { expect(*n == 0, "the counter starts at zero"); *s |= team_gives_up; });
    return cudaSuccess;
}
}

static fdtd_ctx *board(int nx, int ny, int nz, int depth, int prec = FDTD_FP32)
{
    fdtd_grid g{nx, ny, nz, 1e-3, 1e-3, 1e-3, 0.99, 0.0};
    fdtd_boundary b{};
    for (int f = 0; f < 6; ++f) b.depth[f] = depth;
    b.m = 3.0; b.R0 = 1e-6; b.kappa_max = 1.0;
    const std::vector<uint8_t> mat((size_t)nx * ny * nz, 0);
    const double eps = 1.0;
    fdtd_ctx *c = nullptr;
    expect(fdtd_create(&g, mat.data(), &eps, 1, nullptr, 0, nullptr, &b, prec, nullptr, &c) == FDTD_OK, "the board is created");
    return c;
}

static void factors()
{
    fdtd_ctx *c = board(30, 24, 20, 4);
    Axes A;
    build_axes(c, A);
    for (int w = 0; w < 3; ++w)
        for (int s = 0; s < 2; ++s)
            expect(!std::memcmp(c->h.cw[w][s], A.cw[w][s].data(), sizeof(Coef) * A.cw[w][s].size()), "the UPML factors arrive");
    fdtd_destroy(c);
}

// Steps of a call, by path.
struct Took {
    long long tiled, resident;
    Took()
    {
        drain();
        tiled = -tiled_steps;
        resident = -resident_steps;
    }
    bool is(long long t, long long r)
    {
        drain();
        return tiled + tiled_steps == t && resident + resident_steps == r;
    }
};

static void refused()
{
    fdtd_ctx *a = board(30, 24, 20, 4), *c[2] = {board(30, 24, 20, 4), board(25, 24, 20, 4)};
    {
        Took t;
        expect(fdtd_step(a, 20) == FDTD_OK && t.is(0, 20), "the board takes resident launches");
    }
    refuse_cooperative = true;
    a->plan_dirty = true;
    Took t;
    expect(fdtd_step(a, 20) == FDTD_OK && t.is(20, 0), "a board steps where the device takes no resident launch");
    Took u;
    expect(fdtd_step(a, 5) == FDTD_OK && u.is(5, 0), "and goes on so");
    fdtd_batch *b = nullptr;
    int done = 0;
    expect(fdtd_batch_create(nullptr, &b) == FDTD_OK, "the batch is created");
    for (fdtd_ctx *m : c) expect(fdtd_batch_add(b, m, 20) == FDTD_OK, "a board joins");
    Took v;
    expect(fdtd_batch_step(b, 20, &done) == FDTD_OK && v.is(40, 0) && done == 2, "a batch steps there");
    fdtd_batch_destroy(b);
    for (fdtd_ctx *m : c) fdtd_destroy(m);
    fdtd_destroy(a);
}

static bool resident(fdtd_ctx *c, int n)
{
    int r = -1;
    expect(fdtd_is_resident(c, n, &r) == FDTD_OK && (r == 0 || r == 1), "the path is told");
    return r == 1;
}

static void chosen()
{
    fdtd_ctx *a = board(30, 24, 20, 4), *b = board(25, 24, 20, 4), *h = board(25, 24, 20, 4, FDTD_FP16_STORE);
    expect(resident(a, 1) && resident(a, 20) && !resident(h, 20), "the rule before the first step");
    for (int on : {1, 0}) {
        fdtd_set_tiled(a, on);
        Took t;
        expect(resident(a, 20) == !on && fdtd_step(a, 20) == FDTD_OK && t.is(on ? 20 : 0, on ? 0 : 20), "a board steps as set");
    }
    fdtd_batch *g = nullptr;
    expect(fdtd_batch_create(nullptr, &g) == FDTD_OK && fdtd_batch_add(g, a, 30) == FDTD_OK && fdtd_batch_add(g, b, 30) == FDTD_OK,
           "a batch of two");
    Took t;
    expect(fdtd_batch_step(g, 10, nullptr) == FDTD_OK && t.is(0, 20), "both members by the rule");
    fdtd_set_tiled(a, 1);
    Took u;
    expect(!resident(a, 10) && resident(b, 10) && fdtd_batch_step(g, 10, nullptr) == FDTD_OK && u.is(10, 10), "each member as set");
    fdtd_set_tiled(b, 1);
    Took v;
    expect(fdtd_batch_step(g, 10, nullptr) == FDTD_OK && v.is(20, 0), "both set");
    fdtd_batch_destroy(g);
    // a probe on a high wall plane belongs to no block
    fdtd_ctx *p = board(25, 24, 20, 4);
    expect(fdtd_add_probe(p, 25, 3, 3, 2, nullptr) == FDTD_OK && !resident(p, 20), "a port outside the boxes, before the first step");
    Took w;
    expect(fdtd_step(p, 3) == FDTD_OK && w.is(3, 0) && !resident(p, 20), "and after it");
    for (fdtd_ctx *c : {a, b, h, p}) fdtd_destroy(c);
}

// Two parts of a split board take a halo plane from each other after every step.
static void split()
{
    for (int far : {0, 1}) {
        fdtd_ctx *a = board(30, 24, 20, 0);
        device = far;
        fdtd_ctx *b = board(30, 24, 20, 0);
        device = 0;
        expect(fdtd_step(a, 1) == FDTD_OK && fdtd_step(b, 1) == FDTD_OK, "a first step");
        expect(fdtd_halo_copy(a, 24, b, 1, 1, 5) == FDTD_OK && fdtd_halo_copy(b, 0, a, 23, 1, 5) == FDTD_OK, "the exchange");
        Took t;
        expect(fdtd_step(a, 1) == FDTD_OK && fdtd_step(b, 1) == FDTD_OK && t.is(far ? 0 : 2, far ? 2 : 0),
               "parts on one GPU step beside each other, parts on two GPUs by resident launches");
        Took u;
        expect(fdtd_step(a, 3) == FDTD_OK && u.is(3, 0), "several steps after an exchange");
        fdtd_reset(a);
        Took v;
        expect(fdtd_step(a, 3) == FDTD_OK && v.is(0, 3), "a board that starts again");
        fdtd_destroy(a);
        fdtd_destroy(b);
    }
}

static void segments()
{
    fdtd_ctx *a = board(200, 190, 60, 6, FDTD_FP16_STORE);
    fdtd_batch *g = nullptr;
    expect(fdtd_batch_create(nullptr, &g) == FDTD_OK, "the batch is created");
    fdtd_step(a, 1);
    const int rule = a->plan.zseg;
    fdtd_tuning t{}, back{};
    t.zseg = 25;
    back.zseg = FDTD_ZSEG_AUTO;
    fdtd_set_tuning(a, &t);
    fdtd_set_tuning(a, &(t = fdtd_tuning{}));
    fdtd_step(a, 1);
    expect(rule != 25 && a->plan.zseg == 25, "a length that was set, and kept by 0");
    fdtd_set_tuning(a, &back);
    fdtd_step(a, 1);
    expect(a->plan.zseg == rule, "the rule's length again");
    fdtd_batch_add(g, a, 9);
    t.zseg = 25;
    fdtd_batch_set_tuning(g, &t);
    fdtd_batch_step(g, 1, nullptr);
    const int set = g->plan.zseg;
    fdtd_batch_set_tuning(g, &back);
    fdtd_batch_step(g, 1, nullptr);
    expect(set == 25 && g->plan.zseg == rule, "and in a batch");
    fdtd_batch_destroy(g);
    fdtd_destroy(a);
}

// What the host makes of a wait that gave up.
static void waits()
{
    fdtd_ctx *c = board(30, 24, 20, 4);
    expect(fdtd_step(c, 1) == FDTD_OK && fdtd_sync(c) == FDTD_OK, "no wait gave up");
    *c->h.status = kStatusTmaWait;
    expect(fdtd_sync(c) == FDTD_ETIMEOUT && std::strstr(fdtd_last_error(), "TMA wait"), "a TMA wait");
    *c->h.status = kStatusBarrier;
    expect(fdtd_sync(c) == FDTD_ETIMEOUT && std::strstr(fdtd_last_error(), "barrier of a resident launch"), "a barrier");
    fdtd_destroy(c);
    expect(fdtd_selftest_wait_timeout(nullptr, 10) == FDTD_ETIMEOUT, "both kinds gave up");
    team_gives_up = 0;
    expect(fdtd_selftest_wait_timeout(nullptr, 10) == FDTD_OK, "the barrier did not");
    team_gives_up = kStatusBarrier;
    mbarrier_gives_up = 0;
    expect(fdtd_selftest_wait_timeout(nullptr, 10) == FDTD_OK, "the mbarrier did not");
}

// A checkpoint's data say whether a plane was written from outside, also those
// of before resident launches, whose header has 0 in its last word.
static void checkpoint()
{
    fdtd_ctx *a = board(30, 24, 20, 4), *b = board(30, 24, 20, 4);
    fdtd_step(a, 4);
    size_t n = 0;
    fdtd_save(a, nullptr, 0, &n);
    std::vector<unsigned char> clean(n), wrote(n);
    expect(fdtd_save(a, clean.data(), n, &n) == FDTD_OK, "a state of steps alone");
    std::vector<float> plane(2 * 31 * 25, 1.f);
    const int high[3] = {30, 24, 20};
    for (int axis = -1; axis < 3; ++axis) {
        if (axis >= 0) {
            fdtd_load(a, clean.data(), n);
            expect(fdtd_halo_unpack(a, axis, high[axis], 5, plane.data()) == FDTD_OK, "a plane from outside");
            if (axis == 1) fdtd_step(a, 1);   // it then lies in the set of the step before
        }
        expect(fdtd_save(a, wrote.data(), n, &n) == FDTD_OK, "the state is saved");
        std::memset(wrote.data() + offsetof(CkptHeader, scale) + 4, 0, 4);
        expect(fdtd_load(b, wrote.data(), n) == FDTD_OK, "the checkpoint is taken");
        const int tiled = axis < 0 ? 0 : 3;
        Took t;
        expect(fdtd_step(b, 3) == FDTD_OK && t.is(tiled, 3 - tiled), "the launches that continue it");
    }
    fdtd_destroy(a);
    fdtd_destroy(b);
}

// A plan that runs out of memory half-way leaves no copy queued from freed memory.
static void memory()
{
    for (int batched : {0, 1}) {
        fdtd_ctx *c = board(30, 24, 20, 4);
        fdtd_batch *g = nullptr;
        fdtd_step(c, 0);
        c->plan_dirty = true;
        long long **const boards = batched ? nullptr : &c->rplan_buf;
        if (batched) expect(fdtd_batch_create(nullptr, &g) == FDTD_OK && fdtd_batch_add(g, c, 9) == FDTD_OK, "a batch of one");
        else for (long long **b : {&c->rplan_buf, &c->res_buf}) { cudaFree(*b); *b = nullptr; c->rplan_cap = c->res_cap = 0; }
        mallocs_left = 1;
        expect((batched ? fdtd_batch_step(g, 4, nullptr) : fdtd_step(c, 4)) == FDTD_ENOMEM, "the second buffer is refused");
        mallocs_left = -1;
        drain();
        const long long *const buf = boards ? *boards : g->rplan_buf;
        expect(buf && *buf == (long long)(uintptr_t)c->d, "the first holds what was copied to it");
        Took t;
        expect((batched ? fdtd_batch_step(g, 4, nullptr) : fdtd_step(c, 4)) == FDTD_OK && t.is(0, 4), "the next call steps");
        if (g) fdtd_batch_destroy(g);
        fdtd_destroy(c);
    }
}

int main(int, char **argv)
{
    const std::string s = argv[1];
    if (s == "factors") factors();
    else if (s == "refused") refused();
    else if (s == "chosen") chosen();
    else if (s == "split") split();
    else if (s == "segments") segments();
    else if (s == "waits") waits();
    else if (s == "checkpoint") checkpoint();
    else if (s == "memory") memory();
    else expect(false, "a known scenario");
    return bad;
}
