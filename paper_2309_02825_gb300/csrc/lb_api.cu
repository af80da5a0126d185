// C-ABI of the solver (declared in include/lb.h): argument checks, device
// memory, parameters, and the order of kernel launches.  No arithmetic of
// the method runs on the host beyond the scalar relaxation set.
#include <cuda.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "lb_internal.cuh"

namespace {

thread_local std::string g_create_err;

lb_status fail(lb_ctx *c, lb_status s, const std::string &msg)
{
    if (c)
        c->err = msg;
    else
        g_create_err = msg;
    return s;
}

lb_status cuda_fail(lb_ctx *c, cudaError_t e, const char *where)
{
    std::string m = std::string(where) + ": " + cudaGetErrorString(e);
    if (e == cudaErrorMemoryAllocation) return fail(c, LB_ENOMEM, m);
    return fail(c, LB_ECUDA, m);
}

bool finite_pos(double v) { return isfinite(v) && v > 0.0; }

constexpr int kFlags = 4;
constexpr size_t kHostArea = 64 * sizeof(double) + kFlags * sizeof(int);  // results, then the flags' mirrors

// The unique number of the calling thread's CUDA context; false where the driver has none.
bool context_id(unsigned long long *id)
{
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult found{};
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess || !fn) {
        cudaGetLastError();
        return false;
    }
    return ((CUresult(CUDAAPI *)(CUcontext, unsigned long long *))fn)(nullptr, id) == CUDA_SUCCESS;
}

// Page-locked areas, cut from slabs of 64 (page-locking takes about 300 us
// whatever the size).  From any thread, and only within the CUDA context that
// made a slab, so that what a cudaDeviceReset has released is not handed out
// again.  A slab without solvers is released unless it is its context's only one
// with room.
constexpr size_t kAreaPitch = (kHostArea + 127) / 128 * 128;
constexpr int kSlabAreas = 64;
struct AreaSlab {
    char *host, *dev;
    unsigned long long context, used;  // a bit per area
};
std::mutex g_slabs_mutex;
std::vector<AreaSlab> &g_slabs = *new std::vector<AreaSlab>;  // never destroyed: solvers may be closed at exit

cudaError_t take_area(lb_ctx *c)
{
    unsigned long long id = 0;
    const bool shared = context_id(&id);
    std::lock_guard<std::mutex> lock(g_slabs_mutex);
    AreaSlab *slab = nullptr;
    for (AreaSlab &s : g_slabs)
        if (shared && s.context == id && s.used != ~0ull) slab = &s;
    AreaSlab own{};
    if (!slab) {
        cudaError_t e = cudaHostAlloc((void **)&own.host, kAreaPitch * (shared ? kSlabAreas : 1), cudaHostAllocMapped);
        if (e != cudaSuccess) return e;
        if ((e = cudaHostGetDevicePointer((void **)&own.dev, own.host, 0)) != cudaSuccess) {
            cudaFreeHost(own.host);
            return e;
        }
        own.context = id;
        slab = &own;
        if (shared) {
            g_slabs.push_back(own);
            slab = &g_slabs.back();
        }
    }
    int k = 0;
    while ((slab->used >> k) & 1u) ++k;
    slab->used |= 1ull << k;
    c->host_context = id;
    c->host_area = slab->host + k * kAreaPitch;
    c->dout = (double *)(slab->dev + k * kAreaPitch);
    return cudaSuccess;
}

void give_area(lb_ctx *c)  // its stream has been waited for
{
    if (!c->host_area) return;
    char *const p = (char *)c->host_area;
    std::lock_guard<std::mutex> lock(g_slabs_mutex);
    bool room = false;  // in another slab of the same context
    size_t mine = g_slabs.size();
    for (size_t k = 0; k < g_slabs.size(); ++k) {
        const AreaSlab &s = g_slabs[k];
        if (s.context != c->host_context) continue;
        if (p >= s.host && p < s.host + kAreaPitch * kSlabAreas)
            mine = k;
        else
            room = room || s.used != ~0ull;
    }
    if (mine == g_slabs.size()) {  // an area of its own
        cudaFreeHost(p);
        return;
    }
    AreaSlab &s = g_slabs[mine];
    s.used &= ~(1ull << ((p - s.host) / kAreaPitch));
    if (s.used == 0 && room) {
        cudaFreeHost(s.host);
        g_slabs.erase(g_slabs.begin() + (long)mine);
    }
}

void free_ctx(lb_ctx *c)
{
    if (!c) return;
    lbk::blocked_release(c);
    for (auto &g : c->graph)
        if (g) cudaGraphExecDestroy(g);
    cudaFree(c->f[0]);
    cudaFree(c->f[1]);
    cudaFree(c->scratch);
    give_area(c);
    cudaFree(c->gradtmp);
    delete c;
}

// Make the calling thread's current device the context's device.
struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(const lb_ctx *c)
    {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != c->device) cudaSetDevice(c->device);
    }
    ~DeviceGuard()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

constexpr int64_t kGraphSteps = 32;  // sweeps per recorded graph (even: parity unchanged)

// Record kGraphSteps sweeps starting from buffer `from` on a private stream.
cudaError_t record_sweeps(lb_ctx *c, int from)
{
    cudaStream_t cs;
    cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    cudaStream_t user = c->stream;
    c->stream = cs;
    cudaGraph_t graph = nullptr;
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        int p = from;
        for (int64_t k = 0; k < kGraphSteps && e == cudaSuccess; ++k) {
            e = lbk::launch_sweep(c, c->f[p], c->f[p ^ 1]);
            p ^= 1;
        }
        cudaError_t e2 = cudaStreamEndCapture(cs, &graph);
        if (e == cudaSuccess) e = e2;
    }
    c->stream = user;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&c->graph[from], graph, 0);
    if (graph) cudaGraphDestroy(graph);
    cudaStreamDestroy(cs);
    return e;
}

// A status flag, cleared; the stream has been waited for, so nothing is setting it.
int take_flag(lb_ctx *c, int k)
{
    const int f = c->hflag[k];
    if (f) {
        c->hflag[k] = 0;
        cudaMemsetAsync(&c->dflag[k].bits, 0, sizeof(int), c->stream);
    }
    return f;
}

// The same for n flags from `first`, in stream order (sweeps enqueued before may still set them).
cudaError_t clear_flags(lb_ctx *c, int first, int n)
{
    return lbk::launch_clear_flags(c->dflag + first, (int *)(c->dout + 64) + first, n, c->stream);
}

// Read and clear the recovery and range flags (ctx->dflag[1..2]) after
// the work enqueued so far; synchronises the stream.  A staging timeout or a
// fixed-point range overflow leaves the context uninitialised: the state (or
// a staging tile) may be corrupt, so lb_step and lb_macros refuse to run
// until lb_set_theta0 or lb_load_state sets a state again.
lb_status read_flags(lb_ctx *c, const char *who)
{
    const cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, who);
    const int fl[2] = {take_flag(c, lbk::kFlagRecover), take_flag(c, lbk::kFlagRange)};
    const std::string w(who);
    if (fl[0] & 4) {
        c->initialized = false;
        return fail(c, LB_ETIMEOUT, w + ": a shared-memory staging wait of the recovery timed out; set the state "
                                        "again (lb_set_theta0 or lb_load_state)");
    }
    if (fl[1]) {
        c->initialized = false;
        return fail(c, LB_EINVAL, w + ": a fixed-point distribution reached |f| >= 2^61 (the run is unstable: an "
                                      "FP64 run would overflow); set the state again");
    }
    if (fl[0]) return fail(c, LB_ENONPOS, w + ": theta <= 0 or non-finite at some node");
    return LB_OK;
}

constexpr int64_t kTbGraphLaunches = 16;  // blocked launches per recorded graph (even)

// Record kTbGraphLaunches blocked launches of tb_k steps starting from buffer `from`.
cudaError_t record_blocked(lb_ctx *c, int from)
{
    cudaStream_t cs;
    cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    cudaGraph_t graph = nullptr;
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        int p = from;
        for (int64_t k = 0; k < kTbGraphLaunches && e == cudaSuccess; ++k) {
            e = lbk::blocked_launch(c, c->f[p], c->f[p ^ 1], c->tb_k, cs);
            p ^= 1;
        }
        cudaError_t e2 = cudaStreamEndCapture(cs, &graph);
        if (e == cudaSuccess) e = e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&c->tb_graph[from], graph, 0);
    if (graph) cudaGraphDestroy(graph);
    cudaStreamDestroy(cs);
    return e;
}

// The schedule lb_step runs when the caller has set none (kSchedAuto).  On
// periodic 2D and 3D grids large enough to fill the chip, marching sweeps
// (lb_march.cu); on small 2D grids, whose single sweeps last about as long as
// their launch, several steps per launch on square tiles; on short 1D grids
// all steps in one launch; else one sweep per launch.  Every choice gives the
// same bits.
cudaError_t choose_schedule(lb_ctx *c)
{
    if (c->sched != lbk::kSchedAuto) return cudaSuccess;
    c->run = lbk::kSchedSweeps;
    lbk::blocked_release(c);
    c->march = lbk::MarchPlan{};
    c->march_short = false;
    if (lbk::line_fits(c)) {
        c->run = lbk::kSchedLine;
        return cudaSuccess;
    }
    if (c->geom.mirror) return cudaSuccess;
    // FP64 whose collisions take the direct form is bound by the FP64 pipe, which
    // recomputed nodes only load further: us per step, marching / one sweep per
    // launch at eps = 0.01, 1400^2 139 / 122, 2048^2 285 / 254, 4096^2 1062 / 1005.
    const bool direct = c->precision == LB_FP64 && !lbk::coll_f64_aligns(*c);
    lbk::MarchWorth worth = lbk::kMarchNo;
    cudaError_t e = lbk::march_setup(c, &c->march, &worth);
    if (e != cudaSuccess) return e;
    if (direct) worth = lbk::kMarchNo;
    c->march_short = worth == lbk::kMarchShort;
    if (worth != lbk::kMarchNo) c->run = lbk::kSchedMarch;
    if (worth == lbk::kMarchYes) return cudaSuccess;
    if (c->d == 2) {
        // The smallest square tile, from 8 nodes in steps of 4, that leaves at
        // most one tile per SM; 8 steps per launch.  us per step (fixed point,
        // FP32, FP64) against one sweep per launch replayed from a graph:
        // 64^2 1.35, 1.08, 1.9 / 2.9, 2.7, 3.9; 128^2 1.6, 1.1, 2.4 / 2.9, 2.8,
        // 4.0; 192^2 1.6, 1.3, 2.9 / 3.0, 2.7, 4.2; 256^2 2.4, 1.6, 4.4 / 3.4,
        // 2.8, 4.6; 384^2 3.2, 1.9 / 4.7, 3.1.  FP64 tiles above 24 nodes (SMs
        // busy with the recomputed halo) lose: 320^2 5.7 / 5.1; in the direct form
        // those above 8 nodes: 96^2 3.3 / 4.0, 128^2 4.6 / 4.1, 256^2 10.5 / 6.7.
        const int most = c->precision == LB_FP64 ? (direct ? 8 : 24) : (c->precision == LB_FX64 ? 40 : 48);
        for (int tile = 8; tile <= most; tile += 4) {
            if (((c->N[0] + tile - 1) / tile) * ((c->N[1] + tile - 1) / tile) > c->sms) continue;
            bool fits = true;
            if ((e = lbk::blocked_setup(c, 8, tile, tile <= 32 ? 512 : 1024, &fits)) != cudaSuccess) return e;
            if (fits) c->run = lbk::kSchedTiles;
            break;
        }
    }
    return cudaSuccess;
}

bool capturing(cudaStream_t s)
{
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) return true;
    return cap != cudaStreamCaptureStatusNone;
}

}  // namespace

namespace lbk {

bool derive_params(lb_ctx &c, const lb_relax *rs)
{
    const int d = c.d;
    const bool paper = !rs || rs->paper_set;
    c.paper = paper;
    if (paper) {
        const double a = 6.0 * c.eps + 1.0;
        c.s1 = 2.0 / a;
        c.s2x = 24.0 * c.eps / (a * a);
        if (d == 1) {
            c.s22 = 1.0;
            c.w1 = 1.0 / 6.0;
            c.wd = 0.0;
        } else {
            c.s22 = 4.0 / (6.0 * c.eps + 3.0);
            c.w1 = 1.0 / 6.0 - (d - 1) * c.eps / 3.0;
            c.wd = c.eps / 6.0;
        }
    } else {
        c.s1 = rs->s1;
        c.s2x = rs->s2x;
        c.s22 = (d > 1) ? rs->s22 : 1.0;
        c.w1 = rs->w1;
        c.wd = (d > 1) ? rs->wd : 0.0;
    }
    c.theta_ref = rs ? rs->theta_ref : 0.0;
    const bool rates_ok = c.s1 > 0 && c.s1 < 2 && c.s2x > 0 && c.s2x < 2 && (d == 1 || (c.s22 > 0 && c.s22 < 2));
    if (!rates_ok || !isfinite(c.w1) || !isfinite(c.wd) || !isfinite(c.theta_ref)) return false;
    // Eq. (d1-3-weight) and c_s^2 = [2 w1 + 4(d-1) wd] c^2.
    c.w0 = 1.0 - 2.0 * d * c.w1 - 2.0 * d * (d - 1) * c.wd;
    c.sigma = 2.0 * c.w1 + 4.0 * (d - 1) * c.wd;
    c.cs2 = c.sigma * c.c * c.c;
    return true;
}

}  // namespace lbk

extern "C" {

lb_status lb_create(int d, const int64_t *N, double nu, double dx, double dt, const lb_relax *rs, int precision,
                    void *stream, lb_ctx **out)
{
    lbk::NvtxRange nvtx_range("lb_create");
    if (!out) return fail(nullptr, LB_EINVAL, "lb_create: out is NULL");
    *out = nullptr;
    if (d < 1 || d > 4) return fail(nullptr, LB_EINVAL, "lb_create: d must be 1, 2, 3 or 4");
    if (!N) return fail(nullptr, LB_EINVAL, "lb_create: N is NULL");
    if (!finite_pos(nu) || !finite_pos(dx) || !finite_pos(dt))
        return fail(nullptr, LB_EINVAL, "lb_create: nu, dx and dt must be finite and > 0");
    if (precision != LB_FP64 && precision != LB_FP32_SHIFTED && precision != LB_FX64)
        return fail(nullptr, LB_EINVAL, "lb_create: unknown precision");
    int64_t nodes = 1;
    for (int a = 0; a < d; ++a) {
        if (N[a] < 1 || N[a] > (1 << 24)) return fail(nullptr, LB_EINVAL, "lb_create: each N must be in [1, 2^24]");
        nodes *= N[a];
        if (nodes > (int64_t(1) << 31)) return fail(nullptr, LB_EINVAL, "lb_create: more than 2^31 nodes");
    }

    lb_ctx *c = new (std::nothrow) lb_ctx();
    if (!c) return fail(nullptr, LB_ENOMEM, "lb_create: host allocation failed");
    c->d = d;
    c->q = 1 + 2 * d * d;
    for (int a = 0; a < 4; ++a) c->N[a] = (a < d) ? N[a] : 1;
    c->nodes = nodes;
    c->precision = precision;
    c->nu = nu;
    c->dx = dx;
    c->dt = dt;
    c->c = dx / dt;
    c->eps = nu * dt / (dx * dx);
    c->stream = (cudaStream_t)stream;
    cudaGetDevice(&c->device);

    if (!lbk::derive_params(*c, rs)) {
        free_ctx(c);
        return fail(nullptr, LB_EINVAL, "lb_create: relaxation rates must lie in (0, 2) and weights be finite");
    }
    if (precision == LB_FX64 && !lbk::fx_constants_ok(*c)) {
        free_ctx(c);
        return fail(nullptr, LB_EINVAL, "lb_create: a fixed-point collision constant leaves (-1, 1) (weights too large "
                                        "for LB_FX64; use LB_FP64)");
    }

    // Layout.
    const int V = (precision == LB_FP32_SHIFTED) ? lbk::Vec<float>::V : lbk::Vec<double>::V;
    c->elem = (precision == LB_FP32_SHIFTED) ? 4 : 8;
    const int W = lbk::lane_width(c->d, c->elem);
    c->geom = lbk::make_geom(c->N[0], c->N[1], c->N[2], c->N[3], V, W);
    const lbk::Geom &g = c->geom;

    const size_t fbytes = ((size_t)c->q * (size_t)g.slab + lbk::kSlackElems) * c->elem;
    cudaError_t e;
    for (int b = 0; b < 2; ++b) {
        e = cudaMalloc(&c->f[b], fbytes);
        if (e != cudaSuccess) {
            free_ctx(c);
            return cuda_fail(nullptr, e, "lb_create: state allocation");
        }
        e = cudaMemsetAsync(c->f[b], 0, fbytes, c->stream);
        if (e != cudaSuccess) {
            free_ctx(c);
            return cuda_fail(nullptr, e, "lb_create: memset");
        }
    }
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    if (sms > 0) c->sms = sms;
    c->scratch_blocks = c->sms * 4;
    const size_t partials = (size_t)lbk::kRedSlots * c->scratch_blocks;
    if ((e = cudaMalloc(&c->scratch, sizeof(double) * partials + sizeof(lbk::StatusFlag) * kFlags)) != cudaSuccess ||
        (e = take_area(c)) != cudaSuccess) {
        free_ctx(c);
        return cuda_fail(nullptr, e, "lb_create: scratch allocation");
    }
    memset(c->host_area, 0, kHostArea);
    c->hout = (volatile double *)c->host_area;
    c->hflag = (volatile int *)(c->hout + 64);
    c->dflag = (lbk::StatusFlag *)(c->scratch + partials);
    if ((e = clear_flags(c, 0, kFlags)) != cudaSuccess) {
        free_ctx(c);
        return cuda_fail(nullptr, e, "lb_create: status flags");
    }
    if ((e = choose_schedule(c)) != cudaSuccess) {
        free_ctx(c);
        return cuda_fail(nullptr, e, "lb_create: schedule");
    }
    *out = c;
    return LB_OK;
}

lb_status lb_destroy(lb_ctx *c)
{
    lbk::NvtxRange nvtx_range("lb_destroy");
    if (!c) return LB_OK;
    DeviceGuard dg(c);
    cudaStreamSynchronize(c->stream);
    free_ctx(c);
    return LB_OK;
}

lb_status lb_get_params(const lb_ctx *c, double *out)
{
    if (!c || !out) return LB_EINVAL;
    const double v[15] = {c->eps, c->c,  c->cs2, c->s1, c->s2x, c->s22,       c->w0,       c->w1,
                          c->wd,  c->nu, c->dx,  c->dt, (double)c->q, c->theta_ref, (double)c->fx_bits};
    memcpy(out, v, sizeof v);
    return LB_OK;
}

lb_status lb_set_boundary(lb_ctx *c, const int *kind)
{
    lbk::NvtxRange nvtx_range("lb_set_boundary");
    if (!c) return LB_EINVAL;
    if (!kind) return fail(c, LB_EINVAL, "lb_set_boundary: kind is NULL");
    unsigned mask = 0;
    for (int a = 0; a < c->d; ++a) {
        if (kind[a] != LB_PERIODIC && kind[a] != LB_MIRROR)
            return fail(c, LB_EINVAL, "lb_set_boundary: kind must be LB_PERIODIC or LB_MIRROR");
        if (kind[a] == LB_MIRROR) {
            if (c->N[a] < 3) return fail(c, LB_EINVAL, "lb_set_boundary: a mirror axis needs at least 3 nodes");
            mask |= 1u << a;
        }
    }
    DeviceGuard dg(c);
    // recorded sweeps hold the old geometry; drain the stream before dropping them
    cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "lb_set_boundary");
    for (auto &g : c->graph)
        if (g) {
            cudaGraphExecDestroy(g);
            g = nullptr;
        }
    c->geom.mirror = mask;
    c->initialized = false;  // the stored state follows the old walls: initialise again
    ++c->gen;
    if (mask && c->sched != lbk::kSchedAuto) {  // sweeps of several steps per launch are periodic only
        lbk::blocked_release(c);
        c->sched = c->run = lbk::kSchedSweeps;
    }
    if ((e = choose_schedule(c)) != cudaSuccess) return cuda_fail(c, e, "lb_set_boundary: schedule");
    return LB_OK;
}

lb_status lb_set_viscosity(lb_ctx *c, double nu)
{
    lbk::NvtxRange nvtx_range("lb_set_viscosity");
    if (!c) return LB_EINVAL;
    if (!finite_pos(nu)) return fail(c, LB_EINVAL, "lb_set_viscosity: nu must be finite and > 0");
    lb_ctx trial;
    trial.d = c->d;
    trial.dx = c->dx;
    trial.dt = c->dt;
    trial.c = c->c;
    trial.nu = nu;
    trial.eps = nu * c->dt / (c->dx * c->dx);
    const lb_relax rs = {c->paper ? 1 : 0, c->s1, c->s2x, c->s22, c->w1, c->wd, c->theta_ref};
    if (!lbk::derive_params(trial, &rs))
        return fail(c, LB_EINVAL, "lb_set_viscosity: the relaxation set leaves (0, 2) at this nu");
    if (c->precision == LB_FX64 && !lbk::fx_constants_ok(trial))
        return fail(c, LB_EINVAL, "lb_set_viscosity: a fixed-point collision constant leaves (-1, 1) at this nu");
    DeviceGuard dg(c);
    const bool aligned = lbk::coll_f64_aligns(*c);
    // recorded sweeps carry the old collision constants; drain the stream before dropping them
    cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "lb_set_viscosity");
    for (auto &g : c->graph)
        if (g) {
            cudaGraphExecDestroy(g);
            g = nullptr;
        }
    c->nu = nu;
    c->eps = trial.eps;
    c->s1 = trial.s1;
    c->s2x = trial.s2x;
    c->s22 = trial.s22;
    c->w0 = trial.w0;
    c->w1 = trial.w1;
    c->wd = trial.wd;
    c->sigma = trial.sigma;
    c->cs2 = trial.cs2;
    ++c->gen;
    for (auto &g : c->tb_graph)
        if (g) {
            cudaGraphExecDestroy(g);
            g = nullptr;
        }
    if (c->precision == LB_FP64 && aligned != lbk::coll_f64_aligns(*c) && (e = choose_schedule(c)) != cudaSuccess)
        return cuda_fail(c, e, "lb_set_viscosity: schedule");
    return LB_OK;
}

lb_status lb_set_blocking(lb_ctx *c, int steps_per_launch, int tile, int threads)
{
    lbk::NvtxRange nvtx_range("lb_set_blocking");
    if (!c) return LB_EINVAL;
    if (steps_per_launch < 0 || steps_per_launch > 64 ||
        (steps_per_launch > 0 && (tile < 1 || tile > 4096 || !(threads == 256 || threads == 512 || threads == 1024))))
        return fail(c, LB_EINVAL, "lb_set_blocking: steps per launch in 0..64, tile in 1..4096, threads 256, 512 or 1024");
    if (steps_per_launch > 0 && (c->d != 2 || c->geom.mirror))
        return fail(c, LB_EINVAL, "lb_set_blocking: blocked sweeps are built for periodic 2D grids");
    DeviceGuard dg(c);
    cudaError_t e = cudaStreamSynchronize(c->stream);  // tables and graphs may be in use
    if (e != cudaSuccess) return cuda_fail(c, e, "lb_set_blocking");
    bool fits = true;
    if ((e = lbk::blocked_setup(c, steps_per_launch, tile, threads, &fits)) != cudaSuccess)
        return cuda_fail(c, e, "lb_set_blocking");
    c->sched = c->run = c->tb_k ? lbk::kSchedTiles : lbk::kSchedSweeps;
    if (!fits) return fail(c, LB_EINVAL, "lb_set_blocking: tile plus halo exceeds the shared memory per block");
    return LB_OK;
}

lb_status lb_get_blocking(const lb_ctx *c, int *info)
{
    if (!c || !info) return LB_EINVAL;
    info[0] = info[1] = info[2] = info[3] = 0;
    if (c->sched == lbk::kSchedTiles) {
        info[0] = c->tb_k;
        info[1] = c->tb_tile;
        info[2] = c->tb_threads;
        info[3] = c->tb_ntiles;
    } else if (c->sched == lbk::kSchedMarch) {
        info[0] = c->march.steps;
        info[1] = c->march.bx;
        info[2] = c->march.threads;
        info[3] = c->march.nx * c->march.ny * c->march.nc;
    }
    return LB_OK;
}

lb_status lb_autotune(lb_ctx *c, int trial_steps, double *choice)
{
    lbk::NvtxRange nvtx_range("lb_autotune");
    if (!c || trial_steps < 2) return LB_EINVAL;
    if (c->d != 2 || c->geom.mirror) {  // the context keeps its schedule: there are no tiles to choose
        if (choice) {
            choice[0] = 0;
            choice[1] = choice[2] = choice[3] = 0;
        }
        return LB_OK;
    }
    DeviceGuard dg(c);
    cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "lb_autotune");
    struct Cand {
        int sched, K, tile, threads;
    };
    std::vector<Cand> cands = {{lbk::kSchedSweeps, 0, 0, 0}};
    lbk::MarchPlan plan{};
    lbk::MarchWorth worth = lbk::kMarchNo;
    if ((e = lbk::march_setup(c, &plan, &worth)) != cudaSuccess) return cuda_fail(c, e, "lb_autotune");
    if (plan.steps) cands.push_back({lbk::kSchedMarch, plan.steps, plan.bx, plan.threads});
    c->march = plan;
    c->march_short = false;
    int optin = 0;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device)) != cudaSuccess)
        return cuda_fail(c, e, "lb_autotune");
    const int node_bytes = 9 * (int)c->elem;
    for (int K : {2, 3, 4, 5, 6, 8, 12})
        for (int per_sm : {1, 2, 3, 4}) {
            const long avail = per_sm == 1 ? optin : optin / per_sm - 1024;
            int edge = (int)floor(sqrt((double)avail / node_bytes));
            while ((long)edge * edge * node_bytes > avail) --edge;
            // the largest square tile for this many blocks per SM, and one 4 nodes smaller (less work per block)
            for (int tile : {edge - 2 * K, edge - 2 * K - 4}) {
                if (tile < 8) continue;
                for (int th : {256, 512, 1024}) cands.push_back({lbk::kSchedTiles, K, tile, th});
            }
        }
    if (c->precision == LB_FP64) {
        // the trials step whatever the buffers hold: one normal double everywhere
        // (0x3f3f...), which the warm-up relaxes towards w_i theta, so that the timed
        // collisions take the form a run's do (the first steps' equal values do not align)
        const size_t bytes = (size_t)c->q * c->geom.slab * c->elem;
        for (void *p : c->f)
            if ((e = cudaMemsetAsync(p, 0x3f, bytes, c->stream)) != cudaSuccess) return cuda_fail(c, e, "lb_autotune: fill");
    }
    const bool was_init = c->initialized;
    c->initialized = true;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
        return fail(c, LB_ECUDA, "lb_autotune: events");
    double best = 1e300;
    Cand win = cands[0];
    lb_status st = LB_OK;
    for (const Cand &cd : cands) {
        bool fits = true;
        if ((e = lbk::blocked_setup(c, cd.sched == lbk::kSchedTiles ? cd.K : 0, cd.tile, cd.threads, &fits)) != cudaSuccess) {
            st = cuda_fail(c, e, "lb_autotune");
            break;
        }
        if (!fits) continue;
        c->sched = c->run = cd.sched;
        const int64_t n = cd.K ? (trial_steps + cd.K - 1) / cd.K * cd.K : trial_steps;
        if ((st = lb_step(c, n)) != LB_OK) break;  // warm-up
        if ((e = cudaEventRecord(e0, c->stream)) != cudaSuccess) {
            st = cuda_fail(c, e, "lb_autotune");
            break;
        }
        if ((st = lb_step(c, n)) != LB_OK) break;
        float ms = 0.f;
        if ((e = cudaEventRecord(e1, c->stream)) != cudaSuccess || (e = cudaEventSynchronize(e1)) != cudaSuccess ||
            (e = cudaEventElapsedTime(&ms, e0, e1)) != cudaSuccess) {
            st = cuda_fail(c, e, "lb_autotune");
            break;
        }
        if (ms / n < best) {
            best = ms / n;
            win = cd;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaStreamSynchronize(c->stream);
    c->initialized = false;  // the trials overwrote the state: set it again
    c->step = 0;
    (void)was_init;
    if (st != LB_OK) win = cands[0];
    bool fits = true;
    if ((e = lbk::blocked_setup(c, win.sched == lbk::kSchedTiles ? win.K : 0, win.tile, win.threads, &fits)) != cudaSuccess)
        return cuda_fail(c, e, "lb_autotune");
    c->sched = c->run = win.sched;
    if (st != LB_OK) return st;
    if (choice) {
        choice[0] = win.K;
        choice[1] = win.tile;
        choice[2] = win.threads;
        choice[3] = 1e3 * best;
    }
    return LB_OK;
}

lb_status lb_get_boundary(const lb_ctx *c, int *kind)
{
    if (!c || !kind) return LB_EINVAL;
    for (int a = 0; a < c->d; ++a) kind[a] = ((c->geom.mirror >> a) & 1u) ? LB_MIRROR : LB_PERIODIC;
    return LB_OK;
}

lb_status lb_set_theta0(lb_ctx *c, const double *theta0, const double *grad)
{
    lbk::NvtxRange nvtx_range("lb_set_theta0");
    if (!c) return LB_EINVAL;
    if (!theta0) return fail(c, LB_EINVAL, "lb_set_theta0: theta0 is NULL");
    DeviceGuard dg(c);
    cudaError_t e;
    c->initialized = false;
    if (!grad) {
        if (!c->gradtmp) {
            e = cudaMalloc(&c->gradtmp, sizeof(double) * c->d * c->nodes);
            if (e != cudaSuccess) return cuda_fail(c, e, "lb_set_theta0: gradient buffer");
        }
        if ((e = lbk::launch_fd4_grad(c, theta0, c->gradtmp)) != cudaSuccess)
            return cuda_fail(c, e, "lb_set_theta0: fd4 launch");
        grad = c->gradtmp;
    }
    if ((e = clear_flags(c, 0, 3)) != cudaSuccess)
        return cuda_fail(c, e, "lb_set_theta0: flag reset");
    if (c->precision == LB_FX64) {
        // Fixed-point scale: max|theta0| * 2^F < 2^59.  Every moment sum is
        // bounded by sum_k |f_k|, which stays near theta for a stable run, so
        // 4 bits of headroom (16 max|theta0|) cover the sums and transients;
        // the initialisation flags any value beyond 4 max|theta0|.
        if ((e = lbk::launch_maxabs(c, theta0, c->nodes, c->dout)) != cudaSuccess ||
            (e = cudaStreamSynchronize(c->stream)) != cudaSuccess)
            return cuda_fail(c, e, "lb_set_theta0: max|theta0|");
        double mx = c->hout[0];
        if (c->fx_max > 0.0) {  // a slab: the scale of the whole grid (at least this part's maximum)
            if (!isfinite(mx) || mx > c->fx_max)
                return fail(c, LB_EINVAL, "lb_set_theta0: max|theta0| of this part exceeds the grid's maximum");
            mx = c->fx_max;
        }
        if (!(mx > 0.0) || !isfinite(mx)) return fail(c, LB_ENONPOS, "lb_set_theta0: theta0 must be finite and > 0");
        int ex = 0;
        frexp(mx, &ex);  // mx < 2^ex
        c->fx_bits = 59 - ex;
        if (c->fx_bits > 1000 || c->fx_bits < -1000)
            return fail(c, LB_EINVAL, "lb_set_theta0: theta0 magnitude outside the fixed-point range");
    }
    c->cur = 0;
    if ((e = lbk::launch_init(c, theta0, grad, c->dflag)) != cudaSuccess)
        return cuda_fail(c, e, "lb_set_theta0: init launch");
    if ((e = cudaStreamSynchronize(c->stream)) != cudaSuccess) return cuda_fail(c, e, "lb_set_theta0");
    const int flag = c->hflag[lbk::kFlagInit];
    if (flag & 2) return fail(c, LB_EINVAL, "lb_set_theta0: initial distributions exceed the fixed-point range");
    if (flag) return fail(c, LB_ENONPOS, "lb_set_theta0: theta0 must be finite and > 0 (and grad finite)");
    c->initialized = true;
    c->step = 0;
    return LB_OK;
}

lb_status lb_step(lb_ctx *c, int64_t nsteps)
{
    lbk::NvtxRange nvtx_range("lb_step");
    if (!c) return LB_EINVAL;
    if (nsteps < 0) return fail(c, LB_EINVAL, "lb_step: nsteps < 0");
    if (!c->initialized) return fail(c, LB_ESTATE, "lb_step: call lb_set_theta0 first");
    DeviceGuard dg(c);
    // Long runs replay recorded 32-sweep graphs (one host call per 32 sweeps);
    // while the caller's stream is being captured the sweeps are launched
    // directly so that they land in the caller's graph.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(c->stream, &cap) != cudaSuccess) cap = cudaStreamCaptureStatusActive;
    // Every launch below swaps the two buffers once, whatever its number of
    // steps.  A captured call is replayed from the buffer that it read, so there
    // the launches are cut such that an even number of steps ends in that buffer
    // again, as one sweep per launch does, and replays go on from one another.
    const bool held = cap != cudaStreamCaptureStatusNone;
    if (c->run == lbk::kSchedLine) {
        constexpr int64_t kMost = 1 << 20;  // steps per launch
        const int64_t least = lbk::line_least(c);
        while (nsteps >= least) {  // fewer below, one sweep per launch
            int64_t n = nsteps < kMost ? nsteps : kMost;
            if (held && n % 2 == 0 && --n < least) break;
            cudaError_t e = lbk::line_launch(c, c->f[c->cur], c->f[c->cur ^ 1], n);
            if (e != cudaSuccess) return cuda_fail(c, e, "lb_step: resident launch");
            c->cur ^= 1;
            c->step += n;
            nsteps -= n;
        }
    }
    const auto replay = [&]() {  // recorded sweeps
        while (cap == cudaStreamCaptureStatusNone && nsteps >= kGraphSteps) {
            cudaError_t e = cudaSuccess;
            if (!c->graph[c->cur]) e = record_sweeps(c, c->cur);
            if (e == cudaSuccess) e = cudaGraphLaunch(c->graph[c->cur], c->stream);
            if (e != cudaSuccess) return e;
            nsteps -= kGraphSteps;
            c->step += kGraphSteps;
        }
        return cudaSuccess;
    };
    cudaError_t er = cudaSuccess;
    if (c->run == lbk::kSchedMarch && c->march_short && (er = replay()) != cudaSuccess) return cuda_fail(c, er, "lb_step: graph");
    if (c->run == lbk::kSchedMarch && nsteps >= c->march.steps && !(c->march_short && held)) {
        // marching launches; the remainder below, one sweep per launch
        int64_t launches = nsteps / c->march.steps;
        if (held && c->march.steps % 2 == 0) launches -= launches % 2;
        for (; launches > 0; --launches) {
            cudaError_t e = lbk::march_launch(c, c->f[c->cur], c->f[c->cur ^ 1], c->stream);
            if (e != cudaSuccess) return cuda_fail(c, e, "lb_step: marching launch");
            c->cur ^= 1;
            c->step += c->march.steps;
            nsteps -= c->march.steps;
        }
    }
    if (c->run == lbk::kSchedTiles && c->tb_k > 0) {
        // blocked: launches of tb_k steps (recorded in graphs), then one launch for
        // the remainder.  The library's own choice runs a remainder of one step, or
        // two with tiles above 32 nodes, one sweep per launch: us per call, tiles /
        // sweeps, one step FP32 416^2 8.9 / 4.2, 256^2 6.2 / 4.2, fixed point 416^2
        // 10.3 / 6.2, 256^2 6.2 / 4.2; two steps FP32 416^2 10.3 / 8.3, 320^2 6.2 / 8.3.
        const int least = c->sched == lbk::kSchedAuto ? (c->tb_tile > 32 ? 3 : 2) : 1;
        cudaError_t e = cudaSuccess;
        const auto one = [&]() {
            e = least > 1 ? lbk::launch_sweep(c, c->f[c->cur], c->f[c->cur ^ 1])
                          : lbk::blocked_launch(c, c->f[c->cur], c->f[c->cur ^ 1], 1, c->stream);
            if (e != cudaSuccess) return false;
            c->cur ^= 1;
            ++c->step;
            --nsteps;
            return true;
        };
        const auto swaps = [&](int64_t n) {  // of the buffers, in n steps
            const int64_t rem = n % c->tb_k;
            return n / c->tb_k + (rem < least ? rem : 1);
        };
        while (held && (swaps(nsteps) - nsteps) % 2 != 0)  // a few steps on their own
            if (!one()) return cuda_fail(c, e, "lb_step: sweep launch");
        int64_t launches = nsteps / c->tb_k;
        const int rem = (int)(nsteps % c->tb_k);
        while (cap == cudaStreamCaptureStatusNone && launches >= kTbGraphLaunches) {
            if (!c->tb_graph[c->cur]) e = record_blocked(c, c->cur);
            if (e == cudaSuccess) e = cudaGraphLaunch(c->tb_graph[c->cur], c->stream);
            if (e != cudaSuccess) return cuda_fail(c, e, "lb_step: blocked graph");
            launches -= kTbGraphLaunches;
            c->step += kTbGraphLaunches * c->tb_k;
        }
        for (; launches > 0; --launches) {
            if ((e = lbk::blocked_launch(c, c->f[c->cur], c->f[c->cur ^ 1], c->tb_k, c->stream)) != cudaSuccess)
                return cuda_fail(c, e, "lb_step: blocked launch");
            c->cur ^= 1;
            c->step += c->tb_k;
        }
        nsteps = rem;
        if (rem >= least) {
            if ((e = lbk::blocked_launch(c, c->f[c->cur], c->f[c->cur ^ 1], rem, c->stream)) != cudaSuccess)
                return cuda_fail(c, e, "lb_step: blocked launch");
            c->cur ^= 1;
            c->step += rem;
            nsteps = 0;
        }
        while (nsteps > 0)
            if (!one()) return cuda_fail(c, e, "lb_step: sweep launch");
        return LB_OK;
    }
    if ((er = replay()) != cudaSuccess) return cuda_fail(c, er, "lb_step: graph");
    for (int64_t s = 0; s < nsteps; ++s) {
        cudaError_t e = lbk::launch_sweep(c, c->f[c->cur], c->f[c->cur ^ 1]);
        if (e != cudaSuccess) return cuda_fail(c, e, "lb_step: sweep launch");
        c->cur ^= 1;
        ++c->step;
    }
    return LB_OK;
}

lb_status lb_get_step(const lb_ctx *c, int64_t *n)
{
    if (!c || !n) return LB_EINVAL;
    *n = c->step;
    return LB_OK;
}

lb_status lb_macros(lb_ctx *c, double *theta, double *grad, double *u)
{
    lbk::NvtxRange nvtx_range("lb_macros");
    if (!c) return LB_EINVAL;
    if (!c->initialized) return fail(c, LB_ESTATE, "lb_macros: call lb_set_theta0 first");
    if (!theta && !grad && !u) return LB_OK;
    DeviceGuard dg(c);
    cudaError_t e = lbk::launch_macros(c, c->f[c->cur], theta, grad, u, c->dflag + lbk::kFlagRecover);
    if (e != cudaSuccess) return cuda_fail(c, e, "lb_macros: launch");
    // inside the caller's stream capture nothing can be read back: the flags
    // then wait for lb_check, lb_sum_theta or lb_reduce
    if (capturing(c->stream)) return LB_OK;
    return read_flags(c, "lb_macros");
}

lb_status lb_check(lb_ctx *c)
{
    lbk::NvtxRange nvtx_range("lb_check");
    if (!c) return LB_EINVAL;
    DeviceGuard dg(c);
    return read_flags(c, "lb_check");
}

lb_status lb_sum_theta(lb_ctx *c, double *out)
{
    lbk::NvtxRange nvtx_range("lb_sum_theta");
    if (!c || !out) return LB_EINVAL;
    if (!c->initialized) return fail(c, LB_ESTATE, "lb_sum_theta: call lb_set_theta0 first");
    DeviceGuard dg(c);
    cudaError_t e = lbk::launch_sum_state(c, c->f[c->cur], c->dout);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "lb_sum_theta");
    double v = c->hout[0];
    if (take_flag(c, lbk::kFlagRange)) {
        c->initialized = false;
        return fail(c, LB_EINVAL, "lb_sum_theta: a fixed-point distribution reached |f| >= 2^61 (the run is "
                                  "unstable: an FP64 run would overflow); set the state again");
    }
    if (c->precision == LB_FP32_SHIFTED) {
        // sum of the node weights: N_a per periodic axis, N_a - 1 per mirror axis
        double wn = 1.0;
        for (int a = 0; a < c->d; ++a) wn *= (double)(((c->geom.mirror >> a) & 1u) ? c->N[a] - 1 : c->N[a]);
        v += c->theta_ref * wn;
    }
    *out = v;
    return LB_OK;
}

lb_status lb_reduce(lb_ctx *c, const double *theta, const double *u, const double *ex_theta, const double *ex_u,
                    double *out)
{
    lbk::NvtxRange nvtx_range("lb_reduce");
    if (!c || !out) return LB_EINVAL;
    if (!theta || !ex_theta) return fail(c, LB_EINVAL, "lb_reduce: theta and exact_theta are required");
    if ((u == nullptr) != (ex_u == nullptr)) return fail(c, LB_EINVAL, "lb_reduce: u and exact_u go together");
    DeviceGuard dg(c);
    const int ns = 3 * (c->d + 1) + 1;
    cudaError_t e = lbk::launch_norms(c, theta, u, ex_theta, ex_u, c->dout);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "lb_reduce");
    double raw[lbk::kRedSlots];
    for (int k = 0; k < ns; ++k) raw[k] = c->hout[k];
    const int flag = take_flag(c, lbk::kFlagRecover);
    const double n = (double)c->nodes;
    for (int v = 0; v <= c->d; ++v) {
        const double se = raw[3 * v], mx = raw[3 * v + 1], sx = raw[3 * v + 2];
        const bool have = (v == 0) || u;
        out[3 * v + 0] = have ? sqrt(se / n) : NAN;
        out[3 * v + 1] = have ? mx : NAN;
        out[3 * v + 2] = have ? (sx > 0 ? sqrt(se / sx) : (se > 0 ? INFINITY : 0.0)) : NAN;
    }
    out[3 * (c->d + 1)] = raw[ns - 1];
    if (flag & 4) {
        c->initialized = false;
        return fail(c, LB_ETIMEOUT, "lb_macros: a shared-memory staging wait timed out");
    }
    if (flag) return fail(c, LB_ENONPOS, "lb_macros saw theta <= 0 or non-finite");
    return LB_OK;
}

lb_status lb_state_layout(const lb_ctx *c, int64_t *pitch, int64_t *slab, int64_t *elem_bytes)
{
    if (!c) return LB_EINVAL;
    if (pitch) *pitch = c->geom.pitch;
    if (slab) *slab = c->geom.slab;
    if (elem_bytes) *elem_bytes = (int64_t)c->elem;
    return LB_OK;
}

lb_status lb_save_state(lb_ctx *c, void *buf)
{
    lbk::NvtxRange nvtx_range("lb_save_state");
    if (!c || !buf) return LB_EINVAL;
    if (!c->initialized) return fail(c, LB_ESTATE, "lb_save_state: nothing to save");
    DeviceGuard dg(c);
    cudaError_t e = cudaMemcpyAsync(buf, c->f[c->cur], (size_t)c->q * c->geom.slab * c->elem,
                                    cudaMemcpyDeviceToDevice, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "lb_save_state");
    return LB_OK;
}

lb_status lb_load_state(lb_ctx *c, const void *buf, int64_t step)
{
    lbk::NvtxRange nvtx_range("lb_load_state");
    if (!c || !buf || step < 0) return LB_EINVAL;
    DeviceGuard dg(c);
    cudaError_t e = cudaMemcpyAsync(c->f[c->cur], buf, (size_t)c->q * c->geom.slab * c->elem,
                                    cudaMemcpyDeviceToDevice, c->stream);
    if (e == cudaSuccess) e = clear_flags(c, lbk::kFlagRecover, 2);
    if (e != cudaSuccess) return cuda_fail(c, e, "lb_load_state");
    c->initialized = true;
    c->step = step;
    return LB_OK;
}

const char *lb_last_error(const lb_ctx *c)
{
    if (!c) return g_create_err.c_str();
    return c->err.c_str();
}

}  // extern "C"
