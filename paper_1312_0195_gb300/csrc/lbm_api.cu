// lbm_api.cu -- the C ABI of include/lbm.h for grids: validation, ownership,
// CUDA-graph replay of the fused step, residual checks and field read-back.
#include "lbm_internal.h"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <cstdlib>
#include <map>
#include <mutex>
#include <string>
#include <tuple>

namespace lbm {

static std::atomic<int64_t> g_launches{0};
void count_launches(int64_t n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

static thread_local std::string t_err;

lbm_status fail(lbm_status s, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    t_err = buf;
    return s;
}

#define LBM_CUDA(call)                                                                      \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess) {                                                            \
            cudaGetLastError();                                                             \
            return lbm::fail(e_ == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA,      \
                             "%s failed: %s", #call, cudaGetErrorString(e_));               \
        }                                                                                   \
    } while (0)

// Device pointer test without touching the memory.
bool is_device_ptr(const void *p)
{
    if (!p) return false;
    cudaPointerAttributes at;
    cudaError_t e = cudaPointerGetAttributes(&at, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

static bool finite(double v) { return std::isfinite(v); }

lbm_status validate_params(const lbm_params *p)
{
    if (!p) return fail(LBM_EINVAL, "params is NULL");
    if (p->nx < 1 || p->ny < 1) return fail(LBM_EINVAL, "nx, ny must be >= 1 (got %d, %d)", p->nx, p->ny);
    if ((int64_t)p->nx * p->ny > (int64_t)1 << 31)
        return fail(LBM_EINVAL, "nx * ny must be <= 2^31 cells");
    if (!finite(p->tau) || p->tau < 0.5) return fail(LBM_EINVAL, "tau must be finite and >= 0.5 (got %g)", p->tau);
    if (!finite(p->nu)) return fail(LBM_EINVAL, "nu must be finite");
    if (!finite(p->eps) || p->eps < 0.0) return fail(LBM_EINVAL, "eps must be finite and >= 0 (got %g)", p->eps);
    if (!finite(p->gx) || !finite(p->gy)) return fail(LBM_EINVAL, "gx, gy must be finite");
    if (p->bc != LBM_BC_PERIODIC && p->bc != LBM_BC_WALLS_Y) return fail(LBM_EINVAL, "unknown bc %d", p->bc);
    if (p->storage != LBM_F32 && p->storage != LBM_F16 && p->storage != LBM_F64)
        return fail(LBM_EINVAL, "unknown storage %d", p->storage);
    if (!finite(p->scale) || p->scale < 0.0) return fail(LBM_EINVAL, "scale must be finite and >= 0");
    if (p->force_model != 0 && p->force_model != 1) return fail(LBM_EINVAL, "unknown force_model %d", p->force_model);
    if (p->scale > 0.0) {
        int ex2;
        double m = std::frexp(p->scale, &ex2);
        if (m != 0.5) return fail(LBM_EINVAL, "scale must be a power of two (got %g)", p->scale);
    }
    return LBM_OK;
}

double effective_nu(const lbm_params *p) { return p->nu < 0.0 ? (p->tau - 0.5) / 3.0 : p->nu; }

size_t storage_bytes(int storage) { return storage == LBM_F64 ? 8 : (storage == LBM_F16 ? 2 : 4); }

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev)
    {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
        else prev = -1;
    }
    ~DeviceGuard()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

int sm_count(int dev)
{
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        n = 1;
    }
    return n < 1 ? 1 : n;
}

}  // namespace lbm

using namespace lbm;

constexpr int TILE_CHUNK = 4096;     // steps of one launch of the tile kernel at most

// What a call reads back, in one piece of device memory.
struct Outcome {
    double sums[4];        // of moments_kernel: max |du|, max |u|, sum u, sum v
    unsigned flags[2];     // error bits of the coefficients, bits of the largest finite kappa
    unsigned bits[2];      // max |du|, max |u| of a check inside a pass or in the tile kernel, as floats' bits
    int tile_err;          // a wait between the tile kernel's CTAs gave up
    int pad;
};

struct lbm_grid {
    lbm_params p;
    double nu = 0, S = 1;
    int dev = 0;
    int coef_mode = COEF_SCALAR;
    bool has_g = false;
    cudaStream_t stream = nullptr;   // user's stream
    cudaStream_t cap = nullptr;      // private stream used only for graph capture, made when first needed
    int64_t plane = 0;
    void *buf[2] = {nullptr, nullptr};
    int cur = 0;                     // buf[cur] = post-collision state of the last step
    void *coef = nullptr;
    void *gfield = nullptr;
    double *partials = nullptr;
    Outcome *outcome = nullptr;      // device
    Outcome *h_outcome = nullptr;    // pinned, for runs that stop at a tolerance: made when first needed, since it
                                     // costs 0.28 ms with its release; other calls read once, into the stack
    GridLaunch L{};
    int64_t t = 0;
    int sms = 1;
    bool lost = false;               // a step gave up halfway: no valid state until one is loaded
    bool fused = false;              // several steps per pass (multistep.cu) where a call takes several
    TileGeom tiles{0, 0, 0, 0, 0};   // ntx > 0: a small lattice, stepped in shared memory (tiles.cu)
    void *mem = nullptr;             // the one allocation behind every device pointer of the grid
    void *tile_exch = nullptr;       // exchanges between its CTAs
    unsigned tile_base = 0;          // exchanges so far, and more
    unsigned *tile_result = nullptr; // the checks' maxima of one launch, behind the exchanges
    struct Graph {
        cudaGraphExec_t exec;
        int kernels;                 // launches it holds
        int cur;                     // buffer that holds the state after it
    };
    std::map<std::tuple<int, int, int, int>, Graph> graphs;
};

namespace lbm {

// Fills the step / moment argument blocks for one launch of grid g reading src.
template <typename T, typename CT>
static StepArgs<T, CT> make_args(const lbm_grid *g, const void *src, void *dst)
{
    StepArgs<T, CT> a;
    a.nx = g->p.nx;
    a.ny = g->p.ny;
    a.plane = g->plane;
    a.omega = (CT)(1.0 / g->p.tau);
    a.two_tau = (CT)(2.0 * g->p.tau);
    a.one_m_two_tau = (CT)(1.0 - 2.0 * g->p.tau);
    a.half_eps = (CT)(0.5 * g->p.eps);
    a.gx = (CT)g->p.gx;
    a.gy = (CT)g->p.gy;
    a.rho0 = (CT)g->S;
    a.guo = g->p.force_model == 1 ? 1 : 0;
    a.guo_c = (CT)(6.0 * (1.0 - 1.0 / (2.0 * g->p.tau)));
    a.src = static_cast<const T *>(src);
    a.dst = static_cast<T *>(dst);
    a.coef = static_cast<const CT *>(g->coef);
    a.gfield = static_cast<const CT *>(g->gfield);
    return a;
}

static cudaError_t enqueue_step(const lbm_grid *g, int src_idx, cudaStream_t st)
{
    const void *src = g->buf[src_idx];
    void *dst = g->buf[1 - src_idx];
    const bool walls = g->p.bc == LBM_BC_WALLS_Y;
    switch (g->p.storage) {
    case LBM_F32: {
        auto a = make_args<float, float>(g, src, dst);
        return launch_step(LBM_F32, g->coef_mode, g->has_g, walls, &a, g->L, st);
    }
    case LBM_F16: {
        auto a = make_args<__half, float>(g, src, dst);
        return launch_step(LBM_F16, g->coef_mode, g->has_g, walls, &a, g->L, st);
    }
    default: {
        auto a = make_args<double, double>(g, src, dst);
        return launch_step(LBM_F64, g->coef_mode, g->has_g, walls, &a, g->L, st);
    }
    }
}

// Moment pass over buf[cur_idx] (and buf[prev_idx] when prev_idx >= 0).
static cudaError_t enqueue_moments(const lbm_grid *g, int cur_idx, int prev_idx, float *rho, float *u, float *v,
                                   cudaStream_t st)
{
    const bool walls = g->p.bc == LBM_BC_WALLS_Y;
    const void *prev = prev_idx >= 0 ? g->buf[prev_idx] : nullptr;
    switch (g->p.storage) {
    case LBM_F32: {
        MomArgs<float, float> m{make_args<float, float>(g, g->buf[cur_idx], nullptr),
                                static_cast<const float *>(prev), 1.0f, rho, u, v, g->partials};
        return launch_moments(LBM_F32, g->coef_mode, g->has_g, walls, &m, g->L, st);
    }
    case LBM_F16: {
        MomArgs<__half, float> m{make_args<__half, float>(g, g->buf[cur_idx], nullptr),
                                 static_cast<const __half *>(prev), (float)(1.0 / g->S), rho, u, v, g->partials};
        return launch_moments(LBM_F16, g->coef_mode, g->has_g, walls, &m, g->L, st);
    }
    default: {
        MomArgs<double, double> m{make_args<double, double>(g, g->buf[cur_idx], nullptr),
                                  static_cast<const double *>(prev), 1.0, rho, u, v, g->partials};
        return launch_moments(LBM_F64, g->coef_mode, g->has_g, walls, &m, g->L, st);
    }
    }
}

// nlev steps in one pass over memory (multistep.cu); check: with the residual's maxima after the last but one.
static cudaError_t enqueue_multi(const lbm_grid *g, int src_idx, int nlev, unsigned *check, cudaStream_t st)
{
    const void *src = g->buf[src_idx];
    void *dst = g->buf[1 - src_idx];
    const bool walls = g->p.bc == LBM_BC_WALLS_Y;
    if (g->p.storage == LBM_F16) {
        auto a = make_args<__half, float>(g, src, dst);
        return launch_multistep(LBM_F16, g->coef_mode, g->has_g, walls, &a, nlev, g->sms, check, st);
    }
    auto a = make_args<float, float>(g, src, dst);
    return launch_multistep(LBM_F32, g->coef_mode, g->has_g, walls, &a, nlev, g->sms, check, st);
}

// n steps in one launch, the lattice resident in shared memory (tiles.cu), with the checks that fall into them
// (check_every > 0); *checks: how many. Leaves the newest state in buf[cur], the last check's maxima in the
// outcome's bits.
static cudaError_t enqueue_tiles(lbm_grid *g, int n, int check_every, int *checks)
{
    TileRun run{n, 0, check_every, g->tile_result, g->tile_exch, g->tile_base, &g->outcome->tile_err,
                (int)std::min(TILE_POLLS * local_time_limit(), 2e9)};
    *checks = 0;
    if (check_every > 0) {
        run.first_check = (int)(check_every - g->t % check_every);
        *checks = n >= run.first_check ? 1 + (n - run.first_check) / check_every : 0;
        if (*checks == 0) run.check_every = 0;
    }
    cudaError_t e = cudaSuccess;
    if (*checks > 0) e = cudaMemsetAsync(g->tile_result, 0, 2 * sizeof(unsigned) * *checks, g->stream);
    if (e != cudaSuccess) return e;
    const void *src = g->buf[g->cur];
    void *dst = g->buf[1 - g->cur];
    const bool walls = g->p.bc == LBM_BC_WALLS_Y;
    if (g->p.storage == LBM_F16) {
        auto a = make_args<__half, float>(g, src, dst);
        e = launch_tiles(LBM_F16, g->coef_mode, g->has_g, walls, &a, g->tiles, run, g->stream);
    } else {
        auto a = make_args<float, float>(g, src, dst);
        e = launch_tiles(LBM_F32, g->coef_mode, g->has_g, walls, &a, g->tiles, run, g->stream);
    }
    if (e == cudaSuccess && *checks > 0)
        e = cudaMemcpyAsync(g->outcome->bits, g->tile_result + 2 * (*checks - 1), 2 * sizeof(unsigned),
                            cudaMemcpyDeviceToDevice, g->stream);
    if (e != cudaSuccess) return e;
    g->tile_base += n / TILE_HALO + 1;
    g->cur = 1 - g->cur;
    return e;
}

// The tile kernel's launches under way on a device together take no more CTAs than it has SMs, one each: the CTAs of a
// launch wait for one another, and nothing promises that those of two launches, on two streams and short of SMs, become
// resident in turn and not each in part. A call that finds no room steps in passes, with the same bits.
constexpr int TILE_DEVICES = 64;
static std::atomic<int> g_tile_ctas[TILE_DEVICES];
struct TileTurn {
    std::atomic<int> *taken = nullptr;
    int ctas = 0;
    bool take(const lbm_grid *g)
    {
        if (g->tiles.ntx == 0 || g->dev >= TILE_DEVICES) return false;
        std::atomic<int> &n = g_tile_ctas[g->dev];
        if (n.fetch_add(g->tiles.ctas) + g->tiles.ctas > g->sms) {
            n.fetch_sub(g->tiles.ctas);
            return false;
        }
        taken = &n;
        ctas = g->tiles.ctas;
        return true;
    }
    ~TileTurn()
    {
        if (taken) taken->fetch_sub(ctas);
    }
};

// LBM_OK, unless the grid holds no valid state.
static lbm_status valid_state(const lbm_grid *g)
{
    if (!g->lost) return LBM_OK;
    return fail(LBM_ETIMEOUT, "an earlier step of this grid gave up halfway: load a state before going on");
}

// The outcome of the calls so far, after a synchronisation with the grid's stream.
static cudaError_t read_outcome(lbm_grid *g, Outcome *o)
{
    Outcome *to = g->h_outcome ? g->h_outcome : o;
    cudaError_t e = cudaMemcpyAsync(to, g->outcome, sizeof *to, cudaMemcpyDeviceToHost, g->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
    if (e == cudaSuccess && to != o) *o = *to;
    return e;
}

// The residual of the last check, which left its maxima in bits or in sums.
static double residual_of(const Outcome &o, bool as_bits)
{
    float m[2];
    std::memcpy(m, o.bits, sizeof m);
    const double dmax = as_bits ? m[0] : o.sums[0], umax = as_bits ? m[1] : o.sums[1];
    return umax > 0.0 ? dmax / umax : dmax;
}

// Graph of n steps starting from buf[parity], optionally followed by the residual pass (moments of
// the last two states, reduction, copy to pinned host). Where the grid fuses steps, the passes take
// MULTISTEP_MAX steps each; with `pair` the last step is one of its own, so that the two
// buffers end up holding the last two states (the residual and a checkpoint read both). check = CHECK_INSIDE: the
// residual after step n - 1 comes from the last pass, of MULTISTEP_MAX steps, which has both states' velocities at
// hand: 4096 x 4096 with a check every 64 steps then takes 16 equal passes, where a shorter pass, a single
// step and the residual pass used to take the place of the last.
constexpr int CHECK_INSIDE = 2;
static lbm_status get_graph(lbm_grid *g, int n, int parity, int check, int pair, lbm_grid::Graph *out)
{
    if (!g->fused) pair = 0;
    auto key = std::make_tuple(n, parity, check, pair);
    auto it = g->graphs.find(key);
    if (it != g->graphs.end()) {
        *out = it->second;
        return LBM_OK;
    }
    cudaGraph_t graph = nullptr;
    if (!g->cap) LBM_CUDA(cudaStreamCreateWithFlags(&g->cap, cudaStreamNonBlocking));
    LBM_CUDA(cudaStreamBeginCapture(g->cap, cudaStreamCaptureModeThreadLocal));
    cudaError_t err = cudaSuccess;
    int idx = parity, kernels = 0;
    const bool inside = check == CHECK_INSIDE;
    if (inside) err = cudaMemsetAsync(g->outcome->bits, 0, sizeof g->outcome->bits, g->cap);
    for (int left = n; left > 0 && err == cudaSuccess; ++kernels) {
        int take = 1;
        const bool last = inside && left == MULTISTEP_MAX;
        if (g->fused) {
            take = inside && !last ? left - MULTISTEP_MAX : left - (pair || check == 1 ? 1 : 0);
            take = take < 1 ? 1 : (take > MULTISTEP_MAX ? MULTISTEP_MAX : take);
        }
        err = take > 1 ? enqueue_multi(g, idx, take, last ? g->outcome->bits : nullptr, g->cap)
                       : enqueue_step(g, idx, g->cap);
        idx = 1 - idx;
        left -= take;
    }
    if (check == 1 && err == cudaSuccess) {
        err = enqueue_moments(g, idx, 1 - idx, nullptr, nullptr, nullptr, g->cap);
        if (err == cudaSuccess) err = launch_reduce_partials(g->partials, g->L.mom_blocks, g->outcome->sums, g->cap);
        kernels += 2;
    }
    cudaError_t e2 = cudaStreamEndCapture(g->cap, &graph);
    if (err != cudaSuccess || e2 != cudaSuccess) {
        if (graph) cudaGraphDestroy(graph);
        cudaGetLastError();
        return fail(LBM_ECUDA, "graph capture failed: %s",
                    cudaGetErrorString(err != cudaSuccess ? err : e2));
    }
    cudaGraphExec_t exec = nullptr;
    cudaError_t e3 = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e3 != cudaSuccess) {
        cudaGetLastError();
        return fail(LBM_ECUDA, "graph instantiation failed: %s", cudaGetErrorString(e3));
    }
    *out = g->graphs[key] = {exec, kernels, idx};
    return LBM_OK;
}

// ---------------------------------------------------------------- autotuner
// Picks the fused step's launch shape (threads per block, resident blocks per SM,
// cells per thread) by timing candidates on the grid itself right after
// creation, then resets the state to rest. The choice is cached per lattice
// shape and variant for the whole process. Results do not depend on the launch
// shape (every cell's arithmetic and every reduction order are fixed), so
// tuning never changes answers. LBM_AUTOTUNE=0 disables it.
struct TuneKey {
    int nx, ny, storage, coef, gf, walls;
    bool operator<(const TuneKey &o) const
    {
        return std::tie(nx, ny, storage, coef, gf, walls) < std::tie(o.nx, o.ny, o.storage, o.coef, o.gf, o.walls);
    }
};
static std::map<TuneKey, GridLaunch> g_tuned;
static std::mutex g_tune_mu;

static lbm_status autotune(lbm_grid *g)
{
    const char *env = std::getenv("LBM_AUTOTUNE");
    if (env && env[0] == '0') return LBM_OK;
    if (std::getenv("LBM_STEP_VEC")) return LBM_OK;      // a variant was chosen explicitly
    if (g->p.storage == LBM_F64) return LBM_OK;          // bound by the FP64 pipe: see grid_create_impl
    const int64_t n = (int64_t)g->p.nx * g->p.ny;
    if (n < ((int64_t)1 << 20)) return LBM_OK;      // small lattices are launch-bound: keep the default
    const bool walls = g->p.bc == LBM_BC_WALLS_Y;
    const TuneKey key{g->p.nx, g->p.ny, g->p.storage, g->coef_mode, g->has_g, walls};
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tuned.find(key);
        if (it != g_tuned.end()) {
            g->L.step_blocks = it->second.step_blocks;
            g->L.step_threads = it->second.step_threads;
            g->L.step_vec = it->second.step_vec;
            return LBM_OK;
        }
    }
    const int sms = sm_count(g->dev);
    // cells-per-thread candidates: the default for this storage and row length, then the other
    // built packs (FP32: 8; FP16: 4 and 2, fewer registers and more resident warps)
    const int dvec = step_vec(g->p.storage, g->p.nx);
    int vecs[3] = {dvec, 0, 0};
    int nvec = 1;
    const int others[2] = {g->p.storage == LBM_F32 ? 8 : (g->p.storage == LBM_F16 ? 4 : 0),
                           g->p.storage == LBM_F16 ? 2 : 0};
    for (int o : others)
        if (o && o != dvec && step_vec_ok(g->p.storage, g->p.nx, o)) vecs[nvec++] = o;
    GridLaunch best = g->L;
    float best_ms = -1.0f;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    LBM_CUDA(cudaEventCreate(&e0));
    LBM_CUDA(cudaEventCreate(&e1));
    const int warm = 2, timed = 8;
    for (int vi = 0; vi < nvec; ++vi) {
        const int vec = vecs[vi];
        for (int threads : {128, 256, 512}) {
            const int occ = step_blocks_per_sm(g->p.storage, g->coef_mode, g->has_g, walls, g->p.nx, threads, vec);
            const int64_t chunks = n / vec;
            const int64_t want = (chunks + threads - 1) / threads;
            for (int bpsm : {occ, occ > 1 ? occ / 2 : 0}) {
                if (bpsm < 1) continue;
                const int64_t cap = (int64_t)sms * bpsm;
                GridLaunch L = g->L;
                L.step_threads = threads;
                L.step_vec = vec;
                L.step_blocks = (int)(want < cap ? want : cap);
                g->L = L;
                cudaError_t err = cudaSuccess;
                for (int i = 0; i < warm && err == cudaSuccess; ++i) { err = enqueue_step(g, g->cur, g->stream); g->cur ^= 1; }
                cudaEventRecord(e0, g->stream);
                for (int i = 0; i < timed && err == cudaSuccess; ++i) { err = enqueue_step(g, g->cur, g->stream); g->cur ^= 1; }
                cudaEventRecord(e1, g->stream);
                count_launches(warm + timed);
                if (err == cudaSuccess) err = cudaEventSynchronize(e1);
                float ms = 0.0f;
                if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e0, e1);
                if (err != cudaSuccess) {
                    cudaGetLastError();
                    continue;
                }
                if (best_ms < 0.0f || ms < best_ms) {
                    best_ms = ms;
                    best = L;
                }
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    g->L.step_blocks = best.step_blocks;
    g->L.step_threads = best.step_threads;
    g->L.step_vec = best.step_vec;
    // back to rest: zero deviations in both buffers
    const size_t bytes = 9 * g->plane * storage_bytes(g->p.storage);
    LBM_CUDA(cudaMemsetAsync(g->buf[0], 0, bytes, g->stream));
    LBM_CUDA(cudaMemsetAsync(g->buf[1], 0, bytes, g->stream));
    LBM_CUDA(cudaStreamSynchronize(g->stream));
    g->cur = 0;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tuned[key] = g->L;
    return LBM_OK;
}

static void free_grid(lbm_grid *g)
{
    if (!g) return;
    for (auto &kv : g->graphs) cudaGraphExecDestroy(kv.second.exec);
    g->graphs.clear();
    cudaFree(g->mem);
    if (g->h_outcome) cudaFreeHost(g->h_outcome);
    if (g->cap) cudaStreamDestroy(g->cap);
    cudaGetLastError();
    delete g;
}

// Shared by lbm_grid_create (scalar kappa) and the coarse run (tensor K*).
// kstar_scale multiplies K* before the coefficient is formed.
lbm_status grid_create_impl(const lbm_params *p, const float *kappa_dev, const double *kstar_dev,
                            double kstar_scale, const float *g_field_dev, void *cuda_stream, lbm_grid **out)
{
    if (!out) return fail(LBM_EINVAL, "out is NULL");
    *out = nullptr;
    lbm_status s = validate_params(p);
    if (s != LBM_OK) return s;
    if (kappa_dev && !is_device_ptr(kappa_dev)) return fail(LBM_EINVAL, "kappa_dev is not a device pointer");
    if (kstar_dev && !is_device_ptr(kstar_dev)) return fail(LBM_EINVAL, "keff_dev is not a device pointer");
    if (!kappa_dev && !kstar_dev) return fail(LBM_EINVAL, "kappa_dev is NULL");
    if (g_field_dev && !is_device_ptr(g_field_dev)) return fail(LBM_EINVAL, "g_field_dev is not a device pointer");

    lbm_grid *g = new lbm_grid();
    g->p = *p;
    g->nu = effective_nu(p);
    g->coef_mode = kstar_dev ? COEF_TENSOR : COEF_SCALAR;
    g->has_g = g_field_dev != nullptr;
    g->stream = static_cast<cudaStream_t>(cuda_stream);
    if (cudaGetDevice(&g->dev) != cudaSuccess) {
        cudaGetLastError();
        delete g;
        return fail(LBM_ECUDA, "no CUDA device");
    }
    const int64_t n = (int64_t)p->nx * p->ny;
    g->plane = (n + 63) / 64 * 64;
    const size_t sb = storage_bytes(p->storage);
    const size_t cb = p->storage == LBM_F64 ? 8 : 4;
    const int ncoef = kstar_dev ? 4 : 1;

    auto bail = [&](lbm_status st) { free_grid(g); return st; };
#define LBM_GRID_CUDA(call)                                                                 \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess) {                                                            \
            cudaGetLastError();                                                             \
            return bail(fail(e_ == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA,      \
                             "%s failed: %s", #call, cudaGetErrorString(e_)));              \
        }                                                                                   \
    } while (0)

    // launch shapes: persistent step grid, fixed moment grid (fixed reduction order)
    const int sms = sm_count(g->dev);
    g->sms = sms;
    const bool several = !std::getenv("LBM_STEP_VEC") &&
                         multistep_ok(p->storage, g->coef_mode, p->nx, p->ny, p->force_model);
    g->fused = several && multistep_pays(p->storage, p->nx, p->ny, sms);
    const int vec = step_vec(p->storage, p->nx);
    const int64_t chunks = n / vec;
    const bool f64 = p->storage == LBM_F64;
    // FP64 is bound by its arithmetic pipe: one chunk per thread in small blocks keeps every SM busy to the
    // end (1000 x 1000: 0.108 ms a step against 0.116 with a persistent grid's uneven last round)
    g->L.step_threads = f64 ? 128 : 256;
    g->L.step_vec = 0;
    const int64_t want = (chunks + g->L.step_threads - 1) / g->L.step_threads;
    const int64_t cap = (int64_t)sms * step_blocks_per_sm(p->storage, g->coef_mode, g->has_g,
                                                          p->bc == LBM_BC_WALLS_Y, p->nx, g->L.step_threads);
    g->L.step_blocks = (int)(want < 1 ? 1 : (want < cap || f64 ? want : cap));
    // LBM_STEP_VEC=v selects another built cells-per-thread variant of the step (the arithmetic per
    // cell is the same in every variant) and turns the autotuner and the fused passes off for this grid
    if (const char *ev = std::getenv("LBM_STEP_VEC")) {
        const int v = std::atoi(ev);
        if (step_vec_ok(p->storage, p->nx, v)) {
            g->L.step_vec = v;
            const int64_t w2 = (n / v + g->L.step_threads - 1) / g->L.step_threads;
            const int64_t c2 = (int64_t)sms * step_blocks_per_sm(p->storage, g->coef_mode, g->has_g,
                                                                 p->bc == LBM_BC_WALLS_Y, p->nx, g->L.step_threads, v);
            g->L.step_blocks = (int)(w2 < c2 ? (w2 < 1 ? 1 : w2) : c2);
        }
    }
    g->L.mom_threads = 256;
    const int64_t mwant = (chunks + 255) / 256;
    const int64_t mcap = (int64_t)sms * 2;   // 128 registers: two 256-thread blocks per SM
    g->L.mom_blocks = (int)(mwant < mcap ? (mwant < 1 ? 1 : mwant) : mcap);

    if (several) g->tiles = tile_geometry(p->storage, g->coef_mode, g->has_g, p->nx, p->ny, sms);
    // One allocation for everything, zeroed in one go: with one each, a memset each, a capture stream and pinned
    // memory a coarse run of 1250 steps on 256 x 256 took 2.3 ms instead of 1.8. No room for the exchanges of the
    // tile kernel: stepped in passes over memory.
    auto aligned = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
    const size_t b_buf = aligned(9 * g->plane * sb), b_coef = aligned(ncoef * g->plane * cb);
    const size_t b_field = g->has_g ? aligned(2 * g->plane * cb) : 0;
    const size_t b_small = aligned(4 * sizeof(double) * g->L.mom_blocks + sizeof(Outcome));
    const size_t base = 2 * b_buf + b_coef + b_field + b_small;
    size_t exch = 0;
    if (g->tiles.ntx > 0) {
        exch = aligned(tile_exchange_bytes(n));
        if (cudaMalloc(&g->mem, base + exch + 2 * sizeof(unsigned) * TILE_CHUNK) != cudaSuccess) {
            cudaGetLastError();
            g->mem = nullptr;
            g->tiles.ntx = 0;
            exch = 0;
        }
    }
    if (g->tiles.ntx == 0) LBM_GRID_CUDA(cudaMalloc(&g->mem, base));
    char *m = static_cast<char *>(g->mem);
    g->buf[0] = m;
    g->buf[1] = m + b_buf;
    g->coef = m + 2 * b_buf;
    if (g->has_g) g->gfield = m + 2 * b_buf + b_coef;
    g->partials = reinterpret_cast<double *>(m + 2 * b_buf + b_coef + b_field);
    g->outcome = reinterpret_cast<Outcome *>(g->partials + 4 * g->L.mom_blocks);
    g->tile_exch = m + base;
    g->tile_result = reinterpret_cast<unsigned *>(m + base + exch);

    cudaStream_t st = g->stream;
    // rest state: deviations are zero in both buffers (state of step -1 and -2)
    LBM_GRID_CUDA(cudaMemsetAsync(m, 0, base + exch, st));
    if (kstar_dev) {
        // The coarse run passes a K* already divided by r^2 when kstar_scale != 1.
        LBM_GRID_CUDA(launch_coef_tensor(p->storage, kstar_dev, g->coef, n, g->plane,
                                         0.5 * p->eps * g->nu / kstar_scale, g->outcome->flags, st));
        count_launches(1);
    } else {
        LBM_GRID_CUDA(launch_coef_scalar(p->storage, kappa_dev, g->coef, n, g->plane, p->eps * g->nu, g->outcome->flags,
                                         g->outcome->flags + 1, st));
        count_launches(1);
    }
    if (g->has_g) {
        LBM_GRID_CUDA(launch_copy_force(p->storage, g_field_dev, g->gfield, n, g->plane, 1.0, st));
        count_launches(1);
    }
    unsigned hflags[2] = {0, 0};
    LBM_GRID_CUDA(cudaMemcpyAsync(hflags, g->outcome->flags, sizeof hflags, cudaMemcpyDeviceToHost, st));
    LBM_GRID_CUDA(cudaStreamSynchronize(st));
    if (hflags[0] & 1u) return bail(fail(LBM_EINVAL, kstar_dev ? "K* has non-finite entries"
                                                                 : "kappa has negative or NaN entries"));
    if (hflags[0] & 2u) return bail(fail(LBM_EINVAL, "K* + (eps nu / 2) I is singular in some cell"));

    if (p->storage == LBM_F16) {
        if (p->scale > 0.0) {
            g->S = p->scale;
        } else {
            // Largest deviation ~ w_1 * 3 * |u|, |u| <~ kappa_max |G| / nu; aim that at 2^12
            // (headroom of 16x below the FP16 maximum for transients and pressure).
            float kmax;
            std::memcpy(&kmax, &hflags[1], sizeof kmax);
            double gmag = std::fabs(p->gx) + std::fabs(p->gy);
            double umax = (g->nu > 0.0 && kmax > 0.0f) ? (double)kmax * gmag / g->nu : gmag * 1e3;
            if (!(umax > 0.0)) umax = 1e-3;
            if (umax > 0.1) umax = 0.1;
            int e2 = (int)std::floor(std::log2(4096.0 / umax));
            if (e2 > 60) e2 = 60;
            if (e2 < 0) e2 = 0;
            g->S = std::ldexp(1.0, e2);
        }
    }
    s = autotune(g);
    if (s != LBM_OK) return bail(s);
    *out = g;
    return LBM_OK;
#undef LBM_GRID_CUDA
}

}  // namespace lbm

extern "C" {

const char *lbm_last_error(void) { return lbm::t_err.c_str(); }

int64_t lbm_launch_count(void) { return lbm::g_launches.load(); }

lbm_status lbm_grid_create(const lbm_params *p, const float *kappa_dev, const float *g_field_dev, void *cuda_stream,
                           lbm_grid **out)
{
    if (!kappa_dev) {
        if (out) *out = nullptr;
        lbm_status s = validate_params(p);
        return s != LBM_OK ? s : fail(LBM_EINVAL, "kappa_dev is NULL");
    }
    return grid_create_impl(p, kappa_dev, nullptr, 1.0, g_field_dev, cuda_stream, out);
}

lbm_status lbm_grid_destroy(lbm_grid *g)
{
    if (!g) return LBM_OK;
    DeviceGuard dg(g->dev);
    cudaStreamSynchronize(g->stream);
    cudaGetLastError();
    free_grid(g);
    return LBM_OK;
}

lbm_status lbm_step(lbm_grid *g, int64_t max_steps, double tol_rel, int32_t check_every, int64_t *steps_done,
                    double *residual)
{
    if (steps_done) *steps_done = 0;
    if (residual) *residual = -1.0;
    if (!g) return fail(LBM_EINVAL, "grid is NULL");
    if (max_steps < 0) return fail(LBM_EINVAL, "max_steps must be >= 0");
    if (check_every < 0) return fail(LBM_EINVAL, "check_every must be >= 0");
    if (!std::isfinite(tol_rel)) return fail(LBM_EINVAL, "tol_rel must be finite");
    if (tol_rel > 0.0 && check_every == 0) return fail(LBM_EINVAL, "tol_rel > 0 needs check_every > 0");
    const lbm_status valid = valid_state(g);
    if (valid != LBM_OK) return valid;
    DeviceGuard dg(g->dev);
    if (tol_rel > 0.0 && !g->h_outcome) LBM_CUDA(cudaMallocHost(&g->h_outcome, sizeof *g->h_outcome));
    const int CHUNK = 1024;
    int64_t left = max_steps, done = 0;
    double resid = -1.0;
    bool converged = false, checked = false, as_bits = false;       // as_bits: how the last check left its result
    bool tiled = false;
    Outcome o{};
    TileTurn turn;                                                  // until the launches are done
    const bool room = turn.take(g);
    while (left > 0) {
        // one launch of the tile kernel runs up to the next value the host needs
        int64_t m = left < TILE_CHUNK ? left : TILE_CHUNK;
        if (tol_rel > 0.0) m = std::min<int64_t>(m, check_every - g->t % check_every);
        if (room && g->tiles.ntx > 0 && m >= tiles_from(g->tiles)) {
            int checks = 0;
            const cudaError_t e = enqueue_tiles(g, (int)m, check_every, &checks);
            if (e == cudaErrorCooperativeLaunchTooLarge) {       // a stream with a part of the SMs
                cudaGetLastError();
                g->tiles.ntx = 0;
                continue;
            }
            LBM_CUDA(e);
            count_launches(1);
            tiled = true;
            g->t += m;
            done += m;
            left -= m;
            if (checks == 0) continue;
            checked = as_bits = true;
            if (tol_rel > 0.0) {
                LBM_CUDA(read_outcome(g, &o));
                resid = residual_of(o, true);
                if (o.tile_err || resid <= tol_rel) {
                    converged = true;
                    break;
                }
            }
            continue;
        }
        int64_t n = left < CHUNK ? left : CHUNK;
        int check = 0;
        if (check_every > 0) {
            const int64_t to_next = check_every - (g->t % check_every);
            if (g->fused && tol_rel <= 0.0 && to_next + 1 >= MULTISTEP_MAX && to_next < n && to_next + 1 < left) {
                n = to_next + 1;
                check = CHECK_INSIDE;
            } else if (to_next <= n) {
                n = to_next;
                check = 1;
            }
        }
        lbm_grid::Graph gr{};
        lbm_status s = get_graph(g, (int)n, g->cur, check, n == left || tol_rel > 0.0, &gr);
        if (s != LBM_OK) return s;
        LBM_CUDA(cudaGraphLaunch(gr.exec, g->stream));
        count_launches(gr.kernels);
        g->t += n;
        done += n;
        left -= n;
        g->cur = gr.cur;
        if (check) {
            checked = true;
            as_bits = check == CHECK_INSIDE;
            if (tol_rel > 0.0) {      // the stop test needs the value now; otherwise read it at the end
                LBM_CUDA(read_outcome(g, &o));
                resid = residual_of(o, false);
                if (resid <= tol_rel) {
                    converged = true;
                    break;
                }
            }
        }
    }
    if (tiled || (checked && tol_rel <= 0.0)) {
        LBM_CUDA(read_outcome(g, &o));
    } else {
        LBM_CUDA(cudaStreamSynchronize(g->stream));
    }
    if (o.tile_err) {
        g->lost = true;
        LBM_CUDA(cudaMemsetAsync(&g->outcome->tile_err, 0, sizeof(int), g->stream));
        return fail(LBM_ETIMEOUT, "a wait between the tiles of the lattice exceeded %.3g s: the state is not valid any more",
                    local_time_limit());
    }
    if (checked && tol_rel <= 0.0) resid = residual_of(o, as_bits);
    if (steps_done) *steps_done = done;
    if (residual) *residual = resid;
    if (tol_rel > 0.0 && !converged)
        return fail(LBM_ENOTCONV, "residual %.3e above tolerance %.3e after %lld steps", resid, tol_rel,
                    (long long)done);
    return LBM_OK;
}

lbm_status lbm_get_fields(lbm_grid *g, float *rho_dev, float *u_dev, float *v_dev)
{
    if (!g) return fail(LBM_EINVAL, "grid is NULL");
    if ((rho_dev && !is_device_ptr(rho_dev)) || (u_dev && !is_device_ptr(u_dev)) || (v_dev && !is_device_ptr(v_dev)))
        return fail(LBM_EINVAL, "field outputs must be device pointers");
    const lbm_status valid = valid_state(g);
    if (valid != LBM_OK) return valid;
    DeviceGuard dg(g->dev);
    LBM_CUDA(enqueue_moments(g, g->cur, -1, rho_dev, u_dev, v_dev, g->stream));
    count_launches(1);
    LBM_CUDA(cudaStreamSynchronize(g->stream));
    return LBM_OK;
}

lbm_status lbm_mean_velocity(lbm_grid *g, double out_mean_uv[2])
{
    if (!g || !out_mean_uv) return fail(LBM_EINVAL, "grid or output is NULL");
    const lbm_status valid = valid_state(g);
    if (valid != LBM_OK) return valid;
    DeviceGuard dg(g->dev);
    LBM_CUDA(enqueue_moments(g, g->cur, -1, nullptr, nullptr, nullptr, g->stream));
    LBM_CUDA(launch_reduce_partials(g->partials, g->L.mom_blocks, g->outcome->sums, g->stream));
    count_launches(2);
    Outcome o;
    LBM_CUDA(read_outcome(g, &o));
    const double n = (double)g->p.nx * g->p.ny;
    out_mean_uv[0] = o.sums[2] / n;
    out_mean_uv[1] = o.sums[3] / n;
    return LBM_OK;
}

int64_t lbm_grid_steps(const lbm_grid *g) { return g ? g->t : -1; }

int64_t lbm_grid_state_bytes(const lbm_grid *g)
{
    return g ? CKPT_HEADER_BYTES + (int64_t)(2 * 9 * g->plane * storage_bytes(g->p.storage)) : -1;
}

}  // extern "C"

namespace lbm {

// The header a checkpoint of grid g carries (and a loaded one must match).
static CkptHeader grid_header(const lbm_grid *g)
{
    CkptHeader h;
    std::memset(&h, 0, sizeof h);
    std::memcpy(h.magic, "LBM2CKPT", 8);
    h.version = 1;
    h.storage = g->p.storage;
    h.nx = g->p.nx;
    h.ny = g->p.ny;
    h.nz = 1;
    h.scale = g->S;
    const double d[5] = {g->p.tau, g->nu, g->p.eps, g->p.gx, g->p.gy};
    const int32_t i[4] = {g->p.bc, g->p.force_model, g->coef_mode, g->has_g ? 1 : 0};
    h.params_hash = fnv1a(i, sizeof i, fnv1a(d, sizeof d));
    h.steps = g->t;
    return h;
}

}  // namespace lbm

extern "C" {

lbm_status lbm_grid_save_state(lbm_grid *g, void *state_dev, int64_t nbytes, int64_t *steps)
{
    if (!g || !state_dev) return fail(LBM_EINVAL, "grid or state is NULL");
    if (nbytes != lbm_grid_state_bytes(g))
        return fail(LBM_EINVAL, "state buffer holds %lld bytes, the grid's state is %lld", (long long)nbytes,
                    (long long)lbm_grid_state_bytes(g));
    if (!is_device_ptr(state_dev)) return fail(LBM_EINVAL, "state_dev is not a device pointer");
    const lbm_status valid = valid_state(g);
    if (valid != LBM_OK) return valid;
    DeviceGuard dg(g->dev);
    const size_t half = 9 * g->plane * storage_bytes(g->p.storage);
    const CkptHeader h = grid_header(g);
    char *dst = static_cast<char *>(state_dev);
    LBM_CUDA(cudaMemcpyAsync(dst, &h, sizeof h, cudaMemcpyHostToDevice, g->stream));
    LBM_CUDA(cudaMemcpyAsync(dst + CKPT_HEADER_BYTES, g->buf[g->cur], half, cudaMemcpyDeviceToDevice, g->stream));
    LBM_CUDA(cudaMemcpyAsync(dst + CKPT_HEADER_BYTES + half, g->buf[1 - g->cur], half, cudaMemcpyDeviceToDevice,
                             g->stream));
    LBM_CUDA(cudaStreamSynchronize(g->stream));
    if (steps) *steps = g->t;
    return LBM_OK;
}

lbm_status lbm_grid_load_state(lbm_grid *g, const void *state_dev, int64_t nbytes, int64_t steps)
{
    if (!g || !state_dev) return fail(LBM_EINVAL, "grid or state is NULL");
    if (steps < 0) return fail(LBM_EINVAL, "steps must be >= 0");
    if (nbytes != lbm_grid_state_bytes(g))
        return fail(LBM_EINVAL, "state buffer holds %lld bytes, the grid's state is %lld", (long long)nbytes,
                    (long long)lbm_grid_state_bytes(g));
    if (!is_device_ptr(state_dev)) return fail(LBM_EINVAL, "state_dev is not a device pointer");
    DeviceGuard dg(g->dev);
    CkptHeader saved;
    LBM_CUDA(cudaMemcpyAsync(&saved, state_dev, sizeof saved, cudaMemcpyDeviceToHost, g->stream));
    LBM_CUDA(cudaStreamSynchronize(g->stream));
    const CkptHeader mine = grid_header(g);
    if (std::memcmp(saved.magic, mine.magic, 8) || saved.version != mine.version || saved.storage != mine.storage ||
        saved.nx != mine.nx || saved.ny != mine.ny || saved.nz != mine.nz || saved.scale != mine.scale ||
        saved.params_hash != mine.params_hash)
        return fail(LBM_EINVAL, "the state was saved by a grid of another size, storage, scale or parameter set");
    const size_t half = 9 * g->plane * storage_bytes(g->p.storage);
    const char *src = static_cast<const char *>(state_dev);
    LBM_CUDA(cudaMemcpyAsync(g->buf[g->cur], src + CKPT_HEADER_BYTES, half, cudaMemcpyDeviceToDevice, g->stream));
    LBM_CUDA(cudaMemcpyAsync(g->buf[1 - g->cur], src + CKPT_HEADER_BYTES + half, half, cudaMemcpyDeviceToDevice,
                             g->stream));
    LBM_CUDA(cudaStreamSynchronize(g->stream));
    g->lost = false;
    g->t = steps;
    return LBM_OK;
}

double lbm_grid_scale(const lbm_grid *g) { return g ? g->S : 0.0; }

}  // extern "C"
