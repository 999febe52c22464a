// tiles.cu -- many steps of a small lattice in one launch, the state resident in shared memory.
//
// On lattices of up to about 270,000 cells a pass of multistep.cu is short of warps: it takes 8 to 13 us
// whatever the size, most of it launch, first loads and a single warp's issue. Here the lattice is cut into at most two
// tiles per SM, each with a halo of four cells. A CTA keeps two tiles in shared memory, interleaved cell
// by cell (the two tiles' values are the lanes of packed f32x2 operands), steps them four times while the halo is
// used up from outside in, and then exchanges its tiles' outer four rings for its halo through global memory (L2).
// The launch is cooperative, so all CTAs become resident, and wait for one another in bounded time: a thread gives up
// after as many polls in vain as the limit of lbm_set_time_limit has room for, which is long enough for other
// streams' kernels to leave the SMs that some CTAs may still have to wait for. (Reading a clock at each such poll
// made the coarse run of 256 x 256 2 % slower.)
// Two areas take the exchanges in turn: an area is written again two exchanges later, when words of the exchange
// between have come in from every CTA that read it.
// Every cell's arithmetic is that of the one-step kernel, so the bits are the same.
//
// What bounds it: the way of an exchange (about 2 us: a store and a load through L2) and, in between, the latency of a
// step and its barrier; the FMA pipe is a quarter busy. Microseconds a step, single steps / passes of four / here:
// 128 x 64 2.55 / 2.0 / 0.89, 256 x 256 2.58 / 2.2 / 1.37, 517 x 389 3.95 / 2.9 / 1.87, 500 x 500 3.39 / 2.6 / 2.2.
// Flags raised after a fence and polled by one warp, with plain loads of the halo behind them, took 1.11 us at
// 128 x 64 and 2.66 us at 517 x 389. Halos of six or eight cells, with fewer exchanges, were slower (1.07 and 1.27 us
// at 128 x 64; 1.92 and no fit at 517 x 389): the wider halo's cells cost more than the exchanges saved.
#include "pair_step.cuh"

#include <cuda_fp16.h>

namespace lbm {
namespace {

constexpr int TL_THREADS = 768;
constexpr int TL_ROUNDS = 2;                         // cells of a thread at most
constexpr int TL_ITEMS = 3;                          // halo cells (and outer-ring cells) of a thread at most

// Cells of a tile with its halo that fit: two buffers of nine populations and the coefficients, for two tiles.
__host__ __device__ constexpr int tl_cells(int nc) { return nc == 1 ? 1504 : (nc == 3 ? 1360 : (nc == 4 ? 1296 : 1184)); }
template <int COEF, bool GF> constexpr size_t tl_smem()
{
    return (size_t)(2 * Q + ncoef<COEF, GF>()) * tl_cells(ncoef<COEF, GF>()) * sizeof(float2);
}

template <typename T> __device__ __forceinline__ float tl_load(const T *p);
template <> __device__ __forceinline__ float tl_load<float>(const float *p) { return __ldcg(p); }
template <> __device__ __forceinline__ float tl_load<__half>(const __half *p)
{
    return __half2float(__ushort_as_half(__ldcg(reinterpret_cast<const unsigned short *>(p))));
}
template <typename T> __device__ __forceinline__ T tl_cast(float v);
template <> __device__ __forceinline__ float tl_cast<float>(float v) { return v; }
template <> __device__ __forceinline__ __half tl_cast<__half>(float v) { return __float2half_rn(v); }

// A word of the exchange: 16 bytes that are written and seen as one.
__device__ __forceinline__ void tl_store(uint4 *p, float a, float b, float c, unsigned seq)
{
    asm volatile("{\n .reg .b128 w;\n .reg .b64 lo, hi;\n mov.b64 lo, {%1, %2};\n mov.b64 hi, {%3, %4};\n"
                 " mov.b128 w, {lo, hi};\n st.relaxed.gpu.global.b128 [%0], w;\n}" ::"l"(p),
                 "r"(__float_as_uint(a)), "r"(__float_as_uint(b)), "r"(__float_as_uint(c)), "r"(seq)
                 : "memory");
}
__device__ __forceinline__ uint4 tl_poll(const uint4 *p)
{
    uint4 v;
    asm volatile("{\n .reg .b128 w;\n .reg .b64 lo, hi;\n ld.relaxed.gpu.global.b128 w, [%4];\n"
                 " mov.b128 {lo, hi}, w;\n mov.b64 {%0, %1}, lo;\n mov.b64 {%2, %3}, hi;\n}"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

// Threads of a CTA for arrays of np cells.
inline int tl_threads(int np)
{
    const int rounds = (np + TL_THREADS - 1) / TL_THREADS;
    return ((np + rounds - 1) / rounds + 31) / 32 * 32;
}

// One of a CTA's two tiles: cells [x, x + w) x [y, y + h) of the lattice.
struct Tile {
    int x, y, w, h;
};

template <typename T, int COEF, bool GF, bool WALLS>
__global__ void __launch_bounds__(TL_THREADS, 1) tiles_kernel(StepArgs<T, float> a, T *src, T *dst, TileGeom g, int steps,
                                                             int first_check, int check_every, unsigned *result,
                                                             uint4 *exch, unsigned base, int *err, int patience)
{
    constexpr int NC = ncoef<COEF, GF>(), NP = tl_cells(NC), HALO = TILE_HALO;
    extern __shared__ __align__(16) unsigned char tl_raw[];
    float2 *F = reinterpret_cast<float2 *>(tl_raw);              // [2][Q][NP]
    float2 *C = F + 2 * Q * NP;                                  // [NC][NP]
    __shared__ int s_failed;
    const int tid = threadIdx.x, nt = blockDim.x, cta = blockIdx.x;
    const int nx = a.nx, ny = a.ny, W = g.W, np = g.W * g.H, ntiles = g.ntx * g.nty;

    Tile tile[2];
    int index[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        index[k] = cta + k * g.ctas < ntiles ? cta + k * g.ctas : cta;     // an odd tile out is stepped twice
        const int ty = index[k] / g.ntx, tx = index[k] - ty * g.ntx;
        tile[k].x = (int)((int64_t)tx * nx / g.ntx);
        tile[k].y = (int)((int64_t)ty * ny / g.nty);
        tile[k].w = (int)((int64_t)(tx + 1) * nx / g.ntx) - tile[k].x;
        tile[k].h = (int)((int64_t)(ty + 1) * ny / g.nty) - tile[k].y;
    }
    // this thread's cells: local column and row, -1 for none; the lattice cell under it in tile k
    int lx[TL_ROUNDS], ly[TL_ROUNDS];
#pragma unroll
    for (int r = 0; r < TL_ROUNDS; ++r) {
        const int i = tid + r * nt;
        ly[r] = i < np ? i / W : -1;
        lx[r] = i < np ? i - ly[r] * W : -1;
    }
    auto cell = [&](int r, int k, bool &in) -> unsigned {
        int x = tile[k].x - HALO + lx[r], y = tile[k].y - HALO + ly[r];
        x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
        in = !WALLS || (y >= 0 && y < ny);
        y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        return (unsigned)y * nx + x;
    };
    auto lane = [](float2 &v, int k) -> float & { return k == 0 ? v.x : v.y; };
    auto own = [&](int r, int k) {
        return lx[r] >= HALO && lx[r] < HALO + tile[k].w && ly[r] >= HALO && ly[r] < HALO + tile[k].h;
    };
    // the populations of this thread's cells, from global memory to buffer b and back
    auto fetch = [&](const T *from, int b) {
#pragma unroll
        for (int r = 0; r < TL_ROUNDS; ++r) {
            if (ly[r] < 0) continue;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                bool in;
                const unsigned c = cell(r, k, in);
                if (!in) continue;
                float v[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q) v[q] = tl_load(from + q * a.plane + c);
#pragma unroll
                for (int q = 0; q < Q; ++q) lane(F[(b * Q + q) * NP + tid + r * nt], k) = v[q];
            }
        }
    };
    auto put = [&](T *to, int b) {
#pragma unroll
        for (int r = 0; r < TL_ROUNDS; ++r) {
            if (ly[r] < 0) continue;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (!own(r, k)) continue;
                bool in;
                const unsigned c = cell(r, k, in);
#pragma unroll
                for (int q = 0; q < Q; ++q) to[q * a.plane + c] = tl_cast<T>(lane(F[(b * Q + q) * NP + tid + r * nt], k));
            }
        }
    };
    // This thread's share of an exchange: cells of the two tiles' halos to read and of their outer four rings to
    // write, as element of a plane (none: -1) and float of the array. Cell m of the frame, HALO cells thick, along
    // the inside of a w x h box at (x0, y0): the upper and lower rows, then the sides.
    auto frame = [&](int m, int x0, int y0, int w, int h, int &x, int &y) {
        constexpr int D = 2 * HALO;
        if (m < D * w) {
            y = m / w;
            x = x0 + m - y * w;
            y = y0 + (y < HALO ? y : h - D + y);
        } else {
            m -= D * w;
            y = m / D;
            m -= y * D;
            x = x0 + (m < HALO ? m : w - D + m);
            y += y0 + HALO;
        }
    };
    int get_cell[TL_ITEMS], get_at[TL_ITEMS], put_cell[TL_ITEMS], put_at[TL_ITEMS];
#pragma unroll
    for (int j = 0; j < TL_ITEMS; ++j) {
        auto item = [&](bool halo, int &c, int &at) {
            c = -1;
            at = 0;
            int m = tid + j * nt;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int w = tile[k].w + (halo ? 2 * HALO : 0), h = tile[k].h + (halo ? 2 * HALO : 0);
                const int n = 2 * HALO * (w + h - 2 * HALO);
                if (m >= 0 && m < n) {
                    int u, v;
                    frame(m, halo ? 0 : HALO, halo ? 0 : HALO, w, h, u, v);
                    int x = tile[k].x - HALO + u, y = tile[k].y - HALO + v;
                    x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
                    const bool in = !WALLS || (y >= 0 && y < ny);
                    y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
                    c = in ? y * nx + x : -1;
                    at = 2 * (v * W + u) + k;
                }
                m -= n;
            }
        };
        item(true, get_cell[j], get_at[j]);
        item(false, put_cell[j], put_at[j]);
    }
    // Exchange `seq`: the outer rings to the other CTAs' halos. A cell travels as three words of 16 bytes, each with
    // three populations and the exchange's number, written and read as one; a reader polls the words themselves,
    // so that an exchange takes one store and one load's way and no fence.
    const int64_t cells = (int64_t)nx * ny;
    auto exchange = [&](unsigned seq, int b) {
        uint4 *area = exch + (seq & 1) * 3 * cells;
        float *f = reinterpret_cast<float *>(F + b * Q * NP);
#pragma unroll
        for (int j = 0; j < TL_ITEMS; ++j)
            if (put_cell[j] >= 0)
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    const float *v = f + 6 * w * NP + put_at[j];
                    tl_store(area + w * cells + put_cell[j], v[0], v[2 * NP], v[4 * NP], seq);
                }
        int spins = 0;
#pragma unroll
        for (int j = 0; j < TL_ITEMS; ++j) {
            if (get_cell[j] < 0) continue;
            uint4 v[3];
            for (;;) {
#pragma unroll
                for (int w = 0; w < 3; ++w) v[w] = tl_poll(area + w * cells + get_cell[j]);
                if ((v[0].w == seq && v[1].w == seq && v[2].w == seq) || *(volatile int *)&s_failed) break;
                if (++spins > patience) {
                    *(volatile int *)&s_failed = 1;
                    atomicExch(err, 1);
                }
            }
#pragma unroll
            for (int w = 0; w < 3; ++w) {
                float *to = f + 6 * w * NP + get_at[j];
                to[0] = __uint_as_float(v[w].x);
                to[2 * NP] = __uint_as_float(v[w].y);
                to[4 * NP] = __uint_as_float(v[w].z);
            }
        }
    };

    // the whole state with its halo, and the coefficients
    for (int i = tid; i < 2 * Q * NP; i += nt) F[i] = dup2(0.0f);
    for (int i = tid; i < NC * NP; i += nt) C[i] = dup2(0.0f);
    if (tid == 0) s_failed = 0;
    __syncthreads();
    fetch(src, 0);
#pragma unroll
    for (int r = 0; r < TL_ROUNDS; ++r) {
        if (ly[r] < 0) continue;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            bool in;
            const unsigned c = cell(r, k, in);
            if (!in) continue;
            constexpr int CP = COEF == COEF_TENSOR ? 4 : 1;
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                const float *p = j < CP ? a.coef + j * a.plane : a.gfield + (j - CP) * a.plane;
                lane(C[j * NP + tid + r * nt], k) = p[c];
            }
        }
    }
    __syncthreads();

    auto coef_of = [&](int i) {
        PairCoef<COEF, GF> c;
        c.c0 = C[i];
        if constexpr (COEF == COEF_TENSOR) {
            c.c1 = C[NP + i];
            c.c2 = C[2 * NP + i];
            c.c3 = C[3 * NP + i];
        }
        c.gx = GF ? C[(NC - 2) * NP + i] : dup2(a.gx);
        c.gy = GF ? C[(NC - 1) * NP + i] : dup2(a.gy);
        return c;
    };
    // what cell r of this thread pulls from buffer b
    auto pull = [&](int b, int r, float2 (&v)[Q]) {
        const float2 *in = F + b * Q * NP;
        const int i = tid + r * nt;
#pragma unroll
        for (int q = 0; q < Q; ++q) v[q] = in[q * NP + i - ex(q) - ey(q) * W];
        if constexpr (WALLS) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int y = tile[k].y - HALO + ly[r];
                if (y != 0 && y != ny - 1) continue;
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if ((ey(q) == 1 && y == 0) || (ey(q) == -1 && y == ny - 1)) {
                        const float2 o = in[opp(q) * NP + i];
                        lane(v[q], k) = k == 0 ? o.x : o.y;
                    }
            }
        }
    };

    // Step t of the launch takes state t - 1 to state t. A check after step t compares the velocities of states t and
    // t - 1, which are at hand when the next step and this one pull them; a check after the last step pulls once more.
    auto is_check = [&](int t) { return check_every > 0 && t >= first_check && (t - first_check) % check_every == 0; };
    const int turns = steps + (is_check(steps) ? 1 : 0);
    float2 pu[TL_ROUNDS], pv[TL_ROUNDS];             // velocities of the state before a check's
#pragma unroll
    for (int r = 0; r < TL_ROUNDS; ++r) pu[r] = pv[r] = dup2(0.0f);
    int b = 0;                                       // buffer of the newest state
    for (int t = 1; t <= turns; ++t) {
        const bool before = t <= steps && is_check(t), after = t > 1 && is_check(t - 1);
        float dmax = 0.0f, umax = 0.0f;
#pragma unroll
        for (int r = 0; r < TL_ROUNDS; ++r) {
            // cells on the array's border have no sources; what they spoil moves in one cell a step
            if (ly[r] < 1 || lx[r] < 1 || lx[r] >= W - 1 || ly[r] >= g.H - 1) continue;
            const int i = tid + r * nt;
            float2 v[Q];
            pull(b, r, v);
            const PairCoef<COEF, GF> c = coef_of(i);
            if (before || after) {
                const Flow2 m = flow_pair<COEF, GF>(v, c, a.rho0, a.half_eps);
                const float2 u = make_float2(m.rux.x / m.rho.x, m.rux.y / m.rho.y);
                const float2 w = make_float2(m.ruy.x / m.rho.x, m.ruy.y / m.rho.y);
                if (after) {
                    if (own(r, 0)) {
                        dmax = fmaxf(dmax, fmaxf(fabsf(u.x - pu[r].x), fabsf(w.x - pv[r].x)));
                        umax = fmaxf(umax, fmaxf(fabsf(u.x), fabsf(w.x)));
                    }
                    if (own(r, 1)) {
                        dmax = fmaxf(dmax, fmaxf(fabsf(u.y - pu[r].y), fabsf(w.y - pv[r].y)));
                        umax = fmaxf(umax, fmaxf(fabsf(u.y), fabsf(w.y)));
                    }
                }
                pu[r] = u;
                pv[r] = w;
            }
            if (t > steps) continue;
            collide_pair<COEF, GF>(v, c, a.rho0, a.half_eps, a.omega, a.two_tau, a.one_m_two_tau);
            float2 *out = F + (1 - b) * Q * NP;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                if constexpr (sizeof(T) == 2) v[q] = __half22float2(__float22half2_rn(v[q]));   // storage rounding
                out[q * NP + i] = v[q];
            }
        }
        if (after) {                                 // the order of non-negative floats is that of their bits
            const unsigned d = __reduce_max_sync(0xffffffffu, __float_as_uint(dmax));
            const unsigned u = __reduce_max_sync(0xffffffffu, __float_as_uint(umax));
            unsigned *res = result + 2 * ((t - 1 - first_check) / check_every);
            if ((tid & 31) == 0) {
                atomicMax(res, d);
                atomicMax(res + 1, u);
            }
        }
        __syncthreads();
        if (t <= steps) b = 1 - b;
        if (t % HALO == 0 && t < turns) {
            exchange(base + t / HALO, b);
            __syncthreads();
        }
    }
    // The last two states. src is free: an exchange came in from every CTA that read it.
    put(src, 1 - b);
    put(dst, b);
}

template <typename T, int COEF, bool GF, bool WALLS>
cudaError_t launch_tl(const StepArgs<T, float> &a, const TileGeom &g, const TileRun &run, cudaStream_t st)
{
    const auto kern = tiles_kernel<T, COEF, GF, WALLS>;
    constexpr size_t smem = tl_smem<COEF, GF>();
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.gridDim = dim3((unsigned)g.ctas);
    cfg.blockDim = dim3((unsigned)tl_threads(g.W * g.H));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a, const_cast<T *>(a.src), a.dst, g, run.steps, run.first_check,
                              run.check_every, run.result, static_cast<uint4 *>(run.exch), run.base, run.err,
                              run.patience);
}

template <typename T, int COEF>
cudaError_t launch_tc(bool gf, bool walls, const StepArgs<T, float> &a, const TileGeom &g, const TileRun &run,
                      cudaStream_t st)
{
    if (gf) return walls ? launch_tl<T, COEF, true, true>(a, g, run, st)
                         : launch_tl<T, COEF, true, false>(a, g, run, st);
    return walls ? launch_tl<T, COEF, false, true>(a, g, run, st)
                 : launch_tl<T, COEF, false, false>(a, g, run, st);
}

}  // namespace

// The cut into at most two tiles per SM that leaves the smallest tiles with halo (the work of a step and, through the
// exchanged rings, most of an exchange), tiles of at least 2 TILE_HALO cells a side. No cut that fits: ntx = 0.
TileGeom tile_geometry(int storage, int coef_mode, bool gfield, int nx, int ny, int sms)
{
    TileGeom best{0, 0, 0, 0, 0};
    if (!multistep_ok(storage, coef_mode, nx, ny, 0) || nx < 2 * TILE_HALO || ny < 2 * TILE_HALO) return best;
    const int cells = tl_cells((coef_mode == COEF_TENSOR ? 4 : 1) + (gfield ? 2 : 0));
    for (int ntx = 1; ntx <= nx / (2 * TILE_HALO) && ntx <= 2 * sms; ++ntx) {
        int nty = 2 * sms / ntx;
        if (nty > ny / (2 * TILE_HALO)) nty = ny / (2 * TILE_HALO);
        const int W = (nx + ntx - 1) / ntx + 2 * TILE_HALO, H = (ny + nty - 1) / nty + 2 * TILE_HALO;
        const int nt = tl_threads(W * H), halo = 2 * TILE_HALO * (W + H - 2 * TILE_HALO);    // rings are smaller
        if ((int64_t)W * H > cells || 2 * halo > TL_ITEMS * nt) continue;
        if (best.ntx == 0 || W * H < best.W * best.H) best = TileGeom{ntx, nty, W, H, (ntx * nty + 1) / 2};
    }
    return best;
}

cudaError_t launch_tiles(int storage, int coef_mode, bool gfield, bool walls, const void *args, const TileGeom &g,
                         const TileRun &run, cudaStream_t st)
{
    if (storage == LBM_F32) {
        const StepArgs<float, float> &a = *static_cast<const StepArgs<float, float> *>(args);
        return coef_mode == COEF_SCALAR ? launch_tc<float, COEF_SCALAR>(gfield, walls, a, g, run, st)
                                        : launch_tc<float, COEF_TENSOR>(gfield, walls, a, g, run, st);
    }
    if (storage == LBM_F16 && coef_mode == COEF_SCALAR)
        return launch_tc<__half, COEF_SCALAR>(gfield, walls, *static_cast<const StepArgs<__half, float> *>(args), g, run,
                                              st);
    return cudaErrorInvalidValue;
}

}  // namespace lbm
