// multistep.cu -- up to four fused steps of the simplified Shan-Chen LBM per pass over memory.
//
// The one-step kernel of step.cu moves every population through HBM once per step (76 bytes per
// lattice update in FP32) and sits at 0.96 of the measured bandwidth, so the only way past it is to
// move them less often. Here a pass reads the state of step n and writes the state of step n + NLEV:
//  * A warp owns a strip of 64 consecutive columns, two per lane, and marches along y. The two cells of
//    a lane are one packed f32x2 operand throughout (pair_ops.cuh).
//  * At march position i the warp takes row i through step 1, row i - 1 through step 2 (its three source
//    rows have just become available), row i - 2 through step 3 and row i - 3 through step 4, whose
//    result is stored. Rows in flight between two steps are nine values per cell in registers (three
//    populations wait one row, three wait two, three none); the one-column shift of streaming is one warp
//    shuffle per pair. So there is no shared memory and no barrier, and warps never wait for each other.
//  * Columns next to the strip's edges lose one valid column per step on each side, so 64 - 2 * 4 = 56
//    columns of a strip are stored, and a segment of rows needs 2 (NLEV - 1) extra march positions:
//    both are recomputed, not exchanged.
// Every cell's arithmetic is that of step_kernel, operation by operation, and FP16 storage is rounded to
// FP16 after every step, so a fused pass gives the same bits as single steps.
//
// What bounds it, on 4096 x 4096: FP32 moves 1275 MB a pass (76 bytes per cell, 6 % of the reads repeated halo
// rows) at 6.0 TB/s, 0.88 of the measured copy rate; the packed multiply-adds, two clocks each, keep
// the FMA pipe 60 % busy beside that. A pass of four steps takes 0.212 ms against 4 x 0.196 ms for single
// steps. FP16 moves half as much but converts every value after every step and is bound by instruction
// issue: 0.21 ms a pass against 4 x 0.117 ms. Rows reach shared memory through cp.async three positions
// ahead: with one row prefetched into registers a warp waited on memory for 59 % of its time
// (0.30 ms a pass). Warps of one SM take neighbouring strips, which saves 7 % of the time (L1 hits on the
// sectors that two strips share).
#include "lbm_internal.h"
#include "pair_step.cuh"

#include <algorithm>
#include <type_traits>

namespace lbm {
namespace {

constexpr int LEV = MULTISTEP_MAX;       // steps per pass at most
constexpr int STRIP = 64;                // columns of a warp
constexpr int USEFUL = STRIP - 2 * LEV;  // columns of it that are stored

// A stored pair of neighbouring cells and its one-column shifts across the warp. The outermost
// columns of the strip get a value that is not theirs; they are never stored.
template <typename T> struct PairT;
template <> struct PairT<float> { using V = float2; };
template <> struct PairT<__half> { using V = __half2; };
__device__ __forceinline__ float2 from_left(float2 v) { return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x); }
__device__ __forceinline__ float2 from_right(float2 v) { return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1)); }
__device__ __forceinline__ unsigned h2u(__half2 v) { return *reinterpret_cast<unsigned *>(&v); }
__device__ __forceinline__ __half2 u2h(unsigned v) { return *reinterpret_cast<__half2 *>(&v); }
__device__ __forceinline__ __half2 from_left(__half2 v)
{
    const unsigned u = h2u(v);
    return u2h(__byte_perm(__shfl_up_sync(0xffffffffu, u, 1), u, 0x5432));
}
__device__ __forceinline__ __half2 from_right(__half2 v)
{
    const unsigned u = h2u(v);
    return u2h(__byte_perm(u, __shfl_down_sync(0xffffffffu, u, 1), 0x5432));
}
__device__ __forceinline__ float2 to_f2(float2 v) { return v; }
__device__ __forceinline__ float2 to_f2(__half2 v) { return __half22float2(v); }
template <typename V> __device__ __forceinline__ V from_f2(float2 v);
template <> __device__ __forceinline__ float2 from_f2<float2>(float2 v) { return v; }
template <> __device__ __forceinline__ __half2 from_f2<__half2>(float2 v) { return __float22half2_rn(v); }

// Byte offsets within a plane are 32-bit (multistep_ok bounds the plane), added to a uniform base.
template <typename T> __device__ __forceinline__ T *at(T *plane, unsigned byte)
{
    return reinterpret_cast<T *>(reinterpret_cast<uintptr_t>(plane) + byte);
}
// The pair of values at columns x0, x1 of the row at element `row` of a plane (ALIGNED: x1 = x0 + 1
// and the pair is aligned).
template <bool ALIGNED, typename T>
__device__ __forceinline__ typename PairT<T>::V load_pair(const T *plane, unsigned row, int x0, int x1)
{
    using V = typename PairT<T>::V;
    if constexpr (ALIGNED) {
        return *reinterpret_cast<const V *>(at(plane, (row + x0) * (unsigned)sizeof(T)));
    } else {
        V v;
        v.x = *at(plane, (row + x0) * (unsigned)sizeof(T));
        v.y = *at(plane, (row + x1) * (unsigned)sizeof(T));
        return v;
    }
}

// Rows are copied into shared memory AHEAD positions before they are used, each lane its own pairs, so a lane
// waits only for its own copies and no barrier is needed. A slot is overwritten one position after its
// values were last read.
constexpr int AHEAD = 3;
constexpr int RING = 4;       // rows of populations: AHEAD and the one in use
constexpr int CRING = 8;      // rows of coefficients: those of all LEV steps too

template <int BYTES> __device__ __forceinline__ void copy_async(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(BYTES)
                 : "memory");
}
// Copies the pair at columns x0, x1 of the row at element `row` of a plane.
template <bool ALIGNED, typename T>
__device__ __forceinline__ void stage_pair(typename PairT<T>::V *dst, const T *plane, unsigned row, int x0, int x1)
{
    constexpr int E = sizeof(T);
    if constexpr (ALIGNED) {
        copy_async<2 * E>(dst, at(plane, (row + x0) * E));
    } else {
        static_assert(E == 4, "4-byte copies");
        copy_async<E>(&dst->x, at(plane, (row + x0) * E));
        copy_async<E>(&dst->y, at(plane, (row + x1) * E));
    }
}

// Rows on their way from one step to the next: populations with e_y = 0 (0, 1, 3) wait one row, those
// with e_y = +1 (2, 5, 6) two rows (slot = parity of the march position); with walls the last row's
// e_y = -1 populations (4, 7, 8) are kept too, for the bounce-back of row 0.
template <typename V, bool WALLS>
struct RowLine {
    V up[2][3], mid[3], down[3];
};

struct MultiGeom {
    int nlev;        // steps of this pass, 1 .. LEV
    int strips;      // column strips
    int segs;        // row segments
    int seg_rows;    // rows of a segment
    unsigned *check; // CHECK: bits of max |du|, max |u|
};

// Warps per SM: the rows in flight and a collision take up to 168 registers in FP32, 128 in FP16.
template <typename T> constexpr int ms_warps() { return sizeof(T) == 2 ? 16 : 12; }

// Bytes of shared memory of one warp.
template <typename T, int COEF, bool GF>
constexpr size_t warp_smem()
{
    return (size_t)RING * Q * 32 * 2 * sizeof(T) + (size_t)CRING * ncoef<COEF, GF>() * 32 * sizeof(float2);
}

// CHECK (with LEV steps): also raises *m.check to the maxima of the residual after the pass's third step. The third
// and fourth step pull the two states it compares, so their velocities are at hand; the fourth's row is one
// behind, for which the third's velocity waits one position.
// It takes the place of a shorter pass, a single step and a pass of the residual kernel: 4096 x 4096, 256 steps with a
// check every 64, 15.6 -> 14.6 ms (FP16 15.4 -> 14.7); the check alone costs its pass the divisions.
template <typename T, int COEF, bool GF, bool WALLS, bool ALIGNED, bool CHECK>
__global__ void __launch_bounds__(ms_warps<T>() * 32, 1) multi_step_kernel(StepArgs<T, float> a, MultiGeom m)
{
    using V = typename PairT<T>::V;
    constexpr bool ASYNC = ALIGNED || sizeof(T) == 4;    // 2-byte copies do not exist
    constexpr int NC = ncoef<COEF, GF>();
    extern __shared__ __align__(16) unsigned char ms_smem[];
    const int lane = threadIdx.x & 31;
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (w >= m.strips * m.segs) return;
    const int seg = w / m.strips, strip = w - seg * m.strips;
    const int nx = a.nx, ny = a.ny;
    const int ya = seg * m.seg_rows, yb = min(ya + m.seg_rows, ny);
    if (ya >= ny) return;
    unsigned char *mine = ms_smem + (threadIdx.x >> 5) * warp_smem<T, COEF, GF>();
    V *rows = reinterpret_cast<V *>(mine) + lane;                               // [RING][Q][32]
    float2 *coefs = reinterpret_cast<float2 *>(mine + (size_t)RING * Q * 32 * sizeof(V)) + lane;   // [CRING][NC][32]

    // this lane's columns, and which of them are stored
    const int xu = strip * USEFUL - LEV + 2 * lane;
    int x0 = xu % nx, x1 = (xu + 1) % nx;
    x0 += x0 < 0 ? nx : 0;
    x1 += x1 < 0 ? nx : 0;
    const int xend = min((strip + 1) * USEFUL, nx);
    const bool st0 = 2 * lane >= LEV && xu < xend, st1 = 2 * lane >= LEV && xu + 1 < xend;

    auto row_of = [&](int r) {                       // periodic wrap, or any valid row beyond a wall
        if constexpr (WALLS) return min(max(r, 0), ny - 1);
        return r < 0 ? r + ny : (r >= ny ? r - ny : r);
    };
    // population q of the pairs that row r pulls, before the one-column shift: its plane and row
    auto source = [&](int r, int q, unsigned &o) -> const T * {
        int s = q, y = row_of(r - ey(q));
        if (WALLS && ((ey(q) == 1 && r == 0) || (ey(q) == -1 && r == ny - 1))) {
            s = opp(q);
            y = r;
        }
        o = (unsigned)y * nx;
        return a.src + s * a.plane;
    };
    V next[Q];                                       // the next row, where it cannot be copied asynchronously
    auto load_next = [&](int r) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            unsigned o;
            const T *p = source(r, q, o);
            next[q] = load_pair<ALIGNED>(p, o, x0, x1);
        }
    };
    auto stage_row = [&](int r, int j) {             // the j-th row of this warp
        if constexpr (ASYNC) {
            V *d = rows + (j % RING) * (Q * 32);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                unsigned o;
                const T *p = source(r, q, o);
                stage_pair<ALIGNED>(d + q * 32, p, o, x0, x1);
            }
        }
        const unsigned o = (unsigned)row_of(r) * nx;
        float2 *c = coefs + (j % CRING) * (NC * 32);
        constexpr int CP = COEF == COEF_TENSOR ? 4 : 1;
#pragma unroll
        for (int k = 0; k < CP; ++k) stage_pair<ALIGNED>(c + k * 32, a.coef + k * a.plane, o, x0, x1);
        if constexpr (GF) {
            stage_pair<ALIGNED>(c + CP * 32, a.gfield, o, x0, x1);
            stage_pair<ALIGNED>(c + (CP + 1) * 32, a.gfield + a.plane, o, x0, x1);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float2 pu[2], pv[2];                             // velocity at the third step, by parity of the position
    float dmax = 0.0f, umax = 0.0f;
    if constexpr (CHECK) pu[0] = pu[1] = pv[0] = pv[1] = dup2(0.0f);
    // step `lev` of row r, the warp's j-th row, at a position of parity P: p holds its sources before the one-column
    // shift
    auto step_row = [&](int lev, int P, int r, int j, V (&p)[Q]) {
        const float2 *c = coefs + ((unsigned)j % CRING) * (NC * 32);
        PairCoef<COEF, GF> k;
        k.c0 = c[0];
        if constexpr (COEF == COEF_TENSOR) {
            k.c1 = c[32];
            k.c2 = c[64];
            k.c3 = c[96];
        }
        k.gx = GF ? c[(NC - 2) * 32] : dup2(a.gx);
        k.gy = GF ? c[(NC - 1) * 32] : dup2(a.gy);
        const bool lo = WALLS && r == 0, hi = WALLS && r == ny - 1;
        float2 g[Q];
        g[0] = to_f2(p[0]);
        g[1] = to_f2(from_left(p[1]));
        g[3] = to_f2(from_right(p[3]));
        g[2] = to_f2(p[2]);
        g[4] = to_f2(p[4]);
        const V l5 = from_left(p[5]), r6 = from_right(p[6]), r7 = from_right(p[7]), l8 = from_left(p[8]);
        g[5] = to_f2(lo ? p[5] : l5);
        g[6] = to_f2(lo ? p[6] : r6);
        g[7] = to_f2(hi ? p[7] : r7);
        g[8] = to_f2(hi ? p[8] : l8);
        if constexpr (CHECK) {
            if (lev >= LEV - 2) {
                const Flow2 f = flow_pair<COEF, GF>(g, k, a.rho0, a.half_eps);
                const float2 u = make_float2(f.rux.x / f.rho.x, f.rux.y / f.rho.y);
                const float2 v = make_float2(f.ruy.x / f.rho.x, f.ruy.y / f.rho.y);
                if (lev == LEV - 2) {
                    pu[P] = u;
                    pv[P] = v;
                } else if (r >= ya && r < yb) {
                    const float2 du = sub2(u, pu[1 - P]), dv = sub2(v, pv[1 - P]);
                    if (st0) {
                        dmax = fmaxf(dmax, fmaxf(fabsf(du.x), fabsf(dv.x)));
                        umax = fmaxf(umax, fmaxf(fabsf(u.x), fabsf(v.x)));
                    }
                    if (st1) {
                        dmax = fmaxf(dmax, fmaxf(fabsf(du.y), fabsf(dv.y)));
                        umax = fmaxf(umax, fmaxf(fabsf(u.y), fabsf(v.y)));
                    }
                }
            }
        }
        collide_pair<COEF, GF>(g, k, a.rho0, a.half_eps, a.omega, a.two_tau, a.one_m_two_tau);
#pragma unroll
        for (int q = 0; q < Q; ++q) p[q] = from_f2<V>(g[q]);
    };

    RowLine<V, WALLS> line[LEV - 1];
#pragma unroll
    for (int k = 0; k < LEV - 1; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            line[k].up[0][j] = line[k].up[1][j] = line[k].mid[j] = line[k].down[j] = from_f2<V>(dup2(0.0f));

    const int nlev = CHECK ? LEV : m.nlev;
    const int i0 = ya - (nlev - 1), n = yb - ya + 2 * (nlev - 1);
#pragma unroll
    for (int j = 0; j < AHEAD; ++j) stage_row(i0 + j, j);
    if constexpr (!ASYNC) load_next(i0);
    auto march = [&](int j, auto par) {
        constexpr int P = decltype(par)::value;
        const int i = i0 + j;
        asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD - 1) : "memory");
        V p[Q];
        if constexpr (ASYNC) {
            const V *d = rows + (j % RING) * (Q * 32);
#pragma unroll
            for (int q = 0; q < Q; ++q) p[q] = d[q * 32];
        } else {
#pragma unroll
            for (int q = 0; q < Q; ++q) p[q] = next[q];
            load_next(i + 1);
        }
        stage_row(i + AHEAD, j + AHEAD);
        step_row(0, P, i, j, p);
        int r = i;                                   // the row p now holds
#pragma unroll
        for (int k = 0; k < LEV - 1; ++k) {
            if (k + 1 < nlev) {
                RowLine<V, WALLS> &L = line[k];
                r = i - (k + 1);
                const bool lo = WALLS && r == 0, hi = WALLS && r == ny - 1;
                V s[Q];
                s[0] = L.mid[0];
                s[1] = L.mid[1];
                s[3] = L.mid[2];
                s[2] = lo ? L.down[0] : L.up[P][0];
                s[5] = lo ? L.down[1] : L.up[P][1];
                s[6] = lo ? L.down[2] : L.up[P][2];
                s[4] = hi ? L.up[1 - P][0] : p[4];
                s[7] = hi ? L.up[1 - P][1] : p[7];
                s[8] = hi ? L.up[1 - P][2] : p[8];
                L.up[P][0] = p[2];
                L.up[P][1] = p[5];
                L.up[P][2] = p[6];
                L.mid[0] = p[0];
                L.mid[1] = p[1];
                L.mid[2] = p[3];
                if constexpr (WALLS) {
                    L.down[0] = p[4];
                    L.down[1] = p[7];
                    L.down[2] = p[8];
                }
#pragma unroll
                for (int q = 0; q < Q; ++q) p[q] = s[q];
                step_row(k + 1, P, r, j - (k + 1), p);
            }
        }
        if (r >= ya && r < yb) {
            const unsigned o = (unsigned)r * nx;
            if constexpr (ALIGNED) {
                if (st0) {
#pragma unroll
                    for (int q = 0; q < Q; ++q)
                        *reinterpret_cast<V *>(at(a.dst + q * a.plane, (o + x0) * (unsigned)sizeof(T))) = p[q];
                }
            } else {
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    if (st0) *at(a.dst + q * a.plane, (o + x0) * (unsigned)sizeof(T)) = p[q].x;
                    if (st1) *at(a.dst + q * a.plane, (o + x1) * (unsigned)sizeof(T)) = p[q].y;
                }
            }
        }
    };
    // an odd count takes one position more, whose row lies past the segment and is not stored
    for (int j = 0; j < n; j += 2) {
        march(j, std::integral_constant<int, 0>{});
        march(j + 1, std::integral_constant<int, 1>{});
    }
    asm volatile("cp.async.wait_all;" ::: "memory");   // rows staged past the end
    if constexpr (CHECK) {                             // the order of non-negative floats is that of their bits
        const unsigned d = __reduce_max_sync(0xffffffffu, __float_as_uint(dmax));
        const unsigned u = __reduce_max_sync(0xffffffffu, __float_as_uint(umax));
        if (lane == 0) {
            atomicMax(m.check, d);
            atomicMax(m.check + 1, u);
        }
    }
}

template <typename T, int COEF, bool GF, bool WALLS, bool ALIGNED, bool CHECK>
cudaError_t launch_t(const StepArgs<T, float> &a, int nlev, int sms, unsigned *check, cudaStream_t st)
{
    constexpr size_t per_warp = warp_smem<T, COEF, GF>();
    constexpr int by_smem = (int)(231424 / per_warp);            // 227 KB, 1 KB of it reserved per CTA
    constexpr int sm_warps = by_smem < ms_warps<T>() ? by_smem : ms_warps<T>();
    const auto kern = multi_step_kernel<T, COEF, GF, WALLS, ALIGNED, CHECK>;
    const cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(per_warp * sm_warps));
    if (e != cudaSuccess) return e;
    MultiGeom m;
    m.nlev = nlev;
    m.check = check;
    m.strips = (a.nx + USEFUL - 1) / USEFUL;
    // one wave of resident warps; segments of at least MULTISTEP_MIN_ROWS rows
    int segs = sms * sm_warps / m.strips;
    if (segs < 1) segs = 1;
    m.seg_rows = (a.ny + segs - 1) / segs;
    if (m.seg_rows < MULTISTEP_MIN_ROWS) m.seg_rows = MULTISTEP_MIN_ROWS;
    m.segs = (a.ny + m.seg_rows - 1) / m.seg_rows;
    // a large grid fills each SM with one CTA, so that neighbouring strips share the SM's L1 and the
    // sectors their edges overlap on are read once; a small one is spread over the SMs
    const int64_t warps = (int64_t)m.strips * m.segs;
    int cta = (int)((warps + sms - 1) / sms);
    if (cta > sm_warps) cta = sm_warps;
    kern<<<(unsigned)((warps + cta - 1) / cta), cta * 32, per_warp * cta, st>>>(a, m);
    return cudaGetLastError();
}

template <typename T, int COEF>
cudaError_t launch_c(bool gf, bool walls, const StepArgs<T, float> &a, int nlev, int sms, unsigned *check, cudaStream_t st)
{
    const bool al = a.nx % 2 == 0;
#define LBM_MS_CASE(GFv, WLv, ALv)                       \
    if (gf == GFv && walls == WLv && al == ALv)          \
        return check ? launch_t<T, COEF, GFv, WLv, ALv, true>(a, nlev, sms, check, st) \
                     : launch_t<T, COEF, GFv, WLv, ALv, false>(a, nlev, sms, check, st);
    LBM_MS_CASE(false, false, false)
    LBM_MS_CASE(false, false, true)
    LBM_MS_CASE(false, true, false)
    LBM_MS_CASE(false, true, true)
    LBM_MS_CASE(true, false, false)
    LBM_MS_CASE(true, false, true)
    LBM_MS_CASE(true, true, false)
    LBM_MS_CASE(true, true, true)
#undef LBM_MS_CASE
    return cudaErrorInvalidValue;
}

}  // namespace

// Guo's scheme and FP16 with a tensor K* keep the one-step kernel; so do lattices too small for the
// single wrap of a row index.
bool multistep_ok(int storage, int coef_mode, int nx, int ny, int guo)
{
    if ((int64_t)nx * ny >= (int64_t)1 << 30) return false;      // 32-bit byte offsets within a plane
    if (guo || ny < 2 * LEV || nx < 2) return false;
    return storage == LBM_F32 || (storage == LBM_F16 && coef_mode == COEF_SCALAR);
}

// Whether passes of four steps beat single steps, by microseconds a step of either. A pass takes the longest warp's
// march: its positions (rows, and 2 (LEV - 1) of halo), each dearer the more warps share an SM, whatever part of a
// strip's columns the lattice fills. A single step takes a launch and its bytes' way, from L2 up to about a million
// cells. Against 526 measured pairs (both storages, 2 to 131,073 columns, 8 to 400,000 rows, 16 to 29 M cells) the
// choice is at worst 1.13 times the better one, where passes everywhere were up to 17 times it: 2 x 1,048,576 cells 370 us
// a step against 33, 24 x 65,536 in FP16 14.3 against 8.2, 64 x 16,384 in FP16 8.6 against 6.4, 400 x 1000 in FP16
// 4.6 against 4.1. Passes win at 128 x 64 (2.0 against 2.6), 517 x 389 (2.9 against 4.0), 1448 x 1448 (8.9 against
// 24.2) and 4096 x 4096 (53 against 196). Long runs of small lattices go on to tiles.cu.
bool multistep_pays(int storage, int nx, int ny, int sms)
{
    if (nx < 4) return false;
    const bool f16 = storage == LBM_F16, odd = nx % 2 != 0;
    const int warps = f16 ? ms_warps<__half>() : ms_warps<float>();
    const int strips = (nx + USEFUL - 1) / USEFUL;
    const int64_t segs = std::max<int64_t>(1, (int64_t)sms * warps / strips);
    const int64_t rows = std::max<int64_t>(MULTISTEP_MIN_ROWS, (ny + segs - 1) / segs);
    double load = (double)strips * ((ny + rows - 1) / rows) / sms;          // warps on an SM
    load = load > 12.0 ? 16.0 : std::max(load, 1.0);                        // four schedulers
    const double positions = (double)((rows + 2 * (LEV - 1) + 1) / 2 * 2);
    const double fixed = odd ? (f16 ? 0.90 : 0.34) : (f16 ? 0.36 : 0.38), shared = odd ? (f16 ? 0.075 : 0.077) : (f16 ? 0.078 : 0.061);
    const double pass = (fixed + shared * load) * positions + (odd ? (f16 ? 0.0 : 3.5) : 2.5);

    const double n = 1e-6 * nx * ny;                                        // million cells
    double single;
    if (nx % (f16 ? 8 : 4) == 0) {
        if (n < 6e-4) single = 1.8;
        else if (f16) single = n < 2.3 ? 2.9 + 3.4 * n : 7.2 * n;
        else single = n < 1.4 ? 2.5 + 5.6 * n : 12.2 * n;
    } else if (f16 && !odd) {
        single = nx % 4 == 0 && n >= 1.05 && n < 2.3 ? 2.9 + 4.3 * n : 2.0 + 7.2 * n;
    } else {
        single = f16 || n < 1.4 ? (f16 ? 1.80 : 1.95) + 11.7 * n : 14.7 * n;
    }
    return pass < LEV * single;
}

cudaError_t launch_multistep(int storage, int coef_mode, bool gfield, bool walls, const void *args, int nlev, int sms,
                             unsigned *check, cudaStream_t st)
{
    if (nlev < 1 || nlev > LEV || (check && nlev != LEV)) return cudaErrorInvalidValue;
    if (storage == LBM_F32) {
        const StepArgs<float, float> &a = *static_cast<const StepArgs<float, float> *>(args);
        return coef_mode == COEF_SCALAR ? launch_c<float, COEF_SCALAR>(gfield, walls, a, nlev, sms, check, st)
                                        : launch_c<float, COEF_TENSOR>(gfield, walls, a, nlev, sms, check, st);
    }
    if (storage == LBM_F16 && coef_mode == COEF_SCALAR)
        return launch_c<__half, COEF_SCALAR>(gfield, walls, *static_cast<const StepArgs<__half, float> *>(args), nlev,
                                             sms, check, st);
    return cudaErrorInvalidValue;
}

}  // namespace lbm
