// darcy_groups.cuh -- the Darcy K* of leaves of 4 to 64 cells a side (surrogate target base, mode 3), with
// the conjugate-gradient vectors in registers. Included by surrogate.cu.
//
// The system, its preconditioner and its stop rule are those stated in surrogate.cu. Both drives of a leaf are
// solved at once: they share the matrix, and the two right-hand sides are the lanes of packed f32x2 operands.
// A thread holds a block of 4 rows x 2 columns (leaf_groups.cuh): pressure, residual, direction (48
// registers), faces and 1 / diagonal (24). An iteration needs the direction's neighbours along x from the
// neighbouring lanes, along y from shared memory at the block's edges only, and sums over the leaf's group of
// warps: the eight terms of a thread as two chains of four in FP32, everything across threads in pairs of floats (a
// rounded sum and its error, about 46 bits), alpha and beta from those pairs. FP64 sums would keep the pipe's two lanes
// busy for 1500 clocks an iteration of a 64-cell leaf. Pairs cost 5 % over plain FP32 sums, because a lane that takes
// half of its partner's values gives away the other half of its own: four sums over a warp take 6 additions, not 20.
// The faces are scaled by a power of two, so that squares of residuals stay inside FP32's range at any unit of K: with
// unscaled faces and FP32 sums log K* was 2e-4 off at K around 1e-20 and wrong in the first digit at 6e17.
//
// Measured: the leaves of a 512 x 512 quadtree (sigma 1) 12.2 ms with a warp or a CTA per leaf and FP64 sums, 0.625 ms
// here (0.594 with FP32 sums); surrogate inference on a 1024 x 1024 quadtree 29.0 -> 7.5 ms. The largest leaf's
// iterations, a chain of three barriers and two reductions each, are what remains.
#pragma once

#include "leaf_groups.cuh"
#include "pair_ops.cuh"

namespace lbm {
namespace sur {

// Square of the relative residual, 5e-6: half of what the solver with FP64 sums (darcy_leaf) stops at, since a thread's
// eight terms are a longer chain in FP32 than there on small leaves. Mean error of log K* against 64-bit solves, there /
// here: 9e-8 both at sigma <= 1 (the result's own rounding); at sigma 3 1.4e-6 / 1.3e-6 at side 8, 2.5e-6 / 2.4e-6 at 16,
// 5.2e-6 / 3.1e-6 at 32, 3.0e-6 / 2.8e-6 at 64, and 5.1e-7 / 5.4e-7 at side 4.
constexpr float DG_STOP = 2.5e-11f;
constexpr int DG_CLASSES = 5;                // sides 64, 32, 16, 8, 4
__host__ __device__ constexpr int dg_side(int c) { return 64 >> c; }
constexpr int DG_SMALL = DG_CLASSES;          // list of the other sides up to 32
constexpr int DG_BIG = DG_CLASSES + 1;        // list of the other sides above
constexpr int DG_LISTS = DG_CLASSES + 2;
// Scratch of a call: the lists' counts, the classes' queue heads, then the lists.
constexpr int DG_HEADER = 32, DG_HEADS = 16;
inline size_t darcy_scratch_ints(int n) { return DG_HEADER + (size_t)DG_LISTS * n; }

struct DarcyShared {
    double k[RG_WARPS * RG_WCELLS];          // permeability while a leaf is set up
    float4 edge[RG_WARPS][2][32];            // a block's bottom and top row: (column, column + 1) x (drive x, drive y)
    float2 sum4[4][RG_WARPS], sum2[2][RG_WARPS];   // a warp's part of sums over its group
    float kmax[RG_WARPS];
    double flux[2][RG_WARPS];
    int leaf[RG_WARPS][RG_JOBS];
};

// One list of leaves per side.
__global__ void __launch_bounds__(256) darcy_classify_kernel(const float *x, int n, int *scratch)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int s = darcy_size(x + (int64_t)i * IN_PLANES * PIX);
        int c = s <= IMG ? DG_SMALL : DG_BIG;
        for (int k = 0; k < DG_CLASSES; ++k)
            if (s == dg_side(k)) c = k;
        scratch[DG_HEADER + (int64_t)c * n + atomicAdd(&scratch[c], 1)] = i;
    }
}

// A sum carried to twice FP32's precision: hi + lo.
struct Two {
    float hi, lo;
};
// a + b without error (Knuth's two-sum); the same bits whichever comes first
__device__ __forceinline__ Two two_sum(float a, float b)
{
    const float s = a + b, t = s - a;
    return Two{s, (a - (s - t)) + (b - t)};
}
// the low parts are not carried over into the high one: their sum's rounding is 2^-24 of 2^-24
__device__ __forceinline__ Two two_add(Two a, Two b)
{
    const Two s = two_sum(a.hi, b.hi);
    return Two{s.hi, s.lo + (a.lo + b.lo)};
}
__device__ __forceinline__ Two two_norm(Two a)
{
    const float s = a.hi + a.lo;
    return Two{s, a.lo - (s - a.hi)};
}
__device__ __forceinline__ Two two_shfl_xor(Two a, int off)
{
    return Two{__shfl_xor_sync(0xffffffffu, a.hi, off), __shfl_xor_sync(0xffffffffu, a.lo, off)};
}
__device__ __forceinline__ Two two_shfl(Two a, int from)
{
    return Two{__shfl_sync(0xffffffffu, a.hi, from), __shfl_sync(0xffffffffu, a.lo, from)};
}
// a / b, rounded to FP32 once (up to about 2^-40)
__device__ __forceinline__ float two_div(Two a, Two b)
{
    const float q = a.hi / b.hi;
    const float r = fmaf(-q, b.hi, a.hi) + fmaf(-q, b.lo, a.lo);
    return q + __fdividef(r, b.hi);
}

__global__ void __launch_bounds__(RG_THREADS, 1) darcy_group_kernel(const float *x, int n, int *scratch, float4 *cw)
{
    extern __shared__ __align__(16) unsigned char dg_smem[];
    DarcyShared &sh = *reinterpret_cast<DarcyShared *>(dg_smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    for (int cls = 0; cls < DG_CLASSES; ++cls) {
        const int s = dg_side(cls), count = scratch[cls];
        if (count == 0) continue;
        const RegGeo q = reg_geometry(s, warp, lane);
        const int *list = scratch + DG_HEADER + (int64_t)cls * n;
        const int span = q.group == 1 ? 32 / q.jobs : 32;        // lanes of a leaf within a warp
        const int tb = q.below, ta = q.above;
        auto from_right = [&](float2 v) {
            return make_float2(__shfl_sync(0xffffffffu, v.x, q.right), __shfl_sync(0xffffffffu, v.y, q.right));
        };
        auto from_left = [&](float2 v) {
            return make_float2(__shfl_sync(0xffffffffu, v.x, q.left), __shfl_sync(0xffffffffu, v.y, q.left));
        };
        // The sums over the leaf of (a.x, a.y, b.x, b.y), a and b each as two addends, and of c, the same bits in each
        // of its threads. A lane keeps half of what it holds and gives the other half to its partner, until it
        // holds one sum's part (offsets span / 2 and span / 4; a span of 2 lanes stops at two sums each).
        auto totals4 = [&](float2 a0, float2 a1, float2 b0, float2 b1, Two (&t)[4]) {
            Two v[4] = {two_sum(a0.x, a1.x), two_sum(a0.y, a1.y), two_sum(b0.x, b1.x), two_sum(b0.y, b1.y)};
            const int o1 = span / 2, o2 = span / 4;
            const bool up1 = lane & o1, up2 = lane & o2;
            for (int i = 0; i < 2; ++i) v[i] = two_add(up1 ? v[i + 2] : v[i], two_shfl_xor(up1 ? v[i] : v[i + 2], o1));
            if (span > 2) {
                v[0] = two_add(up2 ? v[1] : v[0], two_shfl_xor(up2 ? v[0] : v[1], o2));
                for (int off = span / 8; off > 0; off >>= 1) v[0] = two_add(v[0], two_shfl_xor(v[0], off));
            }
            if (q.group > 1) {                                   // span = 32: lanes 8 k .. 8 k + 7 hold sum k
                if ((lane & 7) == 0) sh.sum4[lane >> 3][warp] = make_float2(v[0].hi, v[0].lo);
                group_sync(q.group, q.w0);
                const int w = lane & 7;
                const float2 *part = sh.sum4[lane >> 3] + q.w0;
                const float2 p0 = w < q.group ? part[w] : dup2(0.0f), p1 = w + 8 < q.group ? part[w + 8] : dup2(0.0f);
                v[0] = two_add(Two{p0.x, p0.y}, Two{p1.x, p1.y});
                for (int off = 4; off > 0; off >>= 1) v[0] = two_add(v[0], two_shfl_xor(v[0], off));
            }
            const int base = lane & ~(span - 1);
            for (int k = 0; k < 4; ++k)
                t[k] = two_norm(two_shfl(span > 2 || !(k & 1) ? v[0] : v[1], base + (k >> 1) * o1 + (k & 1) * o2));
        };
        auto totals2 = [&](float2 c0, float2 c1, Two (&t)[2]) {
            Two v[2] = {two_sum(c0.x, c1.x), two_sum(c0.y, c1.y)};
            const int o1 = span / 2;
            const bool up = lane & o1;
            v[0] = two_add(up ? v[1] : v[0], two_shfl_xor(up ? v[0] : v[1], o1));
            for (int off = span / 4; off > 0; off >>= 1) v[0] = two_add(v[0], two_shfl_xor(v[0], off));
            if (q.group > 1) {
                if ((lane & 15) == 0) sh.sum2[lane >> 4][warp] = make_float2(v[0].hi, v[0].lo);
                group_sync(q.group, q.w0);
                const int w = lane & 15;
                const float2 p = w < q.group ? sh.sum2[lane >> 4][q.w0 + w] : dup2(0.0f);
                v[0] = Two{p.x, p.y};
                for (int off = 8; off > 0; off >>= 1) v[0] = two_add(v[0], two_shfl_xor(v[0], off));
            }
            const int base = lane & ~(span - 1);
            for (int k = 0; k < 2; ++k) t[k] = two_norm(two_shfl(v[0], base + k * o1));
        };
        for (;;) {
            group_sync(q.group, q.w0);                           // the previous leaf's reads are done
            if (warp == q.w0 && lane < q.jobs) {
                const int i = atomicAdd(&scratch[DG_HEADS + cls], 1);
                sh.leaf[q.w0][lane] = i < count ? list[i] : -1;
            }
            group_sync(q.group, q.w0);
            const int leaf = sh.leaf[q.w0][q.job];
            const bool mine = q.cell && leaf >= 0;
            if (!__any_sync(0xffffffffu, leaf >= 0)) break;      // of a group of several warps, all or none
            // permeabilities, read back from the log-K planes
            if (mine) {
                const float *xi = x + (int64_t)leaf * IN_PLANES * PIX;
#pragma unroll
                for (int r = 0; r < RG_ROWS; ++r)
                    for (int c = 0; c < 2; ++c) {
                        const int Y = q.row + r, X = q.col + c;
                        const float v = s <= IMG ? xi[Y * (IMG / s) * IMG + X * (IMG / s)]
                                                 : xi[((Y & 1) * 2 + (X & 1)) * PIX + (Y >> 1) * IMG + (X >> 1)];
                        sh.k[q.scratch + Y * s + X] = exp((double)v);
                    }
            }
            group_sync(q.group, q.w0);
            float kx[RG_ROWS][2], ky[RG_ROWS][2], kb[2], idg[RG_ROWS][2];    // kb: the faces below the block
            float2 p[RG_ROWS][2], res[RG_ROWS][2], d[RG_ROWS][2], ad[RG_ROWS][2];
            Two rz[2];
#pragma unroll
            for (int r = 0; r < RG_ROWS; ++r)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    kx[r][c] = ky[r][c] = idg[r][c] = kb[c] = 0.0f;
                    p[r][c] = res[r][c] = d[r][c] = ad[r][c] = dup2(0.0f);
                }
            if (mine) {
                const double *k = sh.k + q.scratch;
                auto at = [&](int Y, int X) { return k[(Y < 0 ? Y + s : (Y >= s ? Y - s : Y)) * s + (X >= s ? X - s : X)]; };
#pragma unroll
                for (int r = 0; r < RG_ROWS; ++r)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int Y = q.row + r, X = q.col + c;
                        kx[r][c] = harmonic2f(at(Y, X), at(Y, X + 1));
                        ky[r][c] = harmonic2f(at(Y, X), at(Y + 1, X));
                    }
                for (int c = 0; c < 2; ++c) kb[c] = harmonic2f(at(q.row - 1, q.col + c), at(q.row, q.col + c));
            }
            // the faces over the power of two at the leaf's largest one, so that squares of residuals keep clear of
            // FP32's ends whatever the unit of K (exact, and pressures do not depend on it); K* takes it back
            float top = 0.0f;
#pragma unroll
            for (int r = 0; r < RG_ROWS; ++r) top = fmaxf(top, fmaxf(fmaxf(kx[r][0], kx[r][1]), fmaxf(ky[r][0], ky[r][1])));
            for (int off = span / 2; off > 0; off >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
            if (q.group > 1) {
                if (lane == 0) sh.kmax[warp] = top;
                group_sync(q.group, q.w0);
                for (int w = 0; w < q.group; ++w) top = fmaxf(top, sh.kmax[q.w0 + w]);
            }
            int unit = (__float_as_int(top) >> 23) - 127;
            unit = unit > 127 ? 0 : min(max(unit, -126), 126);       // an infinite face: as it is
            const float scale = __int_as_float((127 - unit) << 23);
#pragma unroll
            for (int r = 0; r < RG_ROWS; ++r)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    kx[r][c] *= scale;
                    ky[r][c] *= scale;
                }
            kb[0] *= scale;
            kb[1] *= scale;
            // start: p = 0, r = b (face behind minus face ahead along the drive), d = r / diagonal
            float2 r0 = dup2(0.0f), r1 = dup2(0.0f), g0 = dup2(0.0f), g1 = dup2(0.0f);
#pragma unroll
            for (int r = 0; r < RG_ROWS; ++r) {
                const float kl = __shfl_sync(0xffffffffu, kx[r][1], q.left);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const float xl = c == 0 ? kl : kx[r][0], yb = r == 0 ? kb[c] : ky[r - 1][c];
                    const float dg = kx[r][c] + xl + ky[r][c] + yb;
                    idg[r][c] = dg > 0.0f ? 1.0f / dg : 0.0f;
                    res[r][c] = mine ? make_float2(xl - kx[r][c], yb - ky[r][c]) : dup2(0.0f);
                    d[r][c] = mul2(res[r][c], dup2(idg[r][c]));
                    (c == 0 ? r0 : r1) = fma2(res[r][c], res[r][c], c == 0 ? r0 : r1);
                    (c == 0 ? g0 : g1) = fma2(res[r][c], d[r][c], c == 0 ? g0 : g1);
                }
            }
            Two t[4];                                            // r . r of both drives, r . z of both drives
            totals4(r0, r1, g0, g1, t);
            rz[0] = t[2];
            rz[1] = t[3];
            const float2 stop = mul2(dup2(DG_STOP), make_float2(t[0].hi, t[1].hi));
            bool on0 = mine && t[0].hi > stop.x, on1 = mine && t[1].hi > stop.y;
            auto publish = [&](const float2 (&v)[RG_ROWS][2]) {
                sh.edge[warp][0][lane] = make_float4(v[0][0].x, v[0][0].y, v[0][1].x, v[0][1].y);
                sh.edge[warp][1][lane] = make_float4(v[RG_ROWS - 1][0].x, v[RG_ROWS - 1][0].y, v[RG_ROWS - 1][1].x,
                                                     v[RG_ROWS - 1][1].y);
            };
            // whether any leaf of the group still iterates, the same in all its warps that hold cells
            for (int it = 0; it < DB_MAXIT && __any_sync(0xffffffffu, leaf >= 0 && (on0 || on1)); ++it) {
                if (q.group == 1) __syncwarp();                  // (larger groups: the barriers of the sums)
                publish(d);
                group_sync(q.group, q.w0);
                const float4 below = sh.edge[tb >> 5][1][tb & 31], above = sh.edge[ta >> 5][0][ta & 31];
                // fluxes across the faces; ad = what leaves a cell
                float2 fb[2] = {mul2(dup2(kb[0]), sub2(make_float2(below.x, below.y), d[0][0])),
                                mul2(dup2(kb[1]), sub2(make_float2(below.z, below.w), d[0][1]))};
                float2 t0 = dup2(0.0f), t1 = dup2(0.0f);
#pragma unroll
                for (int r = 0; r < RG_ROWS; ++r) {
                    const float2 f0 = mul2(dup2(kx[r][0]), sub2(d[r][0], d[r][1]));
                    const float2 f1 = mul2(dup2(kx[r][1]), sub2(d[r][1], from_right(d[r][0])));
                    const float2 fl = from_left(f1);
                    const float2 u0 = r < RG_ROWS - 1 ? d[r + 1][0] : make_float2(above.x, above.y);
                    const float2 u1 = r < RG_ROWS - 1 ? d[r + 1][1] : make_float2(above.z, above.w);
                    const float2 g0 = mul2(dup2(ky[r][0]), sub2(d[r][0], u0));
                    const float2 g1 = mul2(dup2(ky[r][1]), sub2(d[r][1], u1));
                    ad[r][0] = add2(sub2(f0, fl), sub2(g0, fb[0]));
                    ad[r][1] = add2(sub2(f1, f0), sub2(g1, fb[1]));
                    fb[0] = g0;
                    fb[1] = g1;
                    t0 = fma2(d[r][0], ad[r][0], t0);
                    t1 = fma2(d[r][1], ad[r][1], t1);
                }
                Two dad[2];
                totals2(t0, t1, dad);
                on0 = on0 && dad[0].hi > 0.0f;                   // else a direction in the null space
                on1 = on1 && dad[1].hi > 0.0f;
                const float2 al = make_float2(on0 ? two_div(rz[0], dad[0]) : 0.0f, on1 ? two_div(rz[1], dad[1]) : 0.0f);
                const float2 nal = make_float2(-al.x, -al.y);
                float2 a0 = dup2(0.0f), a1 = dup2(0.0f), z0 = dup2(0.0f), z1 = dup2(0.0f);
#pragma unroll
                for (int r = 0; r < RG_ROWS; ++r) {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        p[r][c] = fma2(al, d[r][c], p[r][c]);
                        res[r][c] = fma2(nal, ad[r][c], res[r][c]);
                    }
                    const float2 s0 = mul2(res[r][0], res[r][0]), s1 = mul2(res[r][1], res[r][1]);
                    a0 = add2(a0, s0);
                    a1 = add2(a1, s1);
                    z0 = fma2(s0, dup2(idg[r][0]), z0);
                    z1 = fma2(s1, dup2(idg[r][1]), z1);
                }
                totals4(a0, a1, z0, z1, t);
                const float2 be = make_float2(on0 ? two_div(t[2], rz[0]) : 0.0f, on1 ? two_div(t[3], rz[1]) : 0.0f);
                rz[0] = t[2];
                rz[1] = t[3];
                on0 = on0 && t[0].hi > stop.x;
                on1 = on1 && t[1].hi > stop.y;
#pragma unroll
                for (int r = 0; r < RG_ROWS; ++r)
#pragma unroll
                    for (int c = 0; c < 2; ++c) d[r][c] = fma2(be, d[r][c], mul2(res[r][c], dup2(idg[r][c])));
            }
            // K* along the drive is the mean face flux
            group_sync(q.group, q.w0);
            publish(p);
            group_sync(q.group, q.w0);
            const float4 above = sh.edge[ta >> 5][0][ta & 31];
            double qx = 0.0, qy = 0.0;
#pragma unroll
            for (int r = 0; r < RG_ROWS; ++r) {
                const float pr = __shfl_sync(0xffffffffu, p[r][0].x, q.right);
                qx += kx[r][0] * (p[r][0].x - p[r][1].x + 1.0f);
                qx += kx[r][1] * (p[r][1].x - pr + 1.0f);
                qy += ky[r][0] * (p[r][0].y - (r < RG_ROWS - 1 ? p[r + 1][0].y : above.y) + 1.0f);
                qy += ky[r][1] * (p[r][1].y - (r < RG_ROWS - 1 ? p[r + 1][1].y : above.w) + 1.0f);
            }
            for (int off = span / 2; off > 0; off >>= 1) {
                qx += __shfl_xor_sync(0xffffffffu, qx, off);
                qy += __shfl_xor_sync(0xffffffffu, qy, off);
            }
            if (q.group > 1) {
                if (lane == 0) {
                    sh.flux[0][warp] = qx;
                    sh.flux[1][warp] = qy;
                }
                group_sync(q.group, q.w0);
                if (warp == q.w0 && lane == 0) {
                    qx = qy = 0.0;
                    for (int w = 0; w < q.group; ++w) {
                        qx += sh.flux[0][q.w0 + w];
                        qy += sh.flux[1][q.w0 + w];
                    }
                }
            }
            if (mine && warp == q.w0 && q.row == 0 && q.col == 0)
                cw[leaf] = make_float4((float)log(ldexp(qx / (s * s), unit)), 1.0f, (float)log(ldexp(qy / (s * s), unit)), 1.0f);
        }
        // every warp of the group has read that the list is empty before a smaller group of the next class, which
        // some of them may already belong to, puts its leaves into the same words
        group_sync(q.group, q.w0);
    }
}

}  // namespace sur
}  // namespace lbm
