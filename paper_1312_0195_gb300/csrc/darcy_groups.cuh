// darcy_groups.cuh -- the Darcy K* of leaves of 4 to 64 cells a side (surrogate target base, mode 3), with
// the conjugate-gradient vectors in registers. Included by surrogate.cu.
//
// The system, its preconditioner and its stop rule are those stated in surrogate.cu. Both drives of a leaf are
// solved at once: they share the matrix, and the two right-hand sides are the lanes of packed f32x2 operands.
// A thread holds a block of 4 rows x 2 columns (leaf_groups.cuh): pressure, residual, direction (48
// registers), faces and 1 / diagonal (24). An iteration needs the direction's neighbours along x from the
// neighbouring lanes, along y from shared memory at the block's edges only, and three sums over the leaf's
// group of warps: the eight terms of a thread as two chains of four, the threads of a warp and the warps by
// butterflies, all in FP32 (13 roundings at most on the way of a term; the one-CTA-per-leaf solver this
// replaces rounded 16 times in FP32 before its FP64 sums, and its FP64 butterflies and per-cell index
// divisions bounded it).
//
// Measured: a 512 x 512 quadtree's leaves (sigma 1) 13.2 -> 1.4 ms; surrogate inference on a 1024 x 1024
// quadtree 31.2 -> 9.5 ms, the solves in it 22.4 -> 0.6. The largest leaf's iterations, a chain of three
// barriers and two reductions each, are what remains.
#pragma once

#include "leaf_groups.cuh"
#include "pair_ops.cuh"

namespace lbm {
namespace sur {

// Square of the relative residual, 5e-6: half of what the FP64-summed solver stopped at, which makes up for the
// FP32 sums. Against 64-bit solves the mean error of log K* is what it was (1e-7 to 5e-7 at sigma <= 2, any
// scale of K) and on 64-cell leaves at sigma 3 half of it (3.0e-5 against 6.5e-5).
constexpr float DG_STOP = 2.5e-11f;
constexpr int DG_CLASSES = 5;                // sides 64, 32, 16, 8, 4
__host__ __device__ constexpr int dg_side(int c) { return 64 >> c; }
constexpr int DG_TINY = DG_CLASSES;           // list of sides 1 to 3
constexpr int DG_OTHER = DG_CLASSES + 1;      // list of any other side a size plane may say
constexpr int DG_LISTS = DG_CLASSES + 2;
// Scratch of a call: the lists' counts, the classes' queue heads, then the lists.
constexpr int DG_HEADER = 32, DG_HEADS = 16;
inline size_t darcy_scratch_ints(int n) { return DG_HEADER + (size_t)DG_LISTS * n; }

struct DarcyShared {
    double k[RG_WARPS * RG_WCELLS];          // permeability while a leaf is set up
    float4 edge[RG_WARPS][2][32];            // a block's bottom and top row: (column, column + 1) x (drive x, drive y)
    float2 sum[3][RG_WARPS];                 // a warp's part of a sum over its group
    double flux[2][RG_WARPS];
    int leaf[RG_WARPS][RG_JOBS];
};

// One list of leaves per side.
__global__ void __launch_bounds__(256) darcy_classify_kernel(const float *x, int n, int *scratch)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int s = darcy_size(x + (int64_t)i * IN_PLANES * PIX);
        int c = s < 4 ? DG_TINY : DG_OTHER;
        for (int k = 0; k < DG_CLASSES; ++k)
            if (s == dg_side(k)) c = k;
        scratch[DG_HEADER + (int64_t)c * n + atomicAdd(&scratch[c], 1)] = i;
    }
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
        // a sum over the leaf, the same bits in each of its threads
        auto total = [&](float2 v, int slot) {
            for (int off = span / 2; off > 0; off >>= 1)
                v = add2(v, make_float2(__shfl_xor_sync(0xffffffffu, v.x, off), __shfl_xor_sync(0xffffffffu, v.y, off)));
            if (q.group > 1) {
                if (lane == 0) sh.sum[slot][warp] = v;
                group_sync(q.group, q.w0);
                v = sh.sum[slot][q.w0 + (lane & (q.group - 1))];
                for (int off = q.group / 2; off > 0; off >>= 1)
                    v = add2(v, make_float2(__shfl_xor_sync(0xffffffffu, v.x, off), __shfl_xor_sync(0xffffffffu, v.y, off)));
            }
            return v;
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
            float2 rr = dup2(0.0f), rz = dup2(0.0f);
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
            // start: p = 0, r = b (face behind minus face ahead along the drive), d = r / diagonal
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
                    rr = fma2(res[r][c], res[r][c], rr);
                    rz = fma2(res[r][c], d[r][c], rz);
                }
            }
            rr = total(rr, 0);
            rz = total(rz, 1);
            const float2 stop = mul2(dup2(DG_STOP), rr);
            bool on0 = mine && rr.x > stop.x, on1 = mine && rr.y > stop.y;
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
                const float2 dad = total(add2(t0, t1), 2);
                on0 = on0 && dad.x > 0.0f;                       // else a direction in the null space
                on1 = on1 && dad.y > 0.0f;
                const float2 al = make_float2(on0 ? rz.x / dad.x : 0.0f, on1 ? rz.y / dad.y : 0.0f);
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
                rr = total(add2(a0, a1), 0);
                const float2 rz2 = total(add2(z0, z1), 1);
                const float2 be = make_float2(on0 ? rz2.x / rz.x : 0.0f, on1 ? rz2.y / rz.y : 0.0f);
                rz = rz2;
                on0 = on0 && rr.x > stop.x;
                on1 = on1 && rr.y > stop.y;
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
            float fx = 0.0f, fy = 0.0f;
#pragma unroll
            for (int r = 0; r < RG_ROWS; ++r) {
                const float pr = __shfl_sync(0xffffffffu, p[r][0].x, q.right);
                fx += kx[r][0] * (p[r][0].x - p[r][1].x + 1.0f);
                fx += kx[r][1] * (p[r][1].x - pr + 1.0f);
                fy += ky[r][0] * (p[r][0].y - (r < RG_ROWS - 1 ? p[r + 1][0].y : above.y) + 1.0f);
                fy += ky[r][1] * (p[r][1].y - (r < RG_ROWS - 1 ? p[r + 1][1].y : above.w) + 1.0f);
            }
            double qx = fx, qy = fy;
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
                cw[leaf] = make_float4((float)log(qx / (s * s)), 1.0f, (float)log(qy / (s * s)), 1.0f);
        }
        // every warp of the group has read that the list is empty before a smaller group of the next class, which
        // some of them may already belong to, puts its leaves into the same words
        group_sync(q.group, q.w0);
    }
}

}  // namespace sur
}  // namespace lbm
