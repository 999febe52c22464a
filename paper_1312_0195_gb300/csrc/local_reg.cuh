// local_reg.cuh -- the batched local problems from rest with the distributions in registers (FP32,
// leaf sides that are multiples of 4). Included by local.cu, whose solver takes every other side, FP64,
// the Darcy starts and the local-global jobs.
//
// local.cu's solver keeps the distributions in shared memory: 18 shared accesses, 103 instructions and a
// CTA-wide barrier per lattice update and step, so that a single 64-cell leaf also takes 2.2 us a step.
// Here:
//  * A thread holds a block of 4 rows x 2 columns of its leaf, all nine populations, as packed f32x2 pairs
//    of neighbouring columns: 72 registers. The collision does two cells per instruction.
//  * Streaming along x is one warp shuffle per pair (closing on the leaf's row), along y a renaming of the
//    thread's rows; only the three populations that leave the block upwards and the three that leave
//    it downwards go through shared memory (12 eight-byte accesses for 8 cells), double-buffered, so one
//    barrier a step is enough.
//  * A leaf of side s takes s / 2 lanes per row and s / 4 row blocks, packed into the fewest warps, a power
//    of two (64: 16 warps; 32: 4; 16 and 12: 1; 8: a quarter of one). Each such group of warps steps its
//    own leaf and takes the next one from the size's queue by itself; it synchronises with a barrier of its
//    own warps, or none. Between two checks the loop has no bookkeeping at all.
// The arithmetic of a cell, the order of every sum and the stop test are local.cu's, so results are the same
// bit for bit.
//
// Measured (rest start, tau = 1, fixed steps, batches that fill the chip; billions of updates per second,
// local.cu's solver -> this one): side 64 286 -> 488, 48 242 -> 301, 32 312 -> 661, 24 170 -> 370,
// 20 230 -> 493, 16 303 -> 677, 12 258 -> 354, 8 273 -> 636; one 64-cell leaf alone 2.18 -> 1.27 us a step.
// What bounds it: 44 packed multiply-adds of two clocks each per pair keep the FMA pipe 77 % busy at side 16;
// at side 64 all 16 warps meet at one barrier a step and it is 56 %. Announcing rows through mbarriers
// or flags instead, edge rows first, cost more instructions than the waits it saved (446 and 436), and 8 rows a
// thread on 8 warps gained 5 % at side 64 and lost 3 to 12 % below.
#pragma once

#include "leaf_groups.cuh"
#include "pair_ops.cuh"

namespace lbm {
namespace {

struct RegSlot {
    int job;                                 // -1: empty
    int leaf, drive, x0, y0;
    int fresh;                               // its cells are not set up yet
    int next_check;                          // job step of the next steady-state check
    unsigned tstart;                         // group step of the job's step 0
    unsigned tstore;                         // group step at which the cells store their velocity
    double prev;                             // driven mean velocity at the previous check
};

struct RegShared {
    float2 ex[2][RG_WARPS][6][32];           // rows leaving a thread's block: 3 upwards, 3 downwards
    float ux[RG_WARPS * RG_WCELLS], uy[RG_WARPS * RG_WCELLS];
    RegSlot slots[RG_WARPS][RG_JOBS];
    int abort[RG_WARPS];
    unsigned long long t0;
};

// Two cells through collide_d2q9, products and sums fused as there. ne is minus the drag fraction.
template <bool TAU1>
__device__ __forceinline__ void collide_reg(float2 (&g)[Q], float2 ne, float2 hgx, float2 hgy, const LocalArgs &a,
                                            float2 &rux, float2 &ruy, float2 &rho)
{
    const float2 s13 = add2(g[1], g[3]), s24 = add2(g[2], g[4]), s57 = add2(g[5], g[7]), s68 = add2(g[6], g[8]);
    const float2 drho = add2(g[0], add2(add2(s13, s24), add2(s57, s68)));
    const float2 d57 = sub2(g[5], g[7]), d86 = sub2(g[8], g[6]);
    const float2 jx = add2(sub2(g[1], g[3]), add2(d57, d86));
    const float2 jy = add2(sub2(g[2], g[4]), sub2(d57, d86));
    rho = add2(dup2(1.0f), drho);
    const float2 rx = fma2(hgx, rho, jx), ry = fma2(hgy, rho, jy);
    rux = fma2(ne, rx, rx);
    ruy = fma2(ne, ry, ry);
    const float w0 = float(4.0 / 9.0), w1 = float(1.0 / 9.0), w2 = float(1.0 / 36.0);
    float2 nx, ny;                               // -rho u_eq
    if constexpr (TAU1) {
        nx = fma2(dup2(-2.0f), rux, jx);
        ny = fma2(dup2(-2.0f), ruy, jy);
    } else {
        nx = fma2(dup2(-a.kf[K_TWO_TAU]), rux, mul2(dup2(-a.kf[K_OMT]), jx));
        ny = fma2(dup2(-a.kf[K_TWO_TAU]), ruy, mul2(dup2(-a.kf[K_OMT]), jy));
    }
    const float2 ty = mul2(dup2(-3.0f), ny), nty = mul2(dup2(3.0f), ny);
    const float2 sp = fma2(dup2(-3.0f), nx, ty), sm = fma2(dup2(-3.0f), nx, nty);
    float2 q[Q];
    q[0] = drho;
    q[1] = fma2(dup2(-3.0f), nx, drho);
    q[3] = fma2(dup2(3.0f), nx, drho);
    q[2] = add2(drho, ty);
    q[4] = add2(drho, nty);
    q[5] = add2(drho, sp);
    q[7] = sub2(drho, sp);
    q[8] = add2(drho, sm);
    q[6] = sub2(drho, sm);
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        const float w = k == 0 ? w0 : (k <= 4 ? w1 : w2);
        // g + omega (w q - g), the inner difference with its sign turned
        if constexpr (TAU1) g[k] = mul2(dup2(w), q[k]);
        else g[k] = fma2(dup2(-a.kf[K_OMEGA]), fma2(dup2(-w), q[k], g[k]), g[k]);
    }
}

// One lattice step of the group's leaves. f holds the post-collision values of this thread's rows; the rows
// that its neighbours need are in ex[b], this step leaves its own in ex[1 - b]. STORE: lanes with `store`
// also put the flow velocity (Eq. 15) of the state before the collision into the scratch.
template <bool TAU1, bool STORE>
__device__ __forceinline__ void reg_step(float2 (&f)[Q][RG_ROWS], const float2 (&ne)[RG_ROWS], float2 hgx, float2 hgy,
                                         const RegGeo &q, RegShared &sh, float2 *mine, int b, bool store,
                                         const LocalArgs &a)
{
    group_sync(q.group, q.w0);
    const float2 *in = &sh.ex[b][0][0][0];
    float2 up[3], dn[3];                         // e_y = +1 from the row below, e_y = -1 from the row above
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        up[k] = in[q.below + k * 32];
        dn[k] = in[q.above + (3 + k) * 32];
    }
    auto from_left = [&](float2 v) { return make_float2(__shfl_sync(0xffffffffu, v.y, q.left), v.x); };
    auto from_right = [&](float2 v) { return make_float2(v.y, __shfl_sync(0xffffffffu, v.x, q.right)); };
    float2 *out = mine + (1 - b) * (RG_WARPS * 6 * 32);
#pragma unroll
    for (int r = 0; r < RG_ROWS; ++r) {
        float2 g[Q];
        g[0] = f[0][r];
        g[1] = from_left(f[1][r]);
        g[3] = from_right(f[3][r]);
        g[2] = up[0];
        g[5] = from_left(up[1]);
        g[6] = from_right(up[2]);
        g[4] = r < RG_ROWS - 1 ? f[4][r + 1] : dn[0];
        g[7] = from_right(r < RG_ROWS - 1 ? f[7][r + 1] : dn[1]);
        g[8] = from_left(r < RG_ROWS - 1 ? f[8][r + 1] : dn[2]);
        up[0] = f[2][r];                         // what the next row pulls
        up[1] = f[5][r];
        up[2] = f[6][r];
        float2 rux, ruy, rho;
        collide_reg<TAU1>(g, ne[r], hgx, hgy, a, rux, ruy, rho);
#pragma unroll
        for (int k = 0; k < Q; ++k) f[k][r] = g[k];
        if (STORE && store) {
            const int c = q.scratch + (q.row + r) * q.s + q.col;
            *reinterpret_cast<float2 *>(sh.ux + c) = make_float2(rux.x / rho.x, rux.y / rho.y);
            *reinterpret_cast<float2 *>(sh.uy + c) = make_float2(ruy.x / rho.x, ruy.y / rho.y);
        }
        if (r == 0) {
            out[3 * 32] = g[4];
            out[4 * 32] = g[7];
            out[5 * 32] = g[8];
        }
        if (r == RG_ROWS - 1) {
            out[0 * 32] = g[2];
            out[1 * 32] = g[5];
            out[2 * 32] = g[6];
        }
    }
}

// Queue of a size class: jobs qbeg .. qbeg + qn - 1. The first `dealt` of them are dealt out, one per group
// position, when the launch starts; the rest are popped.
struct RegQueue {
    int cls, qbeg, qn, dealt;
};

// Takes job i of the queue (i < 0: the next one) into slot sl at group step T; none: no more jobs.
__device__ __forceinline__ void reg_take(const LocalArgs &a, RegSlot &sl, const RegQueue &u, int i, unsigned T, bool none)
{
    sl.job = -1;
    sl.fresh = 0;
    if (none) return;
    if (i < 0) i = u.dealt + atomicAdd(&a.heads[u.cls], 1);
    if (i >= u.qn) return;
    const int qbeg = u.qbeg;
    sl.job = a.jobs[qbeg + i];
    sl.leaf = sl.job >> 1;
    sl.drive = sl.job & 1;
    sl.x0 = a.leaves[3 * sl.leaf] - a.margin;
    sl.y0 = a.leaves[3 * sl.leaf + 1] - a.margin;
    sl.prev = 0.0;
    sl.fresh = 1;
    sl.next_check = a.check_every;
    sl.tstart = T;
    sl.tstore = T + (unsigned)min(a.check_every, (int)a.max_steps);
}

// The check of one leaf, by one whole warp: mean velocity in FP64 in a fixed order, the stop test on the
// driven component, K* (Eq. 17) and the slot's next job. T: group steps done.
__device__ __forceinline__ void reg_check(const LocalArgs &a, RegShared &sh, RegSlot &slot, int scratch, int s, int lane,
                                          unsigned T, const RegQueue &u, bool abort_now)
{
    RegSlot sl = slot;
    const bool check = sl.tstore + 1 == T;           // the store step has just run
    const int t = (int)((check ? sl.tstore : T) - sl.tstart);
    int st = -1;                                     // -1: keep going
    double ux = 0.0, uy = 0.0;
    if (check) {
        const int m = a.margin, hi = s - m, n = s * s;
        for (int c = lane; c < n; c += 32) {
            const int ly = c / s, lx = c - ly * s;
            if (m == 0 || (lx >= m && lx < hi && ly >= m && ly < hi)) {
                ux += (double)sh.ux[scratch + c];
                uy += (double)sh.uy[scratch + c];
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            ux += __shfl_xor_sync(0xffffffffu, ux, off);
            uy += __shfl_xor_sync(0xffffffffu, uy, off);
        }
        const double inner = (double)(s - 2 * a.margin) * (double)(s - 2 * a.margin);
        ux /= inner;
        uy /= inner;
        const double cur = sl.drive == 0 ? ux : uy;
        const bool regular = t == sl.next_check;
        if (regular) sl.next_check += a.check_every;
        if (a.tol > 0.0 && t > a.check_every && regular && fabs(cur - sl.prev) <= a.tol * a.check_every * fabs(cur))
            st = LBM_OK;
        else if (t == (int)a.max_steps)
            st = a.tol > 0.0 ? LBM_ENOTCONV : LBM_OK;
        sl.prev = cur;
        sl.tstore = sl.tstart + (unsigned)min(sl.next_check, (int)a.max_steps);
    }
    if (abort_now && st < 0) st = LBM_ETIMEOUT;
    if (lane == 0) {
        if (st >= 0) {
            // Eq. 17: column `drive` of K* (NaN if abandoned unchecked)
            const double kx = check ? a.nu_over_g * ux : __longlong_as_double(0x7ff8000000000000LL);
            const double ky = check ? a.nu_over_g * uy : __longlong_as_double(0x7ff8000000000000LL);
            a.keff[4 * (int64_t)sl.leaf + (sl.drive == 0 ? 0 : 1)] = kx;
            a.keff[4 * (int64_t)sl.leaf + (sl.drive == 0 ? 2 : 3)] = ky;
            if (a.steps) a.steps[2 * (int64_t)sl.leaf + sl.drive] = t;
            if (st != LBM_OK) {
                atomicMax(&a.status[sl.leaf], st);
                atomicMax(a.worst, st);
            }
            reg_take(a, sl, u, -1, T, abort_now);
        }
        slot = sl;
    }
    __syncwarp();
}

template <bool TAU1>
__global__ void __launch_bounds__(RG_THREADS, 1) local_reg_kernel(LocalArgs a)
{
    extern __shared__ __align__(16) unsigned char rg_smem[];
    RegShared &sh = *reinterpret_cast<RegShared *>(rg_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        sh.t0 = start_time(a);
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the shared-memory solver needs nothing of this one
    }
    if (lane == 0) sh.abort[warp] = 0;
    __syncthreads();
    const int nclass = a.table ? (a.table[DT_BAD] ? 0 : a.table[DT_NCLASS]) : a.nclass;
    bool stop = false;                               // the wall-clock limit has run out
    bool first = true;                               // no class begun yet
    float2 *mine = &sh.ex[0][warp][0][lane];

    // classes come largest side first, so groups only ever split into smaller ones
    for (int cls = 0; cls < nclass; ++cls) {
        const int s = a.table ? a.table[DT_SIZE + cls] : a.class_size[cls];
        if (!reg_side(s)) continue;
        RegGeo q = reg_geometry(s, warp, lane);
        q.below = (q.below >> 5) * (6 * 32) + (q.below & 31);    // offsets in ex
        q.above = (q.above >> 5) * (6 * 32) + (q.above & 31);
        const bool leader = warp == q.w0;
        RegSlot *slots = sh.slots[q.w0];
        unsigned T = 0;                              // group step
        // every group starts on the first class together: its jobs are dealt out CTA by CTA, so that a small
        // batch spreads over the SMs; groups reach a later class one by one and pop
        RegQueue u;
        u.cls = cls;
        u.qbeg = a.table ? a.table[DT_OFF + cls] : a.class_off[cls];
        u.qn = (a.table ? a.table[DT_OFF + cls + 1] : a.class_off[cls + 1]) - u.qbeg;
        u.dealt = first ? (int)gridDim.x * (RG_WARPS / q.group) * q.jobs : 0;
        if (leader && lane < q.jobs)
            reg_take(a, slots[lane], u, first ? (int)(((warp / q.group) * q.jobs + lane) * gridDim.x + blockIdx.x) : -1,
                     T, stop);
        first = false;
        group_sync(q.group, q.w0);

        float2 f[Q][RG_ROWS], ne[RG_ROWS], hgx = dup2(0.0f), hgy = dup2(0.0f);
#pragma unroll
        for (int r = 0; r < RG_ROWS; ++r) {
            ne[r] = dup2(0.0f);
#pragma unroll
            for (int k = 0; k < Q; ++k) f[k][r] = dup2(0.0f);
        }
        unsigned tstore = 0;
        bool active = false;
        for (;;) {
            // this lane's job: new ones start from rest, with the drag fraction of their cells
            const RegSlot &sl = slots[q.job];
            active = q.cell && sl.job >= 0;
            tstore = sl.tstore;
            if (active && sl.fresh) {
#pragma unroll
                for (int r = 0; r < RG_ROWS; ++r) {
                    float e[2];
                    for (int k = 0; k < 2; ++k) {
                        int gx = sl.x0 + q.col + k, gy = sl.y0 + q.row + r;     // periodic when oversampling
                        gx = gx < 0 ? gx + a.nx : (gx >= a.nx ? gx - a.nx : gx);
                        gy = gy < 0 ? gy + a.ny : (gy >= a.ny ? gy - a.ny : gy);
                        e[k] = (float)coef_e(a.kappa[(int64_t)gy * a.nx + gx], a.eps_nu);
                    }
                    ne[r] = make_float2(-e[0], -e[1]);
#pragma unroll
                    for (int k = 0; k < Q; ++k) f[k][r] = dup2(0.0f);
                }
                hgx = dup2(sl.drive == 0 ? a.kf[K_HG] : 0.0f);
                hgy = dup2(sl.drive == 1 ? a.kf[K_HG] : 0.0f);
#pragma unroll
                for (int k = 0; k < 6; ++k) mine[(T & 1) * (RG_WARPS * 6 * 32) + k * 32] = dup2(0.0f);
            }
            // steps to the next velocity store of any leaf of the group
            const bool any = sl.job >= 0;
            const unsigned todo = __reduce_min_sync(0xffffffffu, any ? tstore - T : 0xffffffffu);
            if (todo == 0xffffffffu) break;
            const unsigned plain = min(todo, 256u);  // the wall clock is read at least every 256 steps
            for (unsigned i = 0; i < plain; ++i, ++T)
                reg_step<TAU1, false>(f, ne, hgx, hgy, q, sh, mine, T & 1, false, a);
            const bool event = plain == todo;
            if (event) {
                reg_step<TAU1, true>(f, ne, hgx, hgy, q, sh, mine, T & 1, active && tstore == T, a);
                ++T;
            }
            group_sync(q.group, q.w0);               // velocities stored, slots read by every warp
            if (leader) {
                if (lane == 0 && !sh.abort[q.w0]) {
                    if (*(volatile int *)a.abort_flag) sh.abort[q.w0] = 1;
                    else if (globaltimer() - sh.t0 > a.time_limit_ns) {
                        sh.abort[q.w0] = 1;
                        atomicExch(a.abort_flag, 1);
                    }
                }
                __syncwarp();
                const bool abort_now = sh.abort[q.w0] != 0;
                for (int j = 0; j < q.jobs; ++j) {
                    if (slots[j].job < 0) continue;
                    if (lane == 0) slots[j].fresh = 0;
                    __syncwarp();
                    if (slots[j].tstore + 1 == T || abort_now)
                        reg_check(a, sh, slots[j], q.w0 * RG_WCELLS + j * s * s, s, lane, T, u, abort_now);
                }
            }
            group_sync(q.group, q.w0);
            stop = sh.abort[q.w0] != 0;
        }
        // the next class may split the group: its warps find the verdict under their own index
        group_sync(q.group, q.w0);
        if (lane == 0) sh.abort[warp] = stop;
        __syncwarp();
    }
}

}  // namespace
}  // namespace lbm
