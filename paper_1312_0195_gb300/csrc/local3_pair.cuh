// local3_pair.cuh -- 3-D local problems (FP32, cubes of up to 18 cells a side) two at a time. Included by d3q19.cu.
//
// local3d_cluster_kernel moves and computes one value per instruction: 216 thread instructions per lattice update
// and 38 shared accesses of 4 bytes. Here a cluster steps two jobs (leaf and drive) side by side, interleaved cell by
// cell: a population of a cell is a float2, job A and job B, so every shared access is 8 bytes, the collision is
// packed f32x2 arithmetic, and addresses are formed once for both. The cube is split into z slabs of at most
// 1024 cells a CTA (twice the CTAs of the one-job kernel for two jobs), stepped in place with the AA
// pattern and one cluster barrier a step, as there. A finished job's place is refilled from the batch's
// queue at once (a new job starts from rest, where every slot is zero, so either half of the AA pattern may
// come first), and the clusters stay for the whole batch. The arithmetic of a cell is the one-job kernel's,
// operation by operation.
//
// What bounds it, at side 16: nothing is full. The shared-memory path is 56 % busy, the FMA pipe 41 %, issue slots 39 %;
// the barrier that ends each step and its release fence are 17 % of the stalls, and loads, arithmetic and stores of a
// CTA's warps, which start each step together, overlap little.
// Which batches come here: pair_pays in d3q19.cu.
#pragma once

#include "pair_ops.cuh"

namespace lbm {
namespace {

// moments19 for two jobs.
__device__ __forceinline__ void moments19_pair(const float2 (&g)[Q19], float2 &drho, float2 &jx, float2 &jy, float2 &jz)
{
    float2 s[9], d[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        s[p] = add2(g[2 * p + 1], g[2 * p + 2]);
        d[p] = sub2(g[2 * p + 1], g[2 * p + 2]);
    }
    drho = add2(g[0], add2(add2(add2(add2(s[0], s[1]), add2(s[2], s[3])), add2(add2(s[4], s[5]), add2(s[6], s[7]))), s[8]));
    jx = add2(d[0], add2(add2(d[3], d[4]), add2(d[5], d[6])));
    jy = add2(d[1], add2(sub2(d[3], d[4]), add2(d[7], d[8])));
    jz = add2(d[2], add2(sub2(d[5], d[6]), sub2(d[7], d[8])));
}

struct Drag2 {
    float2 drho, rho, jx, jy, jz, rux, ruy, ruz;
};
// moments and the drag-reduced momentum (1 - e) r, r = j + hg rho along each job's axis; ne is -e.
__device__ __forceinline__ Drag2 drag_pair(const float2 (&g)[Q19], float2 ne, float2 hgx, float2 hgy, float2 hgz)
{
    Drag2 m;
    moments19_pair(g, m.drho, m.jx, m.jy, m.jz);
    m.rho = add2(dup2(1.0f), m.drho);
    const float2 rx = fma2(hgx, m.rho, m.jx), ry = fma2(hgy, m.rho, m.jy), rz = fma2(hgz, m.rho, m.jz);
    m.rux = fma2(ne, rx, rx);
    m.ruy = fma2(ne, ry, ry);
    m.ruz = fma2(ne, rz, rz);
    return m;
}

__device__ __forceinline__ void collide19_pair(float2 (&g)[Q19], float2 ne, float2 hgx, float2 hgy, float2 hgz, float k_ru,
                                               float k_j, float om)
{
    const Drag2 m = drag_pair(g, ne, hgx, hgy, hgz);
    const float2 ux = fma2(dup2(k_ru), m.rux, mul2(dup2(k_j), m.jx));
    const float2 uy = fma2(dup2(k_ru), m.ruy, mul2(dup2(k_j), m.jy));
    const float2 uz = fma2(dup2(k_ru), m.ruz, mul2(dup2(k_j), m.jz));
    const float w0 = float(1.0 / 3.0), w1 = float(1.0 / 18.0), w2 = float(1.0 / 36.0);
    const float2 d1 = mul2(dup2(w1), m.drho), d2 = mul2(dup2(w2), m.drho);
    // g + om (w drho - g), the inner difference with its sign turned
    g[0] = fma2(dup2(-om), fma2(dup2(-w0), m.drho, g[0]), g[0]);
    auto relax = [&](float2 &p, float2 &q, float2 wd, float w, float2 eu) {
        p = fma2(dup2(om), fma2(dup2(w), eu, sub2(wd, p)), p);
        q = fma2(dup2(om), fma2(dup2(-w), eu, sub2(wd, q)), q);
    };
    relax(g[1], g[2], d1, w1, ux);
    relax(g[3], g[4], d1, w1, uy);
    relax(g[5], g[6], d1, w1, uz);
    relax(g[7], g[8], d2, w2, add2(ux, uy));
    relax(g[9], g[10], d2, w2, sub2(ux, uy));
    relax(g[11], g[12], d2, w2, add2(ux, uz));
    relax(g[13], g[14], d2, w2, sub2(ux, uz));
    relax(g[15], g[16], d2, w2, add2(uy, uz));
    relax(g[17], g[18], d2, w2, sub2(uy, uz));
}

constexpr int CP3_THREADS = 512, CP3_CPT = 2;       // a slab holds at most 1024 cells
constexpr int CP3_MAX_SIDE = 18;

struct Pair3Shared {
    double part[2][4];                               // per job: sums of u; [0][3]: abandon
    double wred[CP3_THREADS / 32][6];
    uint32_t zb[32];                                 // layer z of the cube, in any CTA
    int job[2];                                      // rank 0: the jobs taken last
};
inline size_t pair3_smem_bytes(int ps) { return sizeof(Pair3Shared) + (size_t)ps * Q19 * sizeof(float2); }

// Past the wall-clock limit: the jobs nobody has taken are abandoned too (LBM_ETIMEOUT, no K*, 0 steps).
__device__ __noinline__ void abandon_queue(const Clu3Args<float> &a, int *head)
{
    for (int j; (j = atomicAdd(head, 1)) < a.njobs;) {
        const int leaf = a.ids[j / 3];
        for (int i = 0; i < 3; ++i) a.keff[9 * (int64_t)leaf + 3 * i + j % 3] = __longlong_as_double(0x7ff8000000000000LL);
        atomicMax(&a.status[leaf], (int)LBM_ETIMEOUT);
    }
}

// a.njobs jobs from the queue *head (zeroed), a.s^3 cells each, over as many clusters as are resident.
template <int PS>
__global__ void __launch_bounds__(CP3_THREADS, 1) local3d_pair_kernel(Clu3Args<float> a, int *head)
{
    extern __shared__ __align__(16) unsigned char p3_smem[];
    Pair3Shared &sh = *reinterpret_cast<Pair3Shared *>(p3_smem);
    float2 *own = reinterpret_cast<float2 *>(p3_smem + sizeof(Pair3Shared));      // [19][PS]
    const int C = (int)cluster_size(), r = (int)cluster_rank();
    const int s = a.s, s2 = s * s, L = a.L;
    const int z0 = r * L, ncell = max(0, min(L, s - z0)) * s2;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5;
    for (int z = tid; z < s; z += nt) sh.zb[z] = cluster_addr(own, z / L) + (uint32_t)((z % L) * s2 * sizeof(float2));

    int geo[CP3_CPT];
    float2 ne[CP3_CPT];
#pragma unroll
    for (int i = 0; i < CP3_CPT; ++i) {
        const int c = tid + i * nt;
        geo[i] = -1;
        ne[i] = dup2(0.0f);
        if (c >= ncell) continue;
        const int x = c % s, yz = c / s, y = yz % s, zl = yz / s, z = z0 + zl;
        const int sl = s - 2 * a.m;
        const bool in = x >= a.m && x < a.m + sl && y >= a.m && y < a.m + sl && z >= a.m && z < a.m + sl;
        geo[i] = (zl << 16) | (y << 8) | x | (in ? CLU3_IN : 0);
#pragma unroll
        for (int q = 0; q < Q19; ++q) own[q * PS + c] = dup2(0.0f);
    }
    unsigned long long t0 = 0;
    if (r == 0 && tid == 0) {
        const unsigned long long now = globaltimer3();
        const unsigned long long prev = atomicCAS(a.t_start, 0ull, now);
        t0 = prev == 0ull ? now : prev;
        for (int k = 0; k < 2; ++k) sh.job[k] = atomicAdd(head, 1);
    }
    cluster_sync_all();

    // Per job (the same in every thread of the cluster): leaf, drive, first step, next event, last checked mean.
    int leaf[2], drive[2];
    long long start[2] = {0, 0}, event[2];
    double prev_u[2] = {0.0, 0.0};
    bool on[2], fresh[2];
    float2 hgx = dup2(0.0f), hgy = dup2(0.0f), hgz = dup2(0.0f);
    long long T = 0;                                 // steps the cluster has run
    auto take = [&](int k) {                         // job k's place: what rank 0 took for it
        const int j = ld_cluster<int>(cluster_addr(&sh.job[k], 0));
        on[k] = fresh[k] = j < a.njobs;
        if (!on[k]) return;
        leaf[k] = a.ids[j / 3];
        drive[k] = j % 3;
        start[k] = T;
        event[k] = T + min((long long)a.k, (long long)a.max_steps);
        prev_u[k] = 0.0;
    };
    take(0);
    take(1);
    for (;;) {
        // new jobs: the drag fraction of their cubes, rest
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (!fresh[k]) continue;
            const int4 Lf = a.leaves[leaf[k]];
#pragma unroll
            for (int i = 0; i < CP3_CPT; ++i) {
                if (geo[i] < 0) continue;
                const int x = geo[i] & 255, y = (geo[i] >> 8) & 255, z = z0 + ((geo[i] >> 16) & 255);
                // the grown cube starts margin cells before the leaf, wrapping at the field's edges
                int gx = Lf.x - a.m + x, gy = Lf.y - a.m + y, gz = Lf.z - a.m + z;
                gx = gx < 0 ? gx + a.nx : (gx >= a.nx ? gx - a.nx : gx);
                gy = gy < 0 ? gy + a.ny : (gy >= a.ny ? gy - a.ny : gy);
                gz = gz < 0 ? gz + a.nz : (gz >= a.nz ? gz - a.nz : gz);
                const float kv = a.kappa[((int64_t)gz * a.ny + gy) * a.nx + gx];
                double e;
                if (!(kv >= 0.0f)) e = 1.0;
                else if (a.eps_nu == 0.0 || isinf(kv)) e = 0.0;
                else if (kv == 0.0f) e = 1.0;
                else e = a.eps_nu / (2.0 * (double)kv + a.eps_nu);
                (k == 0 ? ne[i].x : ne[i].y) = -(float)e;
                const int c = tid + i * nt;
#pragma unroll
                for (int q = 0; q < Q19; ++q) (k == 0 ? own[q * PS + c].x : own[q * PS + c].y) = 0.0f;
            }
            (k == 0 ? hgx.x : hgx.y) = drive[k] == 0 ? a.hg : 0.0f;
            (k == 0 ? hgy.x : hgy.y) = drive[k] == 1 ? a.hg : 0.0f;
            (k == 0 ? hgz.x : hgz.y) = drive[k] == 2 ? a.hg : 0.0f;
            fresh[k] = false;
        }
        if (!on[0] && !on[1]) break;
        cluster_sync_all();
        const long long next = on[0] ? (on[1] ? min(event[0], event[1]) : event[0]) : event[1];
        for (; T < next; ++T) {
            const bool odd = (T & 1) != 0;
#pragma unroll
            for (int i = 0; i < CP3_CPT; ++i) {
                if (geo[i] < 0) continue;
                int gj = geo[i];
                asm volatile("" : "+r"(gj));         // keeps the addresses out of registers between steps
                const Cell3<float2> q = cell3_of<float2>(gj, s, sh.zb, z0);
                float2 g[Q19];
                if (odd) {
                    aa_read19<true, PS>(q, own, g);
                    collide19_pair(g, ne[i], hgx, hgy, hgz, a.k_ru, a.k_j, a.omega);
                    aa_write<true, PS, float2, 0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 17, 18>(q, own, g);
                } else {
                    aa_read19<false, PS>(q, own, g);
                    collide19_pair(g, ne[i], hgx, hgy, hgz, a.k_ru, a.k_j, a.omega);
                    aa_write<false, PS, float2, 0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 17, 18>(q, own, g);
                }
            }
            cluster_sync_all();
        }
        // mean flow velocity of the streamed state (Eq. 15) of both jobs, FP64 in a fixed order
        double m[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        const bool odd = (T & 1) != 0;
#pragma unroll
        for (int i = 0; i < CP3_CPT; ++i) {
            if (geo[i] < 0 || !(geo[i] & CLU3_IN)) continue;
            int gj = geo[i];
            asm volatile("" : "+r"(gj));
            const Cell3<float2> q = cell3_of<float2>(gj, s, sh.zb, z0);
            float2 g[Q19];
            if (odd) aa_read19<true, PS>(q, own, g);
            else aa_read19<false, PS>(q, own, g);
            const Drag2 v = drag_pair(g, ne[i], hgx, hgy, hgz);
            m[0] += (double)(v.rux.x / v.rho.x);
            m[1] += (double)(v.ruy.x / v.rho.x);
            m[2] += (double)(v.ruz.x / v.rho.x);
            m[3] += (double)(v.rux.y / v.rho.y);
            m[4] += (double)(v.ruy.y / v.rho.y);
            m[5] += (double)(v.ruz.y / v.rho.y);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < 6; ++j) m[j] += __shfl_down_sync(0xffffffffu, m[j], o);
        if (lane == 0)
            for (int j = 0; j < 6; ++j) sh.wred[wid][j] = m[j];
        __syncthreads();
        if (tid < 6) {
            double u = 0.0;
            for (int w = 0; w < (nt + 31) / 32; ++w) u += sh.wred[w][tid];
            sh.part[tid / 3][tid % 3] = u;
        }
        if (tid == 0) {
            sh.part[0][3] = 0.0;
            if (r == 0) {                            // rank 0 decides the wall-clock limit for the cluster
                if (*(volatile int *)a.abort_flag) sh.part[0][3] = 1.0;
                else if (globaltimer3() - t0 > a.time_limit_ns) {
                    sh.part[0][3] = 1.0;
                    atomicExch(a.abort_flag, 1);
                }
            }
        }
        cluster_sync_all();
        const bool abort_now = ld_cluster<double>(cluster_addr(&sh.part[0][3], 0)) != 0.0;
        const double sl = s - 2 * a.m, inv = 1.0 / (sl * sl * sl);
        bool refill[2] = {false, false};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (!on[k] || !(event[k] == T || abort_now)) continue;
            double u[3] = {0.0, 0.0, 0.0};
            for (int q = 0; q < C; ++q) {
                const uint32_t pq = cluster_addr(sh.part[k], q);
                u[0] += ld_cluster<double>(pq);
                u[1] += ld_cluster<double>(pq + 8);
                u[2] += ld_cluster<double>(pq + 16);
            }
            for (int q = 0; q < 3; ++q) u[q] *= inv;
            const double cur = drive[k] == 0 ? u[0] : (drive[k] == 1 ? u[1] : u[2]);
            const long long t = T - start[k];
            int st = -1;
            if (t % a.k == 0) {
                if (a.tol > 0.0 && t > a.k && fabs(cur - prev_u[k]) <= a.tol * a.k * fabs(cur)) st = LBM_OK;
                prev_u[k] = cur;
            }
            if (st < 0 && t >= a.max_steps) st = a.tol > 0.0 ? LBM_ENOTCONV : LBM_OK;
            if (st < 0 && abort_now) st = LBM_ETIMEOUT;
            event[k] = min(T + a.k - t % a.k, start[k] + (long long)a.max_steps);
            if (st < 0) continue;
            if (r == 0 && tid == 0) {
                for (int i = 0; i < 3; ++i) a.keff[9 * (int64_t)leaf[k] + 3 * i + drive[k]] = a.nu_over_g * u[i];   // Eq. 17
                if (a.steps) a.steps[3 * (int64_t)leaf[k] + drive[k]] = (int)t;
                if (st != LBM_OK) atomicMax(&a.status[leaf[k]], st);
                if (abort_now) abandon_queue(a, head);
                sh.job[k] = abort_now ? INT_MAX : atomicAdd(head, 1);
            }
            refill[k] = true;
        }
        if (refill[0] || refill[1]) {
            cluster_sync_all();                      // rank 0's new jobs; every read of the old sums is done
            if (refill[0]) take(0);
            if (refill[1]) take(1);
        }
    }
    cluster_sync_all();     // no CTA leaves while a peer may still read its shared memory
}

}  // namespace
}  // namespace lbm
