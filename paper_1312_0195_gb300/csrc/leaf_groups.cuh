// leaf_groups.cuh -- how square leaves are laid out over a CTA of 16 warps when each thread holds a block of
// 4 rows x 2 columns of its leaf in registers (the local problems of local_reg.cuh, the Darcy solves of
// darcy_groups.cuh). A leaf of side s takes s / 2 lanes per row and s / 4 row blocks, packed into the fewest
// warps, a power of two of them: 16 for a side of 64, 4 for 32, one for 16 and 12, a quarter of one for 8.
// Such a group of warps works on its own leaf and has a barrier of its own.
#pragma once

#include <cuda_runtime.h>

namespace lbm {
namespace {

constexpr int RG_WARPS = 16;
constexpr int RG_THREADS = RG_WARPS * 32;
constexpr int RG_ROWS = 4;                   // rows of a thread's block
constexpr int RG_JOBS = 16;                  // leaves of one warp at most (side 4)
constexpr int RG_WCELLS = 256;               // cells of a warp at most

// Sides that can be laid out so.
__host__ __device__ constexpr bool reg_side(int s) { return s >= 4 && s <= 64 && s % 4 == 0; }

// Barrier of a group of `g` warps whose first is `w0`: each (size, position) has a hardware barrier of its own.
__device__ __forceinline__ void group_sync(int g, int w0)
{
    if (g == 1) {
        __syncwarp();
    } else {
        const int id = g == 2 ? 1 + w0 / 2 : (g == 4 ? 9 + w0 / 4 : (g == 8 ? 13 + w0 / 8 : 15));
        asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(g * 32) : "memory");
    }
}

// What a thread knows of its leaf size.
struct RegGeo {
    int s, group, w0;            // side; warps of the group and its first warp
    int jobs, job;               // leaves of the group; this lane's
    int row, col;                // first row and first column of this thread's block
    bool cell;                   // has cells
    int left, right;             // lanes of the neighbouring columns
    int below, above;            // threads of the CTA that hold the neighbouring row blocks
    int scratch;                 // first of this lane's leaf's cells in an array of the CTA's 4096
};

__host__ __device__ __forceinline__ RegGeo reg_geometry(int s, int warp, int lane)
{
    RegGeo q;
    const int w = s / 2, per_warp = 32 / w, blocks = s / RG_ROWS;
    q.s = s;
    q.group = 1;
    q.jobs = per_warp / blocks;
    if (q.jobs < 1) {
        q.jobs = 1;
        while (q.group * per_warp < blocks) q.group *= 2;
    }
    q.w0 = warp / q.group * q.group;
    const int c = lane % w, b = lane / w;                    // column pair, row block within the warp
    int rb;                                                  // row block within the leaf
    if (q.group == 1) {
        q.job = b / blocks;
        rb = b - q.job * blocks;
        q.cell = q.job < q.jobs;
        if (!q.cell) q.job = 0;
    } else {
        q.job = 0;
        rb = (warp - q.w0) * per_warp + b;
        q.cell = b < per_warp && rb < blocks;
    }
    q.row = rb * RG_ROWS;
    q.col = 2 * c;
    q.left = q.right = lane;
    q.below = q.above = warp * 32 + lane;
    if (q.cell) {
        q.left = c == 0 ? lane + w - 1 : lane - 1;
        q.right = c == w - 1 ? lane - w + 1 : lane + 1;
        auto place = [&](int r) {
            if (q.group == 1) return warp * 32 + (q.job * blocks + r) * w + c;
            return (q.w0 + r / per_warp) * 32 + (r % per_warp) * w + c;
        };
        q.below = place(rb == 0 ? blocks - 1 : rb - 1);
        q.above = place(rb == blocks - 1 ? 0 : rb + 1);
    }
    q.scratch = q.w0 * RG_WCELLS + q.job * s * s;
    return q;
}

}  // namespace
}  // namespace lbm
