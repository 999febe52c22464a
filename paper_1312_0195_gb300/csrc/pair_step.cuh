// pair_step.cuh -- the fine and coarse grids' collision on two cells at once (multistep.cu, tiles.cu).
#pragma once

#include "lbm_internal.h"
#include "pair_ops.cuh"

namespace lbm {
namespace {

// Drag coefficients and force of a pair.
template <int COEF, bool GF>
struct PairCoef {
    float2 c0, c1, c2, c3, gx, gy;
};
template <int COEF, bool GF> constexpr int ncoef() { return (COEF == COEF_TENSOR ? 4 : 1) + (GF ? 2 : 0); }

// Moments of two cells' streamed deviations and their momentum rho u (Eq. 6 or 18), the products and sums that
// the compiler fuses in collide_cell and cell_uv of step.cu fused here explicitly.
struct Flow2 {
    float2 drho, rho, mx, my, rux, ruy;
};
template <int COEF, bool GF>
__device__ __forceinline__ Flow2 flow_pair(const float2 (&g)[Q], const PairCoef<COEF, GF> &k, float rho0, float half_eps)
{
    Flow2 m;
    m.drho = g[0];
#pragma unroll
    for (int a = 1; a < Q; ++a) m.drho = add2(m.drho, g[a]);
    m.mx = add2(sub2(sub2(add2(sub2(g[1], g[3]), g[5]), g[6]), g[7]), g[8]);
    m.my = sub2(sub2(add2(add2(sub2(g[2], g[4]), g[5]), g[6]), g[7]), g[8]);
    m.rho = add2(dup2(rho0), m.drho);
    const float2 h = mul2(dup2(half_eps), m.rho);
    const float2 rx = fma2(h, k.gx, m.mx), ry = fma2(h, k.gy, m.my);
    if constexpr (COEF == COEF_SCALAR) {
        const float2 n = make_float2(-k.c0.x, -k.c0.y);
        m.rux = fma2(n, rx, rx);
        m.ruy = fma2(n, ry, ry);
    } else {
        m.rux = sub2(rx, fma2(k.c0, rx, mul2(k.c1, ry)));
        m.ruy = sub2(ry, fma2(k.c2, rx, mul2(k.c3, ry)));
    }
    return m;
}

// The collision of two cells: collide_cell of step.cu (simplified scheme).
template <int COEF, bool GF>
__device__ __forceinline__ void collide_pair(float2 (&g)[Q], const PairCoef<COEF, GF> &k, float rho0, float half_eps,
                                             float omega, float two_tau, float omt)
{
    const Flow2 m = flow_pair<COEF, GF>(g, k, rho0, half_eps);
    const float2 drho = m.drho;
    const float2 ux = fma2(dup2(omt), m.mx, mul2(dup2(two_tau), m.rux));
    const float2 uy = fma2(dup2(omt), m.my, mul2(dup2(two_tau), m.ruy));
    const float2 sp = add2(ux, uy), sm = sub2(ux, uy);
    const float w0 = float(4.0 / 9.0), w1 = float(1.0 / 9.0), w2 = float(1.0 / 36.0);
    // g + omega (w q - g): the inner difference is kept with its sign turned, -(w q - g)
    auto relax = [&](float2 &p, float w, float2 q) { p = fma2(dup2(-omega), fma2(dup2(-w), q, p), p); };
    relax(g[0], w0, drho);
    relax(g[1], w1, fma2(dup2(3.0f), ux, drho));
    relax(g[3], w1, fma2(dup2(-3.0f), ux, drho));
    relax(g[2], w1, fma2(dup2(3.0f), uy, drho));
    relax(g[4], w1, fma2(dup2(-3.0f), uy, drho));
    relax(g[5], w2, fma2(dup2(3.0f), sp, drho));
    relax(g[7], w2, fma2(dup2(-3.0f), sp, drho));
    relax(g[8], w2, fma2(dup2(3.0f), sm, drho));
    relax(g[6], w2, fma2(dup2(-3.0f), sm, drho));
}

}  // namespace
}  // namespace lbm
