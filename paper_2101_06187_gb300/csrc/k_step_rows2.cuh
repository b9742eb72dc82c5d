// k_step_rows2.cuh -- the one-column kernel of FP32 storage for any nx (cfl <= 1):
// a thread updates two vertically adjacent nodes (x, y), (x, y + 1) in packed
// FP32 lanes (packed.cuh), one instruction for both.
//
// The kernel for odd nx, where no run of nodes starts aligned in every row,
// and the untuned default.  One node per thread it issued about 700
// instructions per node and was bound by issue; with two rows a class that
// interpolates between rows reads three instead of four of them (72 loads for
// two nodes instead of 106), every load is a whole warp's row segment, and the
// arithmetic is shared.  Taps and order are step_pair's, so results equal the
// packed kernel's bit for bit.  us per step, one node per thread and now: 1023 x
// 769 22.0 and 20.6, 513 x 511 8.0 and 7.0, 4095^2 438 and 417 (85% of the copy
// bandwidth), 1023 x 769 at cfl 0.625 24.2 and 20.8.  At cfl > 1 the choice of
// the corner per class doubles the loads' code and it lost (24.1 and 43.6), so
// that stays with k_step_gather.
#pragma once

#include "k_step_gather.cuh"
#include "packed.cuh"

namespace rlbk {

// Class c at the two nodes: rowoff[k] / cols[k] are rows y - 1 .. y + 2 and
// columns x - 1 .. x + 1 (periodic).  Same corners and weights as gather_class.
template <int c, typename I, int SM>
__device__ __forceinline__ pf2 gather_rows2(const float *__restrict__ qin, I cbase, const I (&rowoff)[4],
                                            const I (&cols)[3], const StepParams &p) {
    static_assert(SM == kStreamCfl1 || SM == kStreamSub1, "halo-1 streaming modes only");
    constexpr bool cfl1 = SM == kStreamCfl1;
    constexpr double cx = cls_cx(c), cy = cls_cy(c), tx = cls_tx(c), ty = cls_ty(c);
    // corner: x - c at CFL 1; below, the cell on the class's upstream side or its own
    constexpr int ox = cfl1 ? cls_ox(c) : (cx > 0 ? -1 : 0), oy = cfl1 ? cls_oy(c) : (cy > 0 ? -1 : 0);
    constexpr bool two_cols = cfl1 ? tx != 0.0 : cx != 0.0, two_rows = cfl1 ? ty != 0.0 : cy != 0.0;
    // one column of the source rows: the lanes' first tap rows (a) and second ones (b)
    auto column = [&](I col, pf2 &a, pf2 &b) {
        auto at = [&](int k) { return __ldg(qin + (cbase + rowoff[oy + 1 + k] + col)); };
        const float u1 = at(1);
        a = pf2(at(0), u1);
        if constexpr (two_rows) b = pf2(u1, at(2));
    };
    pf2 a, b, a1, b1;
    column(cols[ox + 1], a, b);
    if constexpr (two_cols) column(cols[ox + 2], a1, b1);
    if constexpr (!two_cols && !two_rows) {
        return a;  // weight 1
    } else {
        constexpr double w[4] = {(1.0 - tx) * (1.0 - ty), tx * (1.0 - ty), (1.0 - tx) * ty, tx * ty};
        auto wt = [&](int k) { return cfl1 ? pf2((float)w[k]) : pf2(par_wt<float>(p, c, k)); };
        pf2 v = wt(0) * a;
        if constexpr (two_cols) v = fmadd(wt(1), a1, v);
        if constexpr (two_rows) v = fmadd(wt(2), b, v);
        if constexpr (two_cols && two_rows) v = fmadd(wt(3), b1, v);
        return v;
    }
}

template <bool FORCED, typename I, int SM>
__global__ void __launch_bounds__(256, 2) k_step_rows2(const float *__restrict__ qin, float *__restrict__ qout,
                                                       const float *__restrict__ F, StepParams p) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = (blockIdx.y * blockDim.y + threadIdx.y) * 2;
    if (x >= p.nx || y >= p.ny) return;
    const bool second = y + 1 < p.ny;  // an odd ny's last row is updated alone (its upper lane wraps, unwritten)
    I rowoff[4], cols[3];
    for (int d = 0; d < 4; ++d) rowoff[d] = (I)wrap2(y, d - 1, p.ny) * (I)p.pitch;
    for (int d = 0; d < 3; ++d) cols[d] = (I)wrap2(x, d - 1, p.nx);
    const I plane = (I)p.plane, n0 = rowoff[1] + (I)x, n1 = rowoff[2] + (I)x;
    pf2 q[NC];
    static_for<0, NC>([&](auto C) {
        constexpr int c = decltype(C)::value;
        q[c] = gather_rows2<c, I, SM>(qin, (I)c * plane, rowoff, cols, p);
    });
    pf2 Fx = 0.0f, Fy = 0.0f;
    if constexpr (FORCED) {
        Fx = pf2(__ldg(F + n0), __ldg(F + n1));
        Fy = pf2(__ldg(F + (plane + n0)), __ldg(F + (plane + n1)));
    }
    collide_node<pf2, pf2, FORCED, false, true>(q, Fx, Fy, p);
    static_for<0, NC>([&](auto C) {
        constexpr int c = decltype(C)::value;
        qout[(I)c * plane + n0] = q[c].v.x;
        if (second) qout[(I)c * plane + n1] = q[c].v.y;
    });
}

}  // namespace rlbk
