// prc_wall.cuh -- streaming at the walls from TMA-staged windows (cavity walls
// with the moving lid), shared by the kernels that stage wall tiles.
#pragma once

#include <type_traits>

#include "prc_tma.cuh"

namespace prc {

// Windows.  A node at (x, y) pulls population i from row y - y0 + OFF, column
// x - x0 + PADX - e_ix of plane i's window (`cw`), and its own population i sits
// at row y - y0 + OFF + e_iy, column x - x0 + PADX; (x0, y0) is the tile's origin
// and OFF the ring's width below the tile.  A wall tile's windows hold one more
// row below and above the rows that its pulls read, so that its wall nodes' own
// populations are all there (`cw` starts one row into them).

// Ghost cells of a wall tile (half-way bounce-back, reading A3): for every
// node n of the tile or its RING rings that lies inside the grid and every
// population i whose source n - e_i lies beyond a wall, the window of plane i
// at n - e_i -- a position outside the grid, which the copy filled with zeros
// and which no other pull reads -- receives the node's own population
// opp(i), so that the plain pulls then stream with bounce-back.  The cells of
// one wall are those of its nodes (one column or row of the tile and ring)
// and of the three populations that point away from it; a corner cell is
// written twice with the same value.  The moving-lid term is added in the
// collision precision: after the pull (lid_pull), or, where that is also the
// storage precision (LID), to the ghost cell.  All threads take part; the
// caller synchronises before the pulls.
template <typename S, int W, int H, int RING, int OFF, int PE, int BW, int PADX, int THREADS, bool LID = false>
__device__ __forceinline__ void fill_ghosts(S *cw, int tid, int x0, int y0, int nx, int ny, float lid = 0.f)
{
    static_assert(!LID || std::is_same<S, float>::value, "the lid term in the ghost cells is FP32");
    constexpr int NV = (H + 2 * RING) * 3, NH = (W + 2 * RING) * 3;  // cells of a vertical / horizontal wall
    const bool wl = (x0 <= RING) & (x0 + W + RING > 0), wr = (nx - 1 >= x0 - RING) & (nx - 1 < x0 + W + RING);
    const bool wb = (y0 <= RING) & (y0 + H + RING > 0), wt = (ny - 1 >= y0 - RING) & (ny - 1 < y0 + H + RING);
    const int total = (wl ? NV : 0) + (wr ? NV : 0) + (wb ? NH : 0) + (wt ? NH : 0);
    bool wrote = false;
    for (int c = tid; c < total; c += THREADS) {
        int k = c, side;  // 0 left, 1 right, 2 bottom, 3 top
        const int n0 = wl ? NV : 0, n1 = wr ? NV : 0, n2 = wb ? NH : 0;
        if (k < n0) {
            side = 0;
        } else if ((k -= n0) < n1) {
            side = 1;
        } else if ((k -= n1) < n2) {
            side = 2;
        } else {
            k -= n2;
            side = 3;
        }
        const int sel = k % 3, along = k / 3;
        int ax, ay, i;
        if (side < 2) {
            ax = side == 0 ? 0 : nx - 1;
            ay = y0 - RING + along;
            i = side == 0 ? (sel == 0 ? 1 : (sel == 1 ? 5 : 8)) : (sel == 0 ? 3 : (sel == 1 ? 6 : 7));
        } else {
            ax = x0 - RING + along;
            ay = side == 2 ? 0 : ny - 1;
            i = side == 2 ? (sel == 0 ? 2 : (sel == 1 ? 5 : 6)) : (sel == 0 ? 4 : (sel == 1 ? 7 : 8));
        }
        if ((ax < 0) | (ax >= nx) | (ay < 0) | (ay >= ny)) continue;
        // e_i and the opposite direction, for i in 1..8 (Eq. 3 ordering)
        const int exi = (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
        const int eyi = (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
        const int j = i <= 4 ? ((i + 1) % 4) + 1 : ((i - 3) % 4) + 5;
        const int col = ax - x0 + PADX, row = ay - y0 + OFF;
        S v = cw[j * PE + (row - eyi) * BW + col];
        if constexpr (LID) {
            if (ay - eyi == ny) v = i == 7 ? v - lid : (i == 8 ? v + lid : v);
        }
        cw[i * PE + row * BW + col - exi] = v;
        wrote = true;
    }
    // the next copies into this stage (async proxy) come after these writes
    if (wrote) fence_async_shared();
}

// The moving-lid term of the pulls from above the top wall (the two
// diagonal links SW and SE of a node in the top row, reading A3), added to
// the bounced populations in the collision precision as pull9 does.
template <typename V>
__device__ __forceinline__ void lid_pull(V g[9], float lid);
template <>
__device__ __forceinline__ void lid_pull<float>(float g[9], float lid)
{
    g[7] -= lid;
    g[8] += lid;
}
template <>
__device__ __forceinline__ void lid_pull<F2>(F2 g[9], float lid)
{
    g[7].v.x -= lid;
    g[7].v.y -= lid;
    g[8].v.x += lid;
    g[8].v.y += lid;
}

// Density of one ring unit of a wall tile (the units of ring_density) from
// the ghost-filled windows, with the lid term for a unit in the top row.
// Units outside the grid form values that the clamped gradients never read.
template <typename S, int W, int H, int PE, int BW, int RW, int PADX>
__device__ __forceinline__ void ring_density_wall(int tid, const S *cw, float *Rs, int y0, int ny, bool lid_on,
                                                  float lid)
{
    constexpr int PAIRS = W / 2;
    if (tid < 2 * PAIRS) {
        const int ry = tid < PAIRS ? 0 : H + 1;
        const int rx = 2 * (tid < PAIRS ? tid : tid - PAIRS);
        F2 gr[9];
        pull_pair<S, PE>(cw + ry * BW + rx + PADX, gr);
        if (lid_on & (y0 - 1 + ry == ny - 1)) lid_pull(gr, lid);
        *reinterpret_cast<float2 *>(Rs + ry * RW + rx + 2) = sum9(gr).v;
    } else {
        const int c = tid - 2 * PAIRS;
        const int ry = c >> 1, lx = (c & 1) ? W : -1;
        const S *b = cw + ry * BW + lx + PADX;
        float gr[9];
#pragma unroll
        for (int i = 0; i < 9; i++) gr[i] = Pair<S>::one(b + i * PE - ex_of(i));
        if (lid_on & (y0 - 1 + ry == ny - 1)) lid_pull(gr, lid);
        Rs[ry * RW + lx + 2] = sum9(gr);
    }
}

// Density gradients (reading A1) of the node (ax, ay) at tile position
// (lx, ly), its neighbours' positions clamped into the grid (the stencil and
// operation order of general_tile).
template <int RW>
__device__ __forceinline__ void node_gradients_clamped(const float *Rs, int lx, int ly, int ax, int ay, int nx, int ny,
                                                       float i12, float i12r, float &dxr, float &dyr)
{
    const int xc = lx + 2, xw = (ax > 0 ? lx - 1 : lx) + 2, xe = (ax + 1 < nx ? lx + 1 : lx) + 2;
    const int yc = (ly + 1) * RW, ys = (ay > 0 ? ly : ly + 1) * RW, yn = (ay + 1 < ny ? ly + 2 : ly + 1) * RW;
    const float rE = Rs[yc + xe], rW = Rs[yc + xw];
    const float rN = Rs[yn + xc], rS = Rs[ys + xc];
    const float rNE = Rs[yn + xe], rNW = Rs[yn + xw];
    const float rSE = Rs[ys + xe], rSW = Rs[ys + xw];
    drho_stencil<float>(rE, rW, rN, rS, rNE, rNW, rSE, rSW, i12, i12r, dxr, dyr);
}

// Ghost densities of a wall tile (reading A1: the nearest fluid node's density
// beyond a wall): every cell one node outside the grid that lies in the
// (W + 2 RING) x (H + 2 RING) nodes around the tile takes the density at its
// position clamped into the grid, so that the plain stencil applies.  R points
// to the tile's node (0, 0), rows of RW.  The caller synchronises before (the
// densities are complete) and after.
template <int W, int H, int RING, int RW, int THREADS>
__device__ __forceinline__ void fill_ghost_densities(float *R, int tid, int x0, int y0, int nx, int ny)
{
    constexpr int NV = H + 2 * RING, NH = W + 2 * RING;
    for (int c = tid; c < 2 * NV + 2 * NH; c += THREADS) {
        int x, y;  // tile position of the cell
        if (c < 2 * NV) {
            x = (c < NV ? -1 : nx) - x0;
            y = (c < NV ? c : c - NV) - RING;
        } else {
            const int d = c - 2 * NV;
            x = (d < NH ? d : d - NH) - RING;
            y = (d < NH ? -1 : ny) - y0;
        }
        const int ax = x0 + x, ay = y0 + y;
        if ((x < -RING) | (x >= W + RING) | (y < -RING) | (y >= H + RING) | (ax < -1) | (ax > nx) | (ay < -1) | (ay > ny))
            continue;
        R[y * RW + x] = R[(min(max(ay, 0), ny - 1) - y0) * RW + min(max(ax, 0), nx - 1) - x0];
    }
}

template <typename S>
struct Scalar;
template <>
struct Scalar<float> {
    static __device__ __forceinline__ void store(float *p, float v) { *p = v; }
};
template <>
struct Scalar<__half> {
    static __device__ __forceinline__ void store(__half *p, float v) { *p = __float2half_rn(v); }
};

}  // namespace prc
