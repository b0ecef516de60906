// prc_step2.cuh -- two fused time steps per launch (cavities, FP32 collision).
//
// A single step moves every population through memory once (72 B per node for
// FP32 storage), and at that traffic the interior kernel (prc_tma.cuh) runs at
// the memory's copy rate.  This kernel advances two steps per pass: a CTA stages
// the source windows of a W x H tile plus a ring of three nodes, makes the first
// step on the tile plus a ring of two, in place in shared memory, and the second
// on the tile, which it stores.  Memory sees half the traffic per step; the price
// is that the first step is repeated on the ring ((W + 4)(H + 4) / W H nodes).
//
// Bound by the SM: with the copies taken out a launch ran 12 % faster, no more.
// The FP32 pipe is 46 % busy and the shared-memory pipe 45 %, in phases that the
// barriers keep apart.  What that decided:
//   * a pair is two nodes of one column, not of one row: neighbouring lanes then
//     read neighbouring words, where pairs along the row hit every bank twice in
//     the planes of e_x != 0 (shared-memory wavefronts 6840 -> 4680 a tile);
//   * the first step works in place: the pulled values stay in registers across
//     the density barrier, which leaves room for two stages of 64 x 32 tiles;
//   * pairs are dealt to the threads in rounds of whole warps, and the warps
//     without a pair in the last round form the ring's densities;
//   * walls are handled by ghost cells only (populations, lid term, densities):
//     per-lane wall branches around the values held in registers spilled.
// 8192 x 2048 nodes, FP32, us per step: 191.7 (single steps) -> 139.9; 2432 x 1024:
// 30.4 -> 24.2; 1023 x 511: 10.2 -> 7.9; 304 x 256: 6.8 -> 4.0.
//
// Every node goes through the operations of the other kernels in the same order
// (pulls, density sum, gradient stencil, collision, the rounding of the stored
// populations between the two steps included), so the populations are bitwise
// those of two single steps.
//
// Tiles cover the whole grid: wall tiles take windows one row taller on either
// side and stream by ghost cells (prc_wall.cuh), once per step.
#pragma once

#include "prc_wall.cuh"

namespace prc {

// Tiling of the grid: tile (tx, ty) starts at (min(tx W, xlast), min(ty H, ylast)).
// xlast is aligned for the TMA copies; lanes past the grid store nothing.  The
// nodes that a shifted tile shares with its neighbour are stored twice with the
// same values; the owner (the tile they nominally belong to) adds the sums.
struct Tiling2 {
    int ntx, nty, xlast, ylast;
};

template <typename S, int W_, int H_, int THREADS_, int STAGES_>
struct Step2Cfg {
    static constexpr int W = W_, H = H_, THREADS = THREADS_, STAGES = STAGES_;
    static constexpr int PADX = 16 / (int)sizeof(S);  // 16-byte aligned window start, at least 4
    static constexpr int BW = W + 2 * PADX;           // window width
    static constexpr int BH = H + 6, BHW = H + 8;     // window rows: interior and wall tiles
    static constexpr int BOX_BYTES = BW * BH * (int)sizeof(S), BOXW_BYTES = BW * BHW * (int)sizeof(S);
    static constexpr int PLANE_BYTES = (BOXW_BYTES + 127) / 128 * 128;
    static constexpr int STAGE_BYTES = 9 * PLANE_BYTES;
    static constexpr int R_BYTES = (BW * BH * 4 + 127) / 128 * 128;  // density tile: a node at the place of its pulls
    static constexpr int SMEM = STAGES * STAGE_BYTES + 2 * R_BYTES + 128 + 128;  // + barriers, + base alignment
    // row pairs of the first step (tile and a ring of two) and of the second, dealt
    // to the threads in rounds; the last round of each may take only some warps
    static constexpr int N1 = (W + 4) * (H + 4) / 2, NQ1 = (N1 + THREADS - 1) / THREADS;
    static constexpr int N2 = W * H / 2, NQ2 = (N2 + THREADS - 1) / THREADS;
    // the ring's densities go to the warps that have no pair in the last round
    static constexpr int L1 = (N1 - (NQ1 - 1) * THREADS + 31) / 32 * 32, L2 = (N2 - (NQ2 - 1) * THREADS + 31) / 32 * 32;
    static constexpr int FIRST1 = THREADS - L1 >= 64 ? L1 : 0, FIRST2 = THREADS - L2 >= 64 ? L2 : 0;
};

// A node pair: one column, rows y and y + 1 in the two lanes,
// so that a warp's shared-memory accesses are consecutive words (a pair of
// neighbouring columns would make every access to a plane of e_x != 0 hit each
// bank twice).  The nine pulls of the pair whose first node pulls from p.
template <typename S, int PE, int BW>
__device__ __forceinline__ void pull_column(const S *p, F2 g[9])
{
#pragma unroll
    for (int i = 0; i < 9; i++)
        g[i] = F2(Pair<S>::one(p + i * PE - ex_of(i)), Pair<S>::one(p + i * PE - ex_of(i) + BW));
}

// Densities of the ring around the region of the tile extended by E nodes, one
// node at a time (units u = first, first + stride, ...).  LIDP: the moving-lid term
// goes to the pulls of the nodes in tile row `top`.
template <typename S, int W, int H, int E, int PE, int BW, int PADX, bool LIDP = false>
__device__ __forceinline__ void ring_nodes(int first, int stride, const S *cw, float *R, int top = 0, float lid = 0.f)
{
    constexpr int RX = W + 2 * E, N = 2 * RX + 2 * (H + 2 * E + 2);
    for (int u = first; u < N; u += stride) {
        int rx, ry;
        if (u < 2 * RX) {
            ry = u < RX ? -E - 1 : H + E;
            rx = -E + (u < RX ? u : u - RX);
        } else {
            const int c = u - 2 * RX;
            ry = -E - 1 + (c >> 1);
            rx = (c & 1) ? W + E : -E - 1;
        }
        const int o = (ry + 3) * BW + rx + PADX;
        float gr[9];
#pragma unroll
        for (int i = 0; i < 9; i++) gr[i] = Pair<S>::one(cw + o + i * PE - ex_of(i));
        if constexpr (LIDP) {
            if (ry == top) lid_pull(gr, lid);
        }
        R[o] = sum9(gr);
    }
}

// Density gradients of a pair whose first node's density is at c.  A row's
// difference E - W serves the stencils of both nodes; the values are those of
// drho_stencil, operation by operation.
template <int RW>
__device__ __forceinline__ void column_gradients(const float *c, F2 i12, F2 i12r, F2 &dxr, F2 &dyr)
{
    const F2 w = F2(c[-RW - 1], c[-1]), e = F2(c[-RW + 1], c[1]), m = F2(c[-RW], c[0]);
    const F2 w2 = F2(c[RW - 1], c[2 * RW - 1]), e2 = F2(c[RW + 1], c[2 * RW + 1]), m2 = F2(c[RW], c[2 * RW]);
    const F2 d = vsub(e, w), d2 = vsub(e2, w2);
    dxr = vmul(vadd(vfma(F2(4.f), F2(d.v.y, d2.v.x), d2), d), i12);
    dyr = vmul(vadd(vfma(F2(4.f), vsub(m2, m), vsub(e2, e)), vsub(w2, w)), i12r);
}

// Barriers per tile: the first step's densities are complete (A; also the vote
// on the bounded waits), the first step's populations are complete (B), the
// second step's densities are complete and the stage is free (C; the producer
// refills it).  Two density tiles, one per step: each is rewritten two barriers
// after its last read.
template <typename S, int W, int H, int THREADS, int MINB, int STAGES, bool EPI>
__global__ void __launch_bounds__(THREADS, MINB)
k_step2_tma(const __grid_constant__ CUtensorMap tin, const __grid_constant__ CUtensorMap twall, S *__restrict__ dst,
            Grid gd, Coef<F2> k, Coef<float> kf, float *__restrict__ snap, double2 *__restrict__ partials,
            DevStatus *__restrict__ st, Tiling2 tl, int rev)
{
    using C = Step2Cfg<S, W, H, THREADS, STAGES>;
    static_assert(C::PADX >= 4, "windows hold the ring of three nodes and its pulls");
    static_assert(H % 2 == 0, "whole row pairs");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    float *Ra = reinterpret_cast<float *>(smem + STAGES * C::STAGE_BYTES);
    float *Rb = reinterpret_cast<float *>(smem + STAGES * C::STAGE_BYTES + C::R_BYTES);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + STAGES * C::STAGE_BYTES + 2 * C::R_BYTES);
    constexpr int PE = C::PLANE_BYTES / (int)sizeof(S), BW = C::BW, PADX = C::PADX;
    const int tid = threadIdx.x;
    const bool producer = tid == THREADS - 32;
    const int nx = gd.nx, ny = gd.ny, ntiles = tl.ntx * tl.nty;
    if (tid == 0) {
        for (int b = 0; b < STAGES; b++) mbar_init(&bar[b], 1);
        mbar_fence_init();
    }
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    if (st->stop) return;

    // Position q of the tile order.  Every row of tiles starts one column further
    // on, so that a CTA's tiles (strided by the grid size) are not all in one
    // column: wall tiles cost more, and where the row length divides the stride
    // the CTAs of the outer columns would have nothing else.
    auto origin = [&](int q, int &ox, int &oy) {
        const int tile = rev ? ntiles - 1 - q : q;
        const int ty = tile / tl.ntx;
        int tx = tile - ty * tl.ntx + ty % tl.ntx;
        if (tx >= tl.ntx) tx -= tl.ntx;
        ox = tx * W;
        oy = ty * H;
    };
    // every node of the tile and of its ring of three at least one node inside the walls
    auto is_wall = [&](int x0, int y0) { return !((x0 >= 4) & (x0 + W + 4 <= nx) & (y0 >= 4) & (y0 + H + 4 <= ny)); };
    auto issue = [&](int q, int s) {
        int ox, oy;
        origin(q, ox, oy);
        const int x0 = min(ox, tl.xlast), y0 = min(oy, tl.ylast);
        const int wall = is_wall(x0, y0);
        S *stg = reinterpret_cast<S *>(smem + s * C::STAGE_BYTES);
        mbar_arrive_expect_tx(&bar[s], 9u * (wall ? C::BOXW_BYTES : C::BOX_BYTES));
        const CUtensorMap *map = wall ? &twall : &tin;
#pragma unroll
        for (int i = 0; i < 9; i++) tma_load_3d(stg + i * PE, map, &bar[s], x0 - PADX, y0 - 3 - wall - ey_of(i), i);
    };

    RedAcc<float> acc;
    if (producer)
        for (int s = 0; s < STAGES; s++)
            if ((int)blockIdx.x + s * (int)gridDim.x < ntiles) issue(blockIdx.x + s * gridDim.x, s);
    const float lid = gd.lid_on ? kf.lid : 0.f;
    const F2 i12(kf.inv12), i12r(kf.inv12r);
    // this thread's pairs: window (and density tile) offset of the first node's pulls
    int o1[C::NQ1], o2[C::NQ2];
#pragma unroll
    for (int j = 0; j < C::NQ1; j++) {
        const int p = tid + j * THREADS, y = p / (W + 4);
        o1[j] = (2 * y + 1) * BW + p - y * (W + 4) - 2 + PADX;
    }
#pragma unroll
    for (int j = 0; j < C::NQ2; j++) {
        const int p = tid + j * THREADS, y = p / W;
        o2[j] = (2 * y + 3) * BW + p - y * W + PADX;
    }
    auto has1 = [&](int j) { return j + 1 < C::NQ1 || C::N1 % THREADS == 0 || tid + j * THREADS < C::N1; };
    auto has2 = [&](int j) { return j + 1 < C::NQ2 || C::N2 % THREADS == 0 || tid + j * THREADS < C::N2; };
    int it = 0;
    for (int q = blockIdx.x; q < ntiles; it++, q += gridDim.x) {
        const int s = it % STAGES;
        int ox, oy;
        origin(q, ox, oy);
        const int x0 = min(ox, tl.xlast), y0 = min(oy, tl.ylast);
        const bool wall = is_wall(x0, y0);
        S *cw = reinterpret_cast<S *>(smem + s * C::STAGE_BYTES) + (wall ? BW : 0);
        // residual steps: the snapshot is streamed, its loads issued ahead of their use
        float2 snv[C::NQ2];
        if constexpr (EPI) {
#pragma unroll
            for (int j = 0; j < C::NQ2; j++) {
                const int p = tid + j * THREADS, y = p / W;
                const int ax = x0 + p - y * W, ay = y0 + 2 * y;
                const float *sp = snap + (long long)ay * gd.pitch + ax;
                snv[j] = make_float2(0.f, 0.f);
                if (has2(j) & (ax < nx) & (ay < ny)) snv[j].x = __ldcs(sp);
                if (has2(j) & (ax < nx) & (ay + 1 < ny)) snv[j].y = __ldcs(sp + gd.pitch);
            }
        }
        const bool ok = mbar_wait_bounded(&bar[s], (it / STAGES) & 1);

        // ---- first step, on the tile and a ring of two
        if (wall) {
            fill_ghosts<S, W, H, 3, 3, PE, BW, PADX, THREADS, true>(cw, tid, x0, y0, nx, ny, lid);
            __syncthreads();
        }
        {
            F2 g[C::NQ1][9];
#pragma unroll
            for (int j = 0; j < C::NQ1; j++)
                if (has1(j)) {
                    pull_column<S, PE, BW>(cw + o1[j], g[j]);
                    const F2 r = sum9(g[j]);
                    Ra[o1[j]] = r.v.x;
                    Ra[o1[j] + BW] = r.v.y;
                }
            if (tid >= C::FIRST1) ring_nodes<S, W, H, 2, PE, BW, PADX>(tid - C::FIRST1, THREADS - C::FIRST1, cw, Ra);
            if (__syncthreads_or(!ok)) {  // A
                if (producer) {
                    atomicExch(&st->timeout, 1);
                    atomicExch(&st->stop, 1);
                    // the copies of the following tiles may be outstanding
                    for (int d = 1; d < STAGES; d++)
                        if (q + d * (int)gridDim.x < ntiles)
                            mbar_wait_bounded(&bar[(it + d) % STAGES], ((it + d) / STAGES) & 1);
                }
                return;
            }
            if (wall) {
                fill_ghost_densities<W, H, 3, BW, THREADS>(Ra + 3 * BW + PADX, tid, x0, y0, nx, ny);
                __syncthreads();
            }
#pragma unroll
            for (int j = 0; j < C::NQ1; j++)
                if (has1(j)) {
                    F2 dxr, dyr, ux, uy, drho;
                    column_gradients<BW>(Ra + o1[j], i12, i12r, dxr, dyr);
                    collide<F2, true, false>(k, g[j], dxr, dyr, ux, uy, drho);
                    S *m = cw + o1[j];
#pragma unroll
                    for (int i = 0; i < 9; i++) {
                        Scalar<S>::store(m + i * PE + ey_of(i) * BW, g[j][i].v.x);
                        Scalar<S>::store(m + i * PE + (ey_of(i) + 1) * BW, g[j][i].v.y);
                    }
                }
        }
        fence_async_shared();  // these writes come before the next copies into the stage
        __syncthreads();       // B
        // ---- second step, on the tile
        if (wall) {
            fill_ghosts<S, W, H, 1, 3, PE, BW, PADX, THREADS, true>(cw, tid, x0, y0, nx, ny, lid);
            __syncthreads();
        }
        F2 g[C::NQ2][9];
#pragma unroll
        for (int j = 0; j < C::NQ2; j++)
            if (has2(j)) {
                pull_column<S, PE, BW>(cw + o2[j], g[j]);
                const F2 r = sum9(g[j]);
                Rb[o2[j]] = r.v.x;
                Rb[o2[j] + BW] = r.v.y;
            }
        if (tid >= C::FIRST2) ring_nodes<S, W, H, 0, PE, BW, PADX>(tid - C::FIRST2, THREADS - C::FIRST2, cw, Rb);
        __syncthreads();  // C
        if (producer && q + STAGES * (int)gridDim.x < ntiles) issue(q + STAGES * gridDim.x, s);
        if (wall) {
            fill_ghost_densities<W, H, 1, BW, THREADS>(Rb + 3 * BW + PADX, tid, x0, y0, nx, ny);
            __syncthreads();
        }
#pragma unroll
        for (int j = 0; j < C::NQ2; j++)
            if (has2(j)) {
                const int p = tid + j * THREADS, y = p / W;
                const int ax = x0 + p - y * W, ay = y0 + 2 * y;
                F2 dxr, dyr, ux, uy, drho;
                column_gradients<BW>(Rb + o2[j], i12, i12r, dxr, dyr);
                collide<F2, true, false>(k, g[j], dxr, dyr, ux, uy, drho);
                const long long o = (long long)ay * gd.pitch + ax;
                const bool v0 = !wall || ((ax < nx) & (ay < ny)), v1 = !wall || ((ax < nx) & (ay + 1 < ny));
                S *d = dst + o;
#pragma unroll
                for (int i = 0; i < 9; i++, d += gd.plane) {
                    if (v0) Scalar<S>::store(d, g[j][i].v.x);
                    if (v1) Scalar<S>::store(d + gd.pitch, g[j][i].v.y);
                }
                if constexpr (EPI) {
                    if (v0 & (ax >= ox) & (ay >= oy)) {
                        const float da = ux.v.x - snv[j].x;
                        __stcs(snap + o, ux.v.x);
                        acc.add(da * da, drho.v.x);
                    }
                    if (v1 & (ax >= ox) & (ay + 1 >= oy)) {
                        const float db = ux.v.y - snv[j].y;
                        __stcs(snap + o + gd.pitch, ux.v.y);
                        acc.add(db * db, drho.v.y);
                    }
                }
            }
    }
    if constexpr (EPI) {
        __shared__ double red[2 * (THREADS / 32)];
        double a, b;
        acc.block_total(a, b, red);
        if (tid == 0) partials[blockIdx.x] = make_double2(a, b);
    }
}

}  // namespace prc
