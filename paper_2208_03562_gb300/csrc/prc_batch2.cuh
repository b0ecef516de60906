// prc_batch2.cuh -- the batch engine with two fused time steps per pass.
//
// Same contract as k_batch_tma (prc_batch_tma.cuh): one cooperative persistent
// launch, a bounded grid barrier and the instances' bookkeeping after every pass;
// a pass advances every active instance by two steps, tile by tile as k_step2_tma
// does (prc_step2.cuh: windows of the tile and a ring of three nodes, the first
// step in place on the tile and a ring of two, the second on the tile).  Tiles of
// 64 x 24 nodes start at (64 tx, 24 ty), the last column and row reaching past the
// grid.  Compared with k_batch_tma a pass has half the memory traffic and half the
// grid barriers per step, and a fourth of the tile barriers per node.
//
// The host takes it when no active instance can leave within a pair of steps: even
// step counts, an even number of steps, and no step limit an odd number of steps
// away.  Residual steps (multiples of 20) are then second steps.  A pass changes an
// instance's set once, so the host flips the set of an instance whose steps made an
// odd number of passes.
//
// Results do not depend on which body ran: the populations are bitwise those of
// single steps, and the residual's terms are added up as in the 64 x 8 tiles of the
// other two bodies (row by row of 64 nodes, pair by pair, eight rows to a partial
// sum).
//
// What decided the form: registers.  The coefficients, a kernel parameter of the
// single-handle kernel, are read from shared memory here and need registers of their
// own; 512 threads of 128 spilled (about 60 words a thread; the local memory does not
// fit the rest of the L1, and a tile took 9.7 us against k_step2_tma's 5.2).  Hence
// 384 threads of up to 168, and 24 rows: three and two whole rounds of pairs.
//
// Bound by latency: twelve warps meet at three barriers a tile (a third of their time
// is waiting there, the issue slots are 35 % busy).  us per step, k_batch_tma -> here:
// one 4096 x 4096 slot FP32 220 -> 191, FP16 210 -> 193; 24 slots of 768 x 320 87.8 ->
// 78.1 and 83.9 -> 78.5; 228 of 128 x 64 50.1 -> 35.5 and 47.5 -> 33.4; 8 of 96 x 80
// 9.2 -> 6.7 and 8.9 -> 6.7.
#pragma once

#include "prc_batch_tma.cuh"
#include "prc_step2.cuh"

namespace prc {

constexpr int BT2_MAX_INST = 256;  // instances of a launch of k_batch2_tma at most
constexpr int BT2_W = 64, BT2_H = 24, BT2_THREADS = 384, BT2_STAGES = 2;

// A tile of a launch's list: instance, 2 slot + set of the state at t0, x origin (a
// multiple of 64) + 1 for a wall tile, y origin.
using Batch2Tile = int4;

// The tile list: every instance's tiles, row by row, in instance order.
static __global__ void k_batch2_tiles(const BatchInst *__restrict__ inst, Batch2Tile *__restrict__ list)
{
    const BatchInst &I = inst[blockIdx.x];
    const int nx = I.gd.nx, ny = I.gd.ny, ntx = (nx + BT2_W - 1) / BT2_W, n = ntx * ((ny + BT2_H - 1) / BT2_H);
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
        const int ty = q / ntx, x0 = (q - ty * ntx) * BT2_W, y0 = ty * BT2_H;
        // every node of the tile and of its ring of three at least one node inside the walls
        const bool in = (x0 >= 4) & (x0 + BT2_W + 4 <= nx) & (y0 >= 4) & (y0 + BT2_H + 4 <= ny);
        list[I.tile2_start + q] = make_int4(blockIdx.x, 2 * I.slot + (int)((I.t0 + I.flip) & 1), x0 | !in, y0);
    }
}

// The producer's place in the tile order (in shared memory, for want of registers).
struct alignas(16) Batch2Walk {
    Batch2Tile next;   // on its way from the list
    int sought;        // whether there is one
    int nstatic, ns;   // static tiles taken, to take
    unsigned base;     // first claim number of this pass
};

template <typename S>
struct Batch2Cfg : Step2Cfg<S, BT2_W, BT2_H, BT2_THREADS, BT2_STAGES> {
    using Base = Step2Cfg<S, BT2_W, BT2_H, BT2_THREADS, BT2_STAGES>;
    static constexpr int NBUF = BT2_STAGES + 1;  // records, table entries and coefficients: a tile's and those of the tiles in flight
    static constexpr int CB = ((int)sizeof(Coef<F2>) + 15) / 16 * 16, IB = (int)sizeof(BatchInst);
    // after the base's stages, density tiles and barriers: coefficients, table entries, active bits, records
    // and walk
    static constexpr int OFF_COEF = BT2_STAGES * Base::STAGE_BYTES + 2 * Base::R_BYTES + 128;
    static constexpr int OFF_INST = OFF_COEF + NBUF * CB;
    static constexpr int OFF_BITS = OFF_INST + NBUF * IB;
    static constexpr int OFF_REC = OFF_BITS + BT2_MAX_INST / 8;  // 16-byte aligned
    static constexpr int OFF_WALK = (OFF_REC + NBUF * (int)sizeof(Batch2Tile) + 15) / 16 * 16;
    // residual passes: u_x and drho of the tile's nodes, and the totals of its rows
    static constexpr int OFF_RES = (OFF_WALK + (int)sizeof(Batch2Walk) + 15) / 16 * 16;
    static constexpr int SMEM = OFF_RES + 2 * BT2_W * BT2_H * 4 + 2 * BT2_H * 8 + 128;  // + base alignment
    static_assert(BT2_THREADS >= 12 * 32, "eleven warps to issue copies, one to announce them");
    static_assert(OFF_REC % 16 == 0 && OFF_WALK % 16 == 0 && IB % 16 == 0 && OFF_COEF % 16 == 0 && sizeof(BatchCoef<float>) % 16 == 0, "16-byte bulk copies");
    static_assert(SMEM + 256 <= 227 * 1024, "a CTA's shared memory, static variables included");
};

// 16 bytes from global to shared memory without a register in between; the wait is
// for all copies of this thread.
__device__ __forceinline__ void copy_async16(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The moving-lid term of the pulls of a column pair whose first node lies in row y:
// to the lanes in the top row, as lid_pull adds it, and bitwise nothing to the
// others.
__device__ __forceinline__ void lid_pull_column(F2 g[9], int y, int top, float lid)
{
    const bool a = y == top, b = y + 1 == top;
    g[7] = F2(__fsub_rn(g[7].v.x, a ? lid : 0.f), __fsub_rn(g[7].v.y, b ? lid : 0.f));
    g[8] = F2(__fadd_rn(g[8].v.x, a ? lid : -0.f), __fadd_rn(g[8].v.y, b ? lid : -0.f));
}

template <typename S>
__global__ void __launch_bounds__(BT2_THREADS, 1)
k_batch2_tma(const BatchInst *__restrict__ inst, const BatchCoef<float> *__restrict__ coefs,
             const CUtensorMap *__restrict__ tmaps, const Batch2Tile *__restrict__ list, BatchDyn *dyn, int ninst,
             int total_tiles, double2 *partials, BatchCtl *ctl, int passes)
{
    using C = Batch2Cfg<S>;
    constexpr int W = BT2_W, H = BT2_H, THREADS = BT2_THREADS, STAGES = BT2_STAGES, NBUF = C::NBUF;
    constexpr int PE = C::PLANE_BYTES / (int)sizeof(S), BW = C::BW, PADX = C::PADX;
    constexpr bool LIDG = std::is_same<S, float>::value;  // lid term in the ghost cells, else after the pull
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    float *Ra = reinterpret_cast<float *>(smem + STAGES * C::STAGE_BYTES);
    float *Rb = reinterpret_cast<float *>(smem + STAGES * C::STAGE_BYTES + C::R_BYTES);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + STAGES * C::STAGE_BYTES + 2 * C::R_BYTES);
    const BatchInst *ibuf = reinterpret_cast<const BatchInst *>(smem + C::OFF_INST);
    unsigned *bits = reinterpret_cast<unsigned *>(smem + C::OFF_BITS);
    Batch2Tile *rec = reinterpret_cast<Batch2Tile *>(smem + C::OFF_REC);
    Batch2Walk &wk = *reinterpret_cast<Batch2Walk *>(smem + C::OFF_WALK);
    const int tid = threadIdx.x;
    const bool producer = tid == THREADS - 32;
    if (tid == 0) {
        for (int b = 0; b < STAGES; b++) mbar_init(&bar[b], 1);
        mbar_fence_init();
    }
    __syncthreads();
    uint32_t ph = 0;  // bit b: parity of the next completion of bar[b]

    // Tile assignment as in k_batch_tma: static tiles first, then claims.  The
    // producer finds its next tile and requests its list entry (seek) at the start of
    // a tile, and completes the record (take) before barrier C; after it, one lane of
    // every warp issues its share of the tile's copies.
    unsigned kp = 0;  // the claim in flight
    auto seek = [&]() {
        const int G = gridDim.x;
        int k = wk.nstatic;
        long long q;
        if (k < wk.ns) {
            q = blockIdx.x + (long long)k * G;
            wk.nstatic = k + 1;
        } else {
            q = (long long)wk.ns * G + (kp - wk.base);
            if (q < total_tiles) kp = (unsigned)atomicAdd(&ctl->claim, 1ULL);
        }
        wk.sought = q < total_tiles;
        if (q < total_tiles) copy_async16(&wk.next, list + q);
    };
    auto take = [&](int p, Batch2Tile &r) {
        for (;;) {
            Batch2Tile t = make_int4(-1, 0, 0, 0);
            if (wk.sought) {
                copy_async_wait();
                t = wk.next;
                if (!((bits[t.x >> 5] >> (t.x & 31)) & 1u)) {  // retired
                    seek();
                    continue;
                }
                t.y ^= p & 1;
            }
            r = t;
            return;
        }
    };
    // lane 0 of warp w: plane w of the windows, the coefficients, the table entry
    auto issue = [&](const Batch2Tile &r, int s, int cb) {
        const int w = tid >> 5;
        if ((tid & 31) != 0 || r.x < 0) return;
        const int slot = r.y >> 1, wall = r.z & 1;
        if (w < 9) {
            const CUtensorMap *map = tmaps + 8 * slot + 4 + 2 * wall + (r.y & 1);
            tma_load_3d(reinterpret_cast<S *>(smem + s * C::STAGE_BYTES) + w * PE, map, &bar[s], (r.z & ~1) - PADX,
                        r.w - 3 - wall - ey_of(w), w);
        } else if (w == 9) {
            bulk_load(smem + C::OFF_COEF + cb * C::CB, &coefs[slot].k2, C::CB, &bar[s]);
        } else if (w == 10) {
            bulk_load(smem + C::OFF_INST + cb * C::IB, inst + r.x, C::IB, &bar[s]);
        } else if (w == THREADS / 32 - 1) {
            mbar_arrive_expect_tx(&bar[s], 9u * (wall ? C::BOXW_BYTES : C::BOX_BYTES) + C::CB + C::IB);
        }
    };

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

    for (int p = 0; p < passes; p++) {
        // one activity decision per instance and pass for the whole CTA
        for (int k = tid; k < BT2_MAX_INST; k += THREADS) {
            bool on = false;
            if (k < ninst) on = ld_relaxed_i32(&dyn[inst[k].slot].state) == BATCH_ACTIVE && inst[k].t0 + 2 * p < inst[k].max_steps;
            const unsigned m = __ballot_sync(0xffffffffu, on);
            if ((k & 31) == 0) bits[k >> 5] = m;
        }
        __syncthreads();
        if ((tid & 31) == 0) fence_proxy_async_global();  // the copies read what the last pass wrote
        if (producer) {
            const int G = gridDim.x, ns = max(3, total_tiles / G - max(2, total_tiles / (8 * G)));
            const unsigned claims = total_tiles > (long long)ns * G ? total_tiles - ns * G : 0;
            kp = (unsigned)atomicAdd(&ctl->claim, 1ULL);  // taken after the static tiles
            wk.nstatic = 0;
            wk.ns = ns;
            wk.base = (unsigned)p * (claims + G);
            for (int b = 0; b < STAGES; b++) {
                seek();
                take(p, rec[b]);
            }
        }
        __syncthreads();
        for (int b = 0; b < STAGES; b++) issue(rec[b], b, b);
        for (int it = 0;; it++) {
            const int s = it % STAGES, c = it % NBUF;
            const Batch2Tile &r = rec[c];
            if (r.x < 0) break;  // no later record holds a tile either
            const bool wall = r.z & 1;
            const int x0 = r.z & ~1, y0 = r.w;
            // copied in with the windows
            const BatchInst &I = ibuf[c];
            const Coef<F2> &K = *reinterpret_cast<const Coef<F2> *>(smem + C::OFF_COEF + c * C::CB);
            if (producer) seek();
            S *cw = reinterpret_cast<S *>(smem + s * C::STAGE_BYTES) + (wall ? BW : 0);
            const bool ok = mbar_wait_bounded(&bar[s], (ph >> s) & 1u);
            ph ^= 1u << s;
            const int &nx = I.gd.nx, &ny = I.gd.ny;
            const float lid = I.gd.lid_on ? K.lid.v.x : 0.f;
            // the lid term after the pulls (FP16): tiles whose nodes or rings reach the top row
            const bool lidp = !LIDG && wall && I.gd.lid_on && ny - 1 < y0 + H + 3;

            // ---- first step, on the tile and a ring of two
            if (wall) {
                fill_ghosts<S, W, H, 3, 3, PE, BW, PADX, THREADS, LIDG>(cw, tid, x0, y0, nx, ny, lid);
                __syncthreads();
            }
            {
                F2 g[C::NQ1][9];
#pragma unroll
                for (int j = 0; j < C::NQ1; j++)
                    if (has1(j)) {
                        pull_column<S, PE, BW>(cw + o1[j], g[j]);
                        if (lidp) lid_pull_column(g[j], y0 + o1[j] / BW - 3, ny - 1, lid);
                        const F2 d = sum9(g[j]);
                        Ra[o1[j]] = d.v.x;
                        Ra[o1[j] + BW] = d.v.y;
                    }
                if (tid >= C::FIRST1)
                    ring_nodes<S, W, H, 2, PE, BW, PADX, !LIDG>(tid - C::FIRST1, THREADS - C::FIRST1, cw, Ra,
                                                               lidp ? ny - 1 - y0 : -100, lid);
                if (__syncthreads_or(!ok)) {  // A
                    if (producer) {
                        atomicExch(&ctl->error, 1);
                        copy_async_wait();
                        // the copies of the next tiles may be outstanding
                        for (int d = 1; d < STAGES; d++)
                            if (rec[(it + d) % NBUF].x >= 0)
                                mbar_wait_bounded(&bar[(it + d) % STAGES], (ph >> ((it + d) % STAGES)) & 1u);
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
                        column_gradients<BW>(Ra + o1[j], K.inv12, K.inv12r, dxr, dyr);
                        collide<F2, true, false>(K, g[j], dxr, dyr, ux, uy, drho);
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
                fill_ghosts<S, W, H, 1, 3, PE, BW, PADX, THREADS, LIDG>(cw, tid, x0, y0, nx, ny, lid);
                __syncthreads();
            }
            F2 g[C::NQ2][9];
#pragma unroll
            for (int j = 0; j < C::NQ2; j++) {
                if (!has2(j)) break;
                pull_column<S, PE, BW>(cw + o2[j], g[j]);
                if (lidp) lid_pull_column(g[j], y0 + o2[j] / BW - 3, ny - 1, lid);
                const F2 d = sum9(g[j]);
                Rb[o2[j]] = d.v.x;
                Rb[o2[j] + BW] = d.v.y;
            }
            if (tid >= C::FIRST2)
                ring_nodes<S, W, H, 0, PE, BW, PADX, !LIDG>(tid - C::FIRST2, THREADS - C::FIRST2, cw, Rb,
                                                           lidp ? ny - 1 - y0 : -100, lid);
            if (producer) take(p, rec[(it + STAGES) % NBUF]);
            __syncthreads();  // C
            issue(rec[(it + STAGES) % NBUF], s, (it + STAGES) % NBUF);
            if (wall) {
                fill_ghost_densities<W, H, 1, BW, THREADS>(Rb + 3 * BW + PADX, tid, x0, y0, nx, ny);
                __syncthreads();
            }
            const bool epi = (I.t0 + 2 * p + 2) % 20 == 0;
            const int pitch = I.gd.pitch;
            float *res_u = reinterpret_cast<float *>(smem + C::OFF_RES), *res_d = res_u + W * H;
#pragma unroll
            for (int j = 0; j < C::NQ2; j++) {
                if (!has2(j)) break;
                const int q = tid + j * THREADS, y = q / W;
                const int ax = x0 + q - y * W, ay = y0 + 2 * y;
                F2 dxr, dyr, ux, uy, drho;
                column_gradients<BW>(Rb + o2[j], K.inv12, K.inv12r, dxr, dyr);
                collide<F2, true, false>(K, g[j], dxr, dyr, ux, uy, drho);
                const bool v0 = !wall || ((ax < nx) & (ay < ny)), v1 = !wall || ((ax < nx) & (ay + 1 < ny));
                const long long o = (long long)ay * pitch + ax;
                S *d = static_cast<S *>(I.pop[(r.y & 1) ^ 1]) + o;
#pragma unroll
                for (int i = 0; i < 9; i++, d += I.gd.plane) {
                    if (v0) Scalar<S>::store(d, g[j][i].v.x);
                    if (v1) Scalar<S>::store(d + pitch, g[j][i].v.y);
                }
                if (epi) {  // uniform across the CTA
                    float *u = res_u + 2 * y * W + q - y * W, *e = u + W * H;
                    u[0] = ux.v.x;
                    u[W] = ux.v.y;
                    e[0] = drho.v.x;
                    e[W] = drho.v.y;
                }
            }
            if (epi) {
                // The terms of a row of 64 nodes by one warp, a pair to a lane, then
                // the sums of eight rows: a 64 x 8 tile's partial.
                double *red = reinterpret_cast<double *>(res_d + W * H);
                __syncthreads();
                for (int row = tid >> 5; row < H; row += THREADS / 32) {
                    const int x = 2 * (tid & 31), ax = x0 + x, ay = y0 + row;
                    const float2 u = *reinterpret_cast<const float2 *>(res_u + row * W + x);
                    const float2 e = *reinterpret_cast<const float2 *>(res_d + row * W + x);
                    float *sn = static_cast<float *>(I.snap) + (long long)ay * pitch + ax;
                    RedAcc<float> acc;
                    if ((ax + 1 < nx) & (ay < ny)) {
                        const float2 was = __ldcs(reinterpret_cast<const float2 *>(sn));
                        const float da = u.x - was.x, db = u.y - was.y;
                        __stcs(reinterpret_cast<float2 *>(sn), u);
                        acc.add(__fmul_rn(da, da), e.x);
                        acc.add(__fmul_rn(db, db), e.y);
                    } else if ((ax < nx) & (ay < ny)) {
                        const float da = u.x - __ldcs(sn);
                        __stcs(sn, u.x);
                        acc.add(__fmul_rn(da, da), e.x);
                    }
                    acc.warp_total();
                    if ((tid & 31) == 0) {
                        red[row] = (double)acc.ah + (double)acc.al;
                        red[H + row] = (double)acc.bh + (double)acc.bl;
                    }
                }
                __syncthreads();
                if (tid < H / BT_H && y0 + tid * BT_H < ny) {
                    double a = 0.0, b = 0.0;
                    for (int w = 0; w < BT_H; w++) {
                        a += red[tid * BT_H + w];
                        b += red[H + tid * BT_H + w];
                    }
                    partials[I.part_base + (y0 / BT_H + tid) * I.tiles_x + x0 / W] = make_double2(a, b);
                }
            }
        }
        if (!grid_barrier(ctl)) return;
        batch_bookkeeping<2>(inst, dyn, ninst, partials, tid, reinterpret_cast<double *>(Ra));
        // No second barrier, as in k_batch: an instance retired by its residual
        // may be advanced by one more pass, which is not a residual pass, reads the
        // instance's final set and writes only the other one.
        __syncthreads();  // the scratch is a density tile
    }
}

}  // namespace prc
