// prc_cluster.cuh -- cluster-resident engine for small grids.
//
// One thread-block cluster holds a whole instance in distributed shared
// memory for many time steps.  CTA c of the cluster owns the rows
// [c rpc, min((c + 1) rpc, ny)) ("slab"), both population sets of its slab
// and a density tile of the slab plus a one-node ring.  One time step:
//   1. density tile: rho - rho0 of every slab node and of the ring, each from
//      its nine pulled populations (App. A streaming; reading A1 for ghost
//      nodes); pulls of rows outside the slab read the neighbouring CTA's
//      shared memory through the cluster's distributed shared memory;
//   2. CTA barrier;
//   3. every slab node: pull, density gradient from the tile, collision
//      (the same `collide` as every other kernel, on pairs of neighbouring
//      nodes in packed FP32x2 arithmetic for the FP32 collision, as in the
//      general kernel, so the populations are bitwise those of the general
//      kernel), store into the other set;
//   4. cluster barrier: the new set is complete before anyone pulls from it.
// Every 20th step of the absolute step counter the CTAs add their FP64
// residual / mass totals in rank order (identically in every CTA, so the
// stop decision is uniform and no CTA waits on a barrier the others skip).
// The state is read from global memory at launch and written back at the end,
// so a launch of n steps costs one global read and write of the state instead
// of n; steps are separated by cluster barriers instead of kernel launches.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "prc_kernels.cuh"

namespace prc {

constexpr int CL_THREADS = 512;
constexpr int CL_MAX_CTAS = 16;

struct ClusterGeom {
    int nc;    // CTAs (slabs)
    int rpc;   // rows per slab (the last may be shorter, never below 2)
    int smem;  // dynamic shared memory per CTA (bytes)
};

// Shared-memory footprint of a slab of `rows` rows, nx wide.
__host__ __device__ inline size_t cluster_smem_bytes(int rows, int nx, size_t elem, size_t telem)
{
    const size_t f = 2 * 9 * (size_t)rows * nx * elem;
    const size_t fa = (f + 15) / 16 * 16;
    return fa + (size_t)(rows + 2) * (nx + 2) * telem;
}

// Whether a slab has at most two nodes per thread (k_cluster_pairs).
__host__ __device__ inline bool cluster_pairs_fit(int rpc, int nx) { return (long long)rpc * nx <= 2 * CL_THREADS; }

// Load of one stored population through a 32-bit shared::cluster address
// (this CTA's shared memory or another CTA's of the cluster), widened to the
// collision type.  Volatile: the loads must stay between the cluster
// barriers that order them against the neighbours' stores.
template <typename S, typename T>
__device__ __forceinline__ T ld_cl(uint32_t a);
template <>
__device__ __forceinline__ double ld_cl<double, double>(uint32_t a)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
    return v;
}
template <>
__device__ __forceinline__ float ld_cl<float, float>(uint32_t a)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
template <>
__device__ __forceinline__ float ld_cl<__half, float>(uint32_t a)
{
    unsigned short v;
    asm volatile("ld.shared::cluster.b16 %0, [%1];" : "=h"(v) : "r"(a));
    return __half2float(__ushort_as_half(v));
}

// The same from this CTA's own shared memory (shared::cta address).
template <typename S>
__device__ __forceinline__ float ld_cta(uint32_t a);
template <>
__device__ __forceinline__ float ld_cta<float>(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
template <>
__device__ __forceinline__ float ld_cta<__half>(uint32_t a)
{
    unsigned short v;
    asm volatile("ld.shared.b16 %0, [%1];" : "=h"(v) : "r"(a));
    return __half2float(__ushort_as_half(v));
}

// The two halves of a cluster barrier: arrive (releasing this thread's
// earlier writes) and wait for every CTA's arrival (acquiring theirs).  Work
// that needs none of the other CTAs' data can run between them.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// shared::cta address of a pointer into this CTA's shared memory
__device__ __forceinline__ uint32_t cta_smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// the same location in the shared memory of CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_addr(uint32_t cta_addr, int rank)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(cta_addr), "r"(rank));
    return a;
}

// Read access to one population set of the cluster in 32-bit shared::cluster
// addresses: this CTA's slab, the two neighbouring slabs (rows within two of
// the slab) and, across a periodic wrap, any slab.  Every CTA lays its set
// out the same way: plane i, local row ly, column x at i plane_b + ly row_b +
// x sizeof(S) from the set's base.
struct SlabView {
    uint32_t own, prev, next;  // base of the set in this CTA and in the neighbouring CTAs
    uint32_t own_cta;          // base of the set in this CTA's shared::cta window (mapa source on a wrap)
    int y_lo, y_hi, rpc, nc;
    uint32_t row_b, plane_b;   // bytes per row and per plane

    // address of plane 0, column 0 of the in-domain row y (any slab)
    __device__ __forceinline__ uint32_t row(int y) const
    {
        if (y >= y_lo && y < y_hi) return own + (uint32_t)(y - y_lo) * row_b;
        if (y < y_lo && y >= y_lo - 2) return prev + (uint32_t)(y - (y_lo - rpc)) * row_b;
        if (y >= y_hi && y < y_hi + 2) return next + (uint32_t)(y - y_hi) * row_b;
        const int owner = min(y / rpc, nc - 1);  // periodic wrap across the first / last slab
        return cluster_addr(own_cta, owner) + (uint32_t)(y - owner * rpc) * row_b;
    }
};

// Pull-streaming with half-way bounce-back and the lid (as pull9) through
// the slab view.  Nodes whose nine sources are all inside the domain (away
// from the x walls, and away from the y walls unless y is periodic) take the
// fast path: the three source rows are resolved once and the nine pulls are
// fixed offsets from them.
template <typename S, typename T>
__device__ __forceinline__ void pull9_slab(const SlabView &v, const Grid &gd, int x, int y, T lid, T g[9])
{
    constexpr uint32_t es = sizeof(S);
    const bool xin = (x >= 1) & (x <= gd.nx - 2);
    const bool yin = (gd.bc == 2) | ((y >= 1) & (y <= gd.ny - 2));
    if (xin & yin) {
        const int ym = y == 0 ? gd.ny - 1 : y - 1, yp = y == gd.ny - 1 ? 0 : y + 1;
        const uint32_t rr[3] = {v.row(ym), v.row(y), v.row(yp)};  // source row of e_y = +1, 0, -1
#pragma unroll
        for (int i = 0; i < 9; i++)
            g[i] = ld_cl<S, T>(rr[1 - ey_of(i)] + (uint32_t)i * v.plane_b + (uint32_t)(x - ex_of(i)) * es);
        return;
    }
    const uint32_t here = v.row(y) + (uint32_t)x * es;
#pragma unroll
    for (int i = 0; i < 9; i++) {
        int sx = x - ex_of(i), sy = y - ey_of(i);
        if (gd.bc >= 1) sx = sx < 0 ? sx + gd.nx : (sx >= gd.nx ? sx - gd.nx : sx);
        if (gd.bc == 2) sy = sy < 0 ? sy + gd.ny : (sy >= gd.ny ? sy - gd.ny : sy);
        const bool inside = (sx >= 0) & (sx < gd.nx) & (sy >= 0) & (sy < gd.ny);
        if (inside) {
            g[i] = ld_cl<S, T>(v.row(sy) + (uint32_t)i * v.plane_b + (uint32_t)sx * es);
        } else {
            T w = ld_cl<S, T>(here + (uint32_t)opp_of(i) * v.plane_b);
            if (sy >= gd.ny && gd.lid_on) {
                if (i == 7) w -= lid;
                if (i == 8) w += lid;
            }
            g[i] = w;
        }
    }
}

// The nine pulls of the node pair (x, x + 1) in FP32, one pair of source rows
// resolved for both nodes when all eighteen sources are inside the domain.
template <typename S>
__device__ __forceinline__ void pull_pair_slab(const SlabView &v, const Grid &gd, int x, int y, bool v1,
                                               float lid, float ga[9], float gb[9])
{
    constexpr uint32_t es = sizeof(S);
    const bool fast = (x >= 1) & (x + 2 <= gd.nx - 1) & ((gd.bc == 2) | ((y >= 1) & (y <= gd.ny - 2)));
    if (fast) {
        const int ym = y == 0 ? gd.ny - 1 : y - 1, yp = y == gd.ny - 1 ? 0 : y + 1;
        const uint32_t rr[3] = {v.row(ym), v.row(y), v.row(yp)};
#pragma unroll
        for (int i = 0; i < 9; i++) {
            const uint32_t a = rr[1 - ey_of(i)] + (uint32_t)i * v.plane_b + (uint32_t)(x - ex_of(i)) * es;
            ga[i] = ld_cl<S, float>(a);
            gb[i] = ld_cl<S, float>(a + es);
        }
        return;
    }
    pull9_slab<S, float>(v, gd, x, y, lid, ga);
    if (v1) pull9_slab<S, float>(v, gd, x + 1, y, lid, gb);
    else
#pragma unroll
        for (int i = 0; i < 9; i++) gb[i] = ga[i];
}

// n time steps of one instance on one cluster (gridDim.x == cluster size).
// pop_in holds the state after step t0; the state after the last step done
// goes to pop_out[parity of that step]; pop0 is the handle's set `flip`, and a step
// that diverges notes 1 + its set of the handle.
template <typename S, typename T, bool DRHO, bool FORCE, bool RAW>
__global__ void __launch_bounds__(CL_THREADS, 1)
k_cluster(const S *__restrict__ pop0, const S *__restrict__ pop1, Grid gd, Coef<T> k, Coef<F2> k2,
          T *__restrict__ snap, DevStatus *__restrict__ st, long long t0, int nsteps, int rpc,
          int *__restrict__ note, int flip)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char cl_smem[];
    __shared__ double2 part;      // this CTA's residual / mass totals
    __shared__ double red[2 * (CL_THREADS / 32)];
    __shared__ int sh_stop;

    if (st->stop) return;  // uniform: read before any write by this launch
    const int nc = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int nthr = blockDim.x, tid = threadIdx.x;
    const int nx = gd.nx;
    const int plane = rpc * nx;  // elements per plane of a slab (the same layout in every CTA)
    SlabView v;
    v.rpc = rpc;
    v.nc = nc;
    v.y_lo = rank * rpc;
    v.y_hi = min(v.y_lo + rpc, gd.ny);
    v.row_b = (uint32_t)nx * (uint32_t)sizeof(S);
    v.plane_b = (uint32_t)plane * (uint32_t)sizeof(S);
    const int rows = v.y_hi - v.y_lo;
    const size_t fbytes = (2 * 9 * (size_t)rpc * nx * sizeof(S) + 15) / 16 * 16;
    S *F0 = reinterpret_cast<S *>(cl_smem);
    S *F1 = F0 + 9 * plane;
    T *rho = reinterpret_cast<T *>(cl_smem + fbytes);
    const int prv = rank > 0 ? rank - 1 : nc - 1, nxt = rank + 1 < nc ? rank + 1 : 0;
    // 32-bit shared::cluster addresses of both sets in this CTA and its neighbours
    const uint32_t own0c = cta_smem_addr(F0), own1c = cta_smem_addr(F1);  // shared::cta window
    const uint32_t own0 = cluster_addr(own0c, rank), own1 = cluster_addr(own1c, rank);
    const uint32_t prev0 = cluster_addr(own0c, prv), prev1 = cluster_addr(own1c, prv);
    const uint32_t next0 = cluster_addr(own0c, nxt), next1 = cluster_addr(own1c, nxt);

    // load the slab of the current state
    const S *pin = (t0 & 1) ? pop1 : pop0;
    const int nslab = rows * nx;
    // this thread's nodes q = tid + k nthr of the slab (ly = q / nx, x = q % nx)
    // and of the density tile (q / RW, q % RW), advanced without divisions
    const int RW = nx + 2;
    const int s_dly = nthr / nx, s_dx = nthr - s_dly * nx;
    const int s_ly0 = tid / nx, s_x0 = tid - s_ly0 * nx;
    const int r_dly = nthr / RW, r_dx = nthr - r_dly * RW;
    const int r_ly0 = tid / RW, r_x0 = tid - r_ly0 * RW;
    for (int i = 0; i < 9; i++)
        for (int q = tid; q < nslab; q += nthr) {
            const int ly = q / nx, x = q - ly * nx;
            F0[i * plane + ly * nx + x] =
                pin[(long long)i * gd.plane + (long long)(v.y_lo + ly) * gd.pitch + x];
        }
    __syncthreads();
    cluster_arrive();  // matched by the wait at the top of the first step

    int b = 0;  // set holding the state
    int done = 0;
    bool waited = false;  // the last cluster barrier phase has been waited on
    const double nnodes = (double)gd.nx * (double)gd.ny;
    int t20 = (int)((t0 + 1) % 20);  // index of the step being made, modulo 20
    for (; done < nsteps; done++, t20 = t20 == 19 ? 0 : t20 + 1) {
        const long long t = t0 + done + 1;  // absolute index of the step being made
        const bool epi = t20 == 0;
        v.own = b ? own1 : own0;
        v.own_cta = b ? own1c : own0c;
        v.prev = b ? prev1 : prev0;
        v.next = b ? next1 : next0;
        S *Fo = b ? F0 : F1;
        // 1. density tile (slab + ring), one node at a time
        auto density_pass = [&]() {
            const int nr = (rows + 2) * RW;
            int ry = r_ly0, rx = r_x0;
            for (int q = tid; q < nr; q += nthr) {
                const int ly = ry - 1, lx = rx - 1;
                rx += r_dx;
                ry += r_dly;
                if (rx >= RW) {
                    rx -= RW;
                    ry++;
                }
                int gx = lx, gy = v.y_lo + ly;
                map_node(gd, gx, gy);
                T g[9];
                pull9_slab<S, T>(v, gd, gx, gy, k.lid, g);
                rho[q] = sum9(g);
            }
            __syncthreads();
        };
        RedAcc<T> acc;
        if constexpr (std::is_same<T, float>::value) {
            // FP32 collision: pairs of neighbouring nodes (x, x + 1), x even,
            // in packed FP32x2 arithmetic, as in the general kernel
            const int npx = (nx + 1) >> 1, npairs = rows * npx;
            // 2. collide one pair (pulled values in ga, gb) into the other set
            auto pair_body = [&](int ly, int x, const float *ga, const float *gb) {
                const int y = v.y_lo + ly;
                const bool v1 = x + 1 < nx;
                F2 g[9];
#pragma unroll
                for (int i = 0; i < 9; i++) g[i] = F2(ga[i], gb[i]);
                float dx[2] = {0.f, 0.f}, dy[2] = {0.f, 0.f};
                if constexpr (DRHO) {
#pragma unroll
                    for (int j = 0; j < 2; j++) {
                        const float *c = rho + (ly + 1) * RW + x + j + 1;
                        const float rE = c[1], rW = c[-1];
                        const float rN = c[RW], rS = c[-RW];
                        const float rNE = c[RW + 1], rNW = c[RW - 1];
                        const float rSE = c[-RW + 1], rSW = c[-RW - 1];
                        drho_stencil<float>(rE, rW, rN, rS, rNE, rNW, rSE, rSW, k.inv12, k.inv12r, dx[j], dy[j]);
                    }
                }
                F2 ux, uy, drho;
                collide<F2, DRHO, FORCE, RAW>(k2, g, F2(dx[0], dx[1]), F2(dy[0], dy[1]), ux, uy, drho);
                const int o = ly * nx + x;
#pragma unroll
                for (int i = 0; i < 9; i++) {
                    Fo[i * plane + o] = to_s<S, float>(g[i].v.x);
                    if (v1) Fo[i * plane + o + 1] = to_s<S, float>(g[i].v.y);
                }
                if (epi) {
                    const long long og = (long long)y * gd.pitch + x;
                    const float d0 = ux.v.x - snap[og];
                    snap[og] = ux.v.x;
                    acc.add(d0 * d0, drho.v.x);
                    if (v1) {
                        const float d1 = ux.v.y - snap[og + 1];
                        snap[og + 1] = ux.v.y;
                        acc.add(d1 * d1, drho.v.y);
                    }
                }
            };
            cluster_wait();
            if constexpr (DRHO) density_pass();
            const int p_dly = nthr / npx, p_dx = nthr - p_dly * npx;
            int py = tid / npx, pxi = tid - py * npx;
            for (int q = tid; q < npairs; q += nthr) {
                const int ly = py, x = 2 * pxi;
                pxi += p_dx;
                py += p_dly;
                if (pxi >= npx) {
                    pxi -= npx;
                    py++;
                }
                float ga[9], gb[9];
                pull_pair_slab<S>(v, gd, x, v.y_lo + ly, x + 1 < nx, k.lid, ga, gb);
                pair_body(ly, x, ga, gb);
            }
        } else {
            // FP64 collision: one node at a time
            cluster_wait();
            if constexpr (DRHO) density_pass();
            int sy_ = s_ly0, sx_ = s_x0;
            for (int q = tid; q < nslab; q += nthr) {
                const int ly = sy_, x = sx_;
                sx_ += s_dx;
                sy_ += s_dly;
                if (sx_ >= nx) {
                    sx_ -= nx;
                    sy_++;
                }
                const int y = v.y_lo + ly;
                T g[9];
                pull9_slab<S, T>(v, gd, x, y, k.lid, g);
                T dxr = T(0), dyr = T(0);
                if constexpr (DRHO) {
                    const T *c = rho + (ly + 1) * RW + x + 1;
                    const T rE = c[1], rW = c[-1];
                    const T rN = c[RW], rS = c[-RW];
                    const T rNE = c[RW + 1], rNW = c[RW - 1];
                    const T rSE = c[-RW + 1], rSW = c[-RW - 1];
                    drho_stencil<T>(rE, rW, rN, rS, rNE, rNW, rSE, rSW, k.inv12, k.inv12r, dxr, dyr);
                }
                T ux, uy, drho;
                collide<T, DRHO, FORCE, RAW>(k, g, dxr, dyr, ux, uy, drho);
                const int o = ly * nx + x;
#pragma unroll
                for (int i = 0; i < 9; i++) Fo[i * plane + o] = to_s<S, T>(g[i]);
                if (epi) {
                    const long long og = (long long)y * gd.pitch + x;
                    const T d = ux - snap[og];
                    snap[og] = ux;
                    acc.add(d * d, drho);
                }
            }
        }
        if (epi) {
            double a, bb;
            acc.block_total(a, bb, red);
            if (tid == 0) part = make_double2(a, bb);
        }
        // 3. the new set is complete (and every pull of the old one done):
        // this CTA's stores are visible to its own threads, then it arrives;
        // the next step waits for the others
        __syncthreads();
        cluster_arrive();
        b ^= 1;
        if (epi) {
            cluster_wait();  // every CTA's partial sums are written
            if (tid == 0) {
                double a = 0.0, m = 0.0;
                for (int r = 0; r < nc; r++) {  // rank order: the same sums in every CTA
                    const double2 p = *cl.map_shared_rank(&part, r);
                    a += p.x;
                    m += p.y;
                }
                const double res = sqrt(a), mass = nnodes + m;
                int stop = 0;
                if (!isfinite(res) || !isfinite(mass)) stop = 2;
                else if (res < st->tol) stop = 1;
                sh_stop = stop;
                if (rank == 0) {
                    st->res_step = t;
                    st->res = res;
                    st->mass = mass;
                    if (stop == 2) {
                        st->diverged = 1;
                        *note = 1 + (int)((t0 + done + 1 + flip) & 1);
                    }
                    if (stop == 1) st->converged = 1;
                    if (stop) st->stop = 1;
                }
            }
            __syncthreads();  // sh_stop is visible to every thread
            if (sh_stop) {  // the same decision in every CTA
                done++;
                waited = true;
                break;
            }
            cluster_arrive();  // matched by the wait at the top of the next step
        }
    }
    if (!waited) cluster_wait();  // every CTA is done with this CTA's shared memory
    // write the slab of the final state
    const long long tend = t0 + done;
    S *pout = const_cast<S *>((tend & 1) ? pop1 : pop0);
    for (int i = 0; i < 9; i++)
        for (int q = tid; q < nslab; q += nthr) {
            const int ly = q / nx, x = q - ly * nx;
            pout[(long long)i * gd.plane + (long long)(v.y_lo + ly) * gd.pitch + x] =
                (b ? F1 : F0)[i * plane + ly * nx + x];
        }
}

// ---- slabs of at most two nodes per thread (FP32 collision)
//
// Nodes q and q + npairs of a slab are thread q's pair for the whole launch, so
// everything that depends on a node's place is resolved once: the addresses of
// its nine pulls (the neighbouring slab, a periodic seam and the bounce-back of a
// wall are only other addresses), the addresses of its eight neighbour densities
// (clamped at a wall, wrapped at a seam: the density tile needs a ring of rows,
// not of columns) and its lid term.  A step then runs without a branch, where
// the guarded pulls of the wall nodes used to run in nearly every warp (915
// instructions a warp and step).  Lanes address consecutive words.  Bound by
// latency: pulls, CTA barrier, collision, cluster barrier.  us per step before
// and after: 128x128 FP32 5.45 -> 1.88, 100x125 FP16 6.97 -> 2.10, 64x64 FP32 1.28.

// The address of population i's source for node (x, y), relative to a set's
// base in this CTA; for a source in another CTA, in that CTA's shared memory.
__device__ __forceinline__ uint32_t pull_address(const SlabView &v, const Grid &gd, int x, int y, int i, uint32_t es,
                                                 bool &local)
{
    int sx = x - ex_of(i), sy = y - ey_of(i), p = i;
    if (gd.bc >= 1) sx = sx < 0 ? sx + gd.nx : (sx >= gd.nx ? sx - gd.nx : sx);
    if (gd.bc == 2) sy = sy < 0 ? sy + gd.ny : (sy >= gd.ny ? sy - gd.ny : sy);
    if ((sx < 0) | (sx >= gd.nx) | (sy < 0) | (sy >= gd.ny)) {
        sx = x;
        sy = y;
        p = opp_of(i);
    }
    local &= (sy >= v.y_lo) & (sy < v.y_hi);
    return v.row(sy) + (uint32_t)p * v.plane_b + (uint32_t)sx * es;
}

template <typename S, bool DRHO, bool FORCE, bool RAW>
__global__ void __launch_bounds__(CL_THREADS, 1)
k_cluster_pairs(const S *__restrict__ pop0, const S *__restrict__ pop1, Grid gd, Coef<float> k, Coef<F2> k2,
                float *__restrict__ snap, DevStatus *__restrict__ st, long long t0, int nsteps, int rpc,
                int *__restrict__ note, int flip)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char cl_smem[];
    __shared__ double2 part;  // this CTA's residual / mass totals
    __shared__ double red[2 * (CL_THREADS / 32)];
    __shared__ int sh_stop;

    if (st->stop) return;  // uniform: read before any write by this launch
    const int nc = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int tid = threadIdx.x, nx = gd.nx;
    constexpr uint32_t es = sizeof(S);
    const int plane = rpc * nx;  // elements per plane of a slab (the same layout in every CTA)
    const uint32_t set_b = 9u * (uint32_t)plane * es;  // bytes from set 0 to set 1, in every CTA
    S *F0 = reinterpret_cast<S *>(cl_smem);
    float *rho = reinterpret_cast<float *>(cl_smem + (2 * (size_t)set_b + 15) / 16 * 16);  // rows -1 .. rows, nx each
    SlabView v;
    v.rpc = rpc;
    v.nc = nc;
    v.y_lo = rank * rpc;
    v.y_hi = min(v.y_lo + rpc, gd.ny);
    v.row_b = (uint32_t)nx * es;
    v.plane_b = (uint32_t)plane * es;
    v.own_cta = cta_smem_addr(F0);
    v.own = cluster_addr(v.own_cta, rank);
    v.prev = cluster_addr(v.own_cta, rank > 0 ? rank - 1 : nc - 1);
    v.next = cluster_addr(v.own_cta, rank + 1 < nc ? rank + 1 : 0);
    const int rows = v.y_hi - v.y_lo, nslab = rows * nx, npairs = (nslab + 1) >> 1;

    const S *pin = (t0 & 1) ? pop1 : pop0;
    for (int i = 0; i < 9; i++)
        for (int q = tid; q < nslab; q += CL_THREADS) {
            const int ly = q / nx, x = q - ly * nx;
            F0[i * plane + q] = pin[(long long)i * gd.plane + (long long)(v.y_lo + ly) * gd.pitch + x];
        }
    __syncthreads();
    cluster_arrive();  // matched by the wait at the top of the first step

    // this thread's nodes (the second repeats the first where a slab has an odd
    // number of nodes, and stores nothing)
    const bool act = tid < npairs, two = tid + npairs < nslab;
    uint32_t pull[2][9];            // sources in the current set
    uint32_t dy_s[2], dy_0[2], dy_n[2];  // density rows below, at and above the node (bytes in `rho`)
    uint32_t dx_w[2], dx_0[2], dx_e[2];
    float lid[2];
    bool local = true;  // every source lies in this CTA's slab
#pragma unroll
    for (int j = 0; j < 2; j++) {
        const int q = act ? (j && two ? tid + npairs : tid) : 0;
        const int ly = q / nx, x = q - ly * nx, y = v.y_lo + ly;
#pragma unroll
        for (int i = 0; i < 9; i++) pull[j][i] = pull_address(v, gd, x, y, i, es, local);
        const int s = gd.bc != 2 && y == 0 ? 0 : -1, n = gd.bc != 2 && y == gd.ny - 1 ? 0 : 1;
        dy_0[j] = (uint32_t)((ly + 1) * nx) * 4u;
        dy_s[j] = (uint32_t)((ly + 1 + s) * nx) * 4u;
        dy_n[j] = (uint32_t)((ly + 1 + n) * nx) * 4u;
        dx_0[j] = (uint32_t)x * 4u;
        dx_w[j] = (uint32_t)(x > 0 ? x - 1 : (gd.bc >= 1 ? nx - 1 : 0)) * 4u;
        dx_e[j] = (uint32_t)(x < nx - 1 ? x + 1 : (gd.bc >= 1 ? 0 : nx - 1)) * 4u;
        lid[j] = gd.lid_on && gd.bc != 2 && y == gd.ny - 1 ? k.lid : 0.f;
    }
    // Pulls from this CTA only: plain shared-memory addresses, before the other
    // CTAs are waited for.
    if (local)
#pragma unroll
        for (int j = 0; j < 2; j++)
#pragma unroll
            for (int i = 0; i < 9; i++) pull[j][i] += v.own_cta - v.own;
    // the density ring: the rows below and above the slab, except beyond a wall
    const bool ring_s = gd.bc == 2 || v.y_lo > 0, ring_n = gd.bc == 2 || v.y_hi < gd.ny;
    const int nring = (ring_s ? nx : 0) + (ring_n ? nx : 0);
    // its first nodes go to the threads whose pulls do not wait, where there are any
    const int shift = rows > 2 && npairs > 2 * nx ? nx : 0;
    auto ring_node = [&](int u, int &gx, int &gy, int &lr) {
        const bool south = ring_s && u < nx;
        gx = south ? u : u - (ring_s ? nx : 0);
        lr = south ? 0 : rows + 1;  // row of the density tile
        gy = south ? v.y_lo - 1 : v.y_hi;
        if (gy < 0) gy += gd.ny;
        if (gy >= gd.ny) gy -= gd.ny;
    };
    const int u0 = tid >= shift ? tid - shift : tid - shift + CL_THREADS;
    uint32_t rpull[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, rdst = 0;
    float rlid = 0.f;
    if (u0 < nring) {
        int gx, gy, lr;
        bool any = true;
        ring_node(u0, gx, gy, lr);
#pragma unroll
        for (int i = 0; i < 9; i++) rpull[i] = pull_address(v, gd, gx, gy, i, es, any);
        rdst = (uint32_t)(lr * nx + gx);
        rlid = gd.lid_on && gd.bc != 2 && gy == gd.ny - 1 ? k.lid : 0.f;
    }

    const int q0 = tid, q1 = tid + npairs;
    const long long og0 = (long long)(v.y_lo + q0 / nx) * gd.pitch + q0 % nx;
    const long long og1 = (long long)(v.y_lo + q1 / nx) * gd.pitch + q1 % nx;
    uint32_t off = 0;  // set holding the state: 0 or set_b
    int done = 0;
    bool waited = false;  // the last cluster barrier phase has been waited on
    const double nnodes = (double)gd.nx * (double)gd.ny;
    int t20 = (int)((t0 + 1) % 20);  // index of the step being made, modulo 20
    for (; done < nsteps; done++, t20 = t20 == 19 ? 0 : t20 + 1) {
        const bool epi = t20 == 0;
        F2 g[9];
        if (act & local) {
#pragma unroll
            for (int i = 0; i < 9; i++) g[i] = F2(ld_cta<S>(pull[0][i] + off), ld_cta<S>(pull[1][i] + off));
        }
        cluster_wait();
        if (act & !local) {
#pragma unroll
            for (int i = 0; i < 9; i++)
                g[i] = F2(ld_cl<S, float>(pull[0][i] + off), ld_cl<S, float>(pull[1][i] + off));
        }
        if (act) {
            if (lid[0] != 0.f) {
                g[7].v.x -= lid[0];
                g[8].v.x += lid[0];
            }
            if (lid[1] != 0.f) {
                g[7].v.y -= lid[1];
                g[8].v.y += lid[1];
            }
        }
        if constexpr (DRHO) {
            if (act) {
                const F2 r = sum9(g);
                rho[nx + q0] = r.v.x;
                if (two) rho[nx + q1] = r.v.y;
            }
            if (u0 < nring) {
                float gr[9];
#pragma unroll
                for (int i = 0; i < 9; i++) gr[i] = ld_cl<S, float>(rpull[i] + off);
                if (rlid != 0.f) {
                    gr[7] -= rlid;
                    gr[8] += rlid;
                }
                rho[rdst] = sum9(gr);
            }
            for (int u = u0 + CL_THREADS; u < nring; u += CL_THREADS) {  // slabs wider than half the threads
                int gx, gy, lr;
                ring_node(u, gx, gy, lr);
                float gr[9];
                bool any = true;
#pragma unroll
                for (int i = 0; i < 9; i++) gr[i] = ld_cl<S, float>(pull_address(v, gd, gx, gy, i, es, any) + off);
                if (gd.lid_on && gd.bc != 2 && gy == gd.ny - 1) {
                    gr[7] -= k.lid;
                    gr[8] += k.lid;
                }
                rho[lr * nx + gx] = sum9(gr);
            }
            __syncthreads();
        }
        RedAcc<float> acc;
        if (act) {
            F2 dx(0.f), dy(0.f);
            if constexpr (DRHO) {
                auto at = [&](const uint32_t (&r)[2], const uint32_t (&c)[2]) {
                    const char *b = reinterpret_cast<const char *>(rho);
                    return F2(*reinterpret_cast<const float *>(b + r[0] + c[0]),
                              *reinterpret_cast<const float *>(b + r[1] + c[1]));
                };
                drho_stencil<F2>(at(dy_0, dx_e), at(dy_0, dx_w), at(dy_n, dx_0), at(dy_s, dx_0), at(dy_n, dx_e),
                                 at(dy_n, dx_w), at(dy_s, dx_e), at(dy_s, dx_w), F2(k.inv12), F2(k.inv12r), dx, dy);
            }
            F2 ux, uy, drho;
            collide<F2, DRHO, FORCE, RAW>(k2, g, dx, dy, ux, uy, drho);
            S *Fo = reinterpret_cast<S *>(reinterpret_cast<char *>(F0) + (set_b - off)) + q0;
#pragma unroll
            for (int i = 0; i < 9; i++) {
                Fo[i * plane] = to_s<S, float>(g[i].v.x);
                if (two) Fo[i * plane + npairs] = to_s<S, float>(g[i].v.y);
            }
            if (epi) {
                const float d0 = ux.v.x - snap[og0];
                snap[og0] = ux.v.x;
                acc.add(d0 * d0, drho.v.x);
                if (two) {
                    const float d1 = ux.v.y - snap[og1];
                    snap[og1] = ux.v.y;
                    acc.add(d1 * d1, drho.v.y);
                }
            }
        }
        if (epi) {
            double a, b;
            acc.block_total(a, b, red);
            if (tid == 0) part = make_double2(a, b);
        }
        // the new set is complete (and every pull of the old one done): this
        // CTA's stores are visible to its own threads, then it arrives; the next
        // step waits for the others
        __syncthreads();
        cluster_arrive();
        off = set_b - off;
        if (epi) {
            cluster_wait();  // every CTA's partial sums are written
            if (tid == 0) {
                double a = 0.0, m = 0.0;
                for (int r = 0; r < nc; r++) {  // rank order: the same sums in every CTA
                    const double2 p = *cl.map_shared_rank(&part, r);
                    a += p.x;
                    m += p.y;
                }
                const double res = sqrt(a), mass = nnodes + m;
                int stop = 0;
                if (!isfinite(res) || !isfinite(mass)) stop = 2;
                else if (res < st->tol) stop = 1;
                sh_stop = stop;
                if (rank == 0) {
                    st->res_step = t0 + done + 1;
                    st->res = res;
                    st->mass = mass;
                    if (stop == 2) {
                        st->diverged = 1;
                        *note = 1 + (int)((t0 + done + 1 + flip) & 1);
                    }
                    if (stop == 1) st->converged = 1;
                    if (stop) st->stop = 1;
                }
            }
            __syncthreads();  // sh_stop is visible to every thread
            if (sh_stop) {    // the same decision in every CTA
                done++;
                waited = true;
                break;
            }
            cluster_arrive();  // matched by the wait at the top of the next step
        }
    }
    if (!waited) cluster_wait();  // every CTA is done with this CTA's shared memory
    S *pout = const_cast<S *>(((t0 + done) & 1) ? pop1 : pop0);
    const S *fin = reinterpret_cast<const S *>(reinterpret_cast<const char *>(F0) + off);
    for (int i = 0; i < 9; i++)
        for (int q = tid; q < nslab; q += CL_THREADS) {
            const int ly = q / nx, x = q - ly * nx;
            pout[(long long)i * gd.plane + (long long)(v.y_lo + ly) * gd.pitch + x] = fin[i * plane + q];
        }
}

}  // namespace prc
