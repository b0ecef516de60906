// prc_kernels.cuh -- kernels of the single-instance path, templated on the
// storage type S (double, float, __half) and the collision type T.
#pragma once

#include <type_traits>

#include "prc_device.cuh"
#include "prc_reduce.cuh"

namespace prc {

constexpr int BX = 32;  // default tile width  (nodes, one per thread)
constexpr int BY = 8;   // default tile height
constexpr int MAX_RECTS = 4;

// Rectangles of nodes handled by the general tile body (the whole domain, or
// the edge strips around the interior tiles of the TMA kernel), enumerated as
// a 1-D list of tiles.  Each rectangle has its own tile shape: 2^lw nodes wide
// and (CTA threads) >> lw high, so that thin strips are covered without idle
// threads.
struct Rects {
    int n;
    int x0[MAX_RECTS], y0[MAX_RECTS], x1[MAX_RECTS], y1[MAX_RECTS];
    int lw[MAX_RECTS];       // log2 of the tile width
    int tiles_x[MAX_RECTS];
    int start[MAX_RECTS + 1];  // first tile index of each rectangle; start[n] = total
};

// Floats of density tile (+ ring) that general_tile needs for a CTA of
// `threads` threads and any tile width 2 <= 2^lw <= threads / 2.
__host__ __device__ constexpr int srho_floats(int threads) { return 4 * (threads / 2 + 2); }

// Origin and shape of tile `e` of the rectangle list.
__device__ __forceinline__ void rect_tile(const Rects &rc, int e, int &x0, int &y0, int &x1, int &y1, int &lw)
{
    int r = 0;
    while (r + 1 < rc.n && e >= rc.start[r + 1]) r++;
    const int lt = e - rc.start[r];
    lw = rc.lw[r];
    const int th = (int)(blockDim.x * blockDim.y) >> lw;
    x0 = rc.x0[r] + (lt % rc.tiles_x[r]) * (1 << lw);
    y0 = rc.y0[r] + (lt / rc.tiles_x[r]) * th;
    x1 = rc.x1[r];
    y1 = rc.y1[r];
}

// One fused time step on one tile of 2^lw x (threads >> lw) nodes at (x0, y0)
// of the nodes x < x1, y < y1 (all threads of the CTA call it): pull-stream +
// walls, density tile (+1 ring) in shared memory `srho` (srho_floats(threads)
// values of type T) for the density gradient, collision, store.  With EPI the
// thread adds (u_x - u_x,snapshot)^2 and drho of its node to `acc` and
// refreshes the snapshot (residual of Sec. 5.2).  With `stop` (the same for every
// thread) nothing is written: the flag is needed only after the loads are out.
template <typename S, typename T, bool DRHO, bool EPI, bool FORCE, bool CG = false, bool RAW = false>
__device__ __forceinline__ void general_tile(const S *__restrict__ src, S *__restrict__ dst, const Grid &gd,
                                             const Coef<T> &k, T *__restrict__ snap, int x0, int y0, int x1, int y1,
                                             int lw, RedAcc<T> &acc, T *srho, int stop = 0)
{
    const int nthr = blockDim.x * blockDim.y;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int tw = 1 << lw, th = nthr >> lw;
    const int tx = tid & (tw - 1), ty = tid >> lw;
    const int x = x0 + tx, y = y0 + ty;
    const bool valid = (x < x1) & (y < y1);
    T snap_old = T(0);
    if constexpr (EPI) {  // issue early: overlaps the pulls
        if (valid) snap_old = __ldcs(snap + (long long)y * gd.pitch + x);
    }

    T g[9];
    int mx = x, my = y;
    map_node(gd, mx, my);
    const bool top = pull9_load<S, T, CG>(src, gd, mx, my, g);

    T dxr = T(0), dyr = T(0);
    if constexpr (DRHO) {
        const int RW = tw + 2;
        const int nring = 2 * RW + 2 * th;
        auto ring = [&](int q, int &at, T gr[9]) {  // loads of ring node q; its place in srho
            int lx, ly;
            if (q < RW) { lx = q; ly = 0; }
            else if (q < 2 * RW) { lx = q - RW; ly = th + 1; }
            else if (q < 2 * RW + th) { lx = 0; ly = q - 2 * RW + 1; }
            else { lx = tw + 1; ly = q - 2 * RW - th + 1; }
            int gx = x0 - 1 + lx, gy = y0 - 1 + ly;
            map_node(gd, gx, gy);
            at = ly * RW + lx;
            return pull9_load<S, T, CG>(src, gd, gx, gy, gr);
        };
        T gr[9];
        int at = 0, first = tid;
        bool rtop = false;
        // The first ring node's loads are out before the thread's own are used: a small
        // grid's SM has one warp to a scheduler and nothing else to hide them (FP64, us per
        // step, with the late stop flag: 64x64 8.5 -> 8.0, 100x150 8.9 -> 8.4).  The batch
        // engine's tiles (CG) have no registers for it.
        if constexpr (!CG) {
            if (tid < nring) rtop = ring(tid, at, gr);
            first += nthr;
        }
        if (stop) return;
        if (top) pull9_lid(g, k.lid);
        srho[(ty + 1) * RW + tx + 1] = sum9(g);
        if (!CG && tid < nring) {
            if (rtop) pull9_lid(gr, k.lid);
            srho[at] = sum9(gr);
        }
        for (int q = first; q < nring; q += nthr) {
            if (ring(q, at, gr)) pull9_lid(gr, k.lid);
            srho[at] = sum9(gr);
        }
        __syncthreads();
        const T *c = srho + (ty + 1) * RW + tx + 1;
        const T rE = c[1], rW = c[-1];
        const T rN = c[RW], rS = c[-RW];
        const T rNE = c[RW + 1], rNW = c[RW - 1];
        const T rSE = c[-RW + 1], rSW = c[-RW - 1];
        drho_stencil<T>(rE, rW, rN, rS, rNE, rNW, rSE, rSW, k.inv12, k.inv12r, dxr, dyr);
        __syncthreads();  // srho may be refilled by the next tile of this CTA
    } else {
        if (stop) return;
        if (top) pull9_lid(g, k.lid);
    }

    T ux = T(0), uy = T(0), drho = T(0);
    if (valid) {
        collide<T, DRHO, FORCE, RAW>(k, g, dxr, dyr, ux, uy, drho);
        const long long o = (long long)y * gd.pitch + x;
#pragma unroll
        for (int i = 0; i < 9; i++) dst[(long long)i * gd.plane + o] = to_s<S, T>(g[i]);
        if constexpr (EPI) {
            const T d = ux - snap_old;
            __stcs(snap + o, ux);
            acc.add(d * d, drho);
        }
    }
}

// One fused time step on the nodes of `rc` (general kernel, one tile per
// CTA); the CTA totals of a residual step go to partials[part0 + blockIdx.x].
// CTAs of fewer than 256 threads (FP64, one rectangle, tiles of 32 x h nodes with
// h < 8) write the totals of their warps, that is of rows of 32 nodes, instead, at
// the place of the row in the 32 x 8 tiling: eight to a tile, summed as that
// tile's CTA would (k_finalize).
template <typename S, typename T, bool DRHO, bool EPI, bool FORCE, bool RAW>
__global__ void __launch_bounds__(BX * BY)
k_step(const S *__restrict__ src, S *__restrict__ dst, Grid gd, Coef<T> k, T *__restrict__ snap,
       double2 *__restrict__ partials, const DevStatus *__restrict__ st, const __grid_constant__ Rects rc, int part0)
{
    pdl_wait();
    pdl_trigger();
    const int stop = ld_relaxed_i32(&st->stop);
    __shared__ T srho[srho_floats(BX * BY)];
    int x0, y0, x1, y1, lw;
    rect_tile(rc, blockIdx.x, x0, y0, x1, y1, lw);
    RedAcc<T> acc;
    general_tile<S, T, DRHO, EPI, FORCE, false, RAW>(src, dst, gd, k, snap, x0, y0, x1, y1, lw, acc, srho, stop);
    if (stop) return;
    if constexpr (EPI) {
        if constexpr (std::is_same<T, double>::value) {
            if (blockDim.x * blockDim.y < BX * BY) {
                acc.warp_total();
                const int y = y0 + ((int)threadIdx.x >> 5);
                if ((threadIdx.x & 31) == 0 && y < y1)
                    partials[((long long)(y / BY) * rc.tiles_x[0] + x0 / BX) * BY + y % BY] = make_double2(acc.a, acc.b);
                return;
            }
        }
        __shared__ double red[2 * (BX * BY / 32)];
        double a, b;
        acc.block_total(a, b, red);
        if (threadIdx.x == 0 && threadIdx.y == 0) partials[part0 + blockIdx.x] = make_double2(a, b);
    }
}

// ---- transfers of FP64 fields.  The FP64 pipe of this part makes two
// operations per SM and clock, so that these kernels are bound by their FP64
// instructions, conversions between FP64 and FP32 among them, long before they
// are bound by memory (the pipe was 85 % busy in a profile).  They therefore
// share their sums and products, take one reciprocal by Newton's iteration
// instead of two divisions, and convert between the formats in integer
// arithmetic.  On 8192 x 2048 nodes with FP32 storage: fields in 2.61 -> 1.27 ms,
// fields out 1.43 -> 0.81 ms (24 FP64 operations a node; memory alone 0.16 ms); of
// a fluid at rest 2.61 -> 1.24 and 2.16 -> 0.81 (3.68 and 1.08 where zeros went through
// the rounding test and the conversion instructions).

// FP32 -> FP64 (exact) for normal numbers: the exponent moved, the mantissa
// shifted.
__device__ __forceinline__ bool is_normal(float v) { return (__float_as_uint(v) & 0x7fffffffu) - 0x00800000u < 0x7f000000u; }
__device__ __forceinline__ double widen_normal(float v)
{
    const uint32_t u = __float_as_uint(v);
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}

__device__ __forceinline__ bool is_zero(float v) { return (__float_as_uint(v) & 0x7fffffffu) == 0; }
__device__ __forceinline__ double widen_or_zero(float v)
{
    return is_zero(v) ? __hiloint2double((int)__float_as_uint(v), 0) : widen_normal(v);
}

// FP64 -> FP32, round to nearest even, for values of 2^-124 to 2^127: the result is a
// normal number, and so are its half and its quarter.
__device__ __forceinline__ bool narrows_to_normal(double v)
{
    return ((uint32_t)__double2hiint(v) & 0x7fffffffu) - (899u << 20) < (251u << 20);
}
__device__ __forceinline__ float narrow_normal(double v)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const uint32_t q = __funnelshift_l(lo, (hi & 0x7fffffffu) - (896u << 20), 3);  // exponent and 23 mantissa bits
    const uint32_t up = ((lo & 0x1fffffffu) + 0x0fffffffu + (q & 1u)) >> 29;       // above half, or half and odd
    return __uint_as_float((q + up) | (hi & 0x80000000u));
}

__device__ __forceinline__ bool is_zero(double v)
{
    return (((uint32_t)__double2hiint(v) & 0x7fffffffu) | (uint32_t)__double2loint(v)) == 0;
}
__device__ __forceinline__ float narrow_or_zero(double v)
{
    return is_zero(v) ? __uint_as_float((uint32_t)__double2hiint(v)) : narrow_normal(v);
}

// The conversions of a node's values: in integer arithmetic when all of the warp's
// allow it, zeros (a fluid at rest) among them, else (subnormals, infinities, NaN)
// by the conversion instructions.  One branch for all, so that the compiler does
// not run several forms and select.
template <int N>
__device__ __forceinline__ void widen(const float *v, double *d)
{
    bool normal = true;
#pragma unroll
    for (int i = 0; i < N; i++) normal &= is_normal(v[i]);
    if (__all_sync(__activemask(), normal)) {
#pragma unroll
        for (int i = 0; i < N; i++) d[i] = widen_normal(v[i]);
        return;
    }
    normal = true;
#pragma unroll
    for (int i = 0; i < N; i++) normal &= is_normal(v[i]) | is_zero(v[i]);
    if (__all_sync(__activemask(), normal)) {
#pragma unroll
        for (int i = 0; i < N; i++) d[i] = widen_or_zero(v[i]);
    } else {
#pragma unroll
        for (int i = 0; i < N; i++) d[i] = (double)v[i];
    }
}
template <int N>
__device__ __forceinline__ void widen(const double *v, double *d)
{
#pragma unroll
    for (int i = 0; i < N; i++) d[i] = v[i];
}
// scale(i) v[i], rounded once; the scale is a power of two, 1/4 at least.
template <int N, typename F>
__device__ __forceinline__ void narrow(const double *v, float *f, F scale)
{
    bool normal = true;
#pragma unroll
    for (int i = 0; i < N; i++) normal &= narrows_to_normal(v[i]);
    if (__all_sync(__activemask(), normal)) {
#pragma unroll
        for (int i = 0; i < N; i++) f[i] = (float)scale(i) * narrow_normal(v[i]);
        return;
    }
    normal = true;
#pragma unroll
    for (int i = 0; i < N; i++) normal &= narrows_to_normal(v[i]) | is_zero(v[i]);
    if (__all_sync(__activemask(), normal)) {
#pragma unroll
        for (int i = 0; i < N; i++) f[i] = (float)scale(i) * narrow_or_zero(v[i]);
    } else {
#pragma unroll
        for (int i = 0; i < N; i++) f[i] = (float)(scale(i) * v[i]);
    }
}
template <int N, typename F>
__device__ __forceinline__ void narrow(const double *v, double *f, F scale)
{
#pragma unroll
    for (int i = 0; i < N; i++) f[i] = scale(i) * v[i];
}

// Constants of the equilibrium moments of Eq. 12, formed once on the host:
// those of the moments as written, and those in the units of the square
// lattice (e_y = 1).
struct InitCoef {
    double c2, c4, inv_r2, ig, ir;     // c^2, c^4, 1/r^2, 1/gamma, 1/r
    double c2r, c4r, c2g, c2rg, g2;    // c^2/r^2, c^4/r^2, c^2 gamma, c^2 gamma/r^2, gamma^2
};

inline InitCoef make_init_coef(const Coef<double> &k, double gamma)
{
    return InitCoef{k.c2, k.c4, k.inv_r2, 1.0 / gamma, 1.0 / k.r, k.c2 * k.inv_r2, k.c4 * k.inv_r2, k.c2 * gamma,
                    k.c2 * k.inv_r2 * gamma, gamma * gamma};
}

// Rest-shifted equilibrium populations, the moments as written in Eq. 12.
// Reduced storage rounds these values.
static __device__ __noinline__ void equilibrium_as_written(const InitCoef &k, double rho, double ux, double uy, double *f)
{
    const double drho = rho - 1.0;
    // raw equilibrium moments (rectangular) minus the rest-state moments
    const double D00 = drho, D10 = rho * ux, D01 = rho * uy;
    const double D20 = k.c2 * drho + rho * ux * ux * k.ig;
    const double D02 = k.c2 * drho + rho * uy * uy * k.ig;
    const double D11 = rho * ux * uy * k.ig;
    const double D21 = rho * (k.c2 + ux * ux * k.ig * k.ig) * uy;
    const double D12 = rho * (k.c2 + uy * uy * k.ig * k.ig) * ux;
    const double D22 = k.c4 * drho + rho * k.c2 * (ux * ux + uy * uy) + rho * ux * ux * uy * uy;
    const double e01 = D01 * k.ir, e02 = D02 * k.inv_r2, e11 = D11 * k.ir;
    const double e21 = D21 * k.ir, e12 = D12 * k.inv_r2, e22 = D22 * k.inv_r2;
    f[0] = D00 - D20 - e02 + e22;
    f[1] = 0.5 * (D10 + D20 - e12 - e22);
    f[2] = 0.5 * (e01 + e02 - e21 - e22);
    f[3] = 0.5 * (-D10 + D20 + e12 - e22);
    f[4] = 0.5 * (-e01 + e02 + e21 - e22);
    f[5] = 0.25 * (e11 + e21 + e12 + e22);
    f[6] = 0.25 * (-e11 + e21 - e12 + e22);
    f[7] = 0.25 * (e11 - e21 - e12 + e22);
    f[8] = 0.25 * (-e11 - e21 + e12 + e22);
}

__device__ __forceinline__ uint32_t abs_hi(double v) { return (uint32_t)__double2hiint(v) & 0x7fffffffu; }

// Whether v rounds to the same FP32 number as every value within 2^8 ulps of
// a number whose high word is hm (Ziv's rounding test, ACM TOMS 17, 1991): its
// distance from the nearest midpoint between FP32 numbers is larger.  Needs
// v at least 2^-18 of that number and FP32 results, of v and of v / 4, that are normal;
// 2^26 ulps of v are half the smallest distance from an FP32 number to a midpoint
// beside it.
__device__ __forceinline__ bool rounds_safely(double v, uint32_t hm)
{
    const uint32_t hv = abs_hi(v), lo = (uint32_t)__double2loint(v);
    const int s = (int)(hm >> 20) - (int)(hv >> 20) + 8;
    const int d = (int)(lo & 0x1fffffffu) - 0x10000000;
    return narrows_to_normal(v) & (s <= 26) & (abs(d) > (1 << (s & 31)));
}

// f~ = f^eq(rho, u) (Eq. 12, uncorrected), stored shifted; snapshot = u_x.
//
// Bound by FP64 arithmetic.  The equilibria are formed with shared products in
// the units of the square lattice (39 operations instead of about 60, no
// division).  Reduced storage rounds them, and the rounding of a value must not
// depend on the order of the FP64 operations behind it: a node whose value lies
// so close to a midpoint of FP32 numbers that another order could round to the
// other side takes the moments as written.  Both orders differ by less than
// 128 roundings of terms no larger than the largest moment; 2^8 ulps of
// that moment are the test's margin.  A node at rest (rho = 1, u = 0) has zeros in
// either order, which the test does not take.
template <typename S, typename T>
__global__ void k_init_fields(S *__restrict__ dst, Grid gd, const __grid_constant__ InitCoef k,
                              const double *__restrict__ rho_in, const double *__restrict__ ux_in,
                              const double *__restrict__ uy_in, T *__restrict__ snap)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= gd.nx || y >= gd.ny) return;
    const long long n = (long long)y * gd.nx + x;
    const double rho = rho_in[n], ux = ux_in[n], uy = uy_in[n];
    const long long o = (long long)y * gd.pitch + x;
    const double v = uy * k.ir;
    // raw equilibrium moments minus the rest-state ones, y in units of r
    const double drho = rho - 1.0, X = rho * ux, Y = rho * v;
    const double uxg = ux * k.ig, vg = v * k.ig;
    const double xx = X * uxg, yy = Y * vg, E11 = X * vg;  // rho u_x^2 / gamma, rho v^2 / gamma, rho u_x v / gamma
    const double E20 = fma(k.c2, drho, xx), E02 = fma(k.c2r, drho, yy);
    const double t = xx * vg;
    const double E21 = fma(k.c2, Y, t), E12 = fma(k.c2r, X, yy * uxg);
    const double E22 = fma(t, v * k.g2, fma(k.c2g, yy, fma(k.c2rg, xx, k.c4r * drho)));
    const double a = E22 + E21, b = E22 - E21, c = E12 + E11, d = E12 - E11;
    const double a1 = E20 - E22, b1 = X - E12, a2 = E02 - E22, b2 = Y - E21;
    // twice and four times the populations (the factors are exact)
    double f[10] = {(drho - E20) - a2, a1 + b1, a2 + b2, a1 - b1, a2 - b2, a + c, a - c, b - d, b + d, ux};
    T g[10];
    if constexpr (std::is_same<T, float>::value) {
        const uint32_t h0 = max(max(abs_hi(drho), abs_hi(X)), max(abs_hi(Y), abs_hi(E11)));
        const uint32_t h1 = max(max(abs_hi(xx), abs_hi(yy)), max(abs_hi(E20), abs_hi(E02)));
        const uint32_t h2 = max(max(abs_hi(E21), abs_hi(E12)), abs_hi(E22));
        const uint32_t hm = max(max(h0, h1), h2);
        bool safe = true;
#pragma unroll
        for (int i = 0; i < 9; i++) safe &= rounds_safely(f[i], hm);
        if (!safe && !(__double_as_longlong(rho) == __double_as_longlong(1.0) && is_zero(ux) && is_zero(uy))) {
            equilibrium_as_written(k, rho, ux, uy, f);
#pragma unroll
            for (int i = 1; i < 9; i++) f[i] *= i < 5 ? 2.0 : 4.0;
        }
    }
    narrow<10>(f, g, [](int i) { return i == 0 || i == 9 ? 1.0 : (i < 5 ? 0.5 : 0.25); });
#pragma unroll
    for (int i = 0; i < 9; i++) dst[(long long)i * gd.plane + o] = to_s<S, T>(g[i]);
    snap[o] = g[9];
}

// a / b from b's reciprocal ib and q = a ib: the remainder's share added, which rounds the
// quotient correctly (Markstein, IBM J. Res. Dev. 34, 1990); q where a value is not
// finite.
__device__ __forceinline__ double corrected_quotient(double a, double b, double ib, double q)
{
    const double c = fma(fma(-q, b, a), ib, q);
    return abs_hi(c) >= 0x7ff00000u ? q : c;
}

// Fields of the stored post-collision state: rho = 1 + sum g, rho u = sum g e
// - F / (2 gamma) (the rest state carries no momentum).  Quotients of FP64 states are
// rounded correctly; those of reduced storage, the product with the reciprocal, may be
// a unit of 2^-53 off, 2^28 times less than the rounding of a stored population.
template <typename S, typename T>
__global__ void k_fields(const S *__restrict__ src, Grid gd, double r, double hx, double hy,
                         double *__restrict__ rho_out, double *__restrict__ ux_out, double *__restrict__ uy_out,
                         T *__restrict__ snap)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= gd.nx || y >= gd.ny) return;
    const long long o = (long long)y * gd.pitch + x;
    T gs[9];
#pragma unroll
    for (int i = 0; i < 9; i++) gs[i] = ld_s<S, T>(src + (long long)i * gd.plane + o);
    double g[9];
    widen<9>(gs, g);
    const double p56 = g[5] + g[6], p78 = g[7] + g[8];
    const double s00 = ((g[0] + (p56 + p78)) + ((g[1] + g[3]) + (g[2] + g[4])));
    const double s10 = (g[1] - g[3]) + ((g[5] - g[6]) + (g[8] - g[7]));
    const double s01 = (g[2] - g[4]) + (p56 - p78);
    const double rho = 1.0 + s00, jx = s10 - hx, jy = fma(r, s01, -hy);
    const double irho = vrcp(rho);
    double ux = jx * irho, uy = jy * irho;
    if constexpr (std::is_same<T, double>::value) {
        ux = corrected_quotient(jx, rho, irho, ux);
        uy = corrected_quotient(jy, rho, irho, uy);
    }
    const long long n = (long long)y * gd.nx + x;
    if (rho_out) rho_out[n] = rho;
    if (ux_out) ux_out[n] = ux;
    if (uy_out) uy_out[n] = uy;
    if (snap) snap[o] = (T)ux;
}

// Full FP64 populations <-> shifted storage.
template <typename S, typename T>
__global__ void k_set_pop(S *__restrict__ dst, Grid gd, Coef<double> k, const double *__restrict__ f)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= gd.nx || y >= gd.ny) return;
    const long long nn = (long long)gd.nx * gd.ny, n = (long long)y * gd.nx + x;
    const long long o = (long long)y * gd.pitch + x;
#pragma unroll
    for (int i = 0; i < 9; i++) dst[(long long)i * gd.plane + o] = to_s<S, T>((T)(f[i * nn + n] - k.w[i]));
}

template <typename S, typename T>
__global__ void k_get_pop(const S *__restrict__ src, Grid gd, Coef<double> k, double *__restrict__ f)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= gd.nx || y >= gd.ny) return;
    const long long nn = (long long)gd.nx * gd.ny, n = (long long)y * gd.nx + x;
    const long long o = (long long)y * gd.pitch + x;
#pragma unroll
    for (int i = 0; i < 9; i++) f[i * nn + n] = (double)ld_s<S, T>(src + (long long)i * gd.plane + o) + k.w[i];
}

// Uniform density shift: f_i += w_i(r) delta at every node (the rest
// populations carry density and no momentum), rounded to the storage.
template <typename S, typename T>
__global__ void k_add_rest(S *__restrict__ pop, Grid gd, Coef<double> k, double delta)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= gd.nx || y >= gd.ny) return;
    const long long o = (long long)y * gd.pitch + x;
#pragma unroll
    for (int i = 0; i < 9; i++) {
        S *p = pop + (long long)i * gd.plane + o;
        *p = to_s<S, T>((T)((double)ld_s<S, T>(p) + k.w[i] * delta));
    }
}

// Per-CTA FP64 partial sums of sum_i g_i (total mass minus the node count).
template <typename S, typename T>
__global__ void __launch_bounds__(BX * BY) k_mass_partial(const S *__restrict__ src, Grid gd, double2 *__restrict__ partials)
{
    const int x = blockIdx.x * BX + threadIdx.x, y = blockIdx.y * BY + threadIdx.y;
    double dm = 0.0, z = 0.0;
    if (x < gd.nx && y < gd.ny) {
        const long long o = (long long)y * gd.pitch + x;
#pragma unroll
        for (int i = 0; i < 9; i++) dm += (double)ld_s<S, T>(src + (long long)i * gd.plane + o);
    }
    __shared__ double red[2 * (BX * BY / 32)];
    RedAcc<double> acc;
    acc.add(z, dm);
    double a, b;
    acc.block_total(a, b, red);
    if (threadIdx.x == 0 && threadIdx.y == 0) partials[blockIdx.y * gridDim.x + blockIdx.x] = make_double2(a, b);
}

}  // namespace prc
