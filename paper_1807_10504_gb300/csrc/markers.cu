// Lagrangian marker kernels of the method (Sections 2.2, 3 and 4):
//   binning + deterministic (key, id) order, velocity interpolation
//   (Eq. (jump_condu)), conventional spreading (Eq. (delta_vec)) as a gather
//   over markers sorted by cell, the polygon discrete Heaviside and the
//   irrotational face force (Eqs. (delta_hea), (delta_hea_xy)), discrete
//   curvature (Eq. (ten_f)) and least-squares B-spline relocation
//   (Eqs. (bspline), (bcurve), (bspline_ls)).
//
// This translation unit is compiled without multiply-add contraction so that
// integer decisions taken from floating point (cell keys, inside/outside
// crossings, nearest segment) follow the same IEEE operations as a plain
// reading of the definitions.  No floating-point atomics: every sum has a
// fixed order.  All marker work is O(markers x stencil) and small next to the
// pressure solve; the band kernels touch only 8x8-cell blocks that have a
// marker within kSearch cells.
#include <math.h>

#include "ib_internal.cuh"

namespace ibk {
namespace {

constexpr int kT = 256;

// The delta function phi at the four grid lines that a marker reaches along one
// axis: at r = a - 1 - f, a = 0 .. 3, f in [0, 1) the marker's fraction past
// line 1.  The cosine kernel's four values are 1/4 (1 -+ sin, cos(pi f / 2)) of
// one angle: one sincospi instead of four cospi.  Peskin's are 1/8 (3 - 2 f -+ q,
// 1 + 2 f +- q) with q = sqrt(1 + 4 f - 4 f^2), the two branches at 1 + f, f, 1 - f
// and 2 - f: one square root in place of four (the markers' FP64 bounds the
// interpolation: 16384 markers 30.9 -> 16.4 us, 300,000 465 -> 213; one thread a
// marker with a root a factor took 22.6 and 265).
__device__ __forceinline__ void phi4(int kernel, double f, double *p)
{
    if (kernel == 0) {
        double sn, cs;
        sincospi(0.5 * f, &sn, &cs);
        p[0] = 0.25 * (1.0 - sn);
        p[1] = 0.25 * (1.0 + cs);
        p[2] = 0.25 * (1.0 + sn);
        p[3] = 0.25 * (1.0 - cs);
        return;
    }
    const double q = sqrt(fma(4.0 * f, 1.0 - f, 1.0)), s = 3.0 - 2.0 * f, t = 1.0 + 2.0 * f;
    p[0] = 0.125 * (s - q);
    p[1] = 0.125 * (s + q);
    p[2] = 0.125 * (t + q);
    p[3] = 0.125 * (t - q);
}

// Integer key with the order of the doubles (non-NaN; -0 treated as +0), so
// that the many exact comparisons of the inside test run on the integer pipe.
__device__ __forceinline__ unsigned long long okey(double d)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(d + 0.0);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ULL);
}

__device__ __forceinline__ void nbrs(int m, const int32_t *drop_of,
                                     const int32_t *drop_start, int *pm, int *nm)
{
    int d = drop_of[m], s = drop_start[d], e = drop_start[d + 1];
    *pm = (m == s) ? e - 1 : m - 1;
    *nm = (m == e - 1) ? s : m + 1;
}

// ------------------------------------------------------------ validation
// With host (page-locked memory), the last block to finish also moves the three
// flag words there and clears them (flags[3] counts the blocks): a copy and a
// memset fewer behind every time step.
__global__ void k_validate(int M, const double *__restrict__ X, const double *__restrict__ Y,
                           double xlo, double xhi, double ylo, double yhi, uint32_t *flags,
                           uint32_t *host)
{
    int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < M) {
        double x = X[m], y = Y[m];
        if (!(x >= xlo && x <= xhi && y >= ylo && y <= yhi)) atomicOr(&flags[0], 1u);
    }
    if (!host) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&flags[3], 1u) == gridDim.x - 1) {
        __threadfence();
        for (int k = 0; k < 3; k++) host[k] = atomicExch(&flags[k], 0u);
        flags[3] = 0;
    }
}

// ------------------------------------------------------------ geometry
__global__ void k_geometry(int M, const double *__restrict__ X, const double *__restrict__ Y,
                           const int32_t *__restrict__ drop_of,
                           const int32_t *__restrict__ drop_start, double sigma, double x0,
                           double y0, double h, double *__restrict__ kappa,
                           double *__restrict__ nxm, double *__restrict__ nym,
                           double *__restrict__ ds, double *__restrict__ fmag,
                           double *__restrict__ gx, double *__restrict__ gy,
                           float *__restrict__ gxf, float *__restrict__ gyf,
                           unsigned long long *__restrict__ ykey)
{
    int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    ykey[m] = okey(Y[m]);
    {
        double a = (X[m] - x0) / h, b = (Y[m] - y0) / h;
        gx[m] = a; gy[m] = b;
        gxf[m] = d2f_rn(a); gyf[m] = d2f_rn(b);
    }
    int pm, nm;
    nbrs(m, drop_of, drop_start, &pm, &nm);
    double ax = X[m] - X[pm], ay = Y[m] - Y[pm];
    double bx = X[nm] - X[m], by = Y[nm] - Y[m];
    double la = sqrt(ax * ax + ay * ay), lb = sqrt(bx * bx + by * by);
    double tax = ax / la, tay = ay / la, tbx = bx / lb, tby = by / lb;
    double dsm = 0.5 * (la + lb);
    double dx = tbx - tax, dy = tby - tay;
    double cr = tax * tby - tay * tbx;
    double k = sqrt(dx * dx + dy * dy) / dsm;
    k = cr >= 0.0 ? k : -k;
    double nx_ = -tay - tby, ny_ = tax + tbx;
    double ln = sqrt(nx_ * nx_ + ny_ * ny_);
    kappa[m] = k;
    nxm[m] = nx_ / ln;
    nym[m] = ny_ / ln;
    ds[m] = dsm;
    fmag[m] = sigma * k;
}

// 1 / sqrt(s): rsqrt_nr well inside the FP32 range (tested on the bit
// pattern, which orders positive values), square root and division elsewhere.
__device__ __forceinline__ double rsqrt_any(double s)
{
    const unsigned long long a = (unsigned long long)__double_as_longlong(s);
    if (a > (unsigned long long)__double_as_longlong(1e-30) &&
        a < (unsigned long long)__double_as_longlong(1e30))
        return rsqrt_nr(s);
    return 1.0 / sqrt(s);
}
__device__ __forceinline__ double sqrt_any(double s)
{
    const unsigned long long a = (unsigned long long)__double_as_longlong(s);
    if (a > (unsigned long long)__double_as_longlong(1e-30) &&
        a < (unsigned long long)__double_as_longlong(1e30))
        return s * rsqrt_nr(s);
    return sqrt(s);
}

// Segment geometry of (m, next m): the strip corners at offsets -2.5 .. 2.5
// cells along both marker normals (grid units), the strip and slab boxes
// rounded outward to FP32 so that an FP32 test against a cell never rejects
// a strip that touches it, the eight bounding half-planes and whether all
// five strips are convex.
//
// Half-planes {x : a x + b y - c >= 0}, (a, b) the unit left normal of a
// directed line P -> Q (a zero vector, which constrains nothing, if P = Q);
// the quadrilaterals are counter-clockwise: 0: normal edge at m (A5 -> A0), 1:
// normal edge at next m (B0 -> B5), 2 + o: offset line o (A_o -> B_o), inside
// = larger offsets.  Eight lanes per segment, one per line: about 70 FP64
// instructions a lane in place of 650 a segment, which one thread issued at
// 64 cycles each (128 markers: 29 us, now below 7; 16384 markers: 35 us, now 27).
__global__ void __launch_bounds__(128)
k_segments(int M, const int32_t *__restrict__ next, const double *__restrict__ gx,
           const double *__restrict__ gy, const double *__restrict__ nxm,
           const double *__restrict__ nym, float4 *__restrict__ sbox,
           double *__restrict__ sv, float4 *__restrict__ sb5,
           double *__restrict__ sl, float4 *__restrict__ slf,
           uint8_t *__restrict__ scvx, double *__restrict__ sinv)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int t = blockIdx.x * blockDim.x + threadIdx.x, q = t & 7;
    const bool live = (t >> 3) < M;
    const int m = live ? t >> 3 : M - 1, nm = next[m];
    const double gxa = gx[m], gya = gy[m], gxb = gx[nm], gyb = gy[nm];
    const double nax = nxm[m], nay = nym[m], nbx = nxm[nm], nby = nym[nm];
    // the line's ends: corner o (offset o - 2.5 cells) on the normal at m or
    // at next m
    const bool pB = q == 1, qB = q != 0;
    const double off = (double)(q - 2) - 2.5;
    const double oP = q == 0 ? 2.5 : (q == 1 ? -2.5 : off), oQ = q == 0 ? -2.5 : (q == 1 ? 2.5 : off);
    const double px = (pB ? gxb : gxa) + oP * (pB ? nbx : nax), py = (pB ? gyb : gya) + oP * (pB ? nby : nay);
    const double qx = (qB ? gxb : gxa) + oQ * (qB ? nbx : nax), qy = (qB ? gyb : gya) + oQ * (qB ? nby : nay);
    // corner o of m: (2o, 2o+1); of next m: 12 + (2o, 2o+1)
    if (live && q >= 2) {
        double *v = sv + (long)m * 24 + 2 * (q - 2);
        *(double2 *)v = make_double2(px, py);
        *(double2 *)(v + 12) = make_double2(qx, qy);
    }
    // strip k = q - 2 lies between this lane's line and the next lane's
    const double rx = __shfl_down_sync(kAll, qx, 1, 8), ry = __shfl_down_sync(kAll, qy, 1, 8);
    const double sx = __shfl_down_sync(kAll, px, 1, 8), sy = __shfl_down_sync(kAll, py, 1, 8);
    const bool strip = q >= 2 && q < 7;
    // minima and maxima of the (finite) corners compared on their bit
    // patterns, in integer instructions (ordered like the values)
    auto kb = [](double d) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(d);
        return (b >> 63) ? ~b : (b | 0x8000000000000000ULL);
    };
    auto dmin = [&](double a, double b) { return kb(a) <= kb(b) ? a : b; };
    auto dmax = [&](double a, double b) { return kb(a) >= kb(b) ? a : b; };
    const double x0 = dmin(dmin(px, sx), dmin(qx, rx)), x1 = dmax(dmax(px, sx), dmax(qx, rx));
    const double y0 = dmin(dmin(py, sy), dmin(qy, ry)), y1 = dmax(dmax(py, sy), dmax(qy, ry));
    float4 f = make_float4(__double2float_rd(x0) - 1e-3f, __double2float_ru(x1) + 1e-3f,
                           __double2float_rd(y0) - 1e-3f, __double2float_ru(y1) + 1e-3f);
    if (strip) {
        if (live) sb5[(long)m * 5 + q - 2] = f;
    } else {
        f = make_float4(INFINITY, -INFINITY, INFINITY, -INFINITY);
    }
    for (int o = 4; o; o >>= 1) {
        f.x = fminf(f.x, __shfl_xor_sync(kAll, f.x, o)); f.y = fmaxf(f.y, __shfl_xor_sync(kAll, f.y, o));
        f.z = fminf(f.z, __shfl_xor_sync(kAll, f.z, o)); f.w = fmaxf(f.w, __shfl_xor_sync(kAll, f.w, o));
    }
    if (live && q == 0) sbox[m] = f;
    const double dx = qx - px, dy = qy - py, l2 = dx * dx + dy * dy;
    const double il = (__double_as_longlong(l2) & 0x7fffffffffffffffLL) == 0 ? 0.0 : rsqrt_any(l2);
    const double la = -dy * il, lb = dx * il, lc = la * px + lb * py;
    // FP64 record (kSegLine doubles): per line a, b, c, 1/a, 1/b (0 where
    // the component vanishes), then the reciprocals of the determinants
    // a_i b_j - b_i a_j of the two normal edges and of each normal edge with
    // each offset line, which the per-cell area formula would otherwise
    // recompute for every cell the segment meets.
    double *d = sl + (long)m * kSegLine;
    const double ra = recip_any(la), rb = recip_any(lb);
    // |n| in FP32: the normal is normalised (to a few units of 1e-16), so
    // (float)|n| is 1.0f, or 0.0f for the zero vector of a degenerate line
    const bool nz = ((__double_as_longlong(la) | __double_as_longlong(lb)) & 0x7fffffffffffffffLL) != 0;
    if (live) {
        d[5 * q + 0] = la; d[5 * q + 1] = lb; d[5 * q + 2] = lc;
        d[5 * q + 3] = ra; d[5 * q + 4] = rb;
        slf[(long)m * 8 + q] = make_float4(d2f_rn(la), d2f_rn(lb), d2f_rn(lc), nz ? 1.0f : 0.0f);
    }
    const double a0 = __shfl_sync(kAll, la, 0, 8), b0 = __shfl_sync(kAll, lb, 0, 8);
    const double a1 = __shfl_sync(kAll, la, 1, 8), b1 = __shfl_sync(kAll, lb, 1, 8);
    // lane 0: 1 / |segment|^2 (grid units) in the place of a determinant
    const double ex = gxb - gxa, ey = gyb - gya;
    const double r0 = recip_any(q == 0 ? ex * ex + ey * ey : a0 * lb - b0 * la);
    const double r1 = recip_any(a1 * lb - b1 * la);
    if (live) {
        if (q == 0) sinv[m] = r0;
        else if (q == 1) d[40] = r0;
        else { d[41 + 2 * (q - 2)] = r0; d[42 + 2 * (q - 2)] = r1; }
    }
    // The strips are the intersections of those half-planes only when every
    // strip quadrilateral (A_k, B_k, B_k+1, A_k+1) is strictly convex; a
    // radius of curvature below about 2.5 cells folds the inner strips.
    // Segments that fail either test take the edge integrals.
    const double ux = rx - qx, uy = ry - qy, vx = sx - rx, vy = sy - ry, wx = px - sx, wy = py - sy;
    // > 1e-6 on the bit patterns (a negative value has a negative one)
    auto turn = [](double c) { return __double_as_longlong(c) > __double_as_longlong(1e-6); };
    bool ok = !strip || (turn(dx * uy - dy * ux) && turn(ux * vy - uy * vx) &&
                         turn(vx * wy - vy * wx) && turn(wx * dy - wy * dx));
    // The half-plane path also wants every line at least 0.001 rad away from
    // the grid axes (or exactly on one): a line nearly parallel to a cell edge
    // meets it at an ill-conditioned point, which the area formula would use
    // twice (once per boundary piece); the edge integrals have no such
    // sensitivity and take those segments.  |a| == 0 or |a| >= 1e-3, likewise
    // b, on the bit patterns of |a|, |b|.
    const long long k3 = __double_as_longlong(1e-3);
    const long long aa = __double_as_longlong(la) & 0x7fffffffffffffffLL,
                    bb = __double_as_longlong(lb) & 0x7fffffffffffffffLL;
    ok = ok && (aa == 0 || aa >= k3) && (bb == 0 || bb >= k3);
    const unsigned all = __ballot_sync(kAll, ok) >> (threadIdx.x & 24);
    if (live && q == 0) scvx[m] = (all & 0xffu) == 0xffu ? 1 : 0;
}

// One warp per drop: the range of its marker Y.
__global__ void k_drop_yrange(int ndrops, const int32_t *__restrict__ drop_start,
                              const double *__restrict__ Y, double2 *__restrict__ dyr,
                              ulonglong2 *__restrict__ dyk)
{
    int d = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (d >= ndrops) return;
    double lo = INFINITY, hi = -INFINITY;
    for (int m = drop_start[d] + lane; m < drop_start[d + 1]; m += 32) {
        lo = fmin(lo, Y[m]);
        hi = fmax(hi, Y[m]);
    }
    for (int o = 16; o; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) {
        dyr[d] = make_double2(lo, hi);
        dyk[d] = make_ulonglong2(okey(lo), okey(hi));
    }
}

// ------------------------------------------------------------ binning
__global__ void k_keys(int M, const double *__restrict__ X, const double *__restrict__ Y,
                       double x0, double y0, double h, int nx, int ny, int bnx,
                       uint32_t *__restrict__ key, uint32_t *__restrict__ count,
                       uint32_t *__restrict__ bcount)
{
    int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    int kx = (int)floor((X[m] - x0) / h), ky = (int)floor((Y[m] - y0) / h);
    kx = min(max(kx, 0), nx - 1);
    ky = min(max(ky, 0), ny - 1);
    uint32_t k = (uint32_t)ky * (uint32_t)nx + (uint32_t)kx;
    key[m] = k;
    atomicAdd(&count[k], 1u);
    atomicAdd(&bcount[(ky / kBlk) * bnx + kx / kBlk], 1u);
}

constexpr int kScanItems = 8;
constexpr int kScanChunk = kT * kScanItems;

__device__ uint32_t block_excl_scan(uint32_t v, uint32_t *total)
{
    __shared__ uint32_t sh[kT];
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < kT; o <<= 1) {
        uint32_t t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0u;
        __syncthreads();
        sh[threadIdx.x] += t;
        __syncthreads();
    }
    uint32_t incl = sh[threadIdx.x];
    if (total) *total = sh[kT - 1];
    __syncthreads();
    return incl - v;
}

__global__ void k_scan_partial(long n, const uint32_t *__restrict__ a, uint32_t *__restrict__ part)
{
    long base = (long)blockIdx.x * kScanChunk;
    uint32_t s = 0;
    for (int k = 0; k < kScanItems; k++) {
        long q = base + (long)threadIdx.x * kScanItems + k;
        if (q < n) s += a[q];
    }
    uint32_t tot;
    block_excl_scan(s, &tot);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

__global__ void k_scan_parts(int nparts, uint32_t *__restrict__ part)
{
    __shared__ uint32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < nparts; base += kT) {
        int q = base + threadIdx.x;
        uint32_t v = q < nparts ? part[q] : 0u;
        uint32_t tot;
        uint32_t ex = block_excl_scan(v, &tot);
        if (q < nparts) part[q] = ex + carry;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
}

__global__ void k_scan_final(long n, const uint32_t *__restrict__ a,
                             const uint32_t *__restrict__ part, uint32_t *__restrict__ out,
                             uint32_t total_M)
{
    long base = (long)blockIdx.x * kScanChunk + (long)threadIdx.x * kScanItems;
    uint32_t v[kScanItems], s = 0;
    for (int k = 0; k < kScanItems; k++) {
        long q = base + k;
        v[k] = q < n ? a[q] : 0u;
        s += v[k];
    }
    uint32_t ex = block_excl_scan(s, nullptr) + part[blockIdx.x];
    for (int k = 0; k < kScanItems; k++) {
        long q = base + k;
        if (q < n) out[q] = ex;
        ex += v[k];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) out[n] = total_M;
}

__global__ void k_place(int M, const uint32_t *__restrict__ key,
                        const uint32_t *__restrict__ cell_start, uint32_t *__restrict__ count,
                        uint32_t *__restrict__ tmp_ids)
{
    int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    uint32_t k = key[m];
    uint32_t slot = cell_start[k] + atomicSub(&count[k], 1u) - 1u;
    tmp_ids[slot] = (uint32_t)m;
}

// Deterministic rank inside the cell: ids ascending.
__global__ void k_rerank(int M, const uint32_t *__restrict__ key,
                         const uint32_t *__restrict__ cell_start,
                         const uint32_t *__restrict__ tmp_ids, uint32_t *__restrict__ ids)
{
    int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    uint32_t k = key[m], s = cell_start[k], e = cell_start[k + 1], r = 0;
    for (uint32_t t = s; t < e; t++) r += tmp_ids[t] < (uint32_t)m ? 1u : 0u;
    ids[s + r] = (uint32_t)m;
}

// list[0 .. *count): the active blocks, in no fixed order (each block's results
// are its own); *count zero before.  The kernels over active blocks run a
// resident grid over this list: with a CTA for every block of the grid the
// empty ones alone cost 5 us a launch at 1024^2 and 20 at 2048^2.
__global__ void k_block_active(int bnx, int bny, const uint32_t *__restrict__ bcount,
                               uint32_t *__restrict__ list, uint32_t *__restrict__ count)
{
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t any = 0;
    if (b < bnx * bny) {
        int bi = b % bnx, bj = b / bnx;
        for (int dj = -1; dj <= 1; dj++)
            for (int di = -1; di <= 1; di++) {
                int ii = bi + di, jj = bj + dj;
                if (ii >= 0 && ii < bnx && jj >= 0 && jj < bny) any |= bcount[jj * bnx + ii];
            }
    }
    const unsigned vote = __ballot_sync(0xffffffffu, any != 0), lane = threadIdx.x & 31;
    uint32_t at = 0;
    if (lane == 0 && vote) at = atomicAdd(count, (uint32_t)__popc(vote));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (any) list[at + __popc(vote & ((1u << lane) - 1u))] = (uint32_t)b;
}

// ------------------------------------------------------------ interpolation
// Eight lanes per marker: lanes 0-3 the rows of u's 4 x 4 stencil, 4-7 those
// of v's.  The even lanes form their component's factors along x, the odd
// ones those along y, passed on by shuffles; a lane sums its row, and the four
// rows meet in a fixed order.  Few markers are bound by the latency of one
// lane's chain (512: 21 us with one thread per marker, here 6), many by the FP64
// pipe (16384: 25 us with both factors in every lane, 17 so).
__global__ void __launch_bounds__(128)
k_interp(int M, int kernel, int nx, int ny, double ih, double x0, double y0,
         const double *__restrict__ u, const double *__restrict__ v,
         double *__restrict__ X, double *__restrict__ Y,
         double *__restrict__ U, double *__restrict__ V, double dt_move)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 7;
    const int m = min(t >> 3, M - 1);  // whole warps reach the shuffles
    const int b = lane & 3;
    const bool isv = lane >= 4;
    const double Xm = X[m], Ym = Y[m];
    const double sx = (Xm - x0) * ih - (isv ? 0.5 : 0.0), sy = (Ym - y0) * ih - (isv ? 0.0 : 0.5);
    const double fx = floor(sx), fy = floor(sy);
    const int i0 = (int)fx - 1, j = (int)fy - 1 + b;
    // the factors along x by the even lanes, those along y by the odd ones
    double q[4], px[4], py;
    phi4(kernel, b & 1 ? sy - fy : sx - fx, q);
    {
        const int e = threadIdx.x & 31 & ~3;  // the component's first lane
        double w[4];
#pragma unroll
        for (int a = 0; a < 4; a++) {
            px[a] = __shfl_sync(0xffffffffu, q[a], e);
            w[a] = __shfl_sync(0xffffffffu, q[a], e + 1);
        }
        py = b == 0 ? w[0] : (b == 1 ? w[1] : (b == 2 ? w[2] : w[3]));
    }
    const int W = isv ? nx : nx + 1, H = isv ? ny + 1 : ny;
    const double *f = isv ? v : u;
    double acc = 0.0;
    if (j >= 0 && j < H)
#pragma unroll
        for (int a = 0; a < 4; a++) {
            const int i = i0 + a;
            if (i >= 0 && i < W) acc += f[(long)j * W + i] * px[a];
        }
    acc *= py;
    // rows (0 + 1) + (2 + 3), in every lane of the component
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    const double other = __shfl_xor_sync(0xffffffffu, acc, 4);
    if ((t >> 3) >= M || lane != 0) return;
    if (U) U[m] = acc;
    if (V) V[m] = other;
    if (dt_move != 0.0) {
        X[m] = Xm + dt_move * acc;
        Y[m] = Ym + dt_move * other;
    }
}

// ------------------------------------------------------------ conventional spread
// A marker's record for the gather below (kTab doubles): the four factors
// along x and along y towards the x-faces and towards the y-faces, the two
// strengths f n ds / h^2, and the first face it reaches of each kind (two
// ints a double).  Two threads a marker, one for each kind of face.
constexpr int kTab = 20;
__global__ void __launch_bounds__(128)
k_spread_tab(int M, int kernel, double ih, double x0, double y0, const double *__restrict__ X,
             const double *__restrict__ Y, const double *__restrict__ fmag,
             const double *__restrict__ nxm, const double *__restrict__ nym,
             const double *__restrict__ ds, double *__restrict__ tab)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x, m = t >> 1, d = t & 1;
    if (m >= M) return;
    const double sx = (X[m] - x0) * ih - (d ? 0.5 : 0.0), sy = (Y[m] - y0) * ih - (d ? 0.0 : 0.5);
    const double fx = floor(sx), fy = floor(sy);
    double *o = tab + (long)m * kTab + 10 * d;
    double p[4];
    phi4(kernel, sx - fx, p);
    *(double2 *)(o + 0) = make_double2(p[0], p[1]);
    *(double2 *)(o + 2) = make_double2(p[2], p[3]);
    phi4(kernel, sy - fy, p);
    *(double2 *)(o + 4) = make_double2(p[0], p[1]);
    *(double2 *)(o + 6) = make_double2(p[2], p[3]);
    const int2 first = make_int2((int)fx - 1, (int)fy - 1);
    *(double2 *)(o + 8) = make_double2(fmag[m] * (d ? nym[m] : nxm[m]) * ds[m] * (ih * ih),
                                       __longlong_as_double(*(const long long *)&first));
}

// One block per 8 x 8 cells with a marker near, one thread per x-face left of
// and y-face below a cell: the markers of the 4 x 5 (x-faces) or 5 x 4
// (y-faces) cells that can reach the face, visited row by row in (cell, id)
// order, three multiplications and an addition each.  Evaluating the kernel
// per face and marker (two cosines, two divisions) on one thread per face of
// the whole grid took 624 us at 1024^2 with 16384 markers, this 38 us and the
// records 8 us.
__global__ void __launch_bounds__(2 * kBlk * kBlk)
k_spread_conv(int nx, int ny, int bnx, const uint32_t *__restrict__ blist,
              const uint32_t *__restrict__ nact,
              const uint32_t *__restrict__ cell_start, const uint32_t *__restrict__ ids,
              const double *__restrict__ tab, double *__restrict__ Fx, double *__restrict__ Fy)
{
    const int d = threadIdx.x / (kBlk * kBlk), c = threadIdx.x % (kBlk * kBlk);
    for (uint32_t ab = blockIdx.x; ab < *nact; ab += gridDim.x) {
        const int bl = (int)blist[ab], bj = bl / bnx, bi = bl - bj * bnx;
        const int i = bi * kBlk + c % kBlk, j = bj * kBlk + c / kBlk;
        if (i >= nx || j >= ny || (d == 0 ? i == 0 : j == 0)) continue;
        const int ia = max(i - 2, 0), ib = min(d ? i + 2 : i + 1, nx - 1);
        const int ja = max(j - 2, 0), jb = min(d ? j + 1 : j + 2, ny - 1);
        double acc = 0.0;
        for (int jj = ja; jj <= jb; jj++) {
            const uint32_t s = cell_start[(long)jj * nx + ia], e = cell_start[(long)jj * nx + ib + 1];
            for (uint32_t t = s; t < e; t++) {
                const double *o = tab + (long)ids[t] * kTab + 10 * d;
                const double2 cf = *(const double2 *)(o + 8);
                const long long bits = __double_as_longlong(cf.y);
                const int a = i - (int)(unsigned)bits, b = j - (int)(bits >> 32);
                if ((unsigned)a > 3u || (unsigned)b > 3u) continue;
                acc += cf.x * (o[a] * o[4 + b]);
            }
        }
        if (d == 0) Fx[(long)j * (nx + 1) + i] = acc;
        else Fy[(long)j * nx + i] = acc;
    }
}

// ------------------------------------------------------------ inside / outside
// Order-preserving key of the centre x of every column, x0 + (i + 0.5) h,
// formed once per context (the grid does not move; the same FP64 operations
// as the crossing test would use per cell).
__global__ void k_colkeys(int nx, double h, double x0, unsigned long long *__restrict__ ck)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nx) ck[i] = okey(x0 + ((double)i + 0.5) * h);
}

// One CTA per row: crossings of the row's centre line with every segment,
// sorted, then a crossing count per cell centre (the centres' keys from
// k_colkeys).  Writes H = chi.
__global__ void __launch_bounds__(kT)
k_rows_inside(int ndrops, int nx, double h, double x0, double y0, const double *__restrict__ X,
              const double *__restrict__ Y, const unsigned long long *__restrict__ ykey,
              const unsigned long long *__restrict__ colkey,
              const int32_t *__restrict__ next, const int32_t *__restrict__ drop_start,
              const ulonglong2 *__restrict__ dyk, double *__restrict__ H,
              uint32_t *__restrict__ flags)
{
    __shared__ unsigned long long xs[kMaxCross], srt[kMaxCross];
    __shared__ int nc;
    const int j = blockIdx.x;
    const double py = y0 + ((double)j + 0.5) * h;
    const unsigned long long kp = okey(py);
    if (threadIdx.x == 0) nc = 0;
    __syncthreads();
    // a drop entirely above (py < min Y) or not above (py >= max Y) the line
    // has no segment with one end above it and the other not
    for (int d = 0; d < ndrops; d++) {
        const ulonglong2 r = dyk[d];
        if (kp < r.x || kp >= r.y) continue;
        for (int m = drop_start[d] + threadIdx.x; m < drop_start[d + 1]; m += kT) {
            const int nm = next[m];
            if ((ykey[m] > kp) != (ykey[nm] > kp)) {
                double ax = X[m], ay = Y[m], bx = X[nm], by = Y[nm];
                double xc = ax + (py - ay) * (bx - ax) / (by - ay);
                int q = atomicAdd(&nc, 1);
                if (q < kMaxCross) xs[q] = okey(xc);
            }
        }
    }
    __syncthreads();
    int n = nc;
    if (n > kMaxCross) {
        if (threadIdx.x == 0) atomicOr(&flags[1], 1u);
        n = kMaxCross;
    }
    for (int q = threadIdx.x; q < n; q += kT) {
        unsigned long long v = xs[q];
        int r = 0;
        for (int t = 0; t < n; t++) r += (xs[t] < v || (xs[t] == v && t < q)) ? 1 : 0;
        srt[r] = v;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nx; i += kT) {
        const unsigned long long kx = colkey[i];  // okey(x0 + (i + 0.5) h)
        int lo = 0, hi = n;  // first index with srt > px
        while (lo < hi) {
            int mid = (lo + hi) >> 1;
            if (srt[mid] > kx) hi = mid; else lo = mid + 1;
        }
        H[(long)j * nx + i] = ((n - lo) & 1) ? 1.0 : 0.0;
    }
}

// ------------------------------------------------------------ band candidates
// Segments (start-marker ids) whose start marker lies within kSearch cells of
// an 8x8 block, gathered row by row and sorted ascending; with box, only those
// whose box (grid units) meets the block's cells.
__device__ int gather_candidates(int bi, int bj, int nx, int ny,
                                 const uint32_t *__restrict__ cell_start,
                                 const uint32_t *__restrict__ ids, uint32_t *cand,
                                 uint32_t *tmp, uint32_t *flags, const float4 *__restrict__ box = nullptr)
{
    constexpr int kRows = kBlk + 2 * kSearch;  // at most 22 rows: one warp
    __shared__ uint32_t rowoff[kRows + 1], rowsrc[kRows];
    __shared__ int total, nkeep;
    int kept = 0;
    const int ia = max(bi * kBlk - kSearch, 0), ib = min(bi * kBlk + kBlk - 1 + kSearch, nx - 1);
    const int ja = max(bj * kBlk - kSearch, 0), jb = min(bj * kBlk + kBlk - 1 + kSearch, ny - 1);
    const int nrows = jb - ja + 1;
    if (threadIdx.x < 32) {  // per row: first id and count, then an exclusive warp scan
        const int r = threadIdx.x;
        uint32_t src = 0, cnt = 0;
        if (r < nrows) {
            const long base = (long)(ja + r) * nx;
            src = cell_start[base + ia];
            cnt = cell_start[base + ib + 1] - src;
        }
        uint32_t inc = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
            if (r >= o) inc += v;
        }
        if (r < nrows) { rowoff[r] = inc - cnt; rowsrc[r] = src; }
        if (r == 31) { rowoff[nrows] = inc; total = (int)inc; nkeep = 0; }
    }
    __syncthreads();
    int n = total;
    if (n > kMaxCand) {
        if (threadIdx.x == 0) atomicOr(&flags[1], 1u);
        n = kMaxCand;
    }
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
        int r = 0;
        while (r + 1 < nrows && rowoff[r + 1] <= (uint32_t)q) r++;
        uint32_t v = ids[rowsrc[r] + (uint32_t)q - rowoff[r]];
        if (box) {  // rejected: an id above all others
            const float4 b = box[v];
            const float x0 = (float)(bi * kBlk), y0 = (float)(bj * kBlk);
            if (b.x > x0 + (float)kBlk || b.y < x0 || b.z > y0 + (float)kBlk || b.w < y0) v = 0xffffffffu;
            else kept++;
        }
        tmp[q] = v;
    }
    if (box) {
        kept = __reduce_add_sync(0xffffffffu, kept);
        if ((threadIdx.x & 31) == 0 && kept) atomicAdd(&nkeep, kept);
    }
    __syncthreads();
    const int m = box ? nkeep : n;
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
        uint32_t v = tmp[q];
        if (box && v == 0xffffffffu) continue;
        int r = 0;
        for (int t = 0; t < n; t++) r += tmp[t] < v ? 1 : 0;
        cand[r] = v;
    }
    __syncthreads();
    return m;
}

// Integral of clamp(y, 0, 1) dx along the part of the directed edge
// (x0, y0) -> (x1, y1) with 0 <= x <= 1.  The sum over the edges of a closed
// polygon is minus the signed area of its part inside the unit square (minus
// the boundary integral of y dx, y clamped), each point counted as often as
// the polygon winds around it: what clipping the polygon by the square's four
// sides in turn and the shoelace formula give.  Each edge stands alone, and a
// crossing's error enters scaled by the edge's own extent across it, so an
// edge nearly parallel to a side costs no accuracy.
__device__ __forceinline__ double edge_integral(double x0, double y0, double x1, double y1)
{
    const double dx = x1 - x0, dy = y1 - y0;
    const long long kTiny = __double_as_longlong(1e-30), kMask = 0x7fffffffffffffffLL;
    if ((__double_as_longlong(dx) & kMask) <= kTiny) return 0.0;
    // order as numbers, on integers (0, 1 and finite values)
    auto key = [](double x) {
        const long long b = __double_as_longlong(x);
        return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
    };
    auto clampd = [&](double t, double lo, double hi) {
        return key(t) < key(lo) ? lo : (key(t) > key(hi) ? hi : t);
    };
    // parameters t in [ta, tb] of the part with 0 <= x <= 1
    const double rx = recip_any(dx), tx0 = -x0 * rx, tx1 = (1.0 - x0) * rx;
    const bool px = __double_as_longlong(dx) > 0;
    const double ta = clampd(px ? tx0 : tx1, 0.0, 1.0), tb = clampd(px ? tx1 : tx0, ta, 1.0);
    // [u, v] of the part with 0 <= y <= 1; above: length of the part with y > 1
    double u, v, above;
    if ((__double_as_longlong(dy) & kMask) <= kTiny) {
        const bool hi = key(y0) > key(1.0), in = !hi && __double_as_longlong(y0) >= 0;
        u = ta;
        v = in ? tb : ta;
        above = hi ? tb - ta : 0.0;
    } else {
        const double ry = recip_any(dy), ty0 = -y0 * ry, ty1 = (1.0 - y0) * ry;
        const bool py = __double_as_longlong(dy) > 0;
        u = clampd(py ? ty0 : ty1, ta, tb);
        v = clampd(py ? ty1 : ty0, u, tb);
        above = py ? tb - v : u - ta;
    }
    return dx * fma(v - u, fma(0.5 * (u + v), dy, y0), above);
}

// The two integrals of which a strip's area is made, in the frame of cell
// (di, dj): along its inner offset line, v the line's corner at the segment's
// first marker (the one at the next marker 12 values on), and the difference of
// those along its sides on the normals, next marker less first.  Strip k has
// line(k + 1) - line(k) - rails(k), to the bit wherever a pair's area is formed.
__device__ __forceinline__ double line_integral(const double *v, double di, double dj)
{
    return edge_integral(v[0] - di, v[1] - dj, v[12] - di, v[13] - dj);
}
__device__ __forceinline__ double rail_integral(const double *v, double di, double dj)
{
    return edge_integral(v[12] - di, v[13] - dj, v[14] - di, v[15] - dj) -
           edge_integral(v[0] - di, v[1] - dj, v[2] - di, v[3] - dj);
}

__device__ __forceinline__ double strip_value(int k)
{
    // integral of the cosine kernel from -2 to the strip centre r = k - 2:
    // 0 for r = -2, 1 for r = 2, else 1/2 + r/4 + sin(pi r / 2) / (2 pi)
    constexpr double v[5] = {0.0, 0.25 - 1.0 / (2.0 * M_PI), 0.5, 0.75 + 1.0 / (2.0 * M_PI), 1.0};
    return v[k];
}

constexpr int kBT = kBlk * kBlk;  // one thread per cell of the block


// Position of the unit cell [i, i+1] x [j, j+1] against a half-plane
// n.x - c >= 0 evaluated in FP32 with a margin far above the FP32 error:
// -1 entirely outside, +1 entirely inside, 0 cut (or too close to tell).
__device__ __forceinline__ int cell_side(float4 l, float fi, float fj)
{
    const float base = l.x * fi + l.y * fj - l.z;
    const float hi = base + fmaxf(l.x, 0.0f) + fmaxf(l.y, 0.0f);
    const float lo = base + fminf(l.x, 0.0f) + fminf(l.y, 0.0f);
    const float m = 1e-2f * l.w;
    return hi < -m ? -1 : (lo > m ? 1 : 0);
}

// The band Heaviside runs in three launches so that the FP64 clipping, whose
// cost varies from cell to cell, is spread evenly over the GPU:
//  k_band_pairs (one CTA per active 8x8 block): every cell counts the
//    candidate segments whose slab (the four outer half-planes) may meet it,
//    tested in FP32; the block takes a range of the global pair list and
//    writes its (cell, segment) pairs, per cell in ascending segment order;
//  k_band_area (flat over the pair list): the areas of cell and strips;
//  k_band_sum (one CTA per active block): every cell sums its pairs in order,
//    H = sum A_k H_k + max(0, 1 - sum A_k) chi.
// Pair ranges are claimed with an atomic counter, so their place in the list
// varies from run to run, but each cell's pairs and their order do not, and a
// pair's area has the same bits on every route through k_band_area: H is
// deterministic.
constexpr int kPairT = 256, kPairSub = kPairT / kBT;  // 4 threads per cell
// Pairs of non-convex strips or strips along a grid axis (edge integrals, more
// FP64 work than the half-planes) are listed for the first kClipBlocks blocks
// of k_band_area, eight lanes a pair, and marked in the segment id's top bit.
constexpr int kClipBlocks = 128, kClipCap = 16384;
constexpr uint32_t kClipFlag = 0x80000000u;
constexpr int kStage = 256;  // candidates whose slab tests are staged in shared memory
__global__ void __launch_bounds__(kPairT)
k_band_pairs(int nx, int ny, int bnx, const uint32_t *__restrict__ blist,
             const uint32_t *__restrict__ nact, const uint32_t *__restrict__ cell_start, const uint32_t *__restrict__ ids,
             const float4 *__restrict__ slf, const uint8_t *__restrict__ scvx,
             const float4 *__restrict__ sbox, uint32_t cap, uint32_t *__restrict__ npairs,
             uint32_t *__restrict__ pseg, uint32_t *__restrict__ pcell, uint2 *__restrict__ crange,
             uint32_t *__restrict__ clip_list,
             uint32_t *__restrict__ flags)
{
    __shared__ uint32_t cand[kMaxCand], tmp[kMaxCand];
    __shared__ float4 s_box[kStage], s_l[4][kStage];
    __shared__ uint8_t s_cvx[kStage];
    __shared__ uint32_t cnt[kPairT], wsum[kPairT / 32 + 1];
    __shared__ uint32_t base;
    for (uint32_t ab = blockIdx.x; ab < *nact; ab += gridDim.x) {
        const int bl = (int)blist[ab], bj = bl / bnx, bi = bl - bj * bnx;
        __syncthreads();  // the block before is done with the shared arrays
        const int n = gather_candidates(bi, bj, nx, ny, cell_start, ids, cand, tmp, flags, sbox);
        const int ns = min(n, kStage);
        for (int q = threadIdx.x; q < ns; q += kPairT) {
            const uint32_t m = cand[q];
            s_box[q] = sbox[m];
            s_l[0][q] = slf[(long)m * 8 + 0];
            s_l[1][q] = slf[(long)m * 8 + 1];
            s_l[2][q] = slf[(long)m * 8 + 2];
            s_l[3][q] = slf[(long)m * 8 + 7];
            s_cvx[q] = scvx[m];
        }
        __syncthreads();
        const int t = threadIdx.x, cl = t / kPairSub, sub = t - cl * kPairSub;
        const int i = bi * kBlk + (cl % kBlk), j = bj * kBlk + (cl / kBlk);
        const bool live = i < nx && j < ny;
        const float fi = (float)i, fj = (float)j;
        auto meets = [&](int q) {
            const uint32_t m = cand[q];
            const bool st = q < kStage;
            const float4 b = st ? s_box[q] : sbox[m];
            if (b.x > fi + 1.0f || b.y < fi || b.z > fj + 1.0f || b.w < fj) return false;
            if (!(st ? s_cvx[q] : scvx[m])) return true;
            const float4 *L = slf + (long)m * 8;
            return cell_side(st ? s_l[0][q] : L[0], fi, fj) >= 0 &&
                   cell_side(st ? s_l[1][q] : L[1], fi, fj) >= 0 &&
                   cell_side(st ? s_l[2][q] : L[2], fi, fj) >= 0 &&
                   cell_side(st ? s_l[3][q] : L[7], fi, fj) <= 0;
        };
        // this thread's contiguous share of the (ascending) candidate list; its
        // test results are kept as bits in tmp (free after the gathering: four
        // words a thread, word w of thread t at tmp[w * kPairT + t]) for the
        // second pass, when the block has at most 4 x 128 candidates
        const int q0 = (n * sub) / kPairSub, q1 = (n * (sub + 1)) / kPairSub;
        static_assert(kMaxCand >= 4 * kPairT, "four words of tmp per thread");
        const bool keep = n <= kPairSub * 128;
        uint32_t c = 0;
        if (live) {
            uint32_t word = 0;
            for (int q = q0; q < q1; q++) {
                const bool mt = meets(q);
                c += mt ? 1u : 0u;
                if (keep) {
                    const int b = q - q0;
                    word |= (mt ? 1u : 0u) << (b & 31);
                    if ((b & 31) == 31 || q + 1 == q1) { tmp[(b >> 5) * kPairT + t] = word; word = 0; }
                }
            }
        }
        // exclusive scan over threads (cell-major, then share): warp scans, then
        // the warp totals
        const int lane = t & 31, warp = t >> 5;
        uint32_t incl = c;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        if (t == 0) {
            uint32_t acc = 0;
            for (int w = 0; w < kPairT / 32; w++) { const uint32_t v = wsum[w]; wsum[w] = acc; acc += v; }
            wsum[kPairT / 32] = acc;
            const uint32_t b0 = atomicAdd(npairs, acc);
            if (b0 > cap || acc > cap - b0) {
                atomicOr(&flags[1], 1u);
                base = 0xffffffffu;
            } else {
                base = b0;
            }
        }
        __syncthreads();
        const uint32_t excl = wsum[warp] + incl - c;
        cnt[t] = excl;
        __syncthreads();
        if (!live) continue;
        const long cidx = (long)j * nx + i;
        if (base == 0xffffffffu) {
            if (sub == 0) crange[cidx] = make_uint2(0u, 0u);
            continue;
        }
        if (sub == 0) {
            const uint32_t end = (cl + 1 < kBT) ? cnt[t + kPairSub] : wsum[kPairT / 32];
            crange[cidx] = make_uint2(base + excl, end - excl);
        }
        uint32_t o = base + excl;
        for (int q = q0; q < q1; q++)
            if (keep ? ((tmp[((q - q0) >> 5) * kPairT + t] >> ((q - q0) & 31)) & 1u) : meets(q)) {
                uint32_t seg = cand[q];
                // a pair of a non-convex strip goes to the clip list of
                // k_band_area (while it has room), marked in the id's top bit
                if (!(q < kStage ? s_cvx[q] : scvx[seg])) {
                    const uint32_t at = atomicAdd(npairs + 1, 1u);
                    if (at < kClipCap) { clip_list[at] = o; seg |= kClipFlag; }
                }
                pseg[o] = seg;
                pcell[o] = (uint32_t)cidx;
                o++;
            }
    }
}

// A bounding line of a strip in the cell's local frame (the cell is the unit
// square [0,1]^2): f(x, y) = a x + b y - c >= 0 inside, (a, b) a unit vector,
// with the reciprocals of a and b (0 where they vanish); on = false makes the
// slot constrain nothing.
struct CellLine {
    double a, b, c, ra, rb;
    bool on;
};

// l: a, b, c, 1/a, 1/b of the line in grid coordinates.
__device__ __forceinline__ CellLine cell_line(const double *l, double di, double dj, bool on)
{
    CellLine L;
    L.a = on ? l[0] : 0.0;
    L.b = on ? l[1] : 0.0;
    L.c = on ? l[2] - l[0] * di - l[1] * dj : -1.0;
    L.ra = on ? l[3] : 0.0;
    L.rb = on ? l[4] : 0.0;
    L.on = on;
    return L;
}

// Comparisons and selections of doubles on their bit patterns, in integer
// instructions: this part issues FP64 compares and min/max on its reduced
// FP64 pipe.  A double's 64-bit key, flipped below zero, orders like the
// number (finite values and infinities; -0 and +0 adjacent), so the maxima
// and minima below select exactly what fmax / fmin would.
__device__ __forceinline__ long long dkey(double x)
{
    const long long b = __double_as_longlong(x);
    return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
}
__device__ __forceinline__ bool dpos(double x)  // x > 0
{
    return __double_as_longlong(x) > 0;
}
__device__ __forceinline__ bool dneg(double x)  // x < 0
{
    const long long b = __double_as_longlong(x);
    return b < 0 && b != (long long)0x8000000000000000ULL;
}
__device__ __forceinline__ bool dzero(double x)  // x == 0
{
    return (__double_as_longlong(x) & 0x7fffffffffffffffLL) == 0;
}
// fmax(x, 0): x if it is positive (finite or +inf), else 0 (also for a NaN,
// as fmax gives for the empty interval -inf - (-inf))
__device__ __forceinline__ double dmax0(double x)
{
    const long long b = __double_as_longlong(x);
    return (b > 0 && b <= 0x7ff0000000000000LL) ? x : 0.0;
}

// Narrow [lo, hi] to the s with alpha + beta s >= 0, rbeta = 1 / beta (0 for
// beta = 0), which has beta's sign; q = -alpha rbeta where that is known.
__device__ __forceinline__ void narrow(double alpha, double rbeta, double q, double &lo, double &hi)
{
    if (dpos(rbeta)) { if (dkey(q) > dkey(lo)) lo = q; }
    else if (dneg(rbeta)) { if (dkey(q) < dkey(hi)) hi = q; }
    else if (dneg(alpha)) hi = -INFINITY;
}
__device__ __forceinline__ void narrow(double alpha, double rbeta, double &lo, double &hi)
{
    narrow(alpha, rbeta, -alpha * rbeta, lo, hi);
}

// Areas of the unit square cut by half-planes, by Green's theorem: area =
// 1/2 of the boundary integral of x dy - y dx.  On the square's bottom and
// left edges the integrand vanishes; the right edge contributes the length
// of its part inside every half-plane, and so does the top edge; a line,
// traversed with its inside on the left from P(s0) to P(s1), P(s) =
// c (a, b) + s (b, -a), contributes (s1 - s0) cross(P(0), (b, -a)) =
// -(s1 - s0) c.  Each piece is an interval cut down by the other
// constraints.  The result equals clipping the square by the half-planes in
// turn and taking the shoelace area, up to rounding.
//
// A cell meets the two normal edges of a segment and one offset line at a
// time: the pieces' intervals under the normal edges alone are formed once
// (RailCut, which also gives the area a0 of the cell between the normal
// edges) and each cutting offset line only narrows them further.

// A line lying on the top or right edge with the square on its inner side
// traces the same boundary as that edge: its own piece is not counted.
__device__ __forceinline__ bool on_edge(const CellLine &L)
{
    return (dzero(L.a) && dneg(L.b) && dzero(L.b - L.c)) || (dzero(L.b) && dneg(L.a) && dzero(L.a - L.c));
}

// Interval of line L's own piece inside the unit square; (px, py) = c (a, b).
// The FP64 pipe bounds the areas, so the far side's crossing comes from the
// near one's ((1 - px) / b = 1 / b - px / b) and a determinant's sign from its
// reciprocal (170k pairs at 1024^2: 1.19 -> 0.97 million FP64 warp
// instructions, 106 -> 88 us).
__device__ __forceinline__ void square_piece(const CellLine &L, double px, double py, double &lo,
                                             double &hi)
{
    lo = -INFINITY; hi = INFINITY;
    const double qx = -px * L.rb, qy = py * L.ra;
    narrow(px, L.rb, qx, lo, hi);                                       // x >= 0
    if (dzero(L.rb)) narrow(1.0 - px, 0.0, 0.0, lo, hi);
    else narrow(0.0, -L.rb, qx + L.rb, lo, hi);                         // x <= 1
    narrow(py, -L.ra, qy, lo, hi);                                      // y >= 0
    if (dzero(L.ra)) narrow(1.0 - py, 0.0, 0.0, lo, hi);
    else narrow(0.0, L.ra, qy - L.ra, lo, hi);                          // y <= 1
}

// Narrow line J's piece, through (px, py), by half-plane I (rIJ = 1 / (a_I b_J
// - b_I a_J)).
__device__ __forceinline__ void cross_narrow(const CellLine &I, double px, double py, double rIJ,
                                             double &lo, double &hi)
{
    narrow(fma(I.a, px, fma(I.b, py, -I.c)), rIJ, lo, hi);
}

struct RailCut {
    double Rlo, Rhi, Tlo, Thi;  // right edge (y) and top edge (x) inside both normal edges
    double Plo[2], Phi[2];      // normal-edge pieces (s)
    double px[2], py[2];        // c (a, b) of the normal edges
    bool piece[2];              // normal edge j cuts the cell and has a piece of its own
};

// L[0], L[1]: the normal edges (on = cuts the cell); r01 = 1 / D_01.
__device__ __forceinline__ void rail_cut(const CellLine *L, double r01, RailCut &rc)
{
    rc.Rlo = 0.0; rc.Rhi = 1.0; rc.Tlo = 0.0; rc.Thi = 1.0;
#pragma unroll
    for (int j = 0; j < 2; j++) {
        narrow(L[j].a - L[j].c, L[j].rb, rc.Rlo, rc.Rhi);  // x = 1
        narrow(L[j].b - L[j].c, L[j].ra, rc.Tlo, rc.Thi);  // y = 1
    }
#pragma unroll
    for (int j = 0; j < 2; j++) {
        rc.piece[j] = L[j].on && !on_edge(L[j]);
        rc.Plo[j] = 0.0; rc.Phi[j] = 0.0;
        if (!rc.piece[j]) continue;
        rc.px[j] = L[j].c * L[j].a; rc.py[j] = L[j].c * L[j].b;
        square_piece(L[j], rc.px[j], rc.py[j], rc.Plo[j], rc.Phi[j]);
        if (L[1 - j].on)
            cross_narrow(L[1 - j], rc.px[j], rc.py[j], j == 1 ? r01 : -r01, rc.Plo[j], rc.Phi[j]);
    }
}

// Area of the cell between the normal edges (no offset line).
__device__ __forceinline__ double rail_area(const CellLine *L, const RailCut &rc)
{
    double acc = dmax0(rc.Rhi - rc.Rlo);
    acc += dmax0(rc.Thi - rc.Tlo);
#pragma unroll
    for (int j = 0; j < 2; j++)
        if (rc.piece[j]) acc -= L[j].c * dmax0(rc.Phi[j] - rc.Plo[j]);
    return 0.5 * acc;
}

// Area of the cell between the normal edges and inside offset line O;
// r0O, r1O = 1 / D_0O, 1 / D_1O.
__device__ __forceinline__ double rail_line_area(const CellLine *L, const RailCut &rc,
                                                 const CellLine &O, double r0O, double r1O)
{
    double lo = rc.Rlo, hi = rc.Rhi, acc;
    narrow(O.a - O.c, O.rb, lo, hi);
    acc = dmax0(hi - lo);
    lo = rc.Tlo; hi = rc.Thi;
    narrow(O.b - O.c, O.ra, lo, hi);
    acc += dmax0(hi - lo);
#pragma unroll
    for (int j = 0; j < 2; j++) {
        if (!rc.piece[j]) continue;
        lo = rc.Plo[j]; hi = rc.Phi[j];
        cross_narrow(O, rc.px[j], rc.py[j], j == 0 ? -r0O : -r1O, lo, hi);  // D_Oj = -D_jO
        acc -= L[j].c * dmax0(hi - lo);
    }
    if (!on_edge(O)) {
        const double px = O.c * O.a, py = O.c * O.b;
        square_piece(O, px, py, lo, hi);
#pragma unroll
        for (int i = 0; i < 2; i++)
            if (L[i].on) cross_narrow(L[i], px, py, i == 0 ? r0O : r1O, lo, hi);
        acc -= O.c * dmax0(hi - lo);
    }
    return 0.5 * acc;
}

// Area of cell (ci, cj) inside each of the five strips of segment m, weighted
// sum and total.  Convex, well-conditioned strips: P is the cell square cut by the slab's normal
// edges that cross it (area a0), S_o = area(P on the inner side of offset line
// o) for o = 0..5 (a0 or 0 when the FP32 test finds the line clear of the
// cell, else rail_line_area in FP64, the cut lines in ascending o), and strip
// k has area S_k - S_k+1.  Other
// segments (folded strips, lines within 0.001 rad of a grid axis): the edge
// integrals of every quadrilateral.
__device__ __forceinline__ void pair_area(uint32_t m, int ci, int cj, const double *__restrict__ sl,
                                          const float4 *__restrict__ slf,
                                          const uint8_t *__restrict__ scvx,
                                          const double *__restrict__ sv,
                                          const float4 *__restrict__ sb5, const double *Hk,
                                          double &acc, double &cov)
{
    const float gi = (float)ci, gj = (float)cj;
    const double di = (double)ci, dj = (double)cj;
    acc = 0.0;
    cov = 0.0;
    if (!scvx[m]) {
        const double *v = sv + (long)m * 24;
        double line = 0.0;
        bool have = false;  // line is the strip's inner one
        for (int k = 0; k < 5; k++, v += 2) {
            const float4 b = sb5[(long)m * 5 + k];
            const bool hit = !(b.x > gi + 1.0f || b.y < gi || b.z > gj + 1.0f || b.w < gj);
            if (hit) {
                if (!have) line = line_integral(v, di, dj);
                const double next = line_integral(v + 2, di, dj);
                const double A = next - line - rail_integral(v, di, dj);
                acc += A * Hk[k];
                cov += A;
                line = next;
            }
            have = hit;
        }
        return;
    }
    const float4 *Lf = slf + (long)m * 8;
    const double *Ld = sl + (long)m * kSegLine;
    int side[8];
#pragma unroll
    for (int q = 0; q < 8; q++) side[q] = cell_side(Lf[q], gi, gj);
    // the normal edges; one that does not cut the cell constrains nothing
    CellLine L[2];
#pragma unroll
    for (int q = 0; q < 2; q++) L[q] = cell_line(Ld + 5 * q, di, dj, side[q] == 0);
    RailCut rc;
    rail_cut(L, Ld[40], rc);
    const double a0 = (side[0] == 0 || side[1] == 0) ? rail_area(L, rc) : 1.0;
    // lines clear of the cell first; then the cut ones, lowest first: step
    // k of the loop takes the k-th cut line of every lane's pair, so the
    // FP64 area runs on converged warps whichever lines the pairs cut
    double S[6];
    unsigned cut = 0;
#pragma unroll
    for (int o = 0; o < 6; o++) {
        S[o] = side[2 + o] > 0 ? a0 : 0.0;
        if (side[2 + o] == 0) cut |= 1u << o;
    }
    while (cut) {
        const int o = __ffs(cut) - 1;
        cut &= cut - 1;
        const CellLine O = cell_line(Ld + 5 * (2 + o), di, dj, true);
        const double v = rail_line_area(L, rc, O, Ld[41 + 2 * o], Ld[42 + 2 * o]);
#pragma unroll
        for (int r = 0; r < 6; r++)
            if (r == o) S[r] = v;
    }
    // strip k has S[k] - S[k+1]; strip 0's value is zero
#pragma unroll
    for (int k = 1; k < 5; k++) acc = fma(S[k] - S[k + 1], Hk[k], acc);
    cov = S[0] - S[5];
}

// The first kClipBlocks blocks take the listed pairs, a group of 8 lanes per
// pair: lane o < 6 integrates along offset line o, lane k < 5 also along the
// normals' pieces between lines k and k + 1, which together give strip k;
// lane 0 sums the strips in order.  Being dispatched first, their longer FP64
// chains overlap the rest.  The other blocks take one pair per thread (flat
// over the list), skipping the listed ones.  (Strips clipped side by side of
// the square, 1024 pairs listed: 42 us for one drop of 128 markers, 125 us for
// 64 of 256; then 20 and 104, and 88 with the rule at square_piece.)
__global__ void __launch_bounds__(256)
k_band_area(int nx, const uint32_t *__restrict__ npairs, uint32_t cap,
            const uint32_t *__restrict__ pseg, const uint32_t *__restrict__ pcell,
            const uint32_t *__restrict__ clip_list,
            const double *__restrict__ sl, const float4 *__restrict__ slf,
            const uint8_t *__restrict__ scvx, const double *__restrict__ sv,
            const float4 *__restrict__ sb5, double *__restrict__ pacc, double *__restrict__ pcov)
{
    const uint32_t total = min(*npairs, cap);
    double Hk[5];
    for (int k = 0; k < 5; k++) Hk[k] = strip_value(k);
    if (blockIdx.x < kClipBlocks) {
        const uint32_t nc = min(npairs[1], (uint32_t)kClipCap);
        const int k = threadIdx.x % 8;
        // every lane of a warp reaches the shuffles below; a group past the
        // list's end (the same for its 8 lanes) only does no work
        for (uint32_t i0 = blockIdx.x * 32; i0 < nc; i0 += kClipBlocks * 32) {
            const uint32_t idx = i0 + threadIdx.x / 8;
            const bool live = idx < nc;
            const uint32_t p = live ? clip_list[idx] : 0u;
            const uint32_t m = live ? (pseg[p] & ~kClipFlag) : 0u, cell = live ? pcell[p] : 0u;
            const int cj = (int)(cell / (uint32_t)nx), ci = (int)(cell - (uint32_t)cj * (uint32_t)nx);
            const float gi = (float)ci, gj = (float)cj;
            const double di = (double)ci, dj = (double)cj;
            double line = 0.0, rails = 0.0;
            bool hit = false;
            if (live && k < 6) {
                const double *v = sv + (long)m * 24 + 2 * k;
                line = line_integral(v, di, dj);
                if (k < 5) {
                    rails = rail_integral(v, di, dj);
                    const float4 bb = sb5[(long)m * 5 + k];
                    hit = !(bb.x > gi + 1.0f || bb.y < gi || bb.z > gj + 1.0f || bb.w < gj);
                }
            }
            const double next = __shfl_down_sync(0xffffffffu, line, 1, 8);
            const double A = hit ? next - line - rails : 0.0;
            double acc = 0.0, cov = 0.0;
#pragma unroll
            for (int s = 0; s < 5; s++) {
                const double As = __shfl_sync(0xffffffffu, A, s, 8);
                acc += As * Hk[s];
                cov += As;
            }
            if (live && k == 0) { pacc[p] = acc; pcov[p] = cov; }
        }
        return;
    }
    const uint32_t stride = (gridDim.x - kClipBlocks) * blockDim.x;
    for (uint32_t p = (blockIdx.x - kClipBlocks) * blockDim.x + threadIdx.x; p < total; p += stride) {
        const uint32_t seg = pseg[p];
        if (seg & kClipFlag) continue;
        const uint32_t cell = pcell[p];
        const int cj = (int)(cell / (uint32_t)nx), ci = (int)(cell - (uint32_t)cj * (uint32_t)nx);
        double acc, cov;
        pair_area(seg, ci, cj, sl, slf, scvx, sv, sb5, Hk, acc, cov);
        pacc[p] = acc;
        pcov[p] = cov;
    }
}

__global__ void __launch_bounds__(kBT)
k_band_sum(int nx, int ny, int bnx, const uint32_t *__restrict__ blist,
           const uint32_t *__restrict__ nact, const uint2 *__restrict__ crange,
           const double *__restrict__ pacc, const double *__restrict__ pcov, double *__restrict__ H)
{
    for (uint32_t ab = blockIdx.x; ab < *nact; ab += gridDim.x) {
        const int bl = (int)blist[ab], bj = bl / bnx, bi = bl - bj * bnx;
        const int i = bi * kBlk + (threadIdx.x % kBlk), j = bj * kBlk + (threadIdx.x / kBlk);
        if (i >= nx || j >= ny) continue;
        const long cidx = (long)j * nx + i;
        const uint2 r = crange[cidx];
        double acc = 0.0, cov = 0.0;
        for (uint32_t p = r.x; p < r.x + r.y; p++) { acc += pacc[p]; cov += pcov[p]; }
        double unc = 1.0 - cov;
        if (unc < 0.0) unc = 0.0;
        H[cidx] = acc + unc * H[cidx];
    }
}

// Irrotational face force F = f_face (H_ij - H_nb) / h on the x-face left of
// and the y-face below every cell of an active block; f_face from the nearest
// segment (closest point clamped to the segment, ties to the lower id),
// linear in the segment parameter between its two markers.  One thread per
// face: the block's 128 faces are tested for dH != 0, the faces with work
// are packed into a list (so the FP64 part runs on full warps), and each of
// those screens the block's candidates (staged in shared memory in FP32),
// lists the survivors in ascending id and then evaluates them exactly in
// FP64 in that order: step k of the evaluation takes the k-th survivor of
// every face at once, so the FP64 instructions run on converged warps (a
// face with more than kNear survivors evaluates them in a pass of its own).
constexpr int kIrrT = 2 * kBT;  // one thread per face of the block
constexpr int kNear = 8;        // survivors listed per face
__global__ void __launch_bounds__(kIrrT)
k_spread_irrot(int nx, int ny, double ih, int bnx, const uint32_t *__restrict__ blist,
               const uint32_t *__restrict__ nact,
               const uint32_t *__restrict__ cell_start, const uint32_t *__restrict__ ids,
               const int32_t *__restrict__ next, const double *__restrict__ gx,
               const double *__restrict__ gy, const double *__restrict__ sinv,
               const float *__restrict__ gxf, const float *__restrict__ gyf,
               const double *__restrict__ fmag, const double *__restrict__ H,
               double *__restrict__ Fx, double *__restrict__ Fy, uint32_t *__restrict__ flags)
{
    __shared__ uint32_t cand[kMaxCand], tmp[kMaxCand];
    __shared__ float4 seg[kMaxCand];   // FP32 candidate segments: start, direction
    __shared__ float seg_il[kMaxCand]; // 1 / |direction|^2
    __shared__ uint8_t work[kIrrT];     // faces with dH != 0, packed
    __shared__ double wdH[kIrrT];
    __shared__ uint16_t near_q[kNear][kIrrT];  // survivors of the FP32 screen, per face
    __shared__ int nwork;
    for (uint32_t ab = blockIdx.x; ab < *nact; ab += gridDim.x) {
        const int bl = (int)blist[ab], bj = bl / bnx, bi = bl - bj * bnx;
        __syncthreads();  // the block before is done with the shared arrays
        const int n = gather_candidates(bi, bj, nx, ny, cell_start, ids, cand, tmp, flags);
        for (int q = threadIdx.x; q < n; q += blockDim.x) {
            const int m = (int)cand[q], nm = next[m];
            const float ax = gxf[m], ay = gyf[m], ex = gxf[nm] - ax, ey = gyf[nm] - ay;
            seg[q] = make_float4(ax, ay, ex, ey);
            seg_il[q] = 1.0f / (ex * ex + ey * ey);
        }
        if (threadIdx.x == 0) nwork = 0;
        __syncthreads();
        // face f: dir = f / 64 (0: x-face left of the cell, 1: y-face below), cell f % 64
        auto face = [&](int f, int &dir, int &i, int &j) {
            dir = f / kBT;
            const int c = f - dir * kBT;
            i = bi * kBlk + (c % kBlk);
            j = bj * kBlk + (c / kBlk);
        };
        {
            const int f = threadIdx.x;
            int dir, i, j;
            face(f, dir, i, j);
            if (i < nx && j < ny && !(dir == 0 && i == 0) && !(dir == 1 && j == 0)) {
                const double dH = dir == 0 ? H[(long)j * nx + i] - H[(long)j * nx + i - 1]
                                           : H[(long)j * nx + i] - H[(long)(j - 1) * nx + i];
                if (dH != 0.0) {
                    const int w = atomicAdd(&nwork, 1);
                    work[w] = (uint8_t)f;
                    wdH[w] = dH;
                } else if (dir == 0) {
                    Fx[(long)j * (nx + 1) + i] = 0.0;
                } else {
                    Fy[(long)j * nx + i] = 0.0;
                }
            }
        }
        __syncthreads();
        if ((int)threadIdx.x >= nwork) continue;
        int dir, i, j;
        face(work[threadIdx.x], dir, i, j);
        const double dH = wdH[threadIdx.x];
        const double qx = dir == 0 ? (double)i : (double)i + 0.5;
        const double qy = dir == 0 ? (double)j + 0.5 : (double)j;
        // FP32 screen: for faces within the band (distance below ~4 cells) and
        // coordinates below 2^12 cells the FP32 squared distances carry an error
        // below 2e-3 (grid units), so the exact nearest segment is among those
        // within best + 0.01 of the FP32 minimum.
        const float fqx = d2f_rn(qx), fqy = d2f_rn(qy);
        auto d2f = [&](int q) {
            const float4 sg = seg[q];
            float t = ((fqx - sg.x) * sg.z + (fqy - sg.y) * sg.w) * seg_il[q];
            t = fminf(fmaxf(t, 0.0f), 1.0f);
            const float dx = sg.x + t * sg.z - fqx, dy = sg.y + t * sg.w - fqy;
            return dx * dx + dy * dy;
        };
        float best32 = INFINITY;
        for (int q = 0; q < n; q++) best32 = fminf(best32, d2f(q));
        const float lim = best32 + 0.01f;
        static_assert(kMaxCand <= 65536, "candidate index in 16 bits");
        int cnt = 0;
        for (int q = 0; q < n; q++)
            if (!(d2f(q) > lim)) {
                if (cnt < kNear) near_q[cnt][threadIdx.x] = (uint16_t)q;
                cnt++;
            }
        double best = INFINITY, fb = 0.0;
        auto eval = [&](int q) {
            const int m = (int)cand[q], nm = next[m];
            const double ax = gx[m], ay = gy[m];
            const double ex = gx[nm] - ax, ey = gy[nm] - ay;
            double t = ((qx - ax) * ex + (qy - ay) * ey) * sinv[m];
            if (t < 0.0) t = 0.0;
            if (t > 1.0) t = 1.0;
            const double dx = ax + t * ex - qx, dy = ay + t * ey - qy;
            const double d2 = dx * dx + dy * dy;
            if (d2 < best) { best = d2; fb = (1.0 - t) * fmag[m] + t * fmag[nm]; }
        };
        if (cnt <= kNear) {
            for (int k = 0; k < cnt; k++) eval(near_q[k][threadIdx.x]);
        } else {
            for (int q = 0; q < n; q++)
                if (!(d2f(q) > lim)) eval(q);
        }
        const double F = fb * dH * ih;
        if (dir == 0) Fx[(long)j * (nx + 1) + i] = F;
        else Fy[(long)j * nx + i] = F;
    }
}

// ------------------------------------------------------------ B-spline
// Section 4: relocation along a periodic cubic B-spline fitted to each drop
// by least squares: chord-length parameters, g = round(L / 1.5h) spans
// (4 <= g <= n), normal equations accumulated in ascending marker order and
// solved by block elimination, arc length by 8-point Gauss-Legendre per span,
// at most 12 Newton steps per new marker.  Two kernels: the fit (one CTA per
// drop) and the placement of the new markers over the whole grid.
//
// The knots t_k = k tau are uniform, so on span q (u = s / tau - q in [0, 1])
// the four cubic B-splines that do not vanish, of control points q-3 .. q,
// are (1-u)^3/6, (3u^3 - 6u^2 + 4)/6, (-3u^3 + 3u^2 + 3u + 1)/6, u^3/6.
__device__ __forceinline__ int bspl_span(double s, double tau, int g)
{
    int q = (int)floor(s / tau);
    if (q > g - 1) q = g - 1;
    if (q < 0) q = 0;
    return q;
}

__constant__ double cGLX[8] = {-0.9602898564975363, -0.7966664774136267,
                               -0.5255324099163290, -0.1834346424956498,
                               0.1834346424956498,  0.5255324099163290,
                               0.7966664774136267,  0.9602898564975363};
__constant__ double cGLW[8] = {0.1012285362903763, 0.2223810344533745,
                               0.3137066458778873, 0.3626837833783620,
                               0.3626837833783620, 0.3137066458778873,
                               0.2223810344533745, 0.1012285362903763};

// The curve on span q: its control points q-3 .. q (cyclic) and its
// derivative in u, a quadratic d0 + u (d1 + u d2) per coordinate, so that a
// speed costs six FP64 operations before its square root.
struct SpanCurve {
    double x[4], y[4], dx[3], dy[3];
};
__device__ __forceinline__ SpanCurve span_curve(const double *cx, const double *cy, int g, int q)
{
    SpanCurve c;
    for (int r = 0; r < 4; r++) {
        const int k = q - 3 + r, id = k < 0 ? k + g : k;  // q <= g - 1
        c.x[r] = cx[id];
        c.y[r] = cy[id];
    }
    c.dx[0] = 0.5 * (c.x[2] - c.x[0]);
    c.dy[0] = 0.5 * (c.y[2] - c.y[0]);
    c.dx[1] = (c.x[0] - c.x[1]) + (c.x[2] - c.x[1]);
    c.dy[1] = (c.y[0] - c.y[1]) + (c.y[2] - c.y[1]);
    c.dx[2] = 0.5 * fma(3.0, c.x[1] - c.x[2], c.x[3] - c.x[0]);
    c.dy[2] = 0.5 * fma(3.0, c.y[1] - c.y[2], c.y[3] - c.y[0]);
    return c;
}
__device__ __forceinline__ double speed2(const SpanCurve &c, double u)
{
    const double vx = fma(u, fma(u, c.dx[2], c.dx[1]), c.dx[0]);
    const double vy = fma(u, fma(u, c.dy[2], c.dy[1]), c.dy[0]);
    return fma(vx, vx, vy * vy);
}
// out[k] = in[0] + ... + in[k-1], k = 0 .. n, of values >= 0, by the block's
// kT threads; returns the total.  The sums run on 64-bit integers at a power
// of two that keeps n times the largest value below 2^62: exact, so they do
// not depend on the split and ascend with k, and off the FP64 pipe, where one
// thread's running sum took 64 cycles a value.  A value that is not finite
// makes every sum NaN.  scr: scratch of 12 8-byte words.
__device__ double block_scan(int n, const double *in, double *out, void *scr)
{
    long long *ts = (long long *)scr;
    unsigned *hs = (unsigned *)(ts + kT / 32);
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int per = (n + kT - 1) / kT, k0 = min(n, (int)threadIdx.x * per), k1 = min(n, k0 + per);
    unsigned hi = 0;
    for (int k = k0; k < k1; k++) hi = max(hi, (unsigned)__double2hiint(in[k]));
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) hs[wp] = hi;
    __syncthreads();
    for (int w = 0; w < kT / 32; w++) hi = max(hi, hs[w]);
    // every value is below 2^(E - 1022), n below 2^nb
    const int E = (int)(hi >> 20), nb = 32 - __clz(n);
    const int f = max(1, min(2045, 2107 - E - nb));  // exponent field of the scale
    const double sc = __longlong_as_double((long long)f << 52);
    const double inv = E >= 2047 ? __longlong_as_double(0x7ff8000000000000LL)
                                 : __longlong_as_double((long long)(2046 - f) << 52);
    long long s = 0;
    for (int k = k0; k < k1; k++) s += __double2ll_rn(in[k] * sc);
    long long inc = s;
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) ts[wp] = inc;
    __syncthreads();
    long long base = 0, tot = 0;
    for (int w = 0; w < kT / 32; w++) {
        if (w == wp) base = tot;
        tot += ts[w];
    }
    long long run = base + inc - s;
    for (int k = k0; k < k1; k++) {
        out[k] = (double)run * inv;
        run += __double2ll_rn(in[k] * sc);
    }
    const double total = (double)tot * inv;
    if (threadIdx.x == 0) out[n] = total;
    __syncthreads();
    return total;
}

// The normal equations' matrix is a cyclic band of half-width 3.  Its last w
// rows (w = 3 .. 5, so that 3 m rows remain) are the border; the other rows
// form a chain of m 3 x 3 blocks, each coupled to its two neighbours, whose
// ends couple to the border.  A chain block holds, per row, the right-hand
// sides x and y and its (at most five) border entries, seven columns that are
// solved together; its diagonal block, symmetric, then its Cholesky factor
// (diagonal as reciprocals); its coupling to the next chain block still
// there; and, once eliminated, that to the one before.
constexpr int kBR = 0, kBD = 21, kBU = 27, kBW = 36, kBlkLen = 45;
constexpr int kBorder = 5;
constexpr int kEndLen = 7 * kBorder;  // the border's rows: x, y, matrix

// Solves the system by odd-even elimination of the chain (every second block
// that is left goes at once, log2 m times), then the border's 5 x 5 rest,
// then back: 3 log2 m short parallel steps in place of g serial columns and
// 2 g serial rows, each a chain of FP64 latencies (64 cycles an instruction
// on this part; 516 us of the fit for g about 130).  A block elimination in the
// order of a symmetric permutation is a Cholesky factorisation of the
// permuted matrix, as stable as the row by row one.  S: the border's rows, scr: scratch of 30
// values.  Sets *bad if a pivot is not positive.
__device__ void ring_solve(double *blk, int m, int g, double *S, double *scr, double *cx, double *cy,
                           int *bad)
{
    const int t = threadIdx.x;
    // the border entries of the first and the last block, (row, entry)
    double *C0 = scr, *C1 = scr + 3 * kBorder;
    if (m > 0 && t < 2 * 3 * kBorder) {
        const int e = t / (3 * kBorder), k = t % (3 * kBorder), r = k / kBorder, c = k % kBorder;
        scr[t] = blk[kBlkLen * (e ? m - 1 : 0) + kBR + 7 * r + 2 + c];
    }
    __syncthreads();
    int st = 1;
    for (; st <= m; st <<= 1) {
        // eliminated: odd multiples of st among positions 1 .. m; sixteen
        // lanes a block, each with the factor of the block's own 3 x 3 and
        // one of the 13 columns [to the left | to the right | right-hand sides]
        const int ne = (m / st + 1) >> 1;
        for (int e0 = 0; e0 < ne; e0 += kT / 16) {
            const int e = e0 + (t >> 4), lane = t & 15, pos = (2 * e + 1) * st;
            double *B = blk + kBlkLen * (pos - 1);
            double *dst = nullptr;
            int ds = 3;
            double r0 = 0, l10 = 0, r1 = 0, l20 = 0, l21 = 0, r2 = 0, v0 = 0, v1 = 0, v2 = 0;
            if (e < ne) {
                const double *D = B + kBD;
                const double d11 = D[2], d21 = D[4], d22 = D[5];
                const double s0 = D[0];
                l10 = D[1]; l20 = D[3];
                r0 = rsqrt_any(s0);
                l10 *= r0; l20 *= r0;
                const double s1 = fma(-l10, l10, d11);
                r1 = rsqrt_any(s1);
                l21 = fma(-l20, l10, d21) * r1;
                const double s2 = fma(-l21, l21, fma(-l20, l20, d22));
                r2 = rsqrt_any(s2);
                if (lane == 13 && !(s0 > 0.0 && s1 > 0.0 && s2 > 0.0)) *bad = 1;
                const double *src = nullptr;
                int ss = 3;
                if (lane < 3) {
                    if (pos > st) { src = B - kBlkLen * st + kBU + 3 * lane; ss = 1; dst = B + kBW + lane; }
                } else if (lane < 6) {
                    if (pos + st <= m) { dst = B + kBU + lane - 3; src = dst; }
                } else if (lane < 13) {
                    dst = B + kBR + lane - 6; src = dst; ss = ds = 7;
                }
                if (src) {
                    v0 = src[0] * r0;
                    v1 = fma(-l10, v0, src[ss]) * r1;
                    v2 = fma(-l21, v1, fma(-l20, v0, src[2 * ss])) * r2;
                }
            }
            __syncwarp();
            if (dst) {
                dst[0] = v0; dst[ds] = v1; dst[2 * ds] = v2;
            } else if (lane == 13 && e < ne) {
                double *D = B + kBD;
                D[0] = r0; D[1] = l10; D[2] = r1; D[3] = l20; D[4] = l21; D[5] = r2;
            }
        }
        __syncthreads();
        // the blocks left over: their 36 entries less the products of the
        // columns of the neighbours just eliminated, one entry a thread
        const int ns = (m / st) >> 1;
        for (int it = t; it < 36 * ns; it += kT) {
            const int sv = it / 36, k = it - 36 * sv, pos = 2 * (sv + 1) * st;
            double *B = blk + kBlkLen * (pos - 1);
            const double *e1 = B - kBlkLen * st;
            const double *e2 = pos + st <= m ? B + kBlkLen * st : nullptr;
            int r, oc, ow, q = 3;  // row; the column in e1 and in e2, its stride
            if (k < kBD) {
                r = k / 7; oc = ow = kBR + k - 7 * r; q = 7;
            } else if (k < kBU) {
                const int d = k - kBD;
                r = d >= 3 ? 2 : (d >= 1 ? 1 : 0);
                oc = kBU + d - r * (r + 1) / 2; ow = oc - kBU + kBW;
            } else {
                if (pos + 2 * st > m) continue;
                r = (k - kBU) / 3; ow = kBU + (k - kBU) - 3 * r; oc = -1;
            }
            double v = oc < 0 ? 0.0 : B[k];
            if (oc >= 0)
                for (int i = 0; i < 3; i++) v = fma(-e1[kBU + 3 * i + r], e1[oc + q * i], v);
            if (e2)
                for (int i = 0; i < 3; i++) v = fma(-e2[kBW + 3 * i + r], e2[ow + q * i], v);
            B[k] = v;
        }
        __syncthreads();
    }
    for (st >>= 1; st >= 1; st >>= 1) {
        const int ne = (m / st + 1) >> 1;
        for (int it = t; it < 8 * ne; it += kT) {
            const int e = it >> 3, c = it & 7, pos = (2 * e + 1) * st;
            if (c == 7) continue;
            double *B = blk + kBlkLen * (pos - 1), *R = B + kBR + c;
            double y0 = R[0], y1 = R[7], y2 = R[14];
            auto sub = [&](const double *W, const double *x) {
                for (int i = 0; i < 3; i++) {
                    const double xi = x[7 * i];
                    y0 = fma(-W[i], xi, y0);
                    y1 = fma(-W[3 + i], xi, y1);
                    y2 = fma(-W[6 + i], xi, y2);
                }
            };
            if (pos > st) sub(B + kBW, R - kBlkLen * st);
            if (pos + st <= m) sub(B + kBU, R + kBlkLen * st);
            const double *D = B + kBD;
            y2 *= D[5];
            y1 = fma(-D[4], y2, y1) * D[2];
            y0 = fma(-D[3], y2, fma(-D[1], y1, y0)) * D[0];
            R[0] = y0; R[7] = y1; R[14] = y2;
        }
        __syncthreads();
    }
    if (m > 0 && t < 7 * kBorder) {
        const int r = t / 7, c = t % 7;
        double v = S[t];
        for (int i = 0; i < 3; i++) v = fma(-C0[kBorder * i + r], blk[kBR + 7 * i + c], v);
        if (m > 1)
            for (int i = 0; i < 3; i++)
                v = fma(-C1[kBorder * i + r], blk[kBlkLen * (m - 1) + kBR + 7 * i + c], v);
        S[t] = v;
    }
    __syncthreads();
    double *x0 = scr;  // the border's solution, x then y
    if (t < 2) {  // one lane a right-hand side, each with the factor
        double L[kBorder][kBorder], b[kBorder];
#pragma unroll
        for (int c = 0; c < kBorder; c++) {
#pragma unroll
            for (int r = c; r < kBorder; r++) {
                double v = S[7 * r + 2 + c];
#pragma unroll
                for (int k = 0; k < c; k++) v = fma(-L[r][k], L[c][k], v);
                if (r == c) {
                    if (!(v > 0.0)) *bad = 1;
                    L[c][c] = rsqrt_any(v);
                } else {
                    L[r][c] = v * L[c][c];
                }
            }
        }
#pragma unroll
        for (int r = 0; r < kBorder; r++) {
            double v = S[7 * r + t];
#pragma unroll
            for (int k = 0; k < r; k++) v = fma(-L[r][k], b[k], v);
            b[r] = v * L[r][r];
        }
#pragma unroll
        for (int r = kBorder - 1; r >= 0; r--) {
            double v = b[r];
#pragma unroll
            for (int k = r + 1; k < kBorder; k++) v = fma(-L[k][r], b[k], v);
            b[r] = v * L[r][r];
            x0[kBorder * t + r] = b[r];
        }
    }
    __syncthreads();
    for (int it = t; it < 2 * g; it += kT) {
        const int r = it >> 1, a = it & 1, br = r - 3 * m;
        double v;
        if (br >= 0) {
            v = x0[kBorder * a + br];
        } else {
            const double *R = blk + kBlkLen * (r / 3) + kBR + 7 * (r % 3);
            v = R[a];
            for (int k = 0; k < kBorder; k++) v = fma(-R[2 + k], x0[kBorder * a + k], v);
        }
        (a ? cy : cx)[r] = v;
    }
    __syncthreads();
}

// qs[k], k = 0 .. g: the first marker of span >= k (spans ascend with the
// marker), n if none.
__device__ __forceinline__ void span_starts(int n, int g, const int *span, int *qs)
{
    for (int m = threadIdx.x; m < n; m += kT) {
        const int lo = m == 0 ? 0 : span[m - 1] + 1;
        for (int k = lo; k <= span[m]; k++) qs[k] = m;
    }
    for (int k = span[n - 1] + 1 + threadIdx.x; k <= g; k += kT) qs[k] = n;
}

// Normal equations: put(i, dd, value, .) for entry (i, i+dd), dd = 0 .. 3, and
// put(i, 4, x, y) for the right-hand sides of row i, over the markers of spans
// i .. i+3 in ascending order; on span i + t row i has weight 3 - t.
template <typename F>
__device__ __forceinline__ void normal_equations(const double *X, const double *Y, int s0, int g,
                                                 const int *qs, const double *wts, F put)
{
    for (int e = threadIdx.x; e < 5 * g; e += kT) {
        const int i = e / 5, dd = e - 5 * i;
        const int t0 = i + 3 >= g ? g - i : 0;
        double acc = 0.0, accy = 0.0;
        for (int k = 0; k < 4; k++) {
            const int tt = (t0 + k) & 3, a = 3 - tt;
            if (tt == g) continue;  // three spans: i + 3 is span i again
            const int q = i + tt >= g ? i + tt - g : i + tt;
            int b = a + dd;
            if (b > 3) b -= g;  // fewer than seven spans: the band meets itself
            const double *wm = wts + 4L * (s0 + qs[q]);
            const int ke = qs[q + 1];
            if (dd < 4) {
                if (b >= 0)
                    for (int m = qs[q]; m < ke; m++, wm += 4) acc += wm[a] * wm[b];
            } else {
                for (int m = qs[q]; m < ke; m++, wm += 4) {
                    acc += wm[a] * X[s0 + m];
                    accy += wm[a] * Y[s0 + m];
                }
            }
        }
        put(i, dd, acc, accy);
    }
}

// Per-drop fit results: at offset 3 * s0 + d of fit (s0 the drop's first
// marker, n its markers, g <= n) the control points cx[g], cy[g] and the
// cumulative arc length at the knots cum[g + 1]; par[4d .. 4d+3] = (g, tau,
// total arc length, failed).
__device__ __forceinline__ long fit_base(int s0, int d) { return 3L * s0 + d; }

// One CTA per drop; FP64 latency and one SM's FP64 pipe bound it, so that
// every stage is spread over the block and written for few FP64
// instructions.  (With the recursive basis, the sums and the factorisation by
// one thread or warp the fit took 529 us and the placement 173 for 16 drops of
// 256 markers; this form takes 0.6 ms off the 1.73 ms of such a step.)
__global__ void __launch_bounds__(kT)
k_reloc_fit(const double *__restrict__ X, const double *__restrict__ Y,
            const int32_t *__restrict__ drop_start, double h, int maxn,
            double *__restrict__ fit, double *__restrict__ par, double *__restrict__ wts,
            uint32_t *__restrict__ flags)
{
    extern __shared__ double sm[];
    const int d = blockIdx.x, s0 = drop_start[d], n = drop_start[d + 1] - s0;
    // shared layout: sp[n+1] (then scratch, then cum[g+1]), qs[n+1] and
    // span[n] (ints, also the sums' scratch), cx[n], cy[n], the chain's blocks
    // (15 a row, at most n - 3 rows) and behind them the border's rows
    double *sp = sm;
    int *qs = (int *)(sp + maxn + 1);
    int *span = qs + (maxn + 1);
    double *cx = (double *)(qs + 2 * (maxn + 1)), *cy = cx + maxn, *blk = cy + maxn;
    double *S = blk + 15 * maxn - kEndLen;
    __shared__ int bad;
    if (threadIdx.x == 0) bad = 0;
    for (int m = threadIdx.x; m < n; m += kT) {  // chord lengths
        const int a = s0 + m, b = s0 + (m + 1 == n ? 0 : m + 1);
        const double dx = X[b] - X[a], dy = Y[b] - Y[a];
        cx[m] = sqrt(dx * dx + dy * dy);
    }
    __syncthreads();
    const double Lc = block_scan(n, cx, sp, qs);
    int g = (int)floor(Lc / (1.5 * h) + 0.5);
    if (g < 4) g = 4;
    if (g > n) g = n;
    const double tau = Lc / g, itau = 1.0 / tau;
    const int w = 3 + g % 3, nch = (g - w) / 3, gc = 3 * nch;
    // each marker's span and basis weights once (wts, 4 per marker)
    for (int m = threadIdx.x; m < n; m += kT) {
        const double s = sp[m];
        const int q = bspl_span(s, tau, g);
        const double u = fma(-(double)q, tau, s) * itau, v = 1.0 - u, u2 = u * u;
        const double s6 = 1.0 / 6.0;
        double *o = wts + 4L * (s0 + m);
        span[m] = q;
        o[0] = s6 * (v * v * v);
        o[1] = s6 * fma(u2, fma(3.0, u, -6.0), 4.0);
        o[2] = s6 * fma(u, fma(u, fma(-3.0, u, 3.0), 3.0), 1.0);
        o[3] = s6 * (u2 * u);
    }
    for (int k = threadIdx.x; k < kBlkLen * nch; k += kT) blk[k] = 0.0;
    if (threadIdx.x < kEndLen) {
        const int r = threadIdx.x / 7, c = threadIdx.x % 7;
        S[threadIdx.x] = c == 2 + r && r >= w ? 1.0 : 0.0;
    }
    __syncthreads();
    span_starts(n, g, span, qs);
    __syncthreads();
    normal_equations(X, Y, s0, g, qs, wts, [&](int i, int dd, double acc, double accy) {
        if (dd == 4) {
            double *r = i < gc ? blk + kBlkLen * (i / 3) + kBR + 7 * (i % 3) : S + 7 * (i - gc);
            r[0] = acc; r[1] = accy;
            return;
        }
        const int j = i + dd >= g ? i + dd - g : i + dd;
        const int lo = min(i, j), hi = max(i, j);
        if (lo >= gc) {
            S[7 * (lo - gc) + 2 + hi - gc] = acc;
            S[7 * (hi - gc) + 2 + lo - gc] = acc;
        } else {
            const int bl = lo / 3, r = lo - 3 * bl;
            double *B = blk + kBlkLen * bl;
            if (hi >= gc) B[kBR + 7 * r + 2 + hi - gc] = acc;
            else if (hi / 3 == bl) { const int c = hi - 3 * bl; B[kBD + c * (c + 1) / 2 + r] = acc; }
            else B[kBU + 3 * r + hi - 3 * (bl + 1)] = acc;
        }
    });
    __syncthreads();
    ring_solve(blk, nch, g, S, sp, cx, cy, &bad);
    double *out = fit + fit_base(s0, d);
    if (bad) {
        if (threadIdx.x == 0) {
            atomicOr(&flags[2], 1u);
            par[4 * d] = (double)g; par[4 * d + 1] = tau; par[4 * d + 2] = 0.0; par[4 * d + 3] = 1.0;
        }
        return;
    }
    // arc length of every span (blk is free now), its running sum
    for (int q = threadIdx.x; q < g; q += kT) {
        const SpanCurve c = span_curve(cx, cy, g, q);
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < 8; k++)
            s = fma(0.5 * cGLW[k], sqrt_any(speed2(c, fma(0.5, cGLX[k], 0.5))), s);
        blk[q] = s;
    }
    __syncthreads();
    const double len = block_scan(g, blk, sp, qs);
    if (threadIdx.x == 0) {
        par[4 * d] = (double)g; par[4 * d + 1] = tau; par[4 * d + 2] = len; par[4 * d + 3] = 0.0;
    }
    for (int q = threadIdx.x; q < g; q += kT) { out[q] = cx[q]; out[n + q] = cy[q]; }
    for (int q = threadIdx.x; q <= g; q += kT) out[2 * n + q] = sp[q];
}

// New marker m of its drop at arc length L m / n along the fitted curve: the
// span by bisection of the knot arc lengths, then Newton steps on the partial
// arc length in u, kept in the span; at most 12, ended when the iterate
// repeats itself (all later steps would, so the result is that of 12).  LN
// lanes share a marker's eight Gauss-Legendre terms: a step costs about
// 104 / LN + 27 FP64 instructions, and up to four warps an SM the time is
// that of one warp, so LN = 8 below 4096 markers, 4 up to 8192, 1 above
// (with the curve evaluated from control points at every node and always 12
// steps 4096 markers took 173 us, 16384 markers 193).  A drop whose fit failed
// keeps its markers.
constexpr int kPlaceT = 64;
template <int LN>
__global__ void __launch_bounds__(kPlaceT)
k_reloc_place(int M, const int32_t *__restrict__ drop_of, const int32_t *__restrict__ drop_start,
              const double *__restrict__ fit, const double *__restrict__ par,
              double *__restrict__ X, double *__restrict__ Y)
{
    const int lane = threadIdx.x & (LN - 1), j = (blockIdx.x * kPlaceT + threadIdx.x) / LN;
    const unsigned grp = ((1u << LN) - 1u) << (threadIdx.x & 31 & ~(LN - 1));  // this marker's lanes
    if (j >= M) return;  // whole groups leave together
    const int d = drop_of[j], s0 = drop_start[d], n = drop_start[d + 1] - s0, m = j - s0;
    if (par[4 * d + 3] != 0.0) return;
    const int g = (int)par[4 * d];
    const double Lp = par[4 * d + 2];
    const double *cx = fit + fit_base(s0, d), *cy = cx + n, *cum = cx + 2 * n;
    const double target = Lp * (double)m / (double)n;
    int lo = 0, hi = g - 1;  // largest q <= g-1 with cum[q] <= target
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cum[mid] <= target) lo = mid; else hi = mid - 1;
    }
    const int q = lo;
    const SpanCurve c = span_curve(cx, cy, g, q);
    const double c0 = cum[q] - target;
    double node[8 / LN], wgt[8 / LN];
#pragma unroll
    for (int k = 0; k < 8 / LN; k++) {
        node[k] = fma(0.5, cGLX[lane + LN * k], 0.5);
        wgt[k] = 0.5 * cGLW[lane + LN * k];
    }
    double u = -c0 / (cum[q + 1] - cum[q]), prev = u;
    for (int it = 1; it <= 12; it++) {
        double sum = 0.0;
#pragma unroll
        for (int k = 0; k < 8 / LN; k++) sum = fma(wgt[k], sqrt_any(speed2(c, u * node[k])), sum);
        for (int o = LN / 2; o; o >>= 1) sum += __shfl_xor_sync(grp, sum, o);
        double un = fma(-fma(u, sum, c0), rsqrt_any(speed2(c, u)), u);
        if (un < 0.0) un = 0.0;
        if (un > 1.0) un = 1.0;
        const long long bn = __double_as_longlong(un);
        if (bn == __double_as_longlong(u)) break;
        if (it > 1 && bn == __double_as_longlong(prev)) {  // a cycle of two
            if (!((12 - it) & 1)) u = un;
            break;
        }
        prev = u;
        u = un;
    }
    if (lane != 0) return;
    const double v = 1.0 - u, u2 = u * u, u3 = u2 * u;
    const double b0 = v * v * v, b1 = fma(3.0, u3, fma(-6.0, u2, 4.0));
    const double b2 = fma(-3.0, u3, fma(3.0, u2, fma(3.0, u, 1.0))), b3 = u3;
    const double s6 = 1.0 / 6.0;
    X[j] = s6 * (b0 * c.x[0] + b1 * c.x[1] + b2 * c.x[2] + b3 * c.x[3]);
    Y[j] = s6 * (b0 * c.y[0] + b1 * c.y[1] + b2 * c.y[2] + b3 * c.y[3]);
}

// ------------------------------------------------------------ B-spline, serial order
// The same fit and placement in a fixed serial order of operations, for
// axisymmetric contexts.  The falling frame divides differences of the drop's
// centre by the square of the time step: there one unit in the last place of
// a marker shows as 1e-10 of the pressure, and the drop keeps these bits from
// one version to the next.  (Contexts without the frame have no such division;
// they share the path, at 0.3 ms a relocation.)  So the chord lengths and arc
// lengths are summed marker by marker, the basis is the Cox-de Boor recursion on
// knots k tau, the matrix is factored column by column and substituted row by
// row, each sum in ascending order, its products rounded before they are
// subtracted.  FP64 latency bounds the chains (64 cycles an instruction), so that
// operands are loaded a step ahead and nothing but the sums' own instructions is
// on them: one drop of 1024 markers 1114 us with
// every entry looked up on the chain, now 378; the block elimination above 134.
__device__ void bspl_basis(double s, double tau, int g, double *w)
{
    const int q = bspl_span(s, tau, g);
    double N[4][4];
    N[0][0] = 1.0;
    for (int d = 1; d <= 3; d++)
        for (int r = 0; r <= d; r++) {
            int k = q - d + r;
            double tk = k * tau, tkd = (k + d) * tau, tk1 = (k + 1) * tau, tkd1 = (k + d + 1) * tau;
            double left = (r >= 1) ? (s - tk) / (tkd - tk) * N[d - 1][r - 1] : 0.0;
            double right = (r <= d - 1) ? (tkd1 - s) / (tkd1 - tk1) * N[d - 1][r] : 0.0;
            N[d][r] = left + right;
        }
    for (int r = 0; r <= 3; r++) w[r] = N[3][r];
}

struct SpanU {
    int i0, i1, i2, i3;  // control points q-3 .. q (cyclic)
    double u;
};
__device__ __forceinline__ SpanU bspl_span_u(double s, double itau, int g)
{
    const double x = s * itau;
    int q = (int)floor(x);
    q = q > g - 1 ? g - 1 : (q < 0 ? 0 : q);
    SpanU r;
    r.u = x - (double)q;
    const int k = q - 3;  // >= -3, and q <= g - 1
    r.i0 = k < 0 ? k + g : k;
    r.i1 = k + 1 < 0 ? k + 1 + g : k + 1;
    r.i2 = k + 2 < 0 ? k + 2 + g : k + 2;
    r.i3 = q;
    return r;
}

__device__ double bspl_speed(double s, double tau, int g, const double *cx, const double *cy)
{
    const double itau = 1.0 / tau;
    const SpanU p = bspl_span_u(s, itau, g);
    const double u = p.u, v = 1.0 - u;
    // twice the derivatives in u: -(1-u)^2, 3u^2 - 4u, -3u^2 + 2u + 1, u^2
    const double d0 = -v * v, d1 = u * (3.0 * u - 4.0), d2 = fma(u, 2.0 - 3.0 * u, 1.0), d3 = u * u;
    const double dx = d0 * cx[p.i0] + d1 * cx[p.i1] + d2 * cx[p.i2] + d3 * cx[p.i3];
    const double dy = d0 * cy[p.i0] + d1 * cy[p.i1] + d2 * cy[p.i2] + d3 * cy[p.i3];
    return 0.5 * itau * sqrt(dx * dx + dy * dy);
}

// The curve's point at s (closed form, as bspl_speed).
__device__ void bspl_point(double s, double tau, int g, const double *cx, const double *cy,
                           double &px, double &py)
{
    const SpanU p = bspl_span_u(s, 1.0 / tau, g);
    const double u = p.u, v = 1.0 - u, u2 = u * u, u3 = u2 * u;
    const double b0 = v * v * v, b1 = fma(3.0, u3, fma(-6.0, u2, 4.0));
    const double b2 = fma(-3.0, u3, fma(3.0, u2, fma(3.0, u, 1.0))), b3 = u3;
    const double s6 = 1.0 / 6.0;
    px = s6 * (b0 * cx[p.i0] + b1 * cx[p.i1] + b2 * cx[p.i2] + b3 * cx[p.i3]);
    py = s6 * (b0 * cy[p.i0] + b1 * cy[p.i1] + b2 * cy[p.i2] + b3 * cy[p.i3]);
}

__device__ double gl_len(double a, double b, double tau, int g, const double *cx, const double *cy)
{
    double mid = 0.5 * (a + b), half = 0.5 * (b - a), s = 0.0;
    for (int k = 0; k < 8; k++) s += cGLW[k] * bspl_speed(mid + half * cGLX[k], tau, g, cx, cy);
    return s * half;
}

// acc - a b, the product rounded first.
__device__ __forceinline__ double sub_prod(double acc, double a, double b)
{
    return __dsub_rn(acc, __dmul_rn(a, b));
}

// 1/sqrt(x) by two Newton steps y <- y (3/2 - x y^2 / 2) from the FP32 estimate.
__device__ __forceinline__ double rsqrt_newton(double x)
{
    double y = f2d_exact(rsqrtf(d2f_trunc(x)));
    const double hx = -0.5 * x;
    y = y * fma(hx, y * y, 1.5);
    return y * fma(hx, y * y, 1.5);
}

// The lower triangle in its envelope: rows r < g - 3 keep columns r-3 .. r
// (band[4 r + 3 - d] for column r - d), the last three, where the cyclic wrap
// fills in, all columns (dn[(r - (g - 3)) g + c]).  On entry the matrix, on
// return its Cholesky factor, by one warp (lane t): lane 0 the diagonal of
// column c, lanes 1 .. 3 the band rows below it, 4 .. 6 the last rows.  rinv:
// the diagonal's reciprocals.  Returns -1 (in every lane) if not positive
// definite.
__device__ int serial_factor(double *band, double *dn, int g, int t, double *rinv)
{
    const int gb = g - 3;
    const long long lo = __double_as_longlong(1e-30), hi = __double_as_longlong(1e30);
    auto pivot = [&](double s, double &rd) {  // false if not positive
        const long long b = __double_as_longlong(s);
        if (b > lo && b < hi) { rd = rsqrt_newton(s); return true; }
        if (!(s > 0.0)) return false;
        rd = 1.0 / sqrt(s);
        return true;
    };
    for (int c = 0; c < gb; c++) {
        double *slot = nullptr;
        const double *row = nullptr;  // row[k] is the entry of column k
        if (t < 4) {
            if (c + t < gb) { row = band + 4 * (c + t) + 3 - (c + t); slot = band + 4 * (c + t) + 3 - t; }
        } else if (t < 7) {
            row = dn + (t - 4) * g; slot = dn + (t - 4) * g + c;
        }
        const double *pv = band + 4 * c + 3 - c;
        const int first = t < 4 ? max(c + t - 3, 0) : max(c - 3, 0);
        double acc = 0.0;
        if (slot) {
            acc = *slot;
#pragma unroll
            for (int d = 3; d >= 1; d--)
                if (c - d >= first) acc = sub_prod(acc, row[c - d], pv[c - d]);
        }
        const double s = __shfl_sync(0xffffffffu, acc, 0);
        double rd = 0.0;
        if (!pivot(s, rd)) return -1;
        if (slot) *slot = acc * rd;  // the diagonal: s / sqrt(s)
        if (t == 0) rinv[c] = rd;
        __syncwarp();
    }
    for (int c = gb; c < g; c++) {
        // sums over all earlier columns: beyond 32 of them strided partial
        // sums and a shuffle tree (the same total in every lane)
        const int r = c + t;
        const double *pv = dn + (c - gb) * g;
        double acc = 0.0;
        if (c > 32) {
            double pd = 0.0, p1 = 0.0, p2 = 0.0;
            for (int k = t; k < c; k += 32) {
                const double lc = pv[k];
                pd += lc * lc;
                if (c + 1 < g) p1 += pv[g + k] * lc;
                if (c + 2 < g) p2 += pv[2 * g + k] * lc;
            }
            for (int o = 16; o; o >>= 1) {
                pd += __shfl_xor_sync(0xffffffffu, pd, o);
                p1 += __shfl_xor_sync(0xffffffffu, p1, o);
                p2 += __shfl_xor_sync(0xffffffffu, p2, o);
            }
            if (t < 3 && r < g) acc = pv[t * g + c] - (t == 0 ? pd : (t == 1 ? p1 : p2));
        } else if (t < 3 && r < g) {
            acc = pv[t * g + c];
            for (int k = 0; k < c; k++) acc = sub_prod(acc, pv[t * g + k], pv[k]);
        }
        const double s = __shfl_sync(0xffffffffu, acc, 0);
        double rd = 0.0;
        if (!pivot(s, rd)) return -1;
        if (t < 3 && r < g) dn[(r - gb) * g + c] = acc * rd;
        if (t == 0) rinv[c] = rd;
        __syncwarp();
    }
    return 0;
}

// L L^T x = b for the two right-hand sides bx, by (in place) by one warp (lane
// t): even lanes the x side, odd lanes the y side, one instruction for both.
// A lane keeps its side's latest three entries in registers.
__device__ void serial_subst(const double *band, const double *dn, int g, const double *rinv, double *bx,
                             double *by, int t)
{
    const int gb = g - 3;
    double *b = (t & 1) ? by : bx;
    double x1 = 0.0, x2 = 0.0, x3 = 0.0;  // rows r-1, r-2, r-3
    double s = gb > 0 ? b[0] : 0.0, l1 = 0.0, l2 = 0.0, l3 = 0.0, ri = rinv[0];
    for (int r = 0; r < gb; r++) {
        // the next row's operands
        const int n = min(r + 1, gb - 1);
        const double sn = b[n], n1 = band[4 * n + 2], n2 = band[4 * n + 1], n3 = band[4 * n], rn = rinv[n];
        if (r >= 3) s = sub_prod(s, l3, x3);
        if (r >= 2) s = sub_prod(s, l2, x2);
        if (r >= 1) s = sub_prod(s, l1, x1);
        s *= ri;
        __syncwarp();
        if (t < 2) b[r] = s;
        x3 = x2; x2 = x1; x1 = s;
        s = sn; l1 = n1; l2 = n2; l3 = n3; ri = rn;
    }
    for (int r = gb; r < g; r++) {
        const double *row = dn + (r - gb) * g;
        __syncwarp();
        s = b[r];
        if (r > 32) {
            double ps = 0.0, pu = 0.0;
            for (int k = t; k < r; k += 32) { const double l = row[k]; ps += l * bx[k]; pu += l * by[k]; }
            for (int o = 16; o; o >>= 1) {
                ps += __shfl_xor_sync(0xffffffffu, ps, o);
                pu += __shfl_xor_sync(0xffffffffu, pu, o);
            }
            s -= (t & 1) ? pu : ps;
        } else {
            for (int k = 0; k < r; k++) s = sub_prod(s, row[k], b[k]);
        }
        s *= rinv[r];
        __syncwarp();
        if (t < 2) b[r] = s;
    }
    __syncwarp();
    double tl[3];  // rows g-3, g-2, g-1
    for (int q = 2; q >= 0; q--) {
        s = b[gb + q];
        for (int k = q + 1; k < 3; k++) s = sub_prod(s, dn[k * g + gb + q], tl[k]);
        s *= rinv[gb + q];
        __syncwarp();
        if (t < 2) b[gb + q] = s;
        tl[q] = s;
    }
    double f1 = 0.0, f2 = 0.0, f3 = 0.0;  // rows r+1, r+2, r+3 of the band
    double e1 = 0.0, e2 = 0.0, e3 = 0.0, d0 = 0.0, d1 = 0.0, d2 = 0.0;
    auto load = [&](int r) {
        s = b[r]; ri = rinv[r];
        e1 = r + 1 < gb ? band[4 * r + 6] : 0.0;   // (r+1, r)
        e2 = r + 2 < gb ? band[4 * r + 9] : 0.0;   // (r+2, r)
        e3 = r + 3 < gb ? band[4 * r + 12] : 0.0;  // (r+3, r)
        d0 = dn[r]; d1 = dn[g + r]; d2 = dn[2 * g + r];
    };
    if (gb > 0) load(gb - 1);
    for (int r = gb - 1; r >= 0; r--) {
        double v = s;
        const double rr = ri, a1 = e1, a2 = e2, a3 = e3, q0 = d0, q1 = d1, q2 = d2;
        if (r > 0) load(r - 1);
        if (r + 1 < gb) v = sub_prod(v, a1, f1);
        if (r + 2 < gb) v = sub_prod(v, a2, f2);
        if (r + 3 < gb) v = sub_prod(v, a3, f3);
        v = sub_prod(v, q0, tl[0]);
        v = sub_prod(v, q1, tl[1]);
        v = sub_prod(v, q2, tl[2]);
        v *= rr;
        __syncwarp();
        if (t < 2) b[r] = v;
        f3 = f2; f2 = f1; f1 = v;
    }
}

// out[k] = in[0] + ... + in[k-1], k = 0 .. n, one by one; returns the total.
__device__ double serial_sum(int n, const double *in, double *out)
{
    double L = 0.0;
    int m = 0;
    for (; m + 8 <= n; m += 8) {
        double v[8];
#pragma unroll
        for (int k = 0; k < 8; k++) v[k] = in[m + k];
#pragma unroll
        for (int k = 0; k < 8; k++) { out[m + k] = L; L += v[k]; }
    }
    for (; m < n; m++) { const double v = in[m]; out[m] = L; L += v; }
    out[n] = L;
    return L;
}

__global__ void __launch_bounds__(kT)
k_reloc_fit_serial(const double *__restrict__ X, const double *__restrict__ Y,
                   const int32_t *__restrict__ drop_start, double h, int maxn,
                   double *__restrict__ fit, double *__restrict__ par, double *__restrict__ wts,
                   uint32_t *__restrict__ flags)
{
    extern __shared__ double sm[];
    const int d = blockIdx.x, s0 = drop_start[d], n = drop_start[d + 1] - s0;
    // shared layout: sp[n+1] (then cum[g+1]), qs[n+1] and span[n] (ints),
    // cx[n], cy[n], the reciprocals and arc lengths [n], band[4n], the last
    // three rows [3n]
    double *sp = sm;
    int *qs = (int *)(sp + maxn + 1);
    int *span = qs + (maxn + 1);
    double *cx = (double *)(qs + 2 * (maxn + 1)), *cy = cx + maxn, *rinv = cy + maxn;
    double *band = rinv + maxn, *dn = band + 4 * maxn;
    __shared__ double total;
    __shared__ int bad;
    for (int m = threadIdx.x; m < n; m += kT) {  // chord lengths
        const int a = s0 + m, b = s0 + (m + 1 == n ? 0 : m + 1);
        const double dx = X[b] - X[a], dy = Y[b] - Y[a];
        cx[m] = sqrt(dx * dx + dy * dy);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        total = serial_sum(n, cx, sp);
        bad = 0;
    }
    __syncthreads();
    const double Lc = total;
    int g = (int)floor(Lc / (1.5 * h) + 0.5);
    if (g < 4) g = 4;
    if (g > n) g = n;
    const double tau = Lc / g;
    for (int m = threadIdx.x; m < n; m += kT) {
        double w[4];
        bspl_basis(sp[m], tau, g, w);
        span[m] = bspl_span(sp[m], tau, g);
        for (int r = 0; r < 4; r++) wts[4L * (s0 + m) + r] = w[r];
    }
    for (int k = threadIdx.x; k < 3 * g; k += kT) dn[k] = 0.0;
    __syncthreads();
    span_starts(n, g, span, qs);
    __syncthreads();
    normal_equations(X, Y, s0, g, qs, wts, [&](int i, int dd, double acc, double accy) {
        if (dd == 4) { cx[i] = acc; cy[i] = accy; return; }
        const int j = i + dd >= g ? i + dd - g : i + dd;
        const int lo = min(i, j), hi = max(i, j);
        if (hi >= g - 3) dn[(hi - (g - 3)) * g + lo] = acc;
        else band[4 * hi + 3 - (hi - lo)] = acc;
    });
    __syncthreads();
    if (threadIdx.x < 32) {
        const int f = serial_factor(band, dn, g, threadIdx.x, rinv);  // the same in every lane
        if (f != 0) {
            if (threadIdx.x == 0) bad = 1;
        } else {
            serial_subst(band, dn, g, rinv, cx, cy, threadIdx.x);
        }
    }
    __syncthreads();
    double *out = fit + fit_base(s0, d);
    if (bad) {
        if (threadIdx.x == 0) {
            atomicOr(&flags[2], 1u);
            par[4 * d] = (double)g; par[4 * d + 1] = tau; par[4 * d + 2] = 0.0; par[4 * d + 3] = 1.0;
        }
        return;
    }
    for (int q = threadIdx.x; q < g; q += kT) rinv[q] = gl_len(q * tau, (q + 1) * tau, tau, g, cx, cy);
    __syncthreads();
    if (threadIdx.x == 0) {
        const double len = serial_sum(g, rinv, sp);
        par[4 * d] = (double)g; par[4 * d + 1] = tau; par[4 * d + 2] = len; par[4 * d + 3] = 0.0;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < g; q += kT) { out[q] = cx[q]; out[n + q] = cy[q]; }
    for (int q = threadIdx.x; q <= g; q += kT) out[2 * n + q] = sp[q];
}

// The placement of k_reloc_place with the parameter s as the iterate, eight
// lanes a marker: lane k evaluates the k-th Gauss-Legendre term, lane 0 also
// the speed at s, and every lane sums the eight terms in order.
__global__ void __launch_bounds__(kPlaceT)
k_reloc_place_serial(int M, const int32_t *__restrict__ drop_of, const int32_t *__restrict__ drop_start,
                     const double *__restrict__ fit, const double *__restrict__ par,
                     double *__restrict__ X, double *__restrict__ Y)
{
    const int lane = threadIdx.x & 7, j = (blockIdx.x * kPlaceT + threadIdx.x) >> 3;
    const unsigned grp = 0xffu << (threadIdx.x & 24);  // the eight lanes of this marker
    if (j >= M) return;  // whole groups leave together
    const int d = drop_of[j], s0 = drop_start[d], n = drop_start[d + 1] - s0, m = j - s0;
    if (par[4 * d + 3] != 0.0) return;
    const int g = (int)par[4 * d];
    const double tau = par[4 * d + 1], Lp = par[4 * d + 2];
    const double *cx = fit + fit_base(s0, d), *cy = cx + n, *cum = cx + 2 * n;
    const double target = Lp * (double)m / (double)n;
    int lo = 0, hi = g - 1;  // largest q <= g-1 with cum[q] <= target
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cum[mid] <= target) lo = mid; else hi = mid - 1;
    }
    const int q = lo;
    const double a = q * tau, b = (q + 1) * tau;
    const double seg = cum[q + 1] - cum[q];
    double s = a + tau * (target - cum[q]) / seg, prev = s;
    for (int it = 1; it <= 12; it++) {
        const double mid = 0.5 * (a + s), half = 0.5 * (s - a);
        const double term = cGLW[lane] * bspl_speed(mid + half * cGLX[lane], tau, g, cx, cy);
        const double sp_ = lane == 0 ? bspl_speed(s, tau, g, cx, cy) : 0.0;
        double sum = 0.0;
        for (int k = 0; k < 8; k++) sum += __shfl_sync(grp, term, k, 8);
        const double f = cum[q] + sum * half - target;
        double sn = s - f / __shfl_sync(grp, sp_, 0, 8);
        if (sn < a) sn = a;
        if (sn > b) sn = b;
        const long long bn = __double_as_longlong(sn);
        if (bn == __double_as_longlong(s)) break;
        if (it > 1 && bn == __double_as_longlong(prev)) {  // a cycle of two
            if (!((12 - it) & 1)) s = sn;
            break;
        }
        prev = s;
        s = sn;
    }
    if (lane != 0) return;
    double px, py;
    bspl_point(s, tau, g, cx, cy, px, py);
    X[j] = px;
    Y[j] = py;
}

}  // namespace

// --------------------------------------------------------------------- host
static size_t al(size_t b) { return (b + 255) & ~(size_t)255; }

cudaError_t markers_alloc(Markers &mk, int M, int ndrops, int nx, int ny, double h,
                          double x0, double y0, const int32_t *drop_start_host)
{
    mk.M = M; mk.ndrops = ndrops; mk.nx = nx; mk.ny = ny; mk.h = h; mk.x0 = x0; mk.y0 = y0;
    mk.bnx = (nx + kBlk - 1) / kBlk;
    mk.bny = (ny + kBlk - 1) / kBlk;
    mk.drop_start_h.assign(drop_start_host, drop_start_host + ndrops + 1);
    mk.max_drop = 0;
    for (int d = 0; d < ndrops; d++)
        mk.max_drop = std::max(mk.max_drop, drop_start_host[d + 1] - drop_start_host[d]);
    size_t ncell = (size_t)nx * ny, nb = (size_t)mk.bnx * mk.bny;
    size_t nparts = (ncell + kScanChunk - 1) / kScanChunk;
    // (cell, segment) pairs of the band: about (5 + 1) x (segment length + 1)
    // per segment; 64 per segment covers segments up to ~9 cells long.
    const size_t pair_cap = (size_t)M * 64 + 4096;
    mk.pair_cap = (uint32_t)pair_cap;
    size_t bytes = al(M * 8) * 11 + al(M * 4) * 2 + al(M * 16) + al(ndrops * 16) * 2 + al((3 * (size_t)M + ndrops) * 8) + al((size_t)ndrops * 32) + al((size_t)M * 32) +
                   al((size_t)M * 24 * 8) + al((size_t)M * kSegLine * 8) + al((size_t)M * 8 * 16) + al((size_t)M * 5 * 16) + al(M * 8) + al(M) + al(M * 8) +
                   al(64) + al(pair_cap * 4) * 2 + al(pair_cap * 8) * 2 + al(ncell * 8) +
                   al((ndrops + 1) * 4) + al(M * 4) * 5 + al(ncell * 4) +
                   al((ncell + 1) * 4) + al(nparts * 4) + al((nb + 1) * 4) + al(nb * 4) + al(64) +
                   al((size_t)nx * 8) + al((size_t)kClipCap * 4) + al((size_t)M * kTab * 8);
    cudaError_t e = cudaMalloc(&mk.mem, bytes);
    if (e != cudaSuccess) { mk.mem = nullptr; return e; }
    char *q = (char *)mk.mem;
    auto take = [&](size_t b) { char *r = q; q += al(b); return (void *)r; };
    mk.X = (double *)take(M * 8); mk.Y = (double *)take(M * 8);
    mk.kappa = (double *)take(M * 8); mk.nxm = (double *)take(M * 8); mk.nym = (double *)take(M * 8);
    mk.ds = (double *)take(M * 8); mk.fmag = (double *)take(M * 8);
    mk.U = (double *)take(M * 8); mk.V = (double *)take(M * 8);
    mk.gx = (double *)take(M * 8); mk.gy = (double *)take(M * 8);
    mk.gxf = (float *)take(M * 4); mk.gyf = (float *)take(M * 4);
    mk.sbox = (float4 *)take(M * 16);
    mk.dyr = (double2 *)take(ndrops * 16);
    mk.dyk = (ulonglong2 *)take(ndrops * 16);
    mk.rfit = (double *)take((3 * (size_t)M + ndrops) * 8);
    mk.rpar = (double *)take((size_t)ndrops * 32);
    mk.rwts = (double *)take((size_t)M * 32);
    mk.sv = (double *)take((size_t)M * 24 * 8);
    mk.sl = (double *)take((size_t)M * kSegLine * 8);
    mk.slf = (float4 *)take((size_t)M * 8 * 16);
    mk.sb5 = (float4 *)take((size_t)M * 5 * 16);
    mk.scvx = (uint8_t *)take(M);
    mk.sinv = (double *)take(M * 8);
    mk.npairs = (uint32_t *)take(64);
    mk.pseg = (uint32_t *)take(pair_cap * 4); mk.pcell = (uint32_t *)take(pair_cap * 4);
    mk.pacc = (double *)take(pair_cap * 8); mk.pcov = (double *)take(pair_cap * 8);
    mk.crange = (uint2 *)take(ncell * 8);
    mk.ykey = (unsigned long long *)take(M * 8);
    mk.drop_start = (int32_t *)take((ndrops + 1) * 4);
    mk.drop_of = (int32_t *)take(M * 4);
    mk.next = (int32_t *)take(M * 4);
    mk.key = (uint32_t *)take(M * 4); mk.tmp_ids = (uint32_t *)take(M * 4); mk.ids = (uint32_t *)take(M * 4);
    mk.cell_count = (uint32_t *)take(ncell * 4);
    mk.cell_start = (uint32_t *)take((ncell + 1) * 4);
    mk.scan_part = (uint32_t *)take(nparts * 4);
    mk.bcount = (uint32_t *)take((nb + 1) * 4); mk.blist = (uint32_t *)take(nb * 4);
    mk.nact = mk.bcount + nb;
    mk.flags = (uint32_t *)take(64);
    mk.colkey = (unsigned long long *)take((size_t)nx * 8);
    mk.clip_list = (uint32_t *)take((size_t)kClipCap * 4);
    mk.stab = (double *)take((size_t)M * kTab * 8);
    std::vector<int32_t> dof(M), nxt(M);
    for (int d = 0; d < ndrops; d++)
        for (int m = drop_start_host[d]; m < drop_start_host[d + 1]; m++) {
            dof[m] = d;
            nxt[m] = (m + 1 == drop_start_host[d + 1]) ? drop_start_host[d] : m + 1;
        }
    e = cudaMemset(mk.mem, 0, bytes);
    if (e == cudaSuccess) {
        // the column keys of the scanline fill (the grid does not move); the
        // copies below, on the same legacy stream, follow the kernel
        k_colkeys<<<cdiv(nx, kT), kT>>>(nx, h, x0, mk.colkey);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(mk.drop_start, drop_start_host, (ndrops + 1) * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && M > 0) e = cudaMemcpy(mk.drop_of, dof.data(), M * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && M > 0) e = cudaMemcpy(mk.next, nxt.data(), M * 4, cudaMemcpyHostToDevice);
    return e;
}

void markers_free(Markers &mk)
{
    if (mk.mem) cudaFree(mk.mem);
    mk.mem = nullptr;
}

void launch_validate(Markers &mk, uint32_t *flags_host, cudaStream_t s)
{
    double m3 = 3.0 * mk.h;
    note_launch();
    k_validate<<<cdiv(mk.M, kT), kT, 0, s>>>(mk.M, mk.X, mk.Y, mk.x0 + m3, mk.x0 + mk.nx * mk.h - m3,
                                            mk.y0 + m3, mk.y0 + mk.ny * mk.h - m3, mk.flags,
                                            flags_host);
}

void launch_geometry(Markers &mk, double sigma, cudaStream_t s)
{
    note_launch();
    k_geometry<<<cdiv(mk.M, kT), kT, 0, s>>>(mk.M, mk.X, mk.Y, mk.drop_of, mk.drop_start, sigma,
                                            mk.x0, mk.y0, mk.h, mk.kappa, mk.nxm, mk.nym, mk.ds,
                                            mk.fmag, mk.gx, mk.gy, mk.gxf, mk.gyf, mk.ykey);
}

void launch_segments(Markers &mk, cudaStream_t s)
{
    note_launch();
    k_segments<<<cdiv(8L * mk.M, 128), 128, 0, s>>>(mk.M, mk.next, mk.gx, mk.gy, mk.nxm, mk.nym,
                                                    mk.sbox, mk.sv, mk.sb5, mk.sl, mk.slf, mk.scvx,
                                                    mk.sinv);
    note_launch();
    k_drop_yrange<<<cdiv((long)mk.ndrops * 32, kT), kT, 0, s>>>(mk.ndrops, mk.drop_start, mk.Y,
                                                               mk.dyr, mk.dyk);
}

void launch_sort(Markers &mk, cudaStream_t s)
{
    long ncell = (long)mk.nx * mk.ny;
    cudaMemsetAsync(mk.cell_count, 0, ncell * 4, s);
    cudaMemsetAsync(mk.bcount, 0, ((size_t)mk.bnx * mk.bny + 1) * 4, s);  // and *nact
    note_launch();
    k_keys<<<cdiv(mk.M, kT), kT, 0, s>>>(mk.M, mk.X, mk.Y, mk.x0, mk.y0, mk.h, mk.nx, mk.ny,
                                        mk.bnx, mk.key, mk.cell_count, mk.bcount);
    int nparts = (int)cdiv(ncell, kScanChunk);
    note_launch();
    k_scan_partial<<<nparts, kT, 0, s>>>(ncell, mk.cell_count, mk.scan_part);
    note_launch();
    k_scan_parts<<<1, kT, 0, s>>>(nparts, mk.scan_part);
    note_launch();
    k_scan_final<<<nparts, kT, 0, s>>>(ncell, mk.cell_count, mk.scan_part, mk.cell_start,
                                       (uint32_t)mk.M);
    note_launch();
    k_place<<<cdiv(mk.M, kT), kT, 0, s>>>(mk.M, mk.key, mk.cell_start, mk.cell_count, mk.tmp_ids);
    note_launch();
    k_rerank<<<cdiv(mk.M, kT), kT, 0, s>>>(mk.M, mk.key, mk.cell_start, mk.tmp_ids, mk.ids);
    int nb = mk.bnx * mk.bny;
    note_launch();
    k_block_active<<<cdiv(nb, kT), kT, 0, s>>>(mk.bnx, mk.bny, mk.bcount, mk.blist, mk.nact);
}

void launch_interp(const Markers &mk, int kernel, const double *u, const double *v,
                   double *U, double *V, double dt_move, cudaStream_t s)
{
    note_launch();
    k_interp<<<cdiv(8L * mk.M, 128), 128, 0, s>>>(mk.M, kernel, mk.nx, mk.ny, 1.0 / mk.h, mk.x0, mk.y0, u, v,
                                            mk.X, mk.Y, U, V, dt_move);
}

// Multiprocessors of the device (the same on every device this runs on).
static int sm_count()
{
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 152;
    }
    return sms;
}

// Grid of the kernels over active blocks: per CTAs an SM, or one per block.
static int block_grid(const Markers &mk, int per)
{
    return (int)std::min((long)mk.bnx * mk.bny, (long)per * sm_count());
}

void launch_spread_conv(const Markers &mk, int kernel, const double *fmag, double *Fx,
                        double *Fy, cudaStream_t s)
{
    cudaMemsetAsync(Fx, 0, (size_t)(mk.nx + 1) * mk.ny * 8, s);
    cudaMemsetAsync(Fy, 0, (size_t)mk.nx * (mk.ny + 1) * 8, s);
    note_launch();
    k_spread_tab<<<cdiv(2L * mk.M, 128), 128, 0, s>>>(mk.M, kernel, 1.0 / mk.h, mk.x0, mk.y0, mk.X, mk.Y, fmag,
                                                      mk.nxm, mk.nym, mk.ds, mk.stab);
    note_launch();
    k_spread_conv<<<block_grid(mk, 16), 2 * kBlk * kBlk, 0, s>>>(mk.nx, mk.ny, mk.bnx, mk.blist, mk.nact,
                                                                mk.cell_start, mk.ids, mk.stab, Fx, Fy);
}

// Grid of the strip-area kernel: kClipBlocks clip blocks, then 8 CTAs of
// 256 threads per SM for the flat pair loop (grid-stride).
int band_area_grid() { return kClipBlocks + 8 * sm_count(); }

// Strip areas of the current band pair list (idempotent: pacc, pcov only).
void launch_band_area(const Markers &mk, cudaStream_t s)
{
    note_launch();
    k_band_area<<<band_area_grid(), 256, 0, s>>>(mk.nx, mk.npairs, mk.pair_cap, mk.pseg, mk.pcell,
                                                 mk.clip_list, mk.sl, mk.slf, mk.scvx, mk.sv, mk.sb5, mk.pacc,
                                                 mk.pcov);
}

void launch_heaviside(const Markers &mk, double *H, cudaStream_t s, cudaStream_t side,
                      cudaEvent_t ev_fork, cudaEvent_t ev_join)
{
    // the scanline fill of the rows inside the drops needs neither the
    // sort nor the segment records: with a side stream it runs next to the
    // band kernels, joining before the band sum that reads its H
    cudaStream_t sr = s;
    if (side) {
        cudaEventRecord(ev_fork, s);
        cudaStreamWaitEvent(side, ev_fork, 0);
        sr = side;
    }
    note_launch();
    k_rows_inside<<<mk.ny, kT, 0, sr>>>(mk.ndrops, mk.nx, mk.h, mk.x0, mk.y0, mk.X, mk.Y, mk.ykey,
                                        mk.colkey, mk.next, mk.drop_start, mk.dyk, H, mk.flags);
    if (side) cudaEventRecord(ev_join, side);
    cudaMemsetAsync(mk.npairs, 0, 2 * sizeof(uint32_t), s);  // pairs, listed clip pairs
    note_launch();
    k_band_pairs<<<block_grid(mk, 7), kPairT, 0, s>>>(mk.nx, mk.ny, mk.bnx, mk.blist, mk.nact,
                                   mk.cell_start, mk.ids, mk.slf, mk.scvx, mk.sbox, mk.pair_cap, mk.npairs, mk.pseg, mk.pcell,
                                   mk.crange, mk.clip_list, mk.flags);
    launch_band_area(mk, s);
    if (side) cudaStreamWaitEvent(s, ev_join, 0);
    note_launch();
    k_band_sum<<<block_grid(mk, 32), kBT, 0, s>>>(mk.nx, mk.ny, mk.bnx, mk.blist, mk.nact, mk.crange,
                                                  mk.pacc, mk.pcov, H);
}

void launch_spread_irrot(const Markers &mk, const double *fmag, const double *H, double *Fx,
                         double *Fy, cudaStream_t s)
{
    cudaMemsetAsync(Fx, 0, (size_t)(mk.nx + 1) * mk.ny * 8, s);
    cudaMemsetAsync(Fy, 0, (size_t)mk.nx * (mk.ny + 1) * 8, s);
    note_launch();
    k_spread_irrot<<<block_grid(mk, 7), kIrrT, 0, s>>>(mk.nx, mk.ny, 1.0 / mk.h, mk.bnx, mk.blist, mk.nact,
                                       mk.cell_start, mk.ids, mk.next, mk.gx, mk.gy, mk.sinv, mk.gxf, mk.gyf, fmag,
                                       H, Fx, Fy, mk.flags);
}

// Shared memory of k_reloc_fit: 19 doubles a marker.  Its layout takes a drop
// of at least 32 markers, so that the scratch in sp and qs fits.
static int relocate_maxn(int maxn) { return std::max(maxn, 32); }
size_t relocate_smem(int maxn)
{
    const size_t n = (size_t)relocate_maxn(maxn);
    return (19 * n + 11) * 8;
}

// ------------------------------------------------------------ measure correction
// Section 2.5 (conservation of mass).  The measure of a drop: planar, the
// enclosed area by the shoelace sum in marker order; axisymmetric, the volume
// of revolution 2 pi sum (z2 - z1) (r1^2 + r1 r2 + r2^2) / 6 over the right
// half of the meridian (markers 0 .. n/2).  Serial in marker order.
__device__ double drop_measure(int n, const double *X, const double *Y, int axisym)
{
    double a = 0.0;
    if (!axisym) {
        for (int k = 0; k < n; k++) {
            const int q = (k + 1 == n) ? 0 : k + 1;
            a += X[k] * Y[q] - X[q] * Y[k];
        }
        return 0.5 * a;
    }
    for (int k = 0; k < n / 2; k++) {
        const double r1 = X[k], z1 = Y[k], r2 = X[k + 1], z2 = Y[k + 1];
        a += (z2 - z1) * (r1 * r1 + r1 * r2 + r2 * r2) / 6.0;
    }
    return 2.0 * 3.14159265358979323846 * a;
}

// Initial measure of every drop (one thread per drop).
__global__ void k_drop_measure(int ndrops, const int32_t *__restrict__ drop_start,
                               const double *__restrict__ X, const double *__restrict__ Y,
                               int axisym, double *__restrict__ A)
{
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= ndrops) return;
    const int s = drop_start[d], n = drop_start[d + 1] - s;
    A[d] = drop_measure(n, X + s, Y + s, axisym);
}

// Where |A - A0| > tol A0, one offset eps along the inward unit normals (of
// the uncorrected markers) restores the measure: bisection on [-h, h] until
// the bracket is below 1e-13 h or 80 halvings, eps its midpoint; eps_out (may
// be NULL) gets 0 where nothing moved.
//
// One block per drop.  Every decision is the one that the serial sum takes
// (drop_measure: the terms in marker order), to the bit, since near the root
// it is taken on rounding: the block forms the terms (the same operations)
// and first adds them in a tree together with their magnitudes; the serial
// sum differs from that by at most n 2^-52 sum |t|, so where the tree's value
// is further than that from A0 the decision is settled, and only otherwise
// (the last third of the halvings) does one thread add the terms, kept in
// shared memory, in order.  One thread per drop evaluating everything
// serially is a chain of FP64 and memory latencies: 4.87 ms for 16 drops of 256
// markers, here 0.30 ms.
constexpr int kMcT = 256, kMcTile = 2048;
__global__ void __launch_bounds__(kMcT)
k_mass_correct(const int32_t *__restrict__ drop_start, const double *__restrict__ A0, int axisym,
               double tol, double h, const double *__restrict__ nxm,
               const double *__restrict__ nym, double *__restrict__ X, double *__restrict__ Y,
               double *__restrict__ eps_out)
{
    __shared__ double terms[kMcTile], sh[2][kMcT / 32];
    __shared__ double result;
    const int d = blockIdx.x, s = drop_start[d], n = drop_start[d + 1] - s;
    const double *Xd = X + s, *Yd = Y + s, *nx = nxm + s, *ny = nym + s;
    const int nt = axisym ? n / 2 : n;  // terms of the sum
    const double scale = axisym ? 2.0 * 3.14159265358979323846 : 0.5;
    // term k of drop_measure at offset e (off: the markers as they are)
    auto term = [&](int k, double e, bool off) {
        const int q = (k + 1 == n) ? 0 : k + 1;
        const double xk = off ? Xd[k] : Xd[k] + e * nx[k], yk = off ? Yd[k] : Yd[k] + e * ny[k];
        const double xq = off ? Xd[q] : Xd[q] + e * nx[q], yq = off ? Yd[q] : Yd[q] + e * ny[q];
        if (!axisym) return xk * yq - xq * yk;
        return (yq - yk) * (xk * xk + xk * xq + xq * xq) / 6.0;
    };
    // the serial sum, in every thread
    auto serial = [&](double e, bool off) {
        double a = 0.0;
        for (int base = 0; base < nt; base += kMcTile) {
            const int m = min(kMcTile, nt - base);
            __syncthreads();
            for (int k = threadIdx.x; k < m; k += kMcT) terms[k] = term(base + k, e, off);
            __syncthreads();
            if (threadIdx.x == 0) {
#pragma unroll 8
                for (int k = 0; k < m; k++) a += terms[k];
            }
        }
        if (threadIdx.x == 0) result = scale * a;
        __syncthreads();
        return result;
    };
    const double a0 = A0[d];
    const double A = serial(0.0, true);
    if (threadIdx.x == 0 && eps_out) eps_out[d] = 0.0;
    if (!(fabs(A - a0) > tol * a0)) return;
    double lo = -h, hi = h;
    for (int it = 0; it < 80 && hi - lo > 1e-13 * h; it++) {
        const double mid = 0.5 * (lo + hi);
        double t = 0.0, m = 0.0;
        for (int k = threadIdx.x; k < nt; k += kMcT) {
            const double v = term(k, mid, false);
            t += v;
            m += fabs(v);
        }
        for (int o = 16; o; o >>= 1) {
            t += __shfl_xor_sync(0xffffffffu, t, o);
            m += __shfl_xor_sync(0xffffffffu, m, o);
        }
        __syncthreads();
        if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = t; sh[1][threadIdx.x >> 5] = m; }
        __syncthreads();
        t = 0.0; m = 0.0;
        for (int w = 0; w < kMcT / 32; w++) { t += sh[0][w]; m += sh[1][w]; }
        // 2.2204e-16 = 2^-52; the factor 4 covers the rounding of the two
        // sums of magnitudes and of the scaled results
        const double v = scale * t, slack = 4.0 * 2.2204460492503131e-16 * (n * (scale * m) + fabs(a0));
        bool above;
        if (fabs(v - a0) > slack) above = v > a0;
        else above = serial(mid, false) > a0;
        if (above) lo = mid;
        else hi = mid;
    }
    const double eps = 0.5 * (lo + hi);
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += kMcT) {
        X[s + k] = X[s + k] + eps * nx[k];
        Y[s + k] = Y[s + k] + eps * ny[k];
    }
    if (threadIdx.x == 0 && eps_out) eps_out[d] = eps;
}

void launch_drop_measure(const Markers &mk, int axisym, double *A, cudaStream_t s)
{
    note_launch();
    k_drop_measure<<<cdiv(mk.ndrops, 128), 128, 0, s>>>(mk.ndrops, mk.drop_start, mk.X, mk.Y,
                                                        axisym, A);
}

void launch_mass_correct(Markers &mk, const double *A0, int axisym, double tol, double *eps,
                         cudaStream_t s)
{
    note_launch();
    k_mass_correct<<<mk.ndrops, kMcT, 0, s>>>(mk.drop_start, A0, axisym, tol, mk.h, mk.nxm, mk.nym,
                                              mk.X, mk.Y, eps);
}

void launch_relocate(Markers &mk, bool serial, cudaStream_t s)
{
    size_t sm = relocate_smem(mk.max_drop);
    if (serial) {
        raise_smem_limit((const void *)k_reloc_fit_serial, (int)sm);
        note_launch(2);
        k_reloc_fit_serial<<<mk.ndrops, kT, sm, s>>>(mk.X, mk.Y, mk.drop_start, mk.h,
                                                     relocate_maxn(mk.max_drop), mk.rfit, mk.rpar,
                                                     mk.rwts, mk.flags);
        k_reloc_place_serial<<<cdiv(8L * mk.M, kPlaceT), kPlaceT, 0, s>>>(
            mk.M, mk.drop_of, mk.drop_start, mk.rfit, mk.rpar, mk.X, mk.Y);
        return;
    }
    raise_smem_limit((const void *)k_reloc_fit, (int)sm);
    note_launch();
    k_reloc_fit<<<mk.ndrops, kT, sm, s>>>(mk.X, mk.Y, mk.drop_start, mk.h, relocate_maxn(mk.max_drop), mk.rfit,
                                          mk.rpar, mk.rwts, mk.flags);
    note_launch();
    auto place = [&](auto kernel, int ln) {
        kernel<<<cdiv((long)ln * mk.M, kPlaceT), kPlaceT, 0, s>>>(mk.M, mk.drop_of, mk.drop_start,
                                                                  mk.rfit, mk.rpar, mk.X, mk.Y);
    };
    if (mk.M < 4096) place(k_reloc_place<8>, 8);
    else if (mk.M < 8192) place(k_reloc_place<4>, 4);
    else place(k_reloc_place<1>, 1);
}

}  // namespace ibk
