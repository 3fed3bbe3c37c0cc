// Face/cell kernels of one time step: properties and face coefficients
// (Section 2.2 Eq. (indicator), Section 2.1), the pressure right-hand side
// and velocity correction with the force in the projection (Section 2.1
// Eq. (ps), Section 3.2 Eq. (ns2_new)), and the AB2 advection + explicit
// viscous predictor (Section 2.1 Eqs. (ad_bf), (cr_ni)).
//
// All kernels are single-pass, one thread per cell or face, coalesced along
// x.  FP64 arithmetic bounds them on this part before HBM (1.25 TFLOP/s), so
// they are written for few FP64 operations.
#include <utility>

#include "ib_internal.cuh"

namespace ibk {
namespace {

constexpr int kT = 256;

// 2 x for a normal x, and not finite for an infinity or a NaN, by an addition to the
// exponent (x + x where that does not give the double would cost k_coeffs a fifth).
__device__ __forceinline__ double twice(double x)
{
    const int hi = __double2hiint(x);
    return __hiloint2double(hi + ((hi & 0x7ff00000) == 0x7ff00000 ? 0 : 0x00100000), __double2loint(x));
}

// rho and mu of the cells and beta = 1 / (two-cell mean of rho) on the faces.
// A warp takes 31 columns (lane 0 serves its neighbour) of ROWS rows;
// where a row of H equals the one below in all its lanes, as it does off the
// interface, rho, mu and beta are those of the row below, and no FP64
// operation is needed (ten a cell bound the two kernels that this one replaces;
// next to the face force 8 + 41 us at 1024^2, now 15, and 85 + 64 at 2048^2,
// now 49).  ROWS: 1 below 2^18 cells, 4 up to 2^20, 8 from there.  Alone, with one
// row, 4 and 8 (drops; values that never repeat): 64^2 2.4, 4.7, 7.7 us; 256^2
// 3.3, 4.4, 7.0; 512^2 7.9, 6.2, 7.4 (7.9, 7.6, 7.8); 64 x 4096 10.1, 10.5, 13.2;
// 960 x 640 14.9, 10.7, 12.0 (15.0, 16.3, 19.0); 960^2 21.1, 13.5, 12.6 (21.2, 22.0,
// 24.7); 1024^2 24.3, 13.9, 13.7 (24.2, 24.9, 24.7); 2048^2 90, 38.7, 32.0 (90, 86, 88);
// the two kernels: 10.7 at 64 x 4096, 19.5 at 960 x 640, 30.7 at 1024^2.
template <int ROWS>
__global__ void __launch_bounds__(256)
k_coeffs(int nx, int ny, double rho_g, double drho, double mu_g, double dmu,
         const double *__restrict__ H, double *__restrict__ rho, double *__restrict__ mu,
         double *__restrict__ bx, double *__restrict__ by)
{
    const int lane = threadIdx.x & 31, sx = (nx + 30) / 31;
    const int wid = blockIdx.x * (256 / 32) + (threadIdx.x >> 5), ty = wid / sx, j0 = ty * ROWS;
    if (j0 >= ny) return;  // whole warps
    const int i = (wid - ty * sx) * 31 + lane - 1, c = min(max(i, 0), nx - 1);
    const bool out = lane >= 1 && i < nx;
    double h[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; r++) h[r] = H[(long)min(j0 + r, ny - 1) * nx + c];
    double rc = rho_g + drho * H[(long)max(j0 - 1, 0) * nx + c], mc = 0.0, xv = 0.0, yv = 0.0;
    bool steady = false;  // yv is the face between two equal rows
#pragma unroll
    for (int r = 0; r < ROWS; r++) {
        const int j = j0 + r;
        if (j >= ny) break;
        if (r > 0 && __all_sync(0xffffffffu, __double_as_longlong(h[r]) == __double_as_longlong(h[r - 1]))) {
            if (!steady) yv = twice(recip_nr(rc + rc));
            steady = true;
        } else {
            const double rn = rho_g + drho * h[r];
            mc = mu_g + dmu * h[r];
            xv = twice(recip_nr(__shfl_up_sync(0xffffffffu, rn, 1) + rn));
            yv = twice(recip_nr(rc + rn));
            rc = rn;
            steady = false;
        }
        if (out) {
            const long k = (long)j * nx + i, kx = (long)j * (nx + 1) + i;
            rho[k] = rc;
            mu[k] = mc;
            bx[kx] = i == 0 ? 0.0 : xv;
            by[k] = j == 0 ? 0.0 : yv;
            if (i == nx - 1) bx[kx + 1] = 0.0;
            if (j == ny - 1) by[k + nx] = 0.0;
        }
    }
}

// The force is zero on all faces but those of the interface band: where a
// warp's faces carry none, its part is skipped (12 FP64 operations a cell to 4;
// 1024^2 21.1 -> 10.0 us, 19.0 with a force everywhere), unless a coefficient is
// infinite or NaN, which reaches b whatever the force.
__global__ void k_rhs(int nx, int ny, double ih, double ihdt,
                      const double *__restrict__ us, const double *__restrict__ vs,
                      const double *__restrict__ Fx, const double *__restrict__ Fy,
                      const double *__restrict__ bx, const double *__restrict__ by,
                      double *__restrict__ b)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i >= nx) return;
    const long xw = (long)j * (nx + 1) + i, ys = (long)j * nx + i, yn = ys + nx;
    const double fe = Fx[xw + 1], fw = Fx[xw], fn = Fy[yn], fs = Fy[ys];
    const double be = bx[xw + 1], bw = bx[xw], bn = by[yn], bs = by[ys];
    double v = ((us[xw + 1] - us[xw]) + (vs[yn] - vs[ys])) * ihdt;
    if (any_force(fe, fw, fn, fs) || any_unbounded(be, bw, bn, bs))
        v = fma(be * fe - bw * fw + bn * fn - bs * fs, ih, v);
    b[ys] = v;
}

// One face a thread, x-faces (blockIdx.y = 0) and y-faces by their index (below
// 2^32: the arrays of more would not fit the device), whose row and column are one
// unsigned division.  Bound by HBM; a thread for the two faces of a cell, a row of
// cells a block, left memory idle on narrow grids: 128 x 1024 5.8 us, now 3.8, 100 x
// 3000 7.9 and 6.4, 512^2 6.2 and 5.8, 1024^2 18.6 and 17.9, 2048^2 67.3 and 65.9.
__global__ void __launch_bounds__(kT)
k_correct(int nx, int ny, double ih, double dt,
          const double *__restrict__ us, const double *__restrict__ vs,
          const double *__restrict__ p, const double *__restrict__ Fx,
          const double *__restrict__ Fy, const double *__restrict__ bx,
          const double *__restrict__ by, double *__restrict__ u,
          double *__restrict__ v)
{
    const unsigned k = blockIdx.x * kT + threadIdx.x, W = nx;
    if (blockIdx.y == 0) {
        if (k >= (W + 1) * ny) return;
        const unsigned j = k / (W + 1), i = k - j * (W + 1), c = k - j;  // the cell to the east
        u[k] = i == 0 || i == W ? 0.0 : fma(dt, bx[k] * fma(-ih, p[c] - p[c - 1], Fx[k]), us[k]);
    } else {
        const unsigned n = W * (ny + 1);
        if (k >= n) return;
        // the cell to the north
        v[k] = k < W || k >= n - W ? 0.0 : fma(dt, by[k] * fma(-ih, p[k] - p[k - W], Fy[k]), vs[k]);
    }
}

// Predictor: a warp marches up a strip of 30 columns (and one on either side
// for the neighbours' fluxes), rows j0 .. j0 + R - 1, one lane per column; the
// columns that whole strips leave over, where they are at most 14 or 6, are
// marched by 16 or 8 lanes, two or four ranges of rows a warp (64 columns were
// three strips: 64 x 4096 56 us, now 38, 32 x 4096 38 and 26).  A
// lane holds its column's rho, mu, u and v of the current and the next row,
// loads the row after next while it computes, and takes its neighbours'
// values by shuffles; every flux that two faces share is formed once: per
// cell the advective flux rho a^2 and the viscous flux mu du of each
// component, per node (the cell's lower left corner) the advective flux
// rho_n a_v a_u, one product for both components, and the viscous flux mu_n du
// of each.  Then the x-face left of and the y-face below the cell are updated
// (and the wall face on the far side by the last column / row).
//
// FP64 arithmetic bounds it (64 cycles an instruction for one warp, 19 an SM
// with four or more): 44 instructions a cell (40 off the interface), times
// 32/30 and (R + 1) / R.  A
// 32 x 8 tile with the fluxes in shared memory has partly filled warps in
// every pass over its ring and two barriers.  Next to the hierarchy's setup
// and the face force, as in a step: 1024^2 171 -> 127 us, 2048^2 665 -> 429,
// 256 x 1024 axisymmetric 107 -> 52.  R: rows per warp (pred_rows).
//
// Walls: a ghost row or column of the velocity reflected to zero on the wall
// (the outer wall of the axisymmetric form: to wb), of rho and mu equal to the
// row or column inside, makes the wall nodes' formula the inner one: twice the
// two wall cells' mean, and no advective flux through the wall.
//
// The fluxes are kept without their power-of-two factors (the 1/2 of each
// face average, the 1/4 of the node averages): 4 rho a^2 per cell, 16 rho_n a_v
// a_u and 4 mu_n du per node, folded into the factors of their differences.
//
// AXI: axisymmetric form (x = r, y = z).  Every flux carries the radius of its
// face and each balance is divided by the radius of its control volume; these
// ratios, a column's own, are formed once per lane.  The radial component
// adds -mu_face u / r^2.
constexpr int kPredT = 128, kPredCols = 30;
// Lanes for the columns left over by whole strips (0 if none are).
__host__ __device__ inline int pred_lanes(int nx)
{
    const int left = nx % kPredCols;
    return left == 0 ? 0 : (left <= 6 ? 8 : (left <= 14 ? 16 : 32));
}
// Warps of a grid, R rows a range.
inline long pred_warps(int nx, int ny, int R)
{
    const long rows = cdiv(ny, R);
    const int G = pred_lanes(nx);
    return nx / kPredCols * rows + (G ? cdiv(rows, 32 / G) : 0);
}
template <bool AXI>
__global__ void __launch_bounds__(kPredT)
k_predictor(int nx, int ny, int R, double ih, double visc, double dt,
            const double *__restrict__ rho, const double *__restrict__ mu,
            const double *__restrict__ u, const double *__restrict__ v,
            const double *aup, const double *avp,  // may be au, av
            int have_prev, double gx, double gy, const double *__restrict__ frame,
            const double *__restrict__ bx, const double *__restrict__ by,
            double *__restrict__ us, double *__restrict__ vs, double *au, double *av)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int sx = nx / kPredCols, rows = (ny + R - 1) / R, whole = sx * rows;
    const int wid = blockIdx.x * (kPredT / 32) + (threadIdx.x >> 5);
    const bool rest = wid >= whole;             // a warp of the columns left over
    const int GL = rest ? pred_lanes(nx) : 32;  // lanes of a range
    if (GL == 0) return;
    const int lane = threadIdx.x & (GL - 1);
    // the warp's first range, and this lane's
    const int w0 = rest ? (wid - whole) * (32 / GL) : wid / sx;
    const int ty = w0 + (rest ? (threadIdx.x & 31) / GL : 0);
    if (w0 >= rows) return;  // whole warps
    const int n = min(R, ny - w0 * R);
    const int j0 = min(ty * R, ny - 1);  // a range beyond the grid writes nothing
    const int i = (rest ? sx : wid - w0 * sx) * kPredCols + lane - 1;
    const bool out = lane >= 1 && lane <= GL - 2 && i < nx && ty < rows;
    const long nxf = nx + 1;
    // columns to load from: cell and y-face data of column c, x-faces of cu
    const int c = min(max(i, 0), nx - 1), cu = min(max(i, 0), nx);
    const double wb = AXI && frame ? frame[kFrWb] : 0.0;
    if constexpr (AXI) gy += frame ? frame[kFrS] : 0.0;
    auto neg = [](double x) {
        return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ULL);
    };
    auto ld_u = [&](int j) {  // row j, reflected beyond the walls
        if (j < 0) return neg(u[cu]);
        return j < ny ? u[(long)j * nxf + cu] : neg(u[(long)(ny - 1) * nxf + cu]);
    };
    auto ld_v = [&](int j) {  // y-face row j (0 .. ny), reflected beyond the side walls
        const double x = v[(long)j * nx + c];
        if (AXI) return i >= nx ? 2.0 * wb - x : x;
        return i < 0 || i >= nx ? neg(x) : x;
    };
    auto row = [&](int j) { return (long)min(max(j, 0), ny - 1) * nx + c; };
    auto up = [&](double x) { return __shfl_up_sync(kAll, x, 1, GL); };
    auto down = [&](double x) { return __shfl_down_sync(kAll, x, 1, GL); };
    // the factors of the differences
    const double hdt = 0.5 * dt, v2 = 2.0 * visc * ih * ih;
    const double gx2 = 2.0 * gx, gy2 = 2.0 * gy, ca = have_prev ? -3.0 : -2.0;
    double xi = 0.25 * ih, xw = xi, xv = v2, xvw = v2, xm = 0.0;  // x-face: cells i, i-1
    double ge = 0.0625 * ih, gw = ge, we = 0.25 * v2, ww = we;    // y-face: nodes i+1, i
    const double ih4 = 0.25 * ih, ih16 = 0.0625 * ih, v24 = 0.25 * v2;
    if constexpr (AXI) {
        const double rf = i > 0 ? recip_any((double)i) : 0.0, rc = recip_any((double)i + 0.5);
        const double a = ((double)i + 0.5) * rf, b = ((double)i - 0.5) * rf;
        xi = a * ih4; xw = b * ih4; xv = a * v2; xvw = b * v2;
        xm = -(visc * ih * ih) * (rf * rf);
        const double e = ((double)i + 1.0) * rc, w = (double)i * rc;
        ge = i + 1 == nx ? 0.0 : e * ih16;  // no flux through the outer wall
        gw = w * ih16; we = e * v24; ww = w * v24;
    }
    // rows j0 - 1 (m), j0 (0) and j0 + 1 (1)
    double r0, m0, u0, v0, G, Wx, Wy, fyp, vyp, rm, rn = 0.0, mn = 0.0;
    bool steady = false;
    double r1 = rho[row(j0 + 1)], m1 = mu[row(j0 + 1)], u1 = ld_u(j0 + 1), v1 = ld_v(j0 + 1);
    {
        rm = rho[row(j0 - 1)];
        const double mm = mu[row(j0 - 1)], um = ld_u(j0 - 1), vm = ld_v(max(j0 - 1, 0));
        r0 = rho[row(j0)]; m0 = mu[row(j0)]; u0 = ld_u(j0); v0 = ld_v(j0);
        const double rs = rm + r0, ms = mm + m0, vl = up(v0);
        const double rb = rs + up(rs), mb = ms + up(ms), b = vm + v0;
        G = rb * (vl + v0) * (um + u0);
        Wx = mb * (u0 - um);
        Wy = mb * (v0 - vl);
        fyp = rm * b * b;
        vyp = mm * (v0 - vm);
    }
    for (int j = j0; j < j0 + n; j++) {
        const long kx = (long)j * nxf + i, ky = (long)j * nx + i;
        const bool wr = out && j < ny;
        double ap = 0.0, bp = 0.0, irx = 0.0, iry = 0.0;
        if (wr) {
            if (have_prev) { ap = aup[kx]; bp = avp[ky]; }
            if (bx) { irx = bx[kx]; iry = by[ky]; }
        }
        // the row after next (the last one's is not used)
        const int jn = min(j + 2, ny);
        const double r2 = rho[row(jn)], m2 = mu[row(jn)], u2 = ld_u(jn), v2n = ld_v(jn);
        // cell fluxes of row j, node fluxes of node row j + 1
        const double ue = down(u0), a = ue + u0, b = v1 + v0, vl = up(v1);
        const double fx = r0 * a * a, vx = m0 * (ue - u0);
        const double fy = r0 * b * b, vy = m0 * (v1 - v0);
        // rows j and j + 1 alike in all lanes, as rows j - 1 and j were: the
        // nodes' rho and mu are those of the row below
        const bool eq = __all_sync(kAll, __double_as_longlong(r1) == __double_as_longlong(r0) &&
                                             __double_as_longlong(m1) == __double_as_longlong(m0));
        if (!(eq && steady)) {
            const double rs = r0 + r1, ms = m0 + m1;
            rn = rs + up(rs);
            mn = ms + up(ms);
        }
        steady = eq;
        const double G1 = rn * (vl + v1) * (u0 + u1);
        const double Wx1 = mn * (u1 - u0), Wy1 = mn * (v1 - vl);
        const double fw = up(fx), vw = up(vx), Ge = down(G), We = down(Wy);
        const double mw = AXI ? up(m0) : 0.0, rw = bx ? 0.0 : up(r0);
        if (wr) {
            if (!bx) {
                irx = recip_div(0.5 * (rw + r0));
                iry = recip_div(0.5 * (rm + r0));
            }
            if (i == 0) {
                us[kx] = 0.0; au[kx] = 0.0;
            } else {
                double adv, q;
                if constexpr (AXI) adv = fma(xi, fx, fma(-xw, fw, ih16 * (G1 - G)));
                else adv = fma(G1 - G, ih16, (fx - fw) * ih4);
                // twice (viscous - (3/2 adv - 1/2 adv before)), or - adv in the
                // first step; its half in dt / 2
                q = fma(ca, adv, ap);
                if constexpr (AXI)
                    q = fma(xv, vx, fma(-xvw, vw, fma(v24, Wx1 - Wx, fma(xm, (mw + m0) * u0, q))));
                else
                    q = fma(v2, fma(-0.25, Wx, fma(0.25, Wx1, vx - vw)), q);
                us[kx] = fma(hdt, fma(q, irx, gx2), u0);
                au[kx] = adv;
            }
            if (i == nx - 1) { us[kx + 1] = 0.0; au[kx + 1] = 0.0; }  // the right wall's face
            if (j == 0) {
                vs[ky] = wb; av[ky] = 0.0;
            } else {
                double adv, q;
                if constexpr (AXI) adv = fma(ge, Ge, fma(-gw, G, (fy - fyp) * ih4));
                else adv = fma(Ge - G, ih16, (fy - fyp) * ih4);
                q = fma(ca, adv, bp);
                if constexpr (AXI) q = fma(v2, vy - vyp, fma(we, We, fma(-ww, Wy, q)));
                else q = fma(v2, fma(-0.25, Wy, fma(0.25, We, vy - vyp)), q);
                vs[ky] = fma(hdt, fma(q, iry, gy2), v0);
                av[ky] = adv;
            }
            if (j == ny - 1) { vs[ky + nx] = wb; av[ky + nx] = 0.0; }  // the top wall's face
        }
        G = G1; Wx = Wx1; Wy = Wy1; fyp = fy; vyp = vy; rm = r0;
        r0 = r1; m0 = m1; u0 = u1; v0 = v1;
        r1 = r2; m1 = m2; u1 = u2; v1 = v2n;
    }
}

// Crank-Nicolson viscous step (Section 2.1): one red-black colour of a
// Gauss-Seidel sweep on u* - dt / (2 rho_f) D(u*) = u_e for both components
// at once (they do not couple), in place, boundary faces fixed.  D is the
// predictor's div(mu grad): cell mu on normal faces, node averages on
// tangential ones, a no-slip wall by the reflected ghost (moving with the
// frame's axial velocity wb at the axisymmetric outer wall); axisymmetric:
// fluxes times their face radius over the volume radius and -mu_f u / r^2
// on the radial component, zero flux through the axis.
__global__ void k_cn_sweep(int nx, int ny, double h, double dt, const double *__restrict__ rho,
                           const double *__restrict__ mu, int axisym,
                           const double *__restrict__ frame, int color,
                           const double *__restrict__ ue, const double *__restrict__ ve,
                           double *__restrict__ us, double *__restrict__ vs)
{
    const long nxf = nx + 1;
    long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long nu = nxf * ny;
    auto M = [&](int i, int j) { return mu[(long)j * nx + i]; };
    if (k < nu) {
        const int j = (int)(k / nxf), i = (int)(k - (long)j * nxf);
        if (i == 0 || i == nx || ((i + j) & 1) != color) return;
        const double r0 = axisym ? i * h : 1.0, rE = axisym ? (i + 0.5) * h : 1.0,
                     rW = axisym ? (i - 0.5) * h : 1.0;
        const double s = 1.0 / (r0 * h * h);
        const double muN = (j + 1 < ny) ? 0.25 * (M(i - 1, j) + M(i, j) + M(i - 1, j + 1) + M(i, j + 1))
                                        : 0.5 * (M(i - 1, j) + M(i, j));
        const double muS = (j > 0) ? 0.25 * (M(i - 1, j - 1) + M(i, j - 1) + M(i - 1, j) + M(i, j))
                                   : 0.5 * (M(i - 1, j) + M(i, j));
        const double cE = rE * M(i, j) * s, cW = rW * M(i - 1, j) * s;
        const double cN = r0 * muN * s, cS = r0 * muS * s;
        double ex = 0.0, nb = cE * us[k + 1] + cW * us[k - 1], cs = cE + cW;
        if (j + 1 < ny) { nb += cN * us[k + nxf]; cs += cN; } else ex += 2.0 * cN;
        if (j > 0) { nb += cS * us[k - nxf]; cs += cS; } else ex += 2.0 * cS;
        if (axisym) ex += 0.5 * (M(i - 1, j) + M(i, j)) / (r0 * r0);
        const double tau = dt / (2.0 * (0.5 * (rho[(long)j * nx + i - 1] + rho[(long)j * nx + i])));
        us[k] = (ue[k] + tau * nb) / (1.0 + tau * (cs + ex));
        return;
    }
    k -= nu;
    if (k >= (long)nx * (ny + 1)) return;
    const int j = (int)(k / nx), i = (int)(k - (long)j * nx);
    if (j == 0 || j == ny || ((i + j) & 1) != color) return;
    const double r0 = axisym ? (i + 0.5) * h : 1.0, rE = axisym ? (i + 1) * h : 1.0,
                 rW = axisym ? i * h : 1.0;
    const double s = 1.0 / (r0 * h * h);
    const double muE = (i + 1 < nx) ? 0.25 * (M(i, j - 1) + M(i + 1, j - 1) + M(i, j) + M(i + 1, j))
                                    : 0.5 * (M(i, j - 1) + M(i, j));
    const double muW = (i > 0) ? 0.25 * (M(i - 1, j - 1) + M(i, j - 1) + M(i - 1, j) + M(i, j))
                               : 0.5 * (M(i, j - 1) + M(i, j));
    const double cN = r0 * M(i, j) * s, cS = r0 * M(i, j - 1) * s;
    const double cE = rE * muE * s, cW = rW * muW * s;
    const double wb = frame ? frame[kFrWb] : 0.0;
    double ex = 0.0, nb = cN * vs[k + nx] + cS * vs[k - nx], cs = cN + cS;
    if (i + 1 < nx) { nb += cE * vs[k + 1]; cs += cE; } else { ex += 2.0 * cE; nb += 2.0 * cE * wb; }
    if (i > 0) { nb += cW * vs[k - 1]; cs += cW; }
    else if (!axisym) ex += 2.0 * cW;
    const double tau = dt / (2.0 * (0.5 * (rho[(long)(j - 1) * nx + i] + rho[(long)j * nx + i])));
    vs[k] = (ve[k] + tau * nb) / (1.0 + tau * (cs + ex));
}

// The same solve with its coefficients formed once (k_cn_coeffs) and two
// sweeps a launch (k_cn_smooth).  k_cn_sweep forms every coefficient of a
// face, with two divisions, in each of its 2 nsweeps half sweeps: ~60 FP64
// operations where the update itself needs four, and FP64 arithmetic is what
// bounds it on this part (20 sweeps at 512^2: 40 launches, 2.53 ms).
//
// k_cn_coeffs: per face the update u <- r + W u_W + E u_E + S u_S + N u_N of
// k_cn_sweep, u = (u_e + tau nb) / (1 + tau (cs + ex)), as four weights and a
// right-hand side (w[2k], w[2k + 1], r[k]; x-faces then y-faces, blockIdx.z).
// Boundary faces get zero weights and their own value.  Bound by the FP64 pipe,
// some 45 instructions a face.  So a thread takes a column's ROWS rows, and where
// the cells that a face's coefficients depend on equal those of the face below,
// as off the interface, it keeps that face's: one product is left.  Single-warp
// blocks spread the warps along an interface over the SMs (512^2: 52 us with a
// face a thread; 8 rows 43 us in blocks of 128 and 33 in blocks of 32; 16 rows
// 43, 4 rows 36, 2 rows 49).  A thread's 8 rows take 21 us whatever the size, so
// small grids have one row a thread: 160 x 480 cells 22 us with 8 and 21 with 1,
// 320^2 24 and 27, 1024^2 68 and 231.
constexpr int kCnT = 32;
constexpr long kCnRowCells = 90000;  // 8 rows a thread from here up
template <int ROWS>
__global__ void __launch_bounds__(kCnT)
k_cn_coeffs(int nx, int ny, double h, double dt, const double *__restrict__ rho,
            const double *__restrict__ mu, int axisym, const double *__restrict__ frame,
            const double *__restrict__ ue, const double *__restrict__ ve, double2 *__restrict__ w,
            double *__restrict__ r)
{
    const long nxf = nx + 1, nu = nxf * ny;
    const int i = blockIdx.x * kCnT + threadIdx.x, j0 = blockIdx.y * ROWS;
    auto M = [&](int a, int j) { return mu[(long)j * nx + a]; };
    auto same = [](double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); };
    const double2 zero = make_double2(0.0, 0.0);
    double2 we = zero, sn = zero;  // the weights, (W, E) and (S, N)
    double g = 0.0, ghost = 0.0;   // of the right-hand side; of the moving outer wall
    double p0 = 0.0, p1 = 0.0, p2 = 0.0, q0 = 0.0, q1 = 0.0;  // the face below's mu, rho
    bool even = false;             // its cells were alike along y
    if (blockIdx.z == 0) {
        if (i > nx) return;
        const double r0 = axisym ? i * h : 1.0, rE = axisym ? (i + 0.5) * h : 1.0,
                     rW = axisym ? (i - 0.5) * h : 1.0;
#pragma unroll 1
        for (int j = j0; j < min(j0 + ROWS, ny); j++) {
            const long f = (long)j * nxf + i;
            if (i == 0 || i == nx) {
                w[2 * f] = zero; w[2 * f + 1] = zero;
                r[f] = ue[f];
                continue;
            }
            const bool n = j + 1 < ny, b = j > 0;
            const double m0 = M(i - 1, j), m1 = M(i, j);
            const double n0 = n ? M(i - 1, j + 1) : 0.0, n1 = n ? M(i, j + 1) : 0.0;
            const double s0 = b ? M(i - 1, j - 1) : 0.0, s1 = b ? M(i, j - 1) : 0.0;
            const double d0 = rho[(long)j * nx + i - 1], d1 = rho[(long)j * nx + i];
            const bool ev = n && b && same(n0, m0) && same(n1, m1) && same(s0, m0) && same(s1, m1);
            if (!(ROWS > 1 && ev && even && same(m0, p0) && same(m1, p1) && same(d0, q0) && same(d1, q1))) {
                const double s = axisym ? recip_any(r0 * h * h) : recip_any(h * h);
                const double m = m0 + m1;
                const double muN = n ? 0.25 * (m + (n0 + n1)) : 0.5 * m;
                const double muS = b ? 0.25 * ((s0 + s1) + m) : 0.5 * m;
                const double cE = rE * m1 * s, cW = rW * m0 * s, cN = r0 * muN * s, cS = r0 * muS * s;
                // a wall's reflected ghost: twice its weight on the diagonal
                double d = (cE + cW) + (n ? cN : 2.0 * cN) + (b ? cS : 2.0 * cS);
                if (axisym) d += 0.5 * m * recip_any(r0 * r0);
                const double tau = dt * recip_div(d0 + d1);
                g = recip_div(1.0 + tau * d);
                const double tg = tau * g;
                we = make_double2(cW * tg, cE * tg);
                sn = make_double2(b ? cS * tg : 0.0, n ? cN * tg : 0.0);
            }
            even = ev; p0 = m0; p1 = m1; q0 = d0; q1 = d1;
            w[2 * f] = we; w[2 * f + 1] = sn;
            r[f] = ue[f] * g;
        }
        return;
    }
    if (i >= nx) return;
    const double r0 = axisym ? (i + 0.5) * h : 1.0, rE = axisym ? (i + 1) * h : 1.0,
                 rW = axisym ? i * h : 1.0;
    const bool e = i + 1 < nx, b = i > 0;
#pragma unroll 1
    for (int j = j0; j < min(j0 + ROWS, ny + 1); j++) {
        const long k = (long)j * nx + i, f = nu + k;
        if (j == 0 || j == ny) {
            w[2 * f] = zero; w[2 * f + 1] = zero;
            r[f] = ve[k];
            continue;
        }
        const double m0 = M(i, j - 1), m1 = M(i, j);
        const double e0 = e ? M(i + 1, j - 1) : 0.0, e1 = e ? M(i + 1, j) : 0.0;
        const double w0 = b ? M(i - 1, j - 1) : 0.0, w1 = b ? M(i - 1, j) : 0.0;
        const double d0 = rho[(long)(j - 1) * nx + i], d1 = rho[(long)j * nx + i];
        const bool ev = same(m0, m1) && same(e0, e1) && same(w0, w1);
        if (!(ROWS > 1 && ev && even && same(m1, p0) && same(e1, p1) && same(w1, p2) && same(d0, q0) &&
              same(d1, q1))) {
            const double s = axisym ? recip_any(r0 * h * h) : recip_any(h * h);
            const double m = m0 + m1;
            const double muE = e ? 0.25 * (m + (e0 + e1)) : 0.5 * m;
            const double muW = b ? 0.25 * ((w0 + w1) + m) : 0.5 * m;
            const double cN = r0 * m1 * s, cS = r0 * m0 * s, cE = rE * muE * s, cW = rW * muW * s;
            double d = (cN + cS) + (e ? cE : 2.0 * cE);
            if (b) d += cW;
            else if (!axisym) d += 2.0 * cW;
            const double tau = dt * recip_div(d0 + d1);
            g = recip_div(1.0 + tau * d);
            const double tg = tau * g;
            we = make_double2(b ? cW * tg : 0.0, e ? cE * tg : 0.0);
            sn = make_double2(cS * tg, cN * tg);
            ghost = 2.0 * cE * tg;
        }
        even = ev; p0 = m1; p1 = e1; p2 = w1; q0 = d0; q1 = d1;
        w[2 * f] = we; w[2 * f + 1] = sn;
        double v = ve[k] * g;
        if (!e && frame) v += ghost * frame[kFrWb];  // the outer wall moves with the frame
        r[f] = v;
    }
}

// NS red-black sweeps of both components in one launch, out of place: a block
// stages a DW x DH tile of one component with a halo of 2 NS faces, runs the
// 2 NS colour phases in shared memory on shrinking rings (so the tile equals
// NS global sweeps of k_cn_sweep up to rounding), reading the weights from L2
// (40 B a face), and stores the tile.  Blocks below nbu take x-faces, the
// rest y-faces.  Bound by the FP64 pipe (four operations an update, 1.15
// times that with the halo at 64 x 32 and NS = 2).
template <int NS, int DW, int DH>
__global__ void __launch_bounds__(256)
k_cn_smooth(int nx, int ny, int nbu, const double2 *__restrict__ w, const double *__restrict__ r,
            const double *__restrict__ uin, const double *__restrict__ vin,
            double *__restrict__ uout, double *__restrict__ vout)
{
    constexpr int HA = 2 * NS, PW = DW + 2 * HA, PH = DH + 2 * HA;
    __shared__ double ps[PH][PW];
    const bool isv = (int)blockIdx.x >= nbu;
    const int bk = (int)blockIdx.x - (isv ? nbu : 0);
    const int W = isv ? nx : nx + 1, Hh = isv ? ny + 1 : ny;
    const int tw = (W + DW - 1) / DW;
    const int gi0 = (bk % tw) * DW - HA, gj0 = (bk / tw) * DH - HA;
    const double *in = isv ? vin : uin;
    double *out = isv ? vout : uout;
    const long off = isv ? (long)(nx + 1) * ny : 0;
    for (int k = threadIdx.x; k < PH * PW; k += 256) {
        const int a = k / PW, c = k - a * PW, gi = gi0 + c, gj = gj0 + a;
        ps[a][c] = (gi >= 0 && gi < W && gj >= 0 && gj < Hh) ? in[(long)gj * W + gi] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int ph = 0; ph < 2 * NS; ph++) {
        const int q = HA - 1 - ph, color = ph & 1;
        const int hw = (DW + 2 * q) / 2, hq = DH + 2 * q;
        for (int k = threadIdx.x; k < hq * hw; k += 256) {
            const int rr = k / hw, cc = k - rr * hw;
            const int a = HA - q + rr, gj = gj0 + a;
            const int c = HA - q + 2 * cc + ((gi0 + HA - q + gj + color) & 1), gi = gi0 + c;
            if (gi < 0 || gi >= W || gj < 0 || gj >= Hh) continue;
            const long f = off + (long)gj * W + gi;
            const double2 we = w[2 * f], sn = w[2 * f + 1];
            double s = fma(we.x, ps[a][c - 1], r[f]);
            s = fma(we.y, ps[a][c + 1], s);
            s = fma(sn.x, ps[a - 1][c], s);
            ps[a][c] = fma(sn.y, ps[a + 1][c], s);
        }
        __syncthreads();
    }
    for (int k = threadIdx.x; k < DH * DW; k += 256) {
        const int a = HA + k / DW, c = HA + k % DW, gi = gi0 + c, gj = gj0 + a;
        if (gi < W && gj < Hh) out[(long)gj * W + gi] = ps[a][c];
    }
}

// Indicator function of Section 2.2 Eq. (ind_psn), div grad I = div G:
// the right-hand side div G of the face field G (the spread delta vector),
// r_i times the axisymmetric divergence in that form; unit coefficients with
// the walls at zero (r_face for the axisymmetric form).
__global__ void k_div_faces(int nx, int ny, double h, int axisym, const double *__restrict__ Gx,
                            const double *__restrict__ Gy, double *__restrict__ b)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i >= nx) return;
    const long xw = (long)j * (nx + 1) + i, ys = (long)j * nx + i, yn = ys + nx;
    if (!axisym) {
        b[ys] = (Gx[xw + 1] - Gx[xw] + Gy[yn] - Gy[ys]) / h;
        return;
    }
    const double ri = (i + 0.5) * h;
    b[ys] = ri * (((i + 1) * h * Gx[xw + 1] - i * h * Gx[xw]) / (ri * h) + (Gy[yn] - Gy[ys]) / h);
}

__global__ void k_unit_beta(int nx, int ny, double h, int axisym, double *__restrict__ bx,
                            double *__restrict__ by)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (j < ny && i <= nx) bx[(long)j * (nx + 1) + i] = (i == 0 || i == nx) ? 0.0 : (axisym ? i * h : 1.0);
    if (i < nx) by[(long)j * nx + i] = (j == 0 || j == ny) ? 0.0 : (axisym ? (i + 0.5) * h : 1.0);
}

// I = clamp(sol - mean over the cells along the walls (the axis column is not
// a wall), 0, 1): the mean by one block into *ref (each thread a strided
// share of the bottom row, top row, right column and, planar, left column,
// then a fixed tree; one thread alone took 53 us at 256^2, a chain of 1020
// additions), then the shift by a grid of threads.
__global__ void __launch_bounds__(kT)
k_wall_mean(int nx, int ny, int axisym, const double *__restrict__ sol, double *__restrict__ ref)
{
    __shared__ double sh[kT / 32];
    const int side = ny > 2 ? ny - 2 : 0, n = 2 * nx + side * (axisym ? 1 : 2);
    double s = 0.0;
    for (int k = threadIdx.x; k < n; k += kT) {
        long c;
        if (k < nx) c = k;
        else if (k < 2 * nx) c = (long)(ny - 1) * nx + k - nx;
        else if (k < 2 * nx + side) c = (long)(k - 2 * nx + 1) * nx + nx - 1;
        else c = (long)(k - 2 * nx - side + 1) * nx;
        s += sol[c];
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < kT / 32; w++) s += sh[w];
    *ref = s / (double)n;
}

__global__ void k_shift_clip(long n, const double *__restrict__ sol, const double *__restrict__ ref,
                             double *__restrict__ I)
{
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) I[k] = fmin(fmax(sol[k] - *ref, 0.0), 1.0);
}

// Initial guess of the pressure solve extrapolated in time: p <- 2 p - q,
// q <- the old p (p^n and p^(n-1) in, p0 = 2 p^n - p^(n-1) and p^n out).
__global__ void k_extrapolate(long n, double *__restrict__ p, double *__restrict__ q)
{
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double t = p[k];
    p[k] = 2.0 * t - q[k];
    q[k] = t;
}

__global__ void k_fill(long n, double a, double *__restrict__ y)
{
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) y[k] = a;
}

}  // namespace

void launch_cn_solve(int nx, int ny, double h, double dt, const double *rho, const double *mu,
                     int axisym, const double *frame, int nsweeps, const double *ue,
                     const double *ve, double *us, double *vs, cudaStream_t s)
{
    const long nf = (long)(nx + 1) * ny + (long)nx * (ny + 1);
    for (int sw = 0; sw < nsweeps; sw++)
        for (int c = 0; c < 2; c++) {
            note_launch();
            k_cn_sweep<<<cdiv(nf, kT), kT, 0, s>>>(nx, ny, h, dt, rho, mu, axisym, frame, c, ue, ve,
                                                   us, vs);
        }
}

int cn_launches(int nsweeps) { return (nsweeps + 1) / 2; }

// Tiles of 64 x 32 faces once they fill the device four times over, 32 x 16
// below, where a small grid's weights come from L2 with too few blocks in flight
// otherwise.  Two sweeps with 32 x 16 and with 64 x 32: 256^2 6.2 and 13.2 us, 384^2
// 10.4, 14.3, 512^2 15.1, 15.3, 640^2 21.3, 19.8, 768^2 27.5, 30.0, 800^2 (the line) 24.8,
// 26.0, 960^2 41.0, 38.7, 1024^2 47.7, 44.8, 1280 x 1024 58.5, 63.6, 2048^2 170, 157: from
// 512^2 on within 9 % either way as the last wave fills.
void launch_cn_solve_tab(int nx, int ny, double h, double dt, const double *rho, const double *mu,
                         int axisym, const double *frame, int nsweeps, double *w, double *r,
                         double *ua, double *va, double *ub, double *vb, cudaStream_t s)
{
    const long nf = (long)(nx + 1) * ny + (long)nx * (ny + 1);
    note_launch();
    auto coeffs = [&](auto kern, int rows) {
        kern<<<dim3(cdiv(nx + 1, kCnT), cdiv(ny + 1, rows), 2), kCnT, 0, s>>>(nx, ny, h, dt, rho, mu, axisym, frame,
                                                                           ua, va, (double2 *)w, r);
    };
    if ((long)nx * ny >= kCnRowCells) coeffs(k_cn_coeffs<8>, 8);
    else coeffs(k_cn_coeffs<1>, 1);
    auto go = [&](auto kern, int dw, int dh) {
        const int nbu = (int)(cdiv(nx + 1, dw) * cdiv(ny, dh)), nbv = (int)(cdiv(nx, dw) * cdiv(ny + 1, dh));
        note_launch();
        kern<<<nbu + nbv, 256, 0, s>>>(nx, ny, nbu, (const double2 *)w, (const double *)r, (const double *)ua,
                                       (const double *)va, ub, vb);
        std::swap(ua, ub);
        std::swap(va, vb);
    };
    const bool big = nf >= 4L * 152 * 64 * 32;
    int k = 0;
    for (; k + 2 <= nsweeps; k += 2) {
        if (big) go(k_cn_smooth<2, 64, 32>, 64, 32);
        else go(k_cn_smooth<2, 32, 16>, 32, 16);
    }
    if (k < nsweeps) {
        if (big) go(k_cn_smooth<1, 64, 32>, 64, 32);
        else go(k_cn_smooth<1, 32, 16>, 32, 16);
    }
}

void launch_div_faces(int nx, int ny, double h, int axisym, const double *Gx, const double *Gy,
                      double *b, cudaStream_t s)
{
    note_launch();
    k_div_faces<<<dim3(cdiv(nx, 128), ny), 128, 0, s>>>(nx, ny, h, axisym, Gx, Gy, b);
}

void launch_unit_beta(int nx, int ny, double h, int axisym, double *bx, double *by, cudaStream_t s)
{
    note_launch();
    k_unit_beta<<<dim3(cdiv(nx + 1, 128), ny + 1), 128, 0, s>>>(nx, ny, h, axisym, bx, by);
}

void launch_indicator_finish(int nx, int ny, int axisym, const double *sol, double *ref, double *I,
                             cudaStream_t s)
{
    note_launch();
    k_wall_mean<<<1, kT, 0, s>>>(nx, ny, axisym, sol, ref);
    const long n = (long)nx * ny;
    note_launch();
    k_shift_clip<<<cdiv(n, kT), kT, 0, s>>>(n, sol, ref, I);
}

void launch_extrapolate(long n, double *p, double *q, cudaStream_t s)
{
    note_launch();
    k_extrapolate<<<cdiv(n, kT), kT, 0, s>>>(n, p, q);
}

void launch_fill(long n, double a, double *y, cudaStream_t s)
{
    note_launch();
    k_fill<<<cdiv(n, kT), kT, 0, s>>>(n, a, y);
}

void launch_coeffs(int nx, int ny, double rho_g, double rho_l, double mu_g,
                   double mu_l, const double *H, double *rho, double *mu,
                   double *bx, double *by, cudaStream_t s)
{
    auto launch = [&](auto kernel, int rows) {
        const long warps = (long)cdiv(nx, 31) * cdiv(ny, rows);
        kernel<<<cdiv(warps, 256 / 32), 256, 0, s>>>(nx, ny, rho_g, rho_l - rho_g, mu_g, mu_l - mu_g, H, rho,
                                                     mu, bx, by);
    };
    note_launch();
    const long n = (long)nx * ny;
    if (n >= 1L << 20) launch(k_coeffs<8>, 8);
    else if (n >= 1L << 18) launch(k_coeffs<4>, 4);
    else launch(k_coeffs<1>, 1);
}

void launch_rhs(int nx, int ny, double h, double dt, const double *us,
                const double *vs, const double *Fx, const double *Fy,
                const double *bx, const double *by, double *b, cudaStream_t s)
{
    dim3 g(cdiv(nx, 128), ny);
    note_launch();
    k_rhs<<<g, 128, 0, s>>>(nx, ny, 1.0 / h, 1.0 / (h * dt), us, vs, Fx, Fy, bx, by, b);
}

void launch_correct(int nx, int ny, double h, double dt, const double *us,
                    const double *vs, const double *p, const double *Fx,
                    const double *Fy, const double *bx, const double *by,
                    double *u, double *v, cudaStream_t s)
{
    const long n = std::max((long)(nx + 1) * ny, (long)nx * (ny + 1));
    note_launch();
    k_correct<<<dim3(cdiv(n, kT), 2), kT, 0, s>>>(nx, ny, 1.0 / h, dt, us, vs, p, Fx, Fy, bx, by, u, v);
}

// Rows a warp marches: those of the least time by what was measured, (R + 1)
// (4 n + 1) in units of 0.48 us with n the most blocks that an SM gets (n = 1 .. 4:
// 2.45, 4.15, 6.05 and 8.1 us a row; the FP64 pipe's rate, but for one block,
// whose four warps wait for their own chains).  The time steps up with n, so 16
// rows wherever they give 1024 warps cost 103 us at 960 x 640 (320 blocks: three
// on some SMs), the tiles before 87 and 17 rows (two) 74; 768^2 101, 87 and 73;
// 3000 x 100 53, 48 and 41; 1024^2 137, 144 and 130; 2048^2 500, 566 and 491.
static int pred_rows(int nx, int ny)
{
    static const int sms = [] {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            cudaGetLastError();
        return n > 0 ? n : 152;
    }();
    int best = 1;
    long least = 0;
    for (int R = 1; R <= 20; R++) {
        const long blocks = cdiv(pred_warps(nx, ny, R), kPredT / 32);
        const long cost = (R + 1) * (4 * (long)cdiv(blocks, sms) + 1);
        if (R == 1 || cost < least) { best = R; least = cost; }
    }
    return best;
}

static void predictor(bool axi, int nx, int ny, double h, double dt, const double *rho,
                      const double *mu, const double *u, const double *v, const double *au_prev,
                      const double *av_prev, int have_prev, double gx, double gy,
                      const double *frame, const double *bx, const double *by, double *us,
                      double *vs, double *au, double *av, cudaStream_t s, double visc)
{
    const int R = pred_rows(nx, ny);
    const unsigned g = cdiv(pred_warps(nx, ny, R), kPredT / 32);
    note_launch();
    if (axi)
        k_predictor<true><<<g, kPredT, 0, s>>>(nx, ny, R, 1.0 / h, visc, dt, rho, mu, u, v, au_prev, av_prev,
                                               have_prev, gx, gy, frame, bx, by, us, vs, au, av);
    else
        k_predictor<false><<<g, kPredT, 0, s>>>(nx, ny, R, 1.0 / h, visc, dt, rho, mu, u, v, au_prev, av_prev,
                                                have_prev, gx, gy, frame, bx, by, us, vs, au, av);
}

void launch_predictor(int nx, int ny, double h, double dt, const double *rho,
                      const double *mu, const double *u, const double *v,
                      const double *au_prev, const double *av_prev,
                      int have_prev, double gx, double gy, const double *bx,
                      const double *by, double *us, double *vs, double *au, double *av,
                      cudaStream_t s, double visc)
{
    predictor(false, nx, ny, h, dt, rho, mu, u, v, au_prev, av_prev, have_prev, gx, gy, nullptr, bx, by,
              us, vs, au, av, s, visc);
}

void launch_predictor_axi(int nx, int ny, double h, double dt, const double *rho,
                          const double *mu, const double *u, const double *v,
                          const double *au_prev, const double *av_prev, int have_prev,
                          double gx, double gy, const double *frame, const double *bx,
                          const double *by, double *us, double *vs, double *au, double *av,
                          cudaStream_t s, double visc)
{
    predictor(true, nx, ny, h, dt, rho, mu, u, v, au_prev, av_prev, have_prev, gx, gy, frame, bx, by,
              us, vs, au, av, s, visc);
}

}  // namespace ibk
