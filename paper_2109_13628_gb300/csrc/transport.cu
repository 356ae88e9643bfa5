// Vorticity transport on the IIM grid (Sec. 3, Sec. 5.1, 5.3, 5.5, App. B) on the device.
//
//   * velocity extended to the A- nodes at third order with u_b (degree 2, Sec. 5.3);
//   * vorticity boundary condition omega_b = curl of the extended velocity at every control
//     point (Sec. 5.3; the stencil figure is missing, the reading used: along the grid line
//     the derivative at the crossing of the quadratic through the solid node, the fluid node
//     and the next fluid node; across it a one-sided second-order difference of the values
//     interpolated at the crossing on the next two rows (columns), combined with u_b; both
//     sides averaged when both are available);
//   * vorticity extended three times: fourth order with omega_b (diffusion), third order with
//     omega_b (upwind end of advective stencils), third order without a boundary condition
//     (downwind end) (Sec. 3.2);
//   * conservative fluxes (Eq. 2dshuconserve): third-order upwind advective flux of the point
//     flux u w (Eq. upwind; the face velocity selects the stencil), downwind stencil at inflow
//     boundary faces, centred diffusive flux;
//   * Kelvin ODE dGamma_k/dt = -h sum_{dR_k} (f + q).n with the same fluxes (Eq.
//     discreteKelvinChoice);
//   * Williamson low-storage RK3 on (omega, Gamma) with dt = C_stab dt_max from the RK3
//     polygon of App. B.
// Box: velocity Uinf at and beyond the box; vorticity 0 there except at the right (outflow)
// edge, where the last interior column is copied (zero gradient).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <initializer_list>
#include <utility>

#include "common.cuh"

namespace iim {

static constexpr double kRK3A[3] = {0.0, -5.0 / 9.0, -153.0 / 128.0};
static constexpr double kRK3B[3] = {1.0 / 3.0, 15.0 / 16.0, 8.0 / 15.0};
static constexpr double kStabC = 1.620, kStabR = 0.314;

__constant__ int t_dir_i[4] = {1, -1, 0, 0};
__constant__ int t_dir_j[4] = {0, 0, 1, -1};

// Fields of one evaluation in the caller's layout (NY rows of NX), read at fluid nodes only; the
// extensions at the A- nodes are kept per A- index, so no field is copied or rewritten.
struct TrView {
    int NX, NY, nx;
    double h, rh;            // cell size and 1 / h
    int h_pow2;              // 1 / h is exact
    const uint8_t* cls;      // padded
    const int* minus_map;    // padded -> A- index
    const double *w, *ux, *uy;
    const double *gux, *guy; // per A- node: third-order velocity extension with u_b
    const double* g4;        //              fourth-order vorticity extension with omega_b
    const double* g3;        //              third-order with omega_b
    const double* g3n;       //              third-order without boundary condition
    double Ux, Uy;
};

__device__ __forceinline__ bool t_inside(const TrView& v, int i, int j) { return i >= 0 && i < v.NX && j >= 0 && j < v.NY; }
__device__ __forceinline__ long t_pidx(const TrView& v, int i, int j) { return (long)j * v.nx + 1 + i; }
__device__ __forceinline__ long t_uidx(const TrView& v, int i, int j) { return (long)j * v.NX + i; }
__device__ __forceinline__ bool t_solid(const TrView& v, int i, int j) {
    return t_inside(v, i, j) && v.cls[t_pidx(v, i, j)] >= CLS_MINUS;
}
__device__ __forceinline__ double t_vel(const TrView& v, int comp, int i, int j) {
    if (!t_inside(v, i, j)) return comp ? v.Uy : v.Ux;
    const long p = t_pidx(v, i, j);
    const uint8_t c = v.cls[p];
    if (c <= CLS_PLUS) return (comp ? v.uy : v.ux)[t_uidx(v, i, j)];
    return c == CLS_MINUS ? (comp ? v.guy : v.gux)[v.minus_map[p]] : 0.0;
}
// kind 0: fourth-order extension with omega_b, 1: third-order with omega_b, 2: third-order without
__device__ __forceinline__ double t_omega(const TrView& v, int kind, int i, int j) {
    if (!t_inside(v, i, j)) {
        if (!(i >= v.NX && j >= 0 && j < v.NY)) return 0.0;
        i = v.NX - 1;
        return v.cls[t_pidx(v, i, j)] <= CLS_PLUS ? v.w[t_uidx(v, i, j)] : 0.0;
    }
    const long p = t_pidx(v, i, j);
    const uint8_t c = v.cls[p];
    if (c <= CLS_PLUS) return v.w[t_uidx(v, i, j)];
    if (c == CLS_MINUS) {
        const int m = v.minus_map[p];
        return kind == 0 ? v.g4[m] : (kind == 1 ? v.g3[m] : v.g3n[m]);
    }
    return 0.0;
}

// f + q on a face from the point fluxes p of the upwind-biased stencil in order along the axis
// (pos: nodes a - e, a, b; else a, b, b + e) and the vorticity of the face's two nodes (diffusion);
// c = nu / h.
__device__ __forceinline__ double t_flux(bool pos, double p0, double p1, double p2, double wa, double wb, double c) {
    const double k0 = pos ? -1.0 / 6.0 : 1.0 / 3.0, k2 = pos ? 1.0 / 3.0 : -1.0 / 6.0;
    return fma(k0, p0, fma(5.0 / 6.0, p1, k2 * p2)) - c * (wb - wa);
}

// Flux f + q on the face between interior nodes a = (ai, aj) and a + e_axis: the general form, any
// of the stencil's nodes in a solid or beyond the box.
__device__ __noinline__ double t_face_flux(const TrView& v, double c, int axis, int ai, int aj) {
    const int di = axis == 0 ? 1 : 0, dj = axis == 0 ? 0 : 1;
    const int bi = ai + di, bj = aj + dj;
    bool pos = t_vel(v, axis, ai, aj) + t_vel(v, axis, bi, bj) >= 0.0;
    const bool up_left = pos;
    const bool sa = t_solid(v, ai, aj), sb = t_solid(v, bi, bj);
    if (sa != sb) {
        const bool inflow = (sb && !pos) || (sa && pos);
        if (inflow) pos = !pos;   // downwind stencil at inflow boundary faces
    }
    double p[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int o = pos ? k - 1 : k;            // node a + o e_axis
        const int ni = ai + o * di, nj = aj + o * dj;
        const int kind = t_solid(v, ni, nj) ? (((o <= 0) == up_left) ? 1 : 2) : 1;
        p[k] = t_vel(v, axis, ni, nj) * t_omega(v, kind, ni, nj);
    }
    return t_flux(pos, p[0], p[1], p[2], t_omega(v, 0, ai, aj), t_omega(v, 0, bi, bj), c);
}

// a / h: a product when 1 / h is exact, else the product corrected by one residual step (Markstein), which
// an infinite product does not take (its residual is inf - inf).
__device__ __forceinline__ double t_div_h(const TrView& v, double a) {
    const double q = a * v.rh;
    const bool finite = (__double2hiint(q) & 0x7ff00000) != 0x7ff00000;
    return v.h_pow2 || !finite ? q : fma(fma(-q, v.h, a), v.rh, q);
}

// Sums over the four lanes of one A- node in direction order (the lanes of a warp are nodes x
// directions), as a loop over the directions would add them.
__device__ __forceinline__ double sum_dirs(double x) {
    const int base = (threadIdx.x & 31) & ~3;
    double s = __shfl_sync(0xffffffffu, x, base);
#pragma unroll
    for (int d = 1; d < 4; ++d) s += __shfl_sync(0xffffffffu, x, base + d);
    return s;
}

// Third-order velocity extension with u_b at every A- node (both components); four lanes per node,
// one per direction: the kernel is a chain of dependent loads and divisions, so its time is that of
// one direction.
__global__ void k_ext_velocity(int nm, TrView v, const int* __restrict__ minus_node, const int* __restrict__ minus_cp,
                               const uint8_t* __restrict__ minus_mask, const double* __restrict__ cp_t,
                               const double* __restrict__ ubx, const double* __restrict__ uby, double* __restrict__ gux,
                               double* __restrict__ guy) {
    pdl_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x, d = t & 3;
    const int m = min(t >> 2, nm - 1);   // the last warp stays whole for the shuffles
    const int mask = minus_mask[m] >> 4;
    double sx = 0.0, sy = 0.0;
    if (mask & (1 << d)) {
        const int p = minus_node[m], j = p / v.nx, i = p - j * v.nx - 1;
        const int c = minus_cp[4 * m + d];
        const double a = 1.0 - cp_t[c];
        // Lagrange weights at 0 of the quadratic through a (boundary), 2, 3
        const double w0 = 6.0 / ((a - 2.0) * (a - 3.0));
        const double w2 = -3.0 * a / (2.0 - a);
        const double w3 = 2.0 * a / (3.0 - a);
        const long q = t_uidx(v, i, j), step = (long)t_dir_j[d] * v.NX + t_dir_i[d];
        sx = w0 * ubx[c] + w2 * v.ux[q + 2 * step] + w3 * v.ux[q + 3 * step];
        sy = w0 * uby[c] + w2 * v.uy[q + 2 * step] + w3 * v.uy[q + 3 * step];
    }
    sx = sum_dirs(sx);
    sy = sum_dirs(sy);
    if (d == 0 && (t >> 2) < nm) {
        const int cnt = __popc(mask & 15);
        gux[m] = cnt ? sx / cnt : 0.0;
        guy[m] = cnt ? sy / cnt : 0.0;
    }
}

// The three vorticity extensions at every A- node (four lanes per node, as k_ext_velocity).
__global__ void k_ext_vorticity(int nm, TrView v, const int* __restrict__ minus_node, const int* __restrict__ minus_cp,
                                const uint8_t* __restrict__ minus_mask, const double* __restrict__ cp_t,
                                const double* __restrict__ wb, double* __restrict__ g4, double* __restrict__ g3,
                                double* __restrict__ g3n) {
    pdl_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x, d = t & 3;
    const int m = min(t >> 2, nm - 1);
    int mask = minus_mask[m];
    double s4 = 0.0, s3 = 0.0, s3n = 0.0;
    const int c = minus_cp[4 * m + d];
    if (c >= 0 && (mask & (17 << d))) {
        const int p = minus_node[m], j = p / v.nx, i = p - j * v.nx - 1;
        const long q = t_uidx(v, i, j), step = (long)t_dir_j[d] * v.NX + t_dir_i[d];
        const double a = 1.0 - cp_t[c];
        const double x2 = v.w[q + 2 * step], x3 = v.w[q + 3 * step];
        if (mask & (1 << d)) {
            // cubic through a (boundary), 2, 3, 4
            const double w0 = -24.0 / ((a - 2.0) * (a - 3.0) * (a - 4.0));
            const double w2 = -6.0 * a / (2.0 - a);
            const double w3 = 8.0 * a / (3.0 - a);
            const double w4 = -3.0 * a / (4.0 - a);
            s4 = w0 * wb[c] + w2 * x2 + w3 * x3 + w4 * v.w[q + 4 * step];
        }
        if (mask & (16 << d)) {
            const double w0 = 6.0 / ((a - 2.0) * (a - 3.0));
            const double w2 = -3.0 * a / (2.0 - a);
            const double w3 = 2.0 * a / (3.0 - a);
            s3 = w0 * wb[c] + w2 * x2 + w3 * x3;
            // quadratic through the fluid nodes 1, 2, 3 (no boundary condition)
            s3n = 3.0 * v.w[q + step] - 3.0 * x2 + x3;
        }
    }
    s4 = sum_dirs(s4);
    s3 = sum_dirs(s3);
    s3n = sum_dirs(s3n);
    // directions without a control point have no bit in the counts
    const unsigned has = __ballot_sync(0xffffffffu, c >= 0) >> ((threadIdx.x & 31) & ~3);
    if (d == 0 && (t >> 2) < nm) {
        const int c4 = __popc(mask & 15 & has), c3 = __popc((mask >> 4) & 15 & has);
        g4[m] = c4 ? s4 / c4 : 0.0;
        g3[m] = c3 ? s3 / c3 : 0.0;
        g3n[m] = c3 ? s3n / c3 : 0.0;
    }
}

// omega_b = curl of the extended velocity at each control point (Sec. 5.3, reading above).
__global__ void k_vorticity_bc(int ncp, TrView v, int nx_cells, int ny_cells, const int* __restrict__ cp_axis,
                               const int* __restrict__ cp_ei, const int* __restrict__ cp_ej, const double* __restrict__ cp_t,
                               const double* __restrict__ ubx, const double* __restrict__ uby, double* __restrict__ wb) {
    pdl_wait();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncp) return;
    const bool along_x = cp_axis[c] == 0;
    // global node coordinates of the edge ends; interior coordinates are global - 1
    const int ei = cp_ei[c], ej = cp_ej[c];
    const int oi = along_x ? ei + 1 : ei, oj = along_x ? ej : ej + 1;
    const bool lower_solid = t_solid(v, ei - 1, ej - 1);
    const int si = lower_solid ? ei : oi, sj = lower_solid ? ej : oj;
    const int fi = lower_solid ? oi : ei, fj = lower_solid ? oj : ej;
    const int di = fi - si, dj = fj - sj;
    const double t = cp_t[c], h = v.h;
    auto defined = [&](int gi, int gj) {
        if (gi <= 0 || gj <= 0 || gi >= nx_cells || gj >= ny_cells) return true;
        return v.cls[t_pidx(v, gi - 1, gj - 1)] <= CLS_MINUS;
    };
    const int ca = along_x ? 1 : 0;   // component differentiated along the line
    const int cb = along_x ? 0 : 1;   // component differentiated across the line
    const int dsgn = along_x ? di : dj;
    const double Us = t_vel(v, ca, si - 1, sj - 1), Uf = t_vel(v, ca, fi - 1, fj - 1);
    double d_along;
    if (!t_solid(v, fi + di - 1, fj + dj - 1)) {
        const double Un = t_vel(v, ca, fi + di - 1, fj + dj - 1);
        d_along = dsgn / h * ((Un - Us) / 2.0 - t * (Un - 2.0 * Uf + Us));
    } else {
        d_along = dsgn / h * (Uf - Us);
    }
    const double ub = along_x ? ubx[c] : uby[c];
    double est = 0.0, first = 0.0;
    int nest = 0;
    bool have_first = false;
    for (int sgn = 1; sgn >= -1; sgn -= 2) {
        double vals[2];
        bool ok = true;
        for (int k = 1; k <= 2 && ok; ++k) {
            const int pi_ = along_x ? 0 : k * sgn, pj_ = along_x ? k * sgn : 0;
            const int n0i = si + pi_, n0j = sj + pj_, n1i = fi + pi_, n1j = fj + pj_, n2i = fi + di + pi_,
                      n2j = fj + dj + pj_;
            if (!defined(n0i, n0j) || !defined(n1i, n1j) || !defined(n2i, n2j)) { ok = false; break; }
            const double Um = t_vel(v, cb, n0i - 1, n0j - 1), U0 = t_vel(v, cb, n1i - 1, n1j - 1),
                         Up = t_vel(v, cb, n2i - 1, n2j - 1);
            vals[k - 1] = U0 + (-t) * (Up - Um) / 2.0 + t * t * (Up - 2.0 * U0 + Um) / 2.0;
            if (k == 1 && !have_first) {
                first = sgn * (vals[0] - ub) / h;
                have_first = true;
            }
        }
        if (ok) {
            est += sgn * (-3.0 * ub + 4.0 * vals[0] - vals[1]) / (2.0 * h);
            ++nest;
        }
    }
    const double d_cross = nest ? est / nest : (have_first ? first : 0.0);
    wb[c] = along_x ? (d_along - d_cross) : (d_cross - d_along);
}

// ---- total pressure (Sec. 5.4)
// f = -div(u x omega k) = -(d_x(u_y omega) - d_y(u_x omega)) at fluid interior nodes by centred
// differences of the products, the third-order extensions (velocity with u_b, vorticity with
// omega_b) at A- nodes and the box values beyond (caller layout, 0 in the solid).
__global__ void k_pressure_rhs(TrView v, double* __restrict__ f) {
    pdl_wait();
    const long n = (long)v.NX * v.NY;
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int i = (int)(k % v.NX), j = (int)(k / v.NX);
    double r = 0.0;
    if (v.cls[t_pidx(v, i, j)] <= CLS_PLUS) {
        const double qe = t_vel(v, 1, i + 1, j) * t_omega(v, 1, i + 1, j);
        const double qw = t_vel(v, 1, i - 1, j) * t_omega(v, 1, i - 1, j);
        const double rn = t_vel(v, 0, i, j + 1) * t_omega(v, 1, i, j + 1);
        const double rs = t_vel(v, 0, i, j - 1) * t_omega(v, 1, i, j - 1);
        r = -((qe - qw) - (rn - rs)) / (2.0 * v.h);
    }
    f[k] = r;
}

// Wall datum of the Neumann extrapolation at each control point: d . grad H with d along the
// grid line into the fluid.  On a stationary no-slip wall grad H = grad p = nu k x grad omega
// (Eq. pressuregrad1; grad |u|^2 / 2 = (grad u)^T u vanishes where u = 0), so an x-line needs
// d_y omega and a y-line d_x omega at the crossing: the cross-line stencil of the vorticity
// boundary condition applied to the vorticity extended at third order with omega_b.
__global__ void k_pressure_wall_data(int ncp, TrView v, int nx_cells, int ny_cells, const int* __restrict__ cp_axis,
                                     const int* __restrict__ cp_ei, const int* __restrict__ cp_ej,
                                     const double* __restrict__ cp_t, const double* __restrict__ wb, double nu,
                                     double* __restrict__ out) {
    pdl_wait();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncp) return;
    const bool along_x = cp_axis[c] == 0;
    const int ei = cp_ei[c], ej = cp_ej[c];
    const int oi = along_x ? ei + 1 : ei, oj = along_x ? ej : ej + 1;
    const bool lower_solid = t_solid(v, ei - 1, ej - 1);
    const int si = lower_solid ? ei : oi, sj = lower_solid ? ej : oj;
    const int fi = lower_solid ? oi : ei, fj = lower_solid ? oj : ej;
    const int di = fi - si, dj = fj - sj;
    const double t = cp_t[c], h = v.h, w0 = wb[c];
    auto defined = [&](int gi, int gj) {
        if (gi <= 0 || gj <= 0 || gi >= nx_cells || gj >= ny_cells) return true;
        return v.cls[t_pidx(v, gi - 1, gj - 1)] <= CLS_MINUS;
    };
    double est = 0.0, first = 0.0;
    int nest = 0;
    bool have_first = false;
    for (int sgn = 1; sgn >= -1; sgn -= 2) {
        double vals[2];
        bool ok = true;
        for (int k = 1; k <= 2 && ok; ++k) {
            const int pi_ = along_x ? 0 : k * sgn, pj_ = along_x ? k * sgn : 0;
            const int n0i = si + pi_, n0j = sj + pj_, n1i = fi + pi_, n1j = fj + pj_, n2i = fi + di + pi_,
                      n2j = fj + dj + pj_;
            if (!defined(n0i, n0j) || !defined(n1i, n1j) || !defined(n2i, n2j)) { ok = false; break; }
            const double Wm = t_omega(v, 1, n0i - 1, n0j - 1), W0 = t_omega(v, 1, n1i - 1, n1j - 1),
                         Wp = t_omega(v, 1, n2i - 1, n2j - 1);
            vals[k - 1] = W0 + (-t) * (Wp - Wm) / 2.0 + t * t * (Wp - 2.0 * W0 + Wm) / 2.0;
            if (k == 1 && !have_first) {
                first = sgn * (vals[0] - w0) / h;
                have_first = true;
            }
        }
        if (ok) {
            est += sgn * (-3.0 * w0 + 4.0 * vals[0] - vals[1]) / (2.0 * h);
            ++nest;
        }
    }
    const double d_cross = nest ? est / nest : (have_first ? first : 0.0);
    out[c] = along_x ? -nu * di * d_cross : nu * dj * d_cross;
}

// A field (caller layout) at each control point: the quadratic through the fluid node next to
// the crossing and the next two fluid interior nodes on its line, at the crossing (fewer nodes
// where those are not fluid interior nodes).
__global__ void k_wall_values(int ncp, TrView v, const int* __restrict__ cp_axis, const int* __restrict__ cp_ei,
                              const int* __restrict__ cp_ej, const double* __restrict__ cp_t,
                              const double* __restrict__ field, double* __restrict__ out) {
    pdl_wait();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncp) return;
    const bool along_x = cp_axis[c] == 0;
    const int ei = cp_ei[c], ej = cp_ej[c];
    const int oi = along_x ? ei + 1 : ei, oj = along_x ? ej : ej + 1;
    const bool lower_solid = t_solid(v, ei - 1, ej - 1);
    const int si = lower_solid ? ei : oi, sj = lower_solid ? ej : oj;
    const int fi = lower_solid ? oi : ei, fj = lower_solid ? oj : ej;
    const int di = fi - si, dj = fj - sj;
    auto fluid = [&](int gi, int gj) {   // global node coordinates
        return gi >= 1 && gj >= 1 && gi <= v.NX && gj <= v.NY && v.cls[t_pidx(v, gi - 1, gj - 1)] <= CLS_PLUS;
    };
    auto at = [&](int gi, int gj) { return field[(long)(gj - 1) * v.NX + (gi - 1)]; };
    const double x = -cp_t[c];
    const double F0 = at(fi, fj);
    double r;
    if (fluid(fi + di, fj + dj) && fluid(fi + 2 * di, fj + 2 * dj)) {
        const double F1 = at(fi + di, fj + dj), F2 = at(fi + 2 * di, fj + 2 * dj);
        r = F0 * (x - 1.0) * (x - 2.0) * 0.5 - F1 * x * (x - 2.0) + F2 * x * (x - 1.0) * 0.5;
    } else if (fluid(fi + di, fj + dj)) {
        r = F0 * (1.0 - x) + at(fi + di, fj + dj) * x;
    } else {
        r = F0;
    }
    out[c] = r;
}

// Kelvin ODE of body k: dGdt[k] = -h sum_{dR_k}(f+q).n; with rk != 0 also the Williamson update
// dG = a dG + dt dGdt, Gamma += b dG (every body; fixed-psibar bodies do not read Gamma).
struct KelvinArgs {
    const iim_region* R;
    double* dgdt;
    int rk;
    double b;
    double *dG, *gamma;
};
template <int BLOCK>
__device__ __forceinline__ void kelvin_body(const TrView& v, double c, int k, const KelvinArgs& g, double a, double dt) {
    const iim_region r = g.R[k];
    double s = 0.0;
    // interior coordinates = global - 1
    for (int jj = r.ly + threadIdx.x; jj <= r.ry; jj += BLOCK)
        s += t_face_flux(v, c, 0, r.rx - 1, jj - 1) - t_face_flux(v, c, 0, r.lx - 2, jj - 1);
    for (int ii = r.lx + threadIdx.x; ii <= r.rx; ii += BLOCK)
        s += t_face_flux(v, c, 1, ii - 1, r.ry - 1) - t_face_flux(v, c, 1, ii - 1, r.ly - 2);
    __shared__ double red[BLOCK / 32];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < BLOCK / 32; ++w) tot += red[w];
        const double rate = -v.h * tot;
        if (g.dgdt) g.dgdt[k] = rate;
        if (g.rk) {
            g.dG[k] = a * g.dG[k] + dt * rate;
            g.gamma[k] += g.b * g.dG[k];
        }
    }
}

// Transport right-hand side at fluid nodes.  mode 0: out = rhs; mode 1: dw = a * dw + dt * rhs (a = 0
// does not read dw).  Both in the caller's layout.
//
// The FP64 pipe bounds it (two lanes per clock and SM: 1.7 us per instruction and million nodes), so
// every face is evaluated once: a block stages its nodes (and two beyond each side) in shared memory
// with the point fluxes u w formed once per node, evaluates its faces into shared memory, and
// differences them -- about 20 FP64 instructions per node instead of 88 (four faces per node with a
// division each).  Faces whose stencil meets a solid node (found per block, then per face) take the
// general form, from the tile and the extensions, so a face has one value whichever block evaluates
// it.  The first nk blocks integrate one body's Kelvin ODE each (a chain of latencies: started first).
// 1024 x 512, one cylinder: 98 -> 30 us (the whole right-hand side 177 -> 55 us).
constexpr int TR_X = 32, TR_Y = 16, TR_THREADS = 256, TR_W = TR_X + 4, TR_H = TR_Y + 4;
__global__ void __launch_bounds__(TR_THREADS)
k_transport_rhs(TrView v, double c, int mode, double a, double dt, double* __restrict__ out, int tx, int nk,
                KelvinArgs kv) {
    pdl_wait();
    if ((int)blockIdx.x < nk) {
        kelvin_body<TR_THREADS>(v, c, blockIdx.x, kv, a, dt);
        return;
    }
    __shared__ double sw[TR_H][TR_W], sux[TR_H][TR_W], suy[TR_H][TR_W], spx[TR_H][TR_W], spy[TR_H][TR_W];
    __shared__ uint8_t ss[TR_H][TR_W];
    // the faces, once every node has been read, take the place of the point fluxes (29 KB: seven
    // blocks on an SM)
    double(*fx)[TR_X + 1] = reinterpret_cast<double(*)[TR_X + 1]>(&spx[0][0]);
    double(*fy)[TR_X] = reinterpret_cast<double(*)[TR_X]>(&spy[0][0]);
    const int tile = blockIdx.x - nk, by = tile / tx, i0 = (tile - by * tx) * TR_X, j0 = by * TR_Y;
    // nodes: flag 0 fluid or beyond the box, 1 A- node (velocity: its extension), 2 deeper in a solid
    constexpr int NN = TR_H * TR_W, PN = (NN + TR_THREADS - 1) / TR_THREADS;
    int flag[PN];
    double w[PN], ux[PN], uy[PN];
#pragma unroll
    for (int b = 0; b < PN; ++b) {
        const int t = threadIdx.x + b * TR_THREADS, r = t / TR_W, q = t - r * TR_W, i = i0 - 2 + q, j = j0 - 2 + r;
        flag[b] = -1;
        w[b] = ux[b] = uy[b] = 0.0;
        if (t < NN && j >= 0 && j < v.NY && i >= 0) {
            const int ic = min(i, v.NX - 1);     // the right edge copies the last column's vorticity
            const long k = t_uidx(v, ic, j);
            flag[b] = v.cls[t_pidx(v, ic, j)];
            w[b] = v.w[k];
            ux[b] = v.ux[k];
            uy[b] = v.uy[k];
        }
    }
    int solid_any = 0;
#pragma unroll
    for (int b = 0; b < PN; ++b) {
        const int t = threadIdx.x + b * TR_THREADS, r = t / TR_W, q = t - r * TR_W, i = i0 - 2 + q, j = j0 - 2 + r;
        if (t >= NN) continue;
        int sol = 0;
        if (flag[b] >= (int)CLS_MINUS) {
            sol = flag[b] == (int)CLS_MINUS ? 1 : 2;
            w[b] = ux[b] = uy[b] = 0.0;
            if (sol == 1 && i < v.NX) {
                const int m = v.minus_map[t_pidx(v, i, j)];
                ux[b] = v.gux[m];
                uy[b] = v.guy[m];
            }
        }
        if (flag[b] < 0 || i >= v.NX) {
            ux[b] = v.Ux;
            uy[b] = v.Uy;
            sol = 0;
        }
        solid_any |= sol;
        sw[r][q] = w[b];
        sux[r][q] = ux[b];
        suy[r][q] = uy[b];
        spx[r][q] = ux[b] * w[b];
        spy[r][q] = uy[b] * w[b];
        ss[r][q] = (uint8_t)sol;
    }
    solid_any = __syncthreads_or(solid_any);
    // a face next to a solid, from the tile: t_face_flux's form with the A- vorticities from the extensions
    auto solid_face = [&](const double (*su)[TR_W], int y, int x, int dy, int dx) -> double {
        const int fa = ss[y][x], fb = ss[y + dy][x + dx];
        if (fa && fb) return 0.0;   // no fluid node reads it
        bool pos = su[y][x] + su[y + dy][x + dx] >= 0.0;
        const bool up_left = pos;
        if ((fa != 0) != (fb != 0) && ((fb && !pos) || (fa && pos))) pos = !pos;
        auto om = [&](int kind, int o) -> double {
            const int yy = y + o * dy, xx = x + o * dx, fl = ss[yy][xx];
            if (fl == 0) return sw[yy][xx];
            if (fl == 2) return 0.0;
            const int m = v.minus_map[t_pidx(v, i0 - 2 + xx, j0 - 2 + yy)];
            return kind == 0 ? v.g4[m] : kind == 1 ? v.g3[m] : v.g3n[m];
        };
        double p[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int o = pos ? k - 1 : k;
            p[k] = su[y + o * dy][x + o * dx] * om(((o <= 0) == up_left) ? 1 : 2, o);
        }
        return t_flux(pos, p[0], p[1], p[2], om(0, 0), om(0, 1), c);
    };
    constexpr int NFX = TR_Y * (TR_X + 1), NFY = (TR_Y + 1) * TR_X;
    constexpr int PX = (NFX + TR_THREADS - 1) / TR_THREADS, PY = (NFY + TR_THREADS - 1) / TR_THREADS;
    double vx[PX], vy[PY];
    // x faces: face (r, q) between nodes q - 1 and q of row r (tile nodes offset by 2)
#pragma unroll
    for (int b = 0; b < PX; ++b) {
        const int t = threadIdx.x + b * TR_THREADS;
        vx[b] = 0.0;
        if (t < NFX) {
            const int r = t / (TR_X + 1), q = t - r * (TR_X + 1), y = r + 2, x = q + 1;   // nodes x, x + 1
            if (solid_any && (ss[y][x - 1] | ss[y][x] | ss[y][x + 1] | ss[y][x + 2])) {
                vx[b] = solid_face(sux, y, x, 0, 1);
            } else {
                const bool pos = sux[y][x] + sux[y][x + 1] >= 0.0;
                const double* p = &spx[y][pos ? x - 1 : x];
                vx[b] = t_flux(pos, p[0], p[1], p[2], sw[y][x], sw[y][x + 1], c);
            }
        }
    }
#pragma unroll
    for (int b = 0; b < PY; ++b) {
        const int t = threadIdx.x + b * TR_THREADS;
        vy[b] = 0.0;
        if (t < NFY) {
            const int r = t / TR_X, q = t - r * TR_X, y = r + 1, x = q + 2;               // nodes y, y + 1
            if (solid_any && (ss[y - 1][x] | ss[y][x] | ss[y + 1][x] | ss[y + 2][x])) {
                vy[b] = solid_face(suy, y, x, 1, 0);
            } else {
                const bool pos = suy[y][x] + suy[y + 1][x] >= 0.0;
                const double* p = &spy[pos ? y - 1 : y][x];
                vy[b] = t_flux(pos, p[0], p[TR_W], p[2 * TR_W], sw[y][x], sw[y + 1][x], c);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < PX; ++b) {
        const int t = threadIdx.x + b * TR_THREADS;
        if (t < NFX) (&fx[0][0])[t] = vx[b];
    }
#pragma unroll
    for (int b = 0; b < PY; ++b) {
        const int t = threadIdx.x + b * TR_THREADS;
        if (t < NFY) (&fy[0][0])[t] = vy[b];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < TR_Y * TR_X; t += TR_THREADS) {
        const int r = t / TR_X, q = t - r * TR_X;
        if (i0 + q >= v.NX || j0 + r >= v.NY) continue;
        double rate = 0.0;
        if (!ss[r + 2][q + 2])
            rate = -t_div_h(v, (fx[r][q + 1] - fx[r][q]) + (fy[r + 1][q] - fy[r][q]));
        const long k = t_uidx(v, i0 + q, j0 + r);
        if (mode == 0) out[k] = rate;
        else out[k] = a != 0.0 ? a * out[k] + dt * rate : dt * rate;
    }
}

__global__ void k_rk_omega(int NX, int NY, double b, const double* __restrict__ dw, const uint8_t* __restrict__ cls,
                           double* __restrict__ omega) {
    pdl_wait();
    const int n = NX * NY;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int j = k / NX, i = k - j * NX;
    const int p = j * (NX + 1) + 1 + i;
    omega[k] = cls[p] <= CLS_PLUS ? omega[k] + b * dw[k] : 0.0;
}

template <int BLOCK>
__global__ void k_speed_max(long n, const double* __restrict__ ux, const double* __restrict__ uy, double* __restrict__ part) {
    pdl_wait();
    double m = 0.0;
    for (long k = (long)blockIdx.x * BLOCK + threadIdx.x; k < n; k += (long)gridDim.x * BLOCK)
        m = fmax(m, fabs(ux[k]) + fabs(uy[k]));
    __shared__ double red[BLOCK / 32];
    for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < BLOCK / 32; ++w) t = fmax(t, red[w]);
        part[blockIdx.x] = t;
    }
}

// Transport workspace inside g->tr_buf (doubles).
struct TrWork {
    double *dw, *gux, *guy, *g4, *g3, *g3n, *wb, *dG, *part, *psi, *vx, *vy, *zeros, *ub_stage;
};

static iim_status tr_work(iim_geometry g, TrWork* W) {
    const size_t n = (size_t)g->NX * g->NY, nm = (size_t)std::max(g->nminus, 1), ncp = (size_t)std::max(g->ncp, 1);
    const size_t total = 4 * n + 5 * nm + ncp + 64 + 1024 + ncp + 2 * ncp;
    if (!g->tr_buf) {
        IIM_TRY(cudaMalloc(&g->tr_buf, total * sizeof(double)));
        IIM_TRY(cudaMemset(g->tr_buf, 0, total * sizeof(double)));
    }
    double* p = g->tr_buf;
    W->dw = p; p += n;
    W->gux = p; p += nm;
    W->guy = p; p += nm;
    W->g4 = p; p += nm;
    W->g3 = p; p += nm;
    W->g3n = p; p += nm;
    W->wb = p; p += ncp;
    W->dG = p; p += 64;
    W->part = p; p += 1024;
    W->psi = p; p += n;
    W->vx = p; p += n;
    W->vy = p; p += n;
    W->zeros = p; p += ncp;
    W->ub_stage = p; p += 2 * ncp;
    return IIM_OK;
}

static TrView make_view(iim_geometry g, const TrWork& W, const double Uinf[2], const double* omega, const double* ux,
                        const double* uy) {
    TrView v;
    v.NX = g->NX; v.NY = g->NY; v.nx = g->nx; v.h = g->h;
    v.rh = 1.0 / g->h;
    int e = 0;
    v.h_pow2 = std::frexp(g->h, &e) == 0.5;
    v.cls = g->node_class; v.minus_map = g->minus_map;
    v.w = omega; v.ux = ux; v.uy = uy;
    v.gux = W.gux; v.guy = W.guy; v.g4 = W.g4; v.g3 = W.g3; v.g3n = W.g3n;
    v.Ux = Uinf ? Uinf[0] : 0.0;
    v.Uy = Uinf ? Uinf[1] : 0.0;
    return v;
}

// The kernels read the caller's fields, neighbours included, while others write results: a field that an
// output overlaps is read from a copy (outputs in place of inputs are allowed, as with separate arrays).
struct Span {
    const double* p;
    size_t n;
};
static iim_status detach_fields(iim_geometry g, const TrWork& W, std::initializer_list<Span> outs, const double** omega,
                                const double** ux, const double** uy, cudaStream_t s) {
    const size_t n = (size_t)g->NX * g->NY;
    const std::pair<const double**, double*> fields[3] = {{omega, W.psi}, {ux, W.vx}, {uy, W.vy}};
    for (const auto& f : fields) {
        const uintptr_t a = (uintptr_t)*f.first;
        bool hit = false;
        for (const Span& o : outs) {
            const uintptr_t b = (uintptr_t)o.p;
            hit = hit || (o.p && a < b + o.n * sizeof(double) && b < a + n * sizeof(double));
        }
        if (!hit) continue;
        IIM_TRY(cudaMemcpyAsync(f.second, *f.first, n * sizeof(double), cudaMemcpyDefault, s));
        *f.first = f.second;
    }
    return IIM_OK;
}

// Velocity extension; vorticity BC; vorticity extensions (v holds the fields).
static iim_status prepare_stage(iim_geometry g, const TrWork& W, const TrView& v, const double* u_b,
                                const double* wb_in, double* wb_out, cudaStream_t s) {
    const double* ubx = u_b ? u_b : W.zeros;
    const double* uby = u_b ? u_b + g->ncp : W.zeros;
    const unsigned eb = (unsigned)((4 * g->nminus + 127) / 128);   // four lanes per A- node
    if (g->nminus > 0)
        launch_next("tr_ext_velocity", 0.0, 0.0, k_ext_velocity, eb, 128, 0, s, g->nminus, v, g->minus_node, g->minus_cp,
               g->minus_mask, g->cp_t, ubx, uby, W.gux, W.guy);
    if (g->ncp > 0 && wb_in) {
        IIM_TRY(cudaMemcpyAsync(W.wb, wb_in, g->ncp * sizeof(double), cudaMemcpyDeviceToDevice, s));
    } else if (g->ncp > 0)
        launch_next("tr_vorticity_bc", 0.0, 0.0, k_vorticity_bc, (g->ncp + 63) / 64, 64, 0, s, g->ncp, v, g->nx, g->ny,
               g->cp_axis, g->cp_ei, g->cp_ej, g->cp_t, ubx, uby, W.wb);
    if (g->nminus > 0)
        launch_next("tr_ext_vorticity", 0.0, 0.0, k_ext_vorticity, eb, 128, 0, s, g->nminus, v, g->minus_node, g->minus_cp,
               g->minus_mask, g->cp_t, W.wb, W.g4, W.g3, W.g3n);
    IIM_LAUNCHED();
    if (wb_out && g->ncp > 0)
        IIM_TRY(cudaMemcpyAsync(wb_out, W.wb, g->ncp * sizeof(double), cudaMemcpyDeviceToDevice, s));
    return IIM_OK;
}

// The right-hand side (out: rhs, or with rk the Williamson increment dw) and, with bodies and kv.R,
// the Kelvin ODE, in one launch.
static iim_status transport_rhs(iim_geometry g, const TrView& v, double nu, int mode, double a, double dt, double* out,
                                const KelvinArgs& kv, cudaStream_t s) {
    const int tx = (g->NX + TR_X - 1) / TR_X, ty = (g->NY + TR_Y - 1) / TR_Y;
    const int nk = kv.R ? g->nb : 0;
    launch_next("tr_rhs", 40.0 * (double)g->NX * g->NY, 0.0, k_transport_rhs, tx * ty + nk, TR_THREADS, 0, s, v, nu / g->h, mode,
           a, dt, out, tx, nk, kv);
    IIM_LAUNCHED();
    return IIM_OK;
}

}  // namespace iim

using namespace iim;

extern "C" iim_status iim_transport_rhs(iim_geometry g, const double* omega, const double* ux, const double* uy,
                                        const double* u_b, const double Uinf[2], double nu, const double* omega_b_in,
                                        double* omega_b_out, double* rhs_out, double* dgamma_out, iim_stream stream) {
    if (!g || !omega || !ux || !uy || !rhs_out || !(nu >= 0.0)) return IIM_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    TrWork W;
    IIM_CHECK(tr_work(g, &W));
    const size_t n = (size_t)g->NX * g->NY, ncp = (size_t)g->ncp;
    IIM_CHECK(detach_fields(g, W, {{rhs_out, n}, {omega_b_out, ncp}, {dgamma_out, (size_t)g->nb}}, &omega, &ux, &uy, s));
    const TrView v = make_view(g, W, Uinf, omega, ux, uy);
    IIM_CHECK(prepare_stage(g, W, v, u_b, omega_b_in, omega_b_out, s));
    const KelvinArgs kv{dgamma_out ? g->d_regions : nullptr, dgamma_out, 0, 0.0, nullptr, nullptr};
    return transport_rhs(g, v, nu, 0, 0.0, 1.0, rhs_out, kv, s);
}

extern "C" iim_status iim_total_pressure_problem(iim_geometry g, const double* omega, const double* ux,
                                                 const double* uy, const double* u_b, const double Uinf[2], double nu,
                                                 const double* omega_b_in, double* omega_b_out, double* f_out,
                                                 double* data_out, iim_stream stream) {
    if (!g || !omega || !ux || !uy || !f_out || (g->ncp > 0 && !data_out) || !(nu >= 0.0)) return IIM_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    TrWork W;
    IIM_CHECK(tr_work(g, &W));
    const long n = (long)g->NX * g->NY;
    const size_t ncp = (size_t)g->ncp;
    IIM_CHECK(detach_fields(g, W, {{f_out, (size_t)n}, {data_out, ncp}, {omega_b_out, ncp}}, &omega, &ux, &uy, s));
    const TrView v = make_view(g, W, Uinf, omega, ux, uy);
    IIM_CHECK(prepare_stage(g, W, v, u_b, omega_b_in, omega_b_out, s));
    launch_next("pressure_rhs", 48.0 * (double)n, 0.0, k_pressure_rhs, (unsigned)((n + 255) / 256), 256, 0, s, v, f_out);
    if (g->ncp > 0)
        launch_next("pressure_wall_data", 0.0, 0.0, k_pressure_wall_data, (g->ncp + 127) / 128, 128, 0, s, g->ncp, v, g->nx,
               g->ny, g->cp_axis, g->cp_ei, g->cp_ej, g->cp_t, (const double*)W.wb, nu, data_out);
    IIM_LAUNCHED();
    return IIM_OK;
}

extern "C" iim_status iim_wall_values(iim_geometry g, const double* field, double* out, iim_stream stream) {
    if (!g || !field || (g->ncp > 0 && !out)) return IIM_ERR_INVALID_ARG;
    if (g->ncp == 0) return IIM_OK;
    cudaStream_t s = (cudaStream_t)stream;
    TrWork W;
    IIM_CHECK(tr_work(g, &W));
    const TrView v = make_view(g, W, nullptr, nullptr, nullptr, nullptr);
    launch_next("wall_values", 0.0, 0.0, k_wall_values, (g->ncp + 127) / 128, 128, 0, s, g->ncp, v, g->cp_axis, g->cp_ei,
           g->cp_ej, g->cp_t, field, out);
    IIM_LAUNCHED();
    return IIM_OK;
}

extern "C" iim_status iim_total_pressure(iim_geometry g, const double* omega, const double* ux, const double* uy,
                                         const double Uinf[2], double nu, const double* H_box, double* H_out,
                                         double* H_wall_out, const iim_opts* opts, iim_stats* stats, iim_stream stream) {
    if (!g || !omega || !ux || !uy || !H_out || !(nu >= 0.0)) return IIM_ERR_INVALID_ARG;
    if (g->wall != 1) return IIM_ERR_INVALID_ARG;   // the solve needs the Neumann stencils
    const size_t n = (size_t)g->NX * g->NY, ncp = (size_t)std::max(g->ncp, 1);
    if (!g->pr_buf) {
        IIM_TRY(cudaMalloc(&g->pr_buf, (n + ncp) * sizeof(double)));
        IIM_TRY(cudaMemset(g->pr_buf, 0, (n + ncp) * sizeof(double)));
    }
    double* f = g->pr_buf;
    double* data = g->pr_buf + n;
    IIM_CHECK(iim_total_pressure_problem(g, omega, ux, uy, nullptr, Uinf, nu, nullptr, nullptr, f, data, stream));
    IIM_CHECK(iim_poisson_solve(g, f, data, H_box, nullptr, nullptr, H_out, nullptr, nullptr, nullptr, opts, stats,
                                stream));
    if (H_wall_out) IIM_CHECK(iim_wall_values(g, H_out, H_wall_out, stream));
    return IIM_OK;
}

// Stage times of the Williamson scheme: stage st sees the state at t + kRK3C[st] dt.
static constexpr double kRK3C[3] = {0.0, 1.0 / 3.0, 3.0 / 4.0};

// u_b at a stage time: u_b + c dt du_b/dt (u_b NULL = 0)
__global__ void k_ub_stage(int m, const double* __restrict__ ub, const double* __restrict__ rate, double cdt,
                           double* __restrict__ out) {
    pdl_wait();
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < m) out[e] = (ub ? ub[e] : 0.0) + cdt * rate[e];
}

static iim_status rk3_step(iim_geometry g, double* omega, double* gamma, double* psibar, const double* u_b,
                           const double* u_b_rate, const double* psi_b, const double* psi_box, const double Uinf[2],
                           double nu, double c_stab, double* dt_inout, const iim_opts* opts, iim_stats* per_stage,
                           iim_stream stream) {
    if (!g || !omega || !dt_inout || !(nu >= 0.0) || (g->nb > 0 && (!gamma || !psibar))) return IIM_ERR_INVALID_ARG;
    if (*dt_inout <= 0.0 && !(c_stab > 0.0)) return IIM_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    TrWork W;
    IIM_CHECK(tr_work(g, &W));
    const TrView v = make_view(g, W, Uinf, omega, W.vx, W.vy);
    const long n = (long)g->NX * g->NY;
    IIM_TRY(cudaMemsetAsync(W.dG, 0, 64 * sizeof(double), s));
    double dt = *dt_inout;
    for (int st = 0; st < 3; ++st) {
        iim_stats stats;
        const iim_status ps = iim_poisson_solve(g, omega, psi_b ? psi_b : W.zeros, psi_box, gamma, psibar, W.psi, W.vx,
                                                W.vy, nullptr, opts, &stats, stream);
        if (per_stage) per_stage[st] = stats;
        if (ps != IIM_OK) return ps;
        if (st == 0 && dt <= 0.0) {
            launch_next("tr_speed_max", 0.0, 0.0, k_speed_max<256>, 256, 256, 0, s, n, (const double*)W.vx, (const double*)W.vy,
                   W.part);
            IIM_LAUNCHED();
            std::vector<double> part(256);
            IIM_TRY(cudaMemcpyAsync(part.data(), W.part, 256 * sizeof(double), cudaMemcpyDeviceToHost, s));
            IIM_TRY(cudaStreamSynchronize(s));
            double U = 0.0;
            for (double x : part) U = std::max(U, x);
            const double h = g->h;
            dt = c_stab / (U / (kStabC * h) + nu / (kStabR * h * h));
        }
        const double* ub = u_b;
        if (u_b_rate) {
            const int m = 2 * g->ncp;
            if (m > 0)
                launch_next("tr_ub_stage", 0.0, 0.0, k_ub_stage, (unsigned)((m + 255) / 256), 256, 0, s, m, u_b, u_b_rate,
                       kRK3C[st] * dt, W.ub_stage);
            ub = W.ub_stage;
        }
        IIM_CHECK(prepare_stage(g, W, v, ub, nullptr, nullptr, s));
        const KelvinArgs kv{g->d_regions, nullptr, 1, kRK3B[st], W.dG, gamma};
        IIM_CHECK(transport_rhs(g, v, nu, 1, kRK3A[st], dt, W.dw, kv, s));
        launch_next("tr_rk_omega", 24.0 * (double)n, 0.0, k_rk_omega, (unsigned)((n + 255) / 256), 256, 0, s, g->NX, g->NY,
               kRK3B[st], (const double*)W.dw, g->node_class, omega);
        IIM_LAUNCHED();
    }
    IIM_TRY(cudaStreamSynchronize(s));
    *dt_inout = dt;
    return IIM_OK;
}

extern "C" iim_status iim_rk3_step(iim_geometry g, double* omega, double* gamma, double* psibar, const double* u_b,
                                   const double* psi_b, const double* psi_box, const double Uinf[2], double nu,
                                   double c_stab, double* dt_inout, const iim_opts* opts, iim_stats* per_stage,
                                   iim_stream stream) {
    return rk3_step(g, omega, gamma, psibar, u_b, nullptr, psi_b, psi_box, Uinf, nu, c_stab, dt_inout, opts, per_stage,
                    stream);
}

extern "C" iim_status iim_rk3_step_moving_wall(iim_geometry g, double* omega, double* gamma, double* psibar,
                                               const double* u_b, const double* u_b_rate, const double* psi_b,
                                               const double* psi_box, const double Uinf[2], double nu, double c_stab,
                                               double* dt_inout, const iim_opts* opts, iim_stats* per_stage,
                                               iim_stream stream) {
    if (!u_b_rate) return IIM_ERR_INVALID_ARG;
    return rk3_step(g, omega, gamma, psibar, u_b, u_b_rate, psi_b, psi_box, Uinf, nu, c_stab, dt_inout, opts,
                    per_stage, stream);
}
