// One time step of the two-phase wave tank on the GPU (2D, FP64).
//
// Paper (arxiv 2206.07732) passages implemented here:
//   Eq. int_fh ............ heave force as a sum over the faces where the body SDF
//                           changes sign (k_force_partial, k_heave)
//   Eq. newton_u .......... heave update, with an artificial added mass that keeps
//                           the n_cycles = 1 coupling stable (k_heave)
//   Section "Interface tracking" and "Level set advection" .. PPM advection of
//                           sigma (k_advect), Sussman reinitialisation (k_reinit),
//                           analytic body SDF psi by CSG max (psi_box)
//   Eqs. ls_flow, ls_solid, Hflow, Hbody .. materials (k_materials)
//   Eq. c_discrete_momentum .. consistent mass/momentum transport, Crank-Nicolson
//                           viscosity, flow-density gravity, implicit Brinkman term
//                           (Eq. bp_discrete) (k_momentum, k_jacobi)
//   Eq. spongelayer ....... vorticity damping over the top four cells
//   Section "Numerical wave tank" .. Airy inflow at x = 0, wave damping zone
//   Eq. c_discrete_continuity .. incremental projection (k_proj_rhs, solver, k_project)
// Layouts: cells [ny][nx], u [ny][nx+1], v [ny+1][nx]; one thread per cell/face,
// consecutive threads along x (coalesced rows).
#include <algorithm>
#include <cmath>
#include <utility>

#include "limiters.cuh"
#include "tank.cuh"

namespace wec {
namespace {

constexpr int TB = 256;

template <typename R>
__device__ __forceinline__ const TankC<R> &cst(const TankP &P)
{
    if constexpr (sizeof(R) == 4)
        return P.cf;
    else
        return P.cd;
}

__device__ __forceinline__ int clampi(int a, int lo, int hi) { return a < lo ? lo : (a > hi ? hi : a); }
template <typename R>
__device__ __forceinline__ R sq(R a) { return a * a; }

// Smoothed Heaviside of Eqs. Hflow / Hbody, half-width eps = n_cells h (n_cells = 1).
template <typename R>
__device__ __forceinline__ R heav(R phi, R eps)
{
    if (phi < -eps) return R(0.0);
    if (phi > eps) return R(1.0);
    return R(0.5) * (R(1.0) + phi / eps + sin(R(kPi) * phi / eps) / R(kPi));
}

// Box SDF as the CSG intersection (max) of four half-planes.
template <typename R>
__device__ __forceinline__ R psi_box(const TankP &P, R x, R y, R yc)
{
    if (!P.has_body) return R(1.0e3);
    return fmax(fabs(x - cst<R>(P).bxc) - R(0.5) * cst<R>(P).bw, fabs(y - yc) - R(0.5) * cst<R>(P).bh);
}

__device__ double eta_at(const TankP &P, double x, double t)
{
    double e = 0.0;
    for (int c = 0; c < P.ncomp; ++c) e += P.amp[c] * cos(P.kw[c] * x - P.omega[c] * t + P.phase[c]);
    return e;
}

// Linear Airy velocity with Wheeler stretching y' = d y / (d + eta) up to the
// surface, blended to zero in the air by 1 - H(y - d - eta).
__device__ void airy_uv(const TankP &P, double x, double y, double t, double *uo, double *vo)
{
    double d = P.depth;
    double e = eta_at(P, x, t);
    double ys = y < d + e ? y : d + e;
    double yp = d * ys / (d + e);
    double blend = 1.0 - heav(y - d - e, P.h);
    double su = 0.0, sv = 0.0;
    for (int c = 0; c < P.ncomp; ++c) {
        double k = P.kw[c], w = P.omega[c];
        double ph = k * x - w * t + P.phase[c];
        double sk = sinh(k * d);
        su += P.amp[c] * w * cosh(k * yp) / sk * cos(ph);
        sv += P.amp[c] * w * sinh(k * yp) / sk * sin(ph);
    }
    *uo = blend * su;
    *vo = blend * sv;
}

// -------------------------------------------------------- ghost values ----
// sigma: left = incident wave y - d - eta(x, t) (eta precomputed per ghost column),
// right = zero gradient, bottom/top = linear extrapolation.
template <typename R, typename S>
__device__ __forceinline__ R sig_at(const TankP &P, const S *__restrict__ s,
                                         const double *__restrict__ etag, int i, int j)
{
    if (i < 0) return (j + R(0.5)) * cst<R>(P).h - cst<R>(P).depth - R(etag[-1 - i]);
    if (i > P.nx - 1) i = P.nx - 1;
    if (j < 0) return R(s[i]) + j * (R(s[P.nx + i]) - R(s[i]));
    if (j > P.ny - 1) {
        int m = j - (P.ny - 1);
        R a = R(s[(P.ny - 1) * P.nx + i]), b = R(s[(P.ny - 2) * P.nx + i]);
        return a + m * (a - b);
    }
    return R(s[j * P.nx + i]);
}

template <typename R, typename S>
__device__ __forceinline__ R u_at(const TankP &P, const S *__restrict__ u, int i, int j)
{
    return R(u[clampi(j, 0, P.ny - 1) * (P.nx + 1) + clampi(i, 0, P.nx)]);
}

// v: clamp rows; right wall free slip; left: odd reflection about v_in(y_j, t).
template <typename R, typename S>
__device__ __forceinline__ R v_at(const TankP &P, const S *__restrict__ v,
                                       const double *__restrict__ vin, int i, int j)
{
    j = clampi(j, 0, P.ny);
    if (i > P.nx - 1) i = P.nx - 1;
    if (i < 0) return R(2.0) * R(vin[j]) - R(v[j * P.nx + (-1 - i)]);
    return R(v[j * P.nx + i]);
}

template <typename R, typename S>
__device__ __forceinline__ R cell_at(const TankP &P, const S *__restrict__ a, int i, int j)
{
    return R(a[clampi(j, 0, P.ny - 1) * P.nx + clampi(i, 0, P.nx - 1)]);
}

// Damping-zone weight (Jacobsen) and the vorticity-damping shape (cos(pi z~) + 1),
// evaluated once per tank into tables (columns / rows) by k_tables.
__device__ __forceinline__ double damp_alpha_eval(const TankP &P, double x)
{
    if (P.damp_len <= 0.0 || x <= P.damp_x0) return 0.0;
    double xi = (x - P.damp_x0) / P.damp_len;
    if (xi > 1.0) xi = 1.0;
    return (exp(pow(xi, 3.5)) - 1.0) / (exp(1.0) - 1.0);
}

__device__ __forceinline__ double vort_shape_eval(const TankP &P, double y)
{
    double w = 4.0 * P.h;
    if (y < P.ly - w) return 0.0;
    double zt = (y - P.ly) / w;
    return cos(kPi * zt) + 1.0;
}

// g(z~) = rho_a (cos(pi z~) + 1) / (4 dt) (Eq. spongelayer) from the tabulated shape.
template <typename R>
__device__ __forceinline__ R vort_damp(const TankP &P, R shape, R idt)
{
    return cst<R>(P).rho_a * shape * (R(0.25) * idt);
}

// ------------------------------------------------------------- kernels ----
template <typename R>
__device__ __forceinline__ R warp_sum_d(R v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// eta at x = 0 (for the inflow profile) and at the three ghost columns, at t^n
// and t^{n+1}: one block per value, threads over the wave components.  The blocks of
// x = 0 also form what the components' velocities share over the rows (bc.comp): FP64
// transcendentals are some 50 to 80 instructions of a pipe that issues one per 16
// clocks, so every row of k_bc_rows evaluating them for itself bound that kernel.
// With these the two kernels went from 53 to 28 us at 1024x256 and from 37 to 24 at
// 128x64 (64 components, launch gaps included).
constexpr int kEtaT = 128;
__global__ void __launch_bounds__(kEtaT) k_bc_eta(TankP P, const StepScalars *S, const double *__restrict__ inp, Bc bc)
{
    pdl_entry();
    __shared__ double sh[kEtaT / 32];
    const int w = blockIdx.x, lane = threadIdx.x & 31;          // 8 blocks: (time, position)
    const double t = (w & 1) ? S->t + inp[0] : S->t;
    const int pos = w >> 1;                                    // 0: x = 0; 1..3: ghost columns
    const double x = pos == 0 ? 0.0 : (-pos + 0.5) * P.h;
    double e = 0.0;
    for (int c = threadIdx.x; c < P.ncomp; c += kEtaT) {
        const double a = P.amp[c], ph = P.kw[c] * x - P.omega[c] * t + P.phase[c];
        if (pos == 0) {
            double sn, cs;
            sincos(ph, &sn, &cs);
            e += a * cs;
            const double f = a * P.omega[c] / sinh(P.kw[c] * P.depth);
            if (w & 1) {
                bc.comp[c] = f * cs;
                bc.comp[2 * P.ncomp + c] = f * sn;
            } else {
                bc.comp[P.ncomp + c] = f * sn;
            }
        } else {
            e += a * cos(ph);
        }
    }
    e = warp_sum_d(e);
    if (lane == 0) sh[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x) return;
    e = 0.0;
    for (int q = 0; q < kEtaT / 32; ++q) e += sh[q];
    if (pos == 0)
        bc.eta_in[w & 1] = e;
    else
        ((w & 1) ? bc.eta1 : bc.eta0)[pos - 1] = e;
}

// Inflow at x = 0: u_in(y_{j+1/2}, t^{n+1}) and v_in(y_j, t^n), v_in(y_j, t^{n+1}),
// Airy velocities with Wheeler stretching, blended to zero in the air.  A block per
// row j, a warp for each of the three, lanes over the components.
template <typename R>
__global__ void __launch_bounds__(96) k_bc_rows(TankP P, const StepScalars *S, const double *__restrict__ inp, Bc bc)
{
    pdl_entry();
    const int j = blockIdx.x, q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (q == 0 && j == P.ny) return;
    const R d = cst<R>(P).depth;
    const R y = q == 0 ? (j + R(0.5)) * cst<R>(P).h : j * cst<R>(P).h;
    const R e = R(bc.eta_in[q == 1 ? 0 : 1]);
    const R ys = y < d + e ? y : d + e;
    const R yp = d * ys / (d + e);
    R acc = R(0.0);
    if constexpr (sizeof(R) == 4) {
        const R t = q == 1 ? R(S->t) : R(S->t) + R(inp[0]);
        for (int c = lane; c < P.ncomp; c += 32) {
            R k = R(P.kw[c]), w = R(P.omega[c]);
            R ph = -w * t + R(P.phase[c]);
            // cosh(k y') / sinh(k d) and sinh(k y') / sinh(k d), overflow-free in FP32
            // (k d reaches ~120 for short components)
            R e1 = exp(k * (yp - d)), e2 = exp(-k * (yp + d)), den = R(1.0) - exp(R(-2.0) * k * d);
            if (q == 0)
                acc += R(P.amp[c]) * w * ((e1 + e2) / den) * cos(ph);
            else
                acc += R(P.amp[c]) * w * ((e1 - e2) / den) * sin(ph);
        }
    } else {
        const double *f = bc.comp + q * P.ncomp;
        for (int c = lane; c < P.ncomp; c += 32) {
            const R ky = P.kw[c] * yp;
            acc += f[c] * (q == 0 ? cosh(ky) : sinh(ky));
        }
    }
    acc = warp_sum_d<R>(acc);
    if (lane) return;
    (q == 0 ? bc.uin1 : q == 1 ? bc.vin0 : bc.vin1)[j] = (R(1.0) - heav<R>(y - d - e, cst<R>(P).h)) * acc;
}

// Cell materials from sigma and the body at yc (which = 0: y_c^n, 1: y_c^{n+1}).
template <typename R>
__global__ void k_materials(TankP P, const StepScalars *S, int which, const double *__restrict__ sig,
                            R *rho, R *mu, R *rhof, R *chi)
{
    pdl_entry();
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= P.nx * P.ny) return;
    int i = c % P.nx, j = c / P.nx;
    R yc = which ? R(S->yc1) : R(S->yc);
    R ps = psi_box<R>(P, (i + R(0.5)) * cst<R>(P).h, (j + R(0.5)) * cst<R>(P).h, yc);
    R hf = heav<R>(R(sig[c]), cst<R>(P).h), hb = heav<R>(ps, cst<R>(P).h);
    R rf = cst<R>(P).rho_w + (cst<R>(P).rho_a - cst<R>(P).rho_w) * hf;
    R mf = cst<R>(P).mu_w + (cst<R>(P).mu_a - cst<R>(P).mu_w) * hf;
    if (rho) rho[c] = cst<R>(P).rho_s + (rf - cst<R>(P).rho_s) * hb;
    if (mu) mu[c] = cst<R>(P).mu_s + (mf - cst<R>(P).mu_s) * hb;
    if (rhof) rhof[c] = rf;
    if (chi) chi[c] = R(1.0) - hb;
}

__device__ double block_sum(double v, double *sh)
{
    int t = threadIdx.x;
    sh[t] = v;
    __syncthreads();
    for (int s = blockDim.x >> 1; s > 0; s >>= 1) {
        if (t < s) sh[t] += sh[t + s];
        __syncthreads();
    }
    double r = sh[0];
    __syncthreads();
    return r;
}

// Eq. int_fh, heave component: faces whose two cells have opposite psi sign;
// pressure linearly interpolated to the psi = 0 crossing with |psi| weights;
// n_f out of the body; viscous traction by central differences at the face.
template <typename M>
__global__ void k_force_partial(TankP P, const StepScalars *S, const double *__restrict__ p,
                                const double *__restrict__ u, const double *__restrict__ v,
                                const M *__restrict__ mu, const double *__restrict__ vin0,
                                double *__restrict__ part)
{
    pdl_entry();
    __shared__ double sh[TB];
    const int nx = P.nx, ny = P.ny;
    const double h = P.h, yc = S->yc;
    // Only faces whose two cells straddle the box boundary contribute, and those
    // cells lie within one cell of it: walk cells i0..i1 x j0..j1, two cells
    // around the box (the same nonzero terms as a walk over every face).
    const int i0 = max(0, (int)floor((P.bxc - 0.5 * P.bw) / h) - 2);
    const int i1 = min(nx - 1, (int)ceil((P.bxc + 0.5 * P.bw) / h) + 2);
    const int j0 = max(0, (int)floor((yc - 0.5 * P.bh) / h) - 2);
    const int j1 = min(ny - 1, (int)ceil((yc + 0.5 * P.bh) / h) + 2);
    const int bi = i1 - i0 + 1, bj = j1 - j0 + 1;
    // y-faces: j in j0+1..j1, i in i0..i1; x-faces: i in i0+1..i1, j in j0..j1
    const long long ny_faces = bi > 0 && bj > 1 ? (long long)bi * (bj - 1) : 0;
    const long long nx_faces = bi > 1 && bj > 0 ? (long long)(bi - 1) * bj : 0;
    double acc = 0.0;
    if (P.has_body) {
        for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < ny_faces + nx_faces;
             k += (long long)gridDim.x * blockDim.x) {
            if (k < ny_faces) {
                int i = i0 + (int)(k % bi), j = j0 + 1 + (int)(k / bi);
                double x = (i + 0.5) * h;
                double pl = psi_box(P, x, (j - 0.5) * h, yc), pr = psi_box(P, x, (j + 0.5) * h, yc);
                if (!(pl * pr < 0.0)) continue;
                double nrm = pl < 0.0 ? 1.0 : -1.0;
                double wl = fabs(pl), wr = fabs(pr);
                double pf = (p[(j - 1) * nx + i] * wr + p[j * nx + i] * wl) / (wl + wr);
                double muf = 0.5 * (double(mu[(j - 1) * nx + i]) + double(mu[j * nx + i]));
                double dvdy = (v_at<double>(P, v, vin0, i, j + 1) - v_at<double>(P, v, vin0, i, j - 1)) / (2.0 * h);
                acc += (-pf * nrm + muf * 2.0 * dvdy * nrm) * h;
            } else {
                long long q = k - ny_faces;
                int i = i0 + 1 + (int)(q % (bi - 1)), j = j0 + (int)(q / (bi - 1));
                double y = (j + 0.5) * h;
                double pl = psi_box(P, (i - 0.5) * h, y, yc), pr = psi_box(P, (i + 0.5) * h, y, yc);
                if (!(pl * pr < 0.0)) continue;
                double nrm = pl < 0.0 ? 1.0 : -1.0;
                double muf = 0.5 * (double(mu[j * nx + i - 1]) + double(mu[j * nx + i]));
                double dvdx = 0.5 * ((v_at<double>(P, v, vin0, i, j) - v_at<double>(P, v, vin0, i - 1, j)) +
                                     (v_at<double>(P, v, vin0, i, j + 1) - v_at<double>(P, v, vin0, i - 1, j + 1))) / h;
                double dudy = (u_at<double>(P, u, i, j + 1) - u_at<double>(P, u, i, j - 1)) / (2.0 * h);
                acc += muf * (dvdx + dudy) * nrm * h;
            }
        }
    }
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// Sum of the force partials (fixed order), then the stabilised heave update:
// (m + m_a)(zdot^{n+1} - zdot^n) = dt (F - m g + F_PTO) + m_a (zdot^n - zdot^{n-1}).
__global__ void k_heave(TankP P, StepScalars *S, const double *__restrict__ part, const double *__restrict__ inp)
{
    pdl_entry();
    const double dt = inp[0], fpto_in = inp[1];
    __shared__ double sh[TB];
    double s = 0.0;
    for (int b = threadIdx.x; b < kRedBlocks; b += blockDim.x) s += part[b];
    double F = block_sum(s, sh);
    if (threadIdx.x != 0) return;
    double fpto = fpto_in - P.pto_c * S->zdot;
    double zd1 = S->zdot, yc1 = S->yc;
    if (P.has_body) {
        double m = P.mass, ma = P.added_mass;
        zd1 = S->zdot + (dt * (F - m * P.g + fpto) + ma * (S->zdot - S->zdot_prev)) / (m + ma);
        yc1 = S->yc + 0.5 * dt * (S->zdot + zd1);
    }
    S->F = F;
    S->fpto = fpto;
    S->zdot1 = zd1;
    S->yc1 = yc1;
}

// The stencil kernels run one block row per grid row (blockIdx.x the row, which
// may exceed 65535, blockIdx.y the tile along it; no index division) and split
// off the cells and faces whose whole stencil lies inside the grid: those read at
// fixed offsets, the rest through the accessors above with their ghost rules.  In
// FP64 every one of them is bound by the FP64 pipe (two operations per clock and
// SM), so the arithmetic spends as few FP64 instructions as the formulas allow:
// limiter decisions on the integer pipe (limiters.cuh), face quantities formed
// once, the viscous coefficients shared by its two forms.  At 1024x256 in FP64 the step's
// stencils went from 1.15 to 0.43 ms: advection 243 -> 63 us, a reinitialisation
// stage 51 -> 26, the momentum system 246 -> 106 (with the face quantities), a
// Jacobi sweep 69 -> 18.
constexpr int TX = 128;  // threads along a row
inline dim3 row_grid(int nx, int rows) { return dim3(rows, (nx + TX - 1) / TX); }

// The PPM value of sigma on every x-face (block rows 0 .. ny-1) and y-face (the
// ny+1 rows after them), time-centred and upwind: a face value depends on the
// face alone and is read by the two cells beside it.  Formed by each cell for its
// four faces, advection took 243 us at 1024x256 in FP64; the two kernels take 63.
template <typename R>
__global__ void __launch_bounds__(TX) k_ppm_faces(TankP P, const R *__restrict__ s, const R *__restrict__ u,
                                                  const R *__restrict__ v, const double *__restrict__ eta0,
                                                  const double *__restrict__ inp, R *__restrict__ Fx, R *__restrict__ Fy)
{
    pdl_entry();
    const int nx = P.nx, ny = P.ny, i = blockIdx.y * TX + threadIdx.x;
    const bool xf = (int)blockIdx.x < ny;
    const int j = xf ? blockIdx.x : blockIdx.x - ny;
    if (i >= nx + (xf ? 1 : 0)) return;
    const int f = xf ? j * (nx + 1) + i : j * nx + i, c = j * nx + i, sd = xf ? 1 : nx;
    const int cd = xf ? i : j, nd = xf ? nx : ny;
    R a[6];
    if (cd >= 3 && cd + 2 < nd) {
#pragma unroll
        for (int m = 0; m < 6; ++m) a[m] = s[c + (m - 3) * sd];
    } else {
#pragma unroll
        for (int m = 0; m < 6; ++m) a[m] = sig_at<R>(P, s, eta0, xf ? i + m - 3 : i, xf ? j : j + m - 3);
    }
    (xf ? Fx : Fy)[f] = ppm_face3<R>(a, (xf ? u : v)[f], R(inp[0]) * cst<R>(P).ih);
}

// sigma* = sigma^n - dt Q(u^n, sigma^n) from the face values, then damping-zone
// relaxation.
template <typename R>
__global__ void __launch_bounds__(TX) k_advect(TankP P, const R *__restrict__ s, const R *__restrict__ u,
                                               const R *__restrict__ v, const R *__restrict__ Fx,
                                               const R *__restrict__ Fy, const double *__restrict__ inp,
                                               const R *__restrict__ alpha_c, double *__restrict__ out,
                                               R *__restrict__ out_w)
{
    pdl_entry();
    const int nx = P.nx, i = blockIdx.y * TX + threadIdx.x, j = blockIdx.x;
    if (i >= nx) return;
    const int c = j * nx + i, fu = c + j;
    const R dtih = R(inp[0]) * cst<R>(P).ih;
    const R ub = R(0.5) * (u[fu] + u[fu + 1]), vb = R(0.5) * (v[c] + v[c + nx]);
    const R sa = s[c] - dtih * (ub * (Fx[fu + 1] - Fx[fu]) + vb * (Fy[c + nx] - Fy[c]));
    const R al = alpha_c[i];
    const R r = (R(1.0) - al) * sa + al * ((j + R(0.5)) * cst<R>(P).h - cst<R>(P).depth);
    out[c] = r;
    if (out_w) out_w[c] = r;
}

// One TVD-RK2 stage of the Sussman relaxation: y = f - dtau S (|grad f| - 1), the
// Godunov Hamiltonian on ENO-2 (minmod) one-sided differences, taken in units of
// 1/h; stage 1 out = y, stage 2 (fprev) out = (fprev + y) / 2.  S = sigma0 /
// sqrt(sigma0^2 + h^2) is fixed over the pseudo-steps: the first stage (first: f is
// sigma0) forms it and stores it.
template <typename R, typename TO>
__global__ void __launch_bounds__(TX) k_reinit(TankP P, const R *__restrict__ f, R *sgn, const R *__restrict__ fprev,
                                               const double *__restrict__ eta1, R dtau, TO *__restrict__ out, int first)
{
    pdl_entry();
    const int nx = P.nx, ny = P.ny, i = blockIdx.y * TX + threadIdx.x, j = blockIdx.x;
    const bool inner = warp_inside(i >= 2 && i < nx - 2 && j >= 2 && j < ny - 2, i < nx);
    if (i >= nx) return;
    const int c0 = j * nx + i;
    const R ih = cst<R>(P).ih, h = cst<R>(P).h, c = f[c0];
    R S;
    if (first)
        sgn[c0] = S = c / sqrt(c * c + h * h);
    else
        S = sgn[c0];
    const bool pos = positive(S);
    R g2 = R(0.0);
#pragma unroll
    for (int d = 0; d < 2; ++d) {
        const int o = d ? nx : 1, di = d == 0, dj = d;
        R m2, m1, p1, p2;
        if (inner) {
            m2 = f[c0 - 2 * o];
            m1 = f[c0 - o];
            p1 = f[c0 + o];
            p2 = f[c0 + 2 * o];
        } else {
            m2 = sig_at<R>(P, f, eta1, i - 2 * di, j - 2 * dj);
            m1 = sig_at<R>(P, f, eta1, i - di, j - dj);
            p1 = sig_at<R>(P, f, eta1, i + di, j + dj);
            p2 = sig_at<R>(P, f, eta1, i + 2 * di, j + 2 * dj);
        }
        // the three second differences from the four first ones
        const R e0 = c - m1, e1 = p1 - c, dm = e0 - (m1 - m2), d0 = e1 - e0, dp = (p2 - p1) - e1;
        const R a = e0 + R(0.5) * mm3(dm, d0), nb = R(0.5) * mm3(d0, dp) - e1;
        const R m = godunov_max(a, nb, pos);
        g2 += m * m;
    }
    const R y = c - dtau * (S * (ih * sqrt(g2) - R(1.0)));
    out[c0] = fprev ? R(0.5) * (fprev[c0] + y) : y;
}

// ---------------------------------------------------- momentum helpers ----
// Per-tank tables: alpha at cell centres [nx] and at u-faces [nx+1]; vorticity
// shape at cell-centre rows [ny] and at v-face rows [ny+1].
template <typename R>
struct Tabs {
    const R *alpha_c, *alpha_u, *vort_c, *vort_v;
};

// Layout of one table set: alpha_c [nx], alpha_u [nx+1], vort_c [ny], vort_v [ny+1].
// t32 (optional) receives the same tables in FP32.
__global__ void k_tables(TankP P, double *t, float *t32)
{
    pdl_entry();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int nx = P.nx, ny = P.ny, o1 = nx, o2 = 2 * nx + 1, o3 = 2 * nx + 1 + ny;
    auto put = [&](int o, double val) {
        t[o] = val;
        if (t32) t32[o] = (float)val;
    };
    if (k < nx) put(k, damp_alpha_eval(P, (k + 0.5) * P.h));
    if (k <= nx) put(o1 + k, damp_alpha_eval(P, k * P.h));
    if (k < ny) put(o2 + k, vort_shape_eval(P, (k + 0.5) * P.h));
    if (k <= ny) put(o3 + k, vort_shape_eval(P, k * P.h));
}

// u, v with their ghosts where IN is false (the grid's edges); at fixed offsets
// where the stencil is inside
template <bool IN, typename R>
__device__ __forceinline__ R uq2(const TankP &P, const R *__restrict__ u, int i, int j)
{
    if constexpr (IN) return u[j * (P.nx + 1) + i]; else return u_at<R>(P, u, i, j);
}
template <bool IN, typename R>
__device__ __forceinline__ R vq2(const TankP &P, const R *__restrict__ v, const double *__restrict__ vin, int i, int j)
{
    if constexpr (IN) return v[j * P.nx + i]; else return v_at<R>(P, v, vin, i, j);
}
// face densities ru [ny][nx+1], rv [ny+1][nx] (k_faces), clamped
template <bool IN, typename R>
__device__ __forceinline__ R ruq2(const TankP &P, const R *__restrict__ r, int i, int j)
{
    if constexpr (IN) return r[j * (P.nx + 1) + i];
    return r[clampi(j, 0, P.ny - 1) * (P.nx + 1) + clampi(i, 0, P.nx)];
}
template <bool IN, typename R>
__device__ __forceinline__ R rvq2(const TankP &P, const R *__restrict__ r, int i, int j)
{
    if constexpr (IN) return r[j * P.nx + i];
    return r[clampi(j, 0, P.ny) * P.nx + clampi(i, 0, P.nx - 1)];
}

// Densities of rho^n on the u- and v-faces (the mean of the face's cells) and the
// viscosities mu^n and mu^{n+1} at the nodes [ny+1][nx+1] (the mean of the four
// cells around it, clamped into the grid), formed once per step.
template <typename R>
__global__ void __launch_bounds__(TX) k_faces(TankP P, const R *__restrict__ rho, const R *__restrict__ mu_n,
                                              const R *__restrict__ mu_1, R *__restrict__ ru, R *__restrict__ rv,
                                              R *__restrict__ nd_n, R *__restrict__ nd_1)
{
    pdl_entry();
    const int nx = P.nx, ny = P.ny, i = blockIdx.y * TX + threadIdx.x, j = blockIdx.x;
    if (i > nx) return;
    const int i0 = max(i - 1, 0), i1 = min(i, nx - 1), j0 = max(j - 1, 0), j1 = min(j, ny - 1);
    const int c00 = j0 * nx + i0, c01 = j0 * nx + i1, c10 = j1 * nx + i0, c11 = j1 * nx + i1;
    if (j < ny) ru[j * (nx + 1) + i] = R(0.5) * (rho[c10] + rho[c11]);
    if (i < nx) rv[j * nx + i] = R(0.5) * (rho[c01] + rho[c11]);
    nd_n[j * (nx + 1) + i] = R(0.25) * ((mu_n[c00] + mu_n[c01]) + (mu_n[c10] + mu_n[c11]));
    nd_1[j * (nx + 1) + i] = R(0.25) * ((mu_1[c00] + mu_1[c01]) + (mu_1[c10] + mu_1[c11]));
}

// One face of a momentum control volume of component C (0: u-face, 1: v-face) at
// (i, j), in direction d, side s (0 lower, 1 upper): twice the mass flux, m = U r
// with U the sum of two d-velocities, and twice the momentum flux, f = m q (the halves
// are taken once, from the sums over the CV's faces); r and q the Koren-limited upwind
// face density and velocity -- rho-breve and the convection share the mass flux.  Side 1 of a CV is side 0 of
// the next one along d, the same values.
template <bool IN, int C, typename R>
__device__ __forceinline__ void cv_face(const TankP &P, const R *__restrict__ rf, const R *__restrict__ u,
                                        const R *__restrict__ v, const double *__restrict__ vin, int i, int j, int d,
                                        int s, R &m, R &f)
{
    const int o = s - 1;
    R U;
    if (C == 0)
        U = d == 0 ? uq2<IN>(P, u, i + o, j) + uq2<IN>(P, u, i + o + 1, j)
                   : vq2<IN>(P, v, vin, i - 1, j + s) + vq2<IN>(P, v, vin, i, j + s);
    else
        U = d == 0 ? uq2<IN>(P, u, i + s, j - 1) + uq2<IN>(P, u, i + s, j)
                   : vq2<IN>(P, v, vin, i, j + o) + vq2<IN>(P, v, vin, i, j + o + 1);
    const int di = d == 0, dj = d;
    R rr[4], qq[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int a = i + (o - 1 + k) * di, b = j + (o - 1 + k) * dj;
        rr[k] = C == 0 ? ruq2<IN>(P, rf, a, b) : rvq2<IN>(P, rf, a, b);
        qq[k] = C == 0 ? uq2<IN>(P, u, a, b) : vq2<IN>(P, v, vin, a, b);
    }
    m = U * upw3(rr[0], rr[1], rr[2], rr[3], U);
    f = m * upw3(qq[0], qq[1], qq[2], qq[3], U);
}

// The viscous operator div[mu (grad u + grad u^T)] of component C at a face, times h^2,
// in two forms with the same instruction count: as a sum of differences (DIFF: the
// explicit half, whose rounding then scales with the differences), and as S of
// h^2 L_mu(u) = S - Lc u_f, the sum over the face's neighbours (its own component and
// the cross terms; nd: node viscosities), Lc the sum of the coefficients (the
// diagonal, which the Jacobi splitting moves to the left).
template <bool IN, int C, bool DIFF, typename R>
__device__ __forceinline__ R visc_sum(const TankP &P, const R *__restrict__ mu, const R *__restrict__ nd,
                                      const R *__restrict__ u, const R *__restrict__ v, const double *__restrict__ vin,
                                      int i, int j)
{
    const int nn = P.nx + 1;
    if (C == 0) {
        const R c = DIFF ? uq2<IN>(P, u, i, j) : R(0.0);
        auto at = [&](int a, int b) { return DIFF ? uq2<IN>(P, u, a, b) - c : uq2<IN>(P, u, a, b); };
        const R m1 = mu[j * P.nx + i], m0 = mu[j * P.nx + i - 1], n1 = nd[(j + 1) * nn + i], n0 = nd[j * nn + i];
        return R(2.0) * (m1 * at(i + 1, j) + m0 * at(i - 1, j)) +
               (n1 * (at(i, j + 1) + (vq2<IN>(P, v, vin, i, j + 1) - vq2<IN>(P, v, vin, i - 1, j + 1))) +
                n0 * (at(i, j - 1) - (vq2<IN>(P, v, vin, i, j) - vq2<IN>(P, v, vin, i - 1, j))));
    }
    const R c = DIFF ? vq2<IN>(P, v, vin, i, j) : R(0.0);
    auto at = [&](int a, int b) { return DIFF ? vq2<IN>(P, v, vin, a, b) - c : vq2<IN>(P, v, vin, a, b); };
    const R m1 = mu[min(j, P.ny - 1) * P.nx + i], m0 = mu[(j - 1) * P.nx + i], n1 = nd[j * nn + i + 1], n0 = nd[j * nn + i];
    return R(2.0) * (m1 * at(i, j + 1) + m0 * at(i, j - 1)) +
           (n1 * (at(i + 1, j) + (uq2<IN>(P, u, i + 1, j) - uq2<IN>(P, u, i + 1, j - 1))) +
            n0 * (at(i - 1, j) - (uq2<IN>(P, u, i, j) - uq2<IN>(P, u, i, j - 1))));
}
template <int C, typename R>
__device__ __forceinline__ R visc_diag(const TankP &P, const R *__restrict__ mu, const R *__restrict__ nd, int i, int j)
{
    const int nn = P.nx + 1;
    if (C == 0)
        return R(2.0) * (mu[j * P.nx + i] + mu[j * P.nx + i - 1]) + (nd[(j + 1) * nn + i] + nd[j * nn + i]);
    return R(2.0) * (mu[min(j, P.ny - 1) * P.nx + i] + mu[(j - 1) * P.nx + i]) + (nd[j * nn + i + 1] + nd[j * nn + i]);
}

// The stencils reach three cells each way (the transport's upwind triples).
__device__ __forceinline__ bool inside2(const TankP &P, int i, int j)
{
    return i >= 3 && i <= P.nx - 4 && j >= 3 && j <= P.ny - 4;
}

template <typename R>
struct MomArgs {
    const double *inp;
    const StepScalars *S;
    Tabs<R> tb;
    const R *ru, *rv, *mu_n, *mu_1, *nd_n, *nd_1, *chi_1, *rf_1, *u, *v;
    const double *p;
    Bc bc;
    R *Du, *Dv;                // diagonal (without the viscous part)
    R *Ru, *Rv, *Qu, *Qv;      // R / D', (1 / (2 h^2)) / D' with D' = D + Lc / (2 h^2)
    R *ua, *va;                // first Jacobi iterate: u^n with the Dirichlet faces at t^{n+1}
};

// The momentum system at the faces of component C along a row: a warp covers 31
// control volumes, lane l forms the lower x face of its CV and takes the upper one
// from lane l + 1 (lane 31 supplies its lower face only).
template <int C, typename R>
__device__ __forceinline__ void momentum_row(const TankP &P, const MomArgs<R> &M, int j)
{
    const int nx = P.nx, ny = P.ny, lane = threadIdx.x & 31;
    const int ncv = C == 0 ? nx - 1 : nx;  // solved faces of the row
    const int cv = (blockIdx.y * (TX >> 5) + (threadIdx.x >> 5)) * 31 + lane, i = cv + (C == 0 ? 1 : 0);
    const R *rf = C == 0 ? M.ru : M.rv;
    const double *vin = M.bc.vin0;
    const bool in = warp_inside(inside2(P, i, j), cv <= ncv);
    R m0 = R(0.0), f0 = R(0.0);
    if (cv <= ncv) {
        if (in)
            cv_face<true, C, R>(P, rf, M.u, M.v, vin, i, j, 0, 0, m0, f0);
        else
            cv_face<false, C, R>(P, rf, M.u, M.v, vin, i, j, 0, 0, m0, f0);
    }
    const R m1 = shfl_down1<R>(m0), f1 = shfl_down1<R>(f0);
    if (lane == 31 || cv >= ncv) return;
    R my[2], fy[2], S;
    if (in) {
#pragma unroll
        for (int s = 0; s < 2; ++s) cv_face<true, C, R>(P, rf, M.u, M.v, vin, i, j, 1, s, my[s], fy[s]);
        S = visc_sum<true, C, true, R>(P, M.mu_n, M.nd_n, M.u, M.v, vin, i, j);
    } else {
#pragma unroll
        for (int s = 0; s < 2; ++s) cv_face<false, C, R>(P, rf, M.u, M.v, vin, i, j, 1, s, my[s], fy[s]);
        S = visc_sum<false, C, true, R>(P, M.mu_n, M.nd_n, M.u, M.v, vin, i, j);
    }
    const int f = C == 0 ? j * (nx + 1) + i : j * nx + i, c = min(j, ny - 1) * nx + i, cm = C == 0 ? c - 1 : (j - 1) * nx + i;
    const TankC<R> &K = cst<R>(P);
    const R dt = R(M.inp[0]), idt = R(1.0) / dt, ih = K.ih, hi2 = R(0.5) * ih * ih;
    const R r0 = rf[f], w = (C == 0 ? M.u : M.v)[f];
    const R rb = r0 - R(0.5) * (dt * ih) * ((m1 - m0) + (my[1] - my[0]));
    const R Cv = ((f1 - f0) + (fy[1] - fy[0])) * (R(0.5) * ih);
    const R chi = R(0.5) * (M.chi_1[cm] + M.chi_1[c]), rbdt = rb * idt;
    const R al = C == 0 ? M.tb.alpha_u[i] : M.tb.alpha_c[i];
    const R D = rbdt + chi * K.ikp + al * rbdt + vort_damp<R>(P, C == 0 ? M.tb.vort_c[j] : M.tb.vort_v[j], idt);
    R rhs = r0 * w * idt - Cv + hi2 * S;
    if (C == 0) {
        rhs -= R(M.p[c] - M.p[c - 1]) * ih;
    } else {
        const R gp = j < ny ? R(M.p[c] - M.p[cm]) : R(-2.0) * R(M.p[cm]);
        rhs += chi * R(M.S->zdot1) * K.ikp - R(0.5) * (M.rf_1[cm] + M.rf_1[c]) * K.g - gp * ih;
    }
    const R inv = R(1.0) / (D + hi2 * visc_diag<C, R>(P, M.mu_1, M.nd_1, i, j));
    (C == 0 ? M.Du : M.Dv)[f] = D;
    (C == 0 ? M.Ru : M.Rv)[f] = rhs * inv;
    (C == 0 ? M.Qu : M.Qv)[f] = hi2 * inv;
    (C == 0 ? M.ua : M.va)[f] = w;
}

// Block rows 0 .. ny-1: the u-faces; the ny+1 after them: the v-faces.
template <typename R>
__global__ void __launch_bounds__(TX) k_momentum(TankP P, MomArgs<R> M)
{
    pdl_entry();
    const int nx = P.nx, ny = P.ny;
    if ((int)blockIdx.x < ny) {
        const int j = blockIdx.x;
        if (blockIdx.y == 0 && threadIdx.x < 2) M.ua[j * (nx + 1) + threadIdx.x * nx] = threadIdx.x ? R(0.0) : R(M.bc.uin1[j]);
        momentum_row<0, R>(P, M, j);
    } else if ((int)blockIdx.x == ny) {  // v on the bed
        const int cv = (blockIdx.y * (TX >> 5) + (threadIdx.x >> 5)) * 31 + (threadIdx.x & 31);
        if (cv < nx) M.va[cv] = R(0.0);
    } else {
        momentum_row<1, R>(P, M, blockIdx.x - ny);
    }
}

// Working buffers the stencil kernels read, in the compute type R.  An FP64 tank
// points them at its FP64 buffers (sig, u, v are the state itself); a mixed tank
// points them into its FP32 slab, where sig, u, v are mirrors refreshed at the
// start of each step.  Loading FP32 directly keeps the FP32 kernels off the FP64
// pipe, which a per-load FP64 -> FP32 conversion would otherwise saturate.
template <typename R>
struct Work {
    R *sig, *u, *v;                           // state (or its FP32 mirror)
    R *sa, *sgn, *r0, *r1, *rt;               // advected sigma, reinitialisation
    R *rho_n, *mu_n, *mu_1, *rf_1, *chi_1;    // materials
    R *Ru, *Du, *ua, *ub, *uc, *Rv, *Dv, *va, *vb, *vc;  // momentum systems, Jacobi iterates
    R *ru, *rv, *Qu, *Qv, *nd_n, *nd_1;       // face densities, Jacobi factors, node viscosities
};

// sig, u, v -> FP32 mirrors (one thread per cell / face of the largest set).
__global__ void k_mirror(long long nc, long long nu, long long nv, const double *__restrict__ sig,
                         const double *__restrict__ u, const double *__restrict__ v, float *__restrict__ sig32,
                         float *__restrict__ u32, float *__restrict__ v32)
{
    pdl_entry();
    long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (k < nc) sig32[k] = float(sig[k]);
    if (k < nu) u32[k] = float(u[k]);
    if (k < nv) v32[k] = float(v[k]);
}

// One Jacobi sweep of (D - L_mu / 2) u* = R (Crank-Nicolson implicit half), split
// on the diagonal of L_mu: B = R / D' + ((1 / (2 h^2)) / D') S(A), the two factors
// formed with the system (k_momentum); Dirichlet faces are copied.  Block rows as
// k_ppm_faces.
template <typename R, typename TO>
__global__ void __launch_bounds__(TX) k_jacobi(TankP P, const R *__restrict__ mu_1, const R *__restrict__ nd_1,
                                               const double *__restrict__ vin1, const R *__restrict__ Ru,
                                               const R *__restrict__ Qu, const R *__restrict__ Rv,
                                               const R *__restrict__ Qv, const R *__restrict__ ua,
                                               const R *__restrict__ va, TO *__restrict__ ub, TO *__restrict__ vb)
{
    pdl_entry();
    const int nx = P.nx, ny = P.ny, i = blockIdx.y * TX + threadIdx.x;
    if ((int)blockIdx.x < ny) {
        const int j = blockIdx.x, f = j * (nx + 1) + i;
        const bool in = warp_inside(inside2(P, i, j), i > 0 && i < nx);
        if (i > nx) return;
        if (i == 0 || i == nx) {
            ub[f] = ua[f];
            return;
        }
        const R S = in ? visc_sum<true, 0, false, R>(P, mu_1, nd_1, ua, va, vin1, i, j)
                       : visc_sum<false, 0, false, R>(P, mu_1, nd_1, ua, va, vin1, i, j);
        ub[f] = Ru[f] + Qu[f] * S;
    } else {
        const int j = blockIdx.x - ny, f = j * nx + i;
        const bool in = warp_inside(inside2(P, i, j), i < nx);
        if (i >= nx) return;
        if (j == 0) {
            vb[f] = va[f];
            return;
        }
        const R S = in ? visc_sum<true, 1, false, R>(P, mu_1, nd_1, ua, va, vin1, i, j)
                       : visc_sum<false, 1, false, R>(P, mu_1, nd_1, ua, va, vin1, i, j);
        vb[f] = Rv[f] + Qv[f] * S;
    }
}

// b = -h div u*, face coefficients beta = 1 / D (zero on Neumann walls).
template <typename TD>
__global__ void k_proj_rhs(TankP P, const double *__restrict__ us, const double *__restrict__ vs,
                           const TD *__restrict__ Du, const TD *__restrict__ Dv, double *rhs,
                           double *bu, double *bv)
{
    pdl_entry();
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int nx = P.nx, ny = P.ny;
    const int nc = nx * ny, nu = (nx + 1) * ny, nv = nx * (ny + 1);
    if (k < nc) {
        int i = k % nx, j = k / nx;
        rhs[k] = -P.h * (us[j * (nx + 1) + i + 1] - us[j * (nx + 1) + i] + vs[(j + 1) * nx + i] - vs[j * nx + i]);
    } else if (k < nc + nu) {
        int f = k - nc, i = f % (nx + 1);
        bu[f] = (i == 0 || i == nx) ? 0.0 : 1.0 / double(Du[f]);
    } else if (k < nc + nu + nv) {
        int f = k - nc - nu, j = f / nx;
        bv[f] = j == 0 ? 0.0 : 1.0 / double(Dv[f]);
    }
}

// u^{n+1} = u* - beta grad phi; p^{n+1/2} = p^{n-1/2} + phi.
__global__ void k_project(TankP P, const double *__restrict__ us, const double *__restrict__ vs,
                          const double *__restrict__ bu, const double *__restrict__ bv,
                          const double *__restrict__ phi, double *u, double *v, double *p)
{
    pdl_entry();
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int nx = P.nx, ny = P.ny;
    const int nc = nx * ny, nu = (nx + 1) * ny, nv = nx * (ny + 1);
    if (k < nu) {
        int i = k % (nx + 1), j = k / (nx + 1);
        double uu = us[k];
        if (i > 0 && i < nx) uu -= bu[k] * (phi[j * nx + i] - phi[j * nx + i - 1]) * P.ih;
        u[k] = uu;
    } else if (k < nu + nv) {
        int f = k - nu, i = f % nx, j = f / nx;
        double vv = vs[f];
        if (j > 0 && j < ny) vv -= bv[f] * (phi[j * nx + i] - phi[(j - 1) * nx + i]) * P.ih;
        if (j == ny) vv += 2.0 * bv[f] * phi[(ny - 1) * nx + i] * P.ih;
        v[f] = vv;
    } else if (k < nu + nv + nc) {
        int c = k - nu - nv;
        p[c] += phi[c];
    }
}

__global__ void k_div_partial(TankP P, const double *__restrict__ u, const double *__restrict__ v,
                              double *__restrict__ part)
{
    pdl_entry();
    __shared__ double sh[TB];
    const int nx = P.nx;
    double acc = 0.0;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nx * P.ny; c += gridDim.x * blockDim.x) {
        int i = c % nx, j = c / nx;
        acc += sq(P.h * (u[j * (nx + 1) + i + 1] - u[j * (nx + 1) + i] + v[(j + 1) * nx + i] - v[j * nx + i]));
    }
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// Close the step: divergence norm, probe elevation, advance time and body state,
// and account the kernels a graph replay executed (fixed part + per-iteration
// and per-cycle parts of the solve).
__global__ void k_finalize(TankP P, StepScalars *S, const double *__restrict__ part,
                           const double *__restrict__ sig, const double *__restrict__ inp, const KState *ks,
                           int n_fixed, int n_body, int n_close)
{
    pdl_entry();
    __shared__ double sh[TB];
    double s = 0.0;
    for (int b = threadIdx.x; b < kRedBlocks; b += blockDim.x) s += part[b];
    double d2 = block_sum(s, sh);
    // probe: the lowest row j of the probe column with sigma_j < 0 <= sigma_{j+1}
    __shared__ int jmin;
    if (threadIdx.x == 0) jmin = P.ny;
    __syncthreads();
    const int ip = clampi((int)floor(P.probe_x / P.h), 0, P.nx - 1);
    for (int j = threadIdx.x; j + 1 < P.ny; j += blockDim.x) {
        double a = sig[j * P.nx + ip], b = sig[(j + 1) * P.nx + ip];
        if (a < 0.0 && b >= 0.0) atomicMin(&jmin, j);
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    double eta = nan("");
    if (jmin < P.ny) {
        const int j = jmin;
        double a = sig[j * P.nx + ip], b = sig[(j + 1) * P.nx + ip];
        eta = (j + 0.5) * P.h + P.h * a / (a - b) - P.depth;
    }
    S->div2 = d2;
    S->eta = eta;
    S->t = S->t + inp[0];
    S->yc = S->yc1;
    S->zdot_prev = S->zdot;
    S->zdot = S->zdot1;
    S->launches = (long long)n_fixed + (long long)ks->its * n_body + (long long)ks->ncycles * n_close;
}

// Initial state: sigma = y - (d + eta(x, 0)); Airy velocities (u = 0 on the
// right wall, v = 0 on the bed).
__global__ void k_init_fields(TankP P, double *sig, double *u, double *v)
{
    pdl_entry();
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int nx = P.nx, ny = P.ny;
    const int nc = nx * ny, nu = (nx + 1) * ny, nv = nx * (ny + 1);
    const double h = P.h;
    double uu, vv;
    if (k < nc) {
        int i = k % nx, j = k / nx;
        sig[k] = (j + 0.5) * h - P.depth - eta_at(P, (i + 0.5) * h, 0.0);
    } else if (k < nc + nu) {
        int f = k - nc, i = f % (nx + 1), j = f / (nx + 1);
        airy_uv(P, i * h, (j + 0.5) * h, 0.0, &uu, &vv);
        u[f] = i == nx ? 0.0 : uu;
    } else if (k < nc + nu + nv) {
        int f = k - nc - nu, i = f % nx, j = f / nx;
        airy_uv(P, (i + 0.5) * h, j * h, 0.0, &uu, &vv);
        v[f] = j == 0 ? 0.0 : vv;
    }
}

// p^{-1/2}: discrete hydrostatic pressure of the flow density (p = 0 at the top
// face): p_{ny-1} = rho_f g h / 2, p_{j-1} = p_j + (face mean rho_f) g h.
__global__ void k_init_pressure(TankP P, const double *__restrict__ rf, double *p)
{
    pdl_entry();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int nx = P.nx, ny = P.ny;
    if (i >= nx) return;
    double pj = 0.5 * rf[(ny - 1) * nx + i] * P.g * P.h;
    p[(ny - 1) * nx + i] = pj;
    for (int j = ny - 1; j >= 1; --j) {
        pj += 0.5 * (rf[(j - 1) * nx + i] + rf[j * nx + i]) * P.g * P.h;
        p[(j - 1) * nx + i] = pj;
    }
}

inline size_t pad64(size_t n) { return (n + 63) & ~size_t(63); }

// A tank's face and node arrays in its working type (ru, rv, Qu, Qv, nd_n, nd_1),
// and the FP32 slab of a mixed tank: those, 11 cell arrays, 6 u-face and 6 v-face
// arrays, each starting on a 256-byte boundary.
size_t face_elems(size_t nu, size_t nv, size_t nn) { return 2 * (pad64(nu) + pad64(nv) + pad64(nn)); }
size_t work_floats(size_t nc, size_t nu, size_t nv, size_t nn)
{
    return 11 * pad64(nc) + 6 * pad64(nu) + 6 * pad64(nv) + face_elems(nu, nv, nn);
}
size_t nodes(const wec_tank *T) { return (size_t)(T->P.nx + 1) * (T->P.ny + 1); }

template <typename R>
void take_faces(const wec_tank *T, Work<R> &W, R *q)
{
    const size_t n[6] = {T->nu, T->nv, T->nu, T->nv, nodes(T), nodes(T)};
    R **dst[6] = {&W.ru, &W.rv, &W.Qu, &W.Qv, &W.nd_n, &W.nd_1};
    for (int k = 0; k < 6; ++k) {
        *dst[k] = q;
        q += pad64(n[k]);
    }
}

Work<double> work64(wec_tank *T)
{
    Work<double> W{T->sig, T->u, T->v, T->sa, T->sgn, T->r0, T->r1, T->rt, T->rho_n, T->mu_n, T->mu_1,
                   T->rf_1, T->chi_1, T->Ru, T->Du, T->ua, T->ub, T->uc, T->Rv, T->Dv, T->va, T->vb,
                   T->vc, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    take_faces(T, W, T->w64);
    return W;
}

Work<float> work32(wec_tank *T)
{
    float *q = T->w32;
    auto take = [&q](size_t n) { float *r = q; q += pad64(n); return r; };
    Work<float> W;
    float **cells[] = {&W.sig, &W.sa, &W.sgn, &W.r0, &W.r1, &W.rt, &W.rho_n, &W.mu_n, &W.mu_1, &W.rf_1, &W.chi_1};
    for (float **c : cells) *c = take(T->nc);
    float **uf[] = {&W.u, &W.Ru, &W.Du, &W.ua, &W.ub, &W.uc};
    for (float **c : uf) *c = take(T->nu);
    float **vf[] = {&W.v, &W.Rv, &W.Dv, &W.va, &W.vb, &W.vc};
    for (float **c : vf) *c = take(T->nv);
    take_faces(T, W, q);
    return W;
}

}  // namespace

int tank_alloc_and_init(wec_tank *T)
{
    const TankP &P = T->P;
    T->nc = (size_t)P.nx * P.ny;
    T->nu = (size_t)(P.nx + 1) * P.ny;
    T->nv = (size_t)P.nx * (P.ny + 1);
    size_t nc = T->nc, nu = T->nu, nv = T->nv;
    WEC_CK(cudaStreamCreateWithFlags(&T->gst, cudaStreamNonBlocking));
    WEC_CK(cudaStreamCreateWithFlags(&T->h1, cudaStreamNonBlocking));
    WEC_CK(cudaStreamCreateWithFlags(&T->h2, cudaStreamNonBlocking));
    WEC_CK(cudaEventCreateWithFlags(&T->ev_in, cudaEventDisableTiming));
    WEC_CK(cudaEventCreateWithFlags(&T->ev_out, cudaEventDisableTiming));
    WEC_CK(cudaStreamCreateWithFlags(&T->nst, cudaStreamNonBlocking));
    WEC_CK(cudaEventCreateWithFlags(&T->ev_nf, cudaEventDisableTiming));
    WEC_CK(cudaEventCreateWithFlags(&T->ev_nj, cudaEventDisableTiming));
    double **cells[] = {&T->sig, &T->sa, &T->r0, &T->r1, &T->rt, &T->p, &T->phi, &T->rhs,
                        &T->rho_n, &T->mu_n, &T->mu_1, &T->rf_1, &T->chi_1};
    for (double **q : cells) {
        WEC_CK(cudaMalloc(q, nc * 8));
        WEC_CK(cudaMemset(*q, 0, nc * 8));
    }
    double **ufaces[] = {&T->u, &T->us, &T->ua, &T->ub, &T->uc, &T->Ru, &T->Du};
    for (double **q : ufaces) {
        WEC_CK(cudaMalloc(q, nu * 8));
        WEC_CK(cudaMemset(*q, 0, nu * 8));
    }
    double **vfaces[] = {&T->v, &T->vs, &T->va, &T->vb, &T->vc, &T->Rv, &T->Dv};
    if (T->opts.precision == WEC_PREC_MIXED) {
        const size_t e = work_floats(nc, nu, nv, nodes(T));
        WEC_CK(cudaMalloc(&T->w32, e * 4));
        WEC_CK(cudaMemset(T->w32, 0, e * 4));
    } else {
        const size_t e = face_elems(nu, nv, nodes(T));
        WEC_CK(cudaMalloc(&T->w64, e * 8));
        WEC_CK(cudaMemset(T->w64, 0, e * 8));
    }
    for (double **q : vfaces) {
        WEC_CK(cudaMalloc(q, nv * 8));
        WEC_CK(cudaMemset(*q, 0, nv * 8));
    }
    size_t nbc = (size_t)P.ny + 2 * (P.ny + 1) + 8 + 3 * (size_t)P.ncomp;
    WEC_CK(cudaMalloc(&T->bcbuf, nbc * 8));
    T->bc.uin1 = T->bcbuf;
    T->bc.vin0 = T->bc.uin1 + P.ny;
    T->bc.vin1 = T->bc.vin0 + P.ny + 1;
    T->bc.eta0 = T->bc.vin1 + P.ny + 1;
    T->bc.eta1 = T->bc.eta0 + 3;
    T->bc.eta_in = T->bc.eta1 + 3;
    T->bc.comp = T->bc.eta_in + 2;
    WEC_CK(cudaMalloc(&T->part, kRedBlocks * 8));
    WEC_CK(cudaMalloc(&T->tabs, (size_t)(2 * P.nx + 1 + 2 * P.ny + 1) * 8));
    if (T->opts.precision == WEC_PREC_MIXED) WEC_CK(cudaMalloc(&T->tabs32, (size_t)(2 * P.nx + 1 + 2 * P.ny + 1) * 4));
    WEC_CK(cudaMalloc(&T->sgn, nc * 8));
    {
        WEC_PROF("init", -1, 8.0 * (2 * P.nx + 2 * P.ny + 2), T->gst);
        launch_k(k_tables, nblk(std::max(P.nx, P.ny) + 1, 128), 128, 0, T->gst, P, T->tabs, T->tabs32);
    }
    WEC_CK(cudaMalloc(&T->inp, 2 * 8));
    WEC_CK(cudaMemset(T->inp, 0, 2 * 8));
    WEC_CK(cudaMalloc(&T->S, sizeof(StepScalars)));
    WEC_CK(cudaMallocHost(&T->Sh, sizeof(StepScalars)));
    *T->Sh = StepScalars{};
    // the solver runs FP32 V-cycles for both mixed modes
    const int sprec = T->opts.precision == WEC_PREC_FP64 ? WEC_PREC_FP64 : WEC_PREC_MIXED;
    if (int e = poisson_init(&T->solver, P.nx, P.ny, sprec, T->opts.restart, T->opts.mg_pre,
                             T->opts.mg_post, T->gst))
        return e;
    long long ninit = (long long)nc + nu + nv;
    WEC_PROF("init", -1, 8.0 * ninit, T->gst);
    launch_k(k_init_fields, nblk(ninit, TB), TB, 0, T->gst, P, T->sig, T->u, T->v);
    WEC_CK(cudaGetLastError());
    return WEC_OK;
}

// Called after the host filled Sh (initial body state): hydrostatic p from the initial sigma.
int tank_init_pressure(wec_tank *T)
{
    WEC_CK(cudaMemcpyAsync(T->S, T->Sh, sizeof(StepScalars), cudaMemcpyHostToDevice, T->gst));
    const TankP &P = T->P;
    {
        WEC_PROF("materials", -1, 16.0 * T->nc, T->gst);
        launch_k(k_materials<double>, nblk(T->nc, TB), TB, 0, T->gst, P, T->S, 0, T->sig, (double *)nullptr,
                 (double *)nullptr, T->rf_1, (double *)nullptr);
    }
    {
        WEC_PROF("init", -1, 16.0 * T->nc, T->gst);
        launch_k(k_init_pressure, nblk(P.nx, 128), 128, 0, T->gst, P, T->rf_1, T->p);
    }
    WEC_CK(cudaGetLastError());
    WEC_CK(cudaStreamSynchronize(T->gst));
    return WEC_OK;
}

namespace {

template <typename R>
Tabs<R> tabs(const wec_tank *T)
{
    const int nx = T->P.nx, ny = T->P.ny;
    const R *t;
    if constexpr (sizeof(R) == 4)
        t = T->tabs32;
    else
        t = T->tabs;
    return Tabs<R>{t, t + nx, t + 2 * nx + 1, t + 2 * nx + 1 + ny};
}

// Everything before the pressure solve: steps (1)-(7) of the step, stencils in
// the compute type R over the working set W.
template <typename R>
void enqueue_front_t(wec_tank *T, const Work<R> &W, cudaStream_t st)
{
    const TankP &P = T->P;
    const long long nc = T->nc, nu = T->nu, nv = T->nv;
    const double fb = 8.0, rb = sizeof(R);  // bytes of FP64 storage / of the working type
    constexpr bool f32 = sizeof(R) == 4;
    if constexpr (f32) {
        WEC_PROF("mirror", -1, (fb + rb) * (nc + nu + nv), st);
        launch_k(k_mirror, nblk(std::max(nc, std::max(nu, nv)), TB), TB, 0, st, nc, nu, nv, T->sig, T->u, T->v, W.sig,
                                                                            W.u, W.v);
    }
    // (1) inflow / ghost data at t^n and t^{n+1}
    {
        WEC_PROF("bc", -1, fb * 8.0, st);
        launch_k(k_bc_eta, 8, kEtaT, 0, st, P, T->S, T->inp, T->bc);
    }
    {
        WEC_PROF("bc", -1, fb * (3.0 * P.ny + 2), st);
        launch_k(k_bc_rows<R>, P.ny + 1, 96, 0, st, P, T->S, T->inp, T->bc);
    }
    // (2) materials at n, force from p^{n-1/2}, u^n (Eq. int_fh), heave (Eq. newton_u)
    {
        WEC_PROF("materials", -1, (fb + 2.0 * rb) * nc, st);
        launch_k(k_materials<R>, nblk(nc, TB), TB, 0, st, P, T->S, 0, T->sig, W.rho_n, W.mu_n, nullptr, nullptr);
    }
    {
        WEC_PROF("force", -1, fb * kRedBlocks, st);
        launch_k(k_force_partial<R>, kRedBlocks, TB, 0, st, P, T->S, T->p, T->u, T->v, W.mu_n, T->bc.vin0, T->part);
    }
    {
        WEC_PROF("scalar", -1, fb * kRedBlocks, st);
        launch_k(k_heave, 1, TB, 0, st, P, T->S, T->part, T->inp);
    }
    // (3) sigma advection + damping-zone relaxation, then reinitialisation; the
    // last pseudo-step writes sigma^{n+1} over sigma^n (no longer needed).
    {
        // (the Jacobi buffers are free until the momentum system)
        WEC_PROF("advect_faces", -1, rb * (nc + 2.0 * (nu + nv)), st);
        launch_k(k_ppm_faces<R>, row_grid(P.nx + 1, 2 * P.ny + 1), TX, 0, st, P, W.sig, W.u, W.v, T->bc.eta0, T->inp, W.ub,
                 W.vb);
    }
    {
        WEC_PROF("advect", -1, rb * (nc + 2.0 * (nu + nv)) + (fb + (f32 ? rb : 0.0)) * nc, st);
        launch_k(k_advect<R>, row_grid(P.nx, P.ny), TX, 0, st, P, W.sig, W.u, W.v, W.ub, W.vb, T->inp, tabs<R>(T).alpha_c,
                 T->sa, f32 ? W.sa : nullptr);
    }
    const R dtau = R(0.3 * P.h);
    const dim3 rg = row_grid(P.nx, P.ny);
    const R *f = W.sa;
    R *bufs[2] = {W.r0, W.r1};
    const int nr = T->opts.n_reinit;
    for (int it = 0; it < nr; ++it) {
        {
            WEC_PROF("reinit", -1, rb * 3.0 * nc, st);
            launch_k(k_reinit<R, R>, rg, TX, 0, st, P, f, W.sgn, nullptr, T->bc.eta1, dtau, W.rt, it == 0 ? 1 : 0);
        }
        WEC_PROF("reinit", -1, rb * 3.0 * nc + (it == nr - 1 ? fb : rb) * nc, st);
        if (it == nr - 1) {
            launch_k(k_reinit<R, double>, rg, TX, 0, st, P, W.rt, W.sgn, f, T->bc.eta1, dtau, T->sig, 0);
        } else {
            R *dst = bufs[it & 1];
            launch_k(k_reinit<R, R>, rg, TX, 0, st, P, W.rt, W.sgn, f, T->bc.eta1, dtau, dst, 0);
            f = dst;
        }
    }
    if (nr == 0) cudaMemcpyAsync(T->sig, T->sa, nc * 8, cudaMemcpyDeviceToDevice, st);
    // (4) materials at n+1 (psi at the new body position)
    {
        WEC_PROF("materials", -1, (fb + 3.0 * rb) * nc, st);
        launch_k(k_materials<R>, nblk(nc, TB), TB, 0, st, P, T->S, 1, T->sig, nullptr, W.mu_1, W.rf_1, W.chi_1);
    }
    // (5) momentum right-hand side and diagonal, (6) Crank-Nicolson Jacobi sweeps
    {
        WEC_PROF("faces", -1, rb * (3.0 * nc + 2.0 * (nu + nv)), st);
        launch_k(k_faces<R>, row_grid(P.nx + 1, P.ny + 1), TX, 0, st, P, W.rho_n, W.mu_n, W.mu_1, W.ru, W.rv, W.nd_n,
                 W.nd_1);
    }
    {
        WEC_PROF("momentum", -1, rb * (6.0 * nc + 6.0 * (nu + nv)) + fb * nc, st);
        const MomArgs<R> M{T->inp, T->S, tabs<R>(T), W.ru, W.rv, W.mu_n, W.mu_1, W.nd_n, W.nd_1, W.chi_1, W.rf_1, W.u, W.v,
                           T->p, T->bc, W.Du, W.Dv, W.Ru, W.Rv, W.Qu, W.Qv, W.ua, W.va};
        // (31 control volumes per warp, one face more per row)
        launch_k(k_momentum<R>, dim3(2 * P.ny + 1, (P.nx + 1 + 31 * (TX / 32) - 1) / (31 * (TX / 32))), TX, 0, st, P, M);
    }
    const R *ju = W.ua, *jv = W.va;
    R *tu[2] = {W.ub, W.uc}, *tv[2] = {W.vb, W.vc};
    const int nj = T->opts.n_jacobi;
    const dim3 jg = row_grid(P.nx + 1, 2 * P.ny + 1);
    for (int it = 0; it < nj; ++it) {
        const bool last = it == nj - 1;
        WEC_PROF("jacobi", -1, rb * (nc + 4.0 * (nu + nv)) + fb * (nu + nv) + (last ? fb - rb : 0.0) * (nu + nv),
                 st);
        if (last) {
            launch_k(k_jacobi<R, double>, jg, TX, 0, st, P, W.mu_1, W.nd_1, T->bc.vin1, W.Ru, W.Qu, W.Rv, W.Qv, ju, jv,
                     T->us, T->vs);
        } else {
            launch_k(k_jacobi<R, R>, jg, TX, 0, st, P, W.mu_1, W.nd_1, T->bc.vin1, W.Ru, W.Qu, W.Rv, W.Qv, ju, jv,
                     tu[it & 1], tv[it & 1]);
            ju = tu[it & 1];
            jv = tv[it & 1];
        }
    }
    // (7) pressure increment: A phi = -h div u*, beta = 1/D; phi from zero
    wec_poisson *S = &T->solver;
    {
        WEC_PROF("proj_rhs", -1, fb * (nc + 3.0 * (nu + nv)), st);
        launch_k(k_proj_rhs<R>, nblk(nc + nu + nv, TB), TB, 0, st, P, T->us, T->vs, W.Du, W.Dv, T->rhs, S->L64[0].bu,
                                                          S->L64[0].bv);
    }
    if (T->net) {
        // the guess reads the right-hand side and the level-0 coefficients only:
        // it runs on the net's stream while this one builds the hierarchy
        // (launch errors surface at the capture / the step's error check)
        cudaEventRecord(T->ev_nf, st);
        cudaStreamWaitEvent(T->nst, T->ev_nf, 0);
        net_enqueue_guess(T, T->nst);
        cudaEventRecord(T->ev_nj, T->nst);
        poisson_build(S, st);
        cudaStreamWaitEvent(st, T->ev_nj, 0);
    } else {
        poisson_build(S, st);
        cudaMemsetAsync(T->phi, 0, nc * 8, st);
    }
}

void enqueue_front(wec_tank *T, cudaStream_t st)
{
    if (T->opts.precision == WEC_PREC_MIXED)
        enqueue_front_t<float>(T, work32(T), st);
    else
        enqueue_front_t<double>(T, work64(T), st);
}

// (8) projection and the close of the step.
void enqueue_back(wec_tank *T, cudaStream_t st)
{
    const TankP &P = T->P;
    const long long nc = T->nc, nu = T->nu, nv = T->nv;
    const double fb = 8.0;
    wec_poisson *S = &T->solver;
    {
        WEC_PROF("project", -1, fb * (3.0 * nc + 3.0 * (nu + nv)), st);
        launch_k(k_project, nblk(nu + nv + nc, TB), TB, 0, st, P, T->us, T->vs, S->L64[0].bu, S->L64[0].bv, T->phi,
                                                         T->u, T->v, T->p);
    }
    {
        WEC_PROF("divergence", -1, fb * (nu + nv), st);
        launch_k(k_div_partial, kRedBlocks, TB, 0, st, P, T->u, T->v, T->part);
    }
    WEC_PROF("scalar", -1, fb * (kRedBlocks + P.ny), st);
    launch_k(k_finalize, 1, TB, 0, st, P, T->S, T->part, T->sig, T->inp, S->ks, T->n_fixed, T->n_body, T->n_close);
}

// Kernels per replay (front + the solve's opening + back once, then the
// Arnoldi-step kernels per iteration and the cycle-closing kernels per cycle),
// counted on a throwaway capture; k_finalize uses them to report launches.
int count_kernels(wec_tank *T)
{
    wec_poisson *S = &T->solver;
    cudaGraph_t tmp = nullptr;
    WEC_CK(cudaStreamBeginCapture(T->h1, cudaStreamCaptureModeThreadLocal));
    prof::begin_capture();
    enqueue_front(T, T->h1);
    enqueue_back(T, T->h1);
    long long nfb = prof::captured();
    prof::end_capture();
    WEC_CK(cudaStreamEndCapture(T->h1, &tmp));
    if (tmp) cudaGraphDestroy(tmp);
    int nbeg = 0, nb = 0, ncl = 0;
    if (int e = poisson_count_kernels(S, T->h1, &nbeg, &nb, &ncl)) return e;
    T->n_fixed = (int)nfb + nbeg;
    T->n_body = nb;
    T->n_close = ncl;
    return WEC_OK;
}

int build_graph(wec_tank *T)
{
    if (int e = count_kernels(T)) return e;
    WEC_CK(cudaStreamBeginCapture(T->gst, cudaStreamCaptureModeThreadLocal));
    int e = tank_capture_step(T, T->gst);
    cudaGraph_t g = nullptr;
    cudaError_t ce = cudaStreamEndCapture(T->gst, &g);
    if (e) {
        if (g) cudaGraphDestroy(g);
        return e;
    }
    if (ce != cudaSuccess) return cuda_fail(ce, "cudaStreamEndCapture (step graph)");
    T->graph = g;
    WEC_CK(cudaGraphInstantiate(&T->exec, g, 0));
    return WEC_OK;
}

int finish_step(wec_tank *T, int status, wec_step_result *out)
{
    const StepScalars &s = *T->Sh;
    int iters = 0;
    double relres = 0.0;
    int st = solve_result(&T->solver, &iters, &relres);
    if (status == WEC_OK) status = st;
    T->stepped = true;
    T->last_iters = iters;
    T->last_relres = relres;
    if (status == WEC_OK && !(std::isfinite(s.zdot) && std::isfinite(s.F) && std::isfinite(relres)))
        status = fail(WEC_ERR_NONFINITE, "step: non-finite body state or residual");
    if (out) {
        out->t = s.t;
        out->z = s.yc - s.yc0;
        out->zdot = s.zdot;
        out->f_hydro = s.F;
        out->f_pto = s.fpto;
        out->eta_probe = s.eta;
        out->residual = relres;
        out->div_norm = sqrt(s.div2);
        out->iters = iters;
        out->status = status;
    }
    return status;
}

}  // namespace

int tank_prepare_capture(wec_tank *T) { return count_kernels(T); }

int tank_capture_step(wec_tank *T, cudaStream_t st)
{
    wec_poisson *S = &T->solver;
    S->st = st;
    prof::begin_capture();
    enqueue_front(T, st);
    int e = poisson_capture_solve(S, T->rhs, T->phi, T->opts.rtol, T->opts.max_iters, st, T->h1, T->h2);
    enqueue_back(T, st);
    cudaMemcpyAsync(T->Sh, T->S, sizeof(StepScalars), cudaMemcpyDeviceToHost, st);
    poisson_state_to_host(S, st);
    prof::end_capture();
    return e;
}

int tank_finish_step(wec_tank *T, wec_step_result *out)
{
    prof::add_launches(T->Sh->launches);
    return finish_step(T, WEC_OK, out);
}

int tank_step(wec_tank *T, double dt, double fpto, wec_step_result *out)
{
    cudaStream_t st = T->gst;
    // order after the caller's stream, and the caller's stream after this step
    WEC_CK(cudaEventRecord(T->ev_in, T->st));
    WEC_CK(cudaStreamWaitEvent(st, T->ev_in, 0));
    double in[2] = {dt, fpto};
    WEC_CK(cudaMemcpyAsync(T->inp, in, sizeof(in), cudaMemcpyHostToDevice, st));  // pageable: staged before return
    const bool graph = T->use_graph && !prof::enabled();
    int status = WEC_OK;
    if (T->net)
        if (int e = net_sync_weights(T->net)) return e;
    if (graph) {
        if (!T->exec)
            if (int e = build_graph(T)) return e;
        WEC_CK(cudaGraphLaunch(T->exec, st));
        WEC_CK(cudaStreamSynchronize(st));
        prof::add_launches(T->Sh->launches);
    } else {
        wec_poisson *S = &T->solver;
        S->st = st;
        enqueue_front(T, st);
        WEC_CK(cudaGetLastError());
        int iters = 0;
        double relres = 0.0;
        status = poisson_solve(S, T->rhs, T->phi, T->opts.rtol, T->opts.max_iters, &iters, &relres);
        if (status != WEC_OK && status != WEC_ERR_NOT_CONVERGED) return status;
        enqueue_back(T, st);
        WEC_CK(cudaGetLastError());
        WEC_CK(cudaMemcpyAsync(T->Sh, T->S, sizeof(StepScalars), cudaMemcpyDeviceToHost, st));
        WEC_CK(cudaStreamSynchronize(st));
        status = WEC_OK;
    }
    WEC_CK(cudaEventRecord(T->ev_out, st));
    WEC_CK(cudaStreamWaitEvent(T->st, T->ev_out, 0));
    return finish_step(T, status, out);
}

void tank_free(wec_tank *T)
{
    if (T->exec) cudaGraphExecDestroy(T->exec);
    if (T->graph) cudaGraphDestroy(T->graph);
    double *all[] = {T->sig, T->sa, T->r0, T->r1, T->rt, T->p, T->phi, T->rhs, T->rho_n, T->mu_n, T->mu_1,
                     T->rf_1, T->chi_1, T->u, T->us, T->ua, T->ub, T->uc, T->Ru, T->Du, T->v, T->vs,
                     T->va, T->vb, T->vc, T->Rv, T->Dv, T->bcbuf, T->part, T->waves,
                     T->tabs, T->sgn};
    for (double *q : all) cudaFree(q);
    if (T->inp_owned) cudaFree(T->inp);
    cudaFree(T->w32);
    cudaFree(T->w64);
    cudaFree(T->tabs32);
    cudaFree(T->net_stats);
    cudaFree(T->S);
    if (T->Sh) cudaFreeHost(T->Sh);
    poisson_free(&T->solver);
    if (T->ev_in) cudaEventDestroy(T->ev_in);
    if (T->ev_out) cudaEventDestroy(T->ev_out);
    if (T->ev_nf) cudaEventDestroy(T->ev_nf);
    if (T->ev_nj) cudaEventDestroy(T->ev_nj);
    if (T->nst) cudaStreamDestroy(T->nst);
    if (T->h1) cudaStreamDestroy(T->h1);
    if (T->h2) cudaStreamDestroy(T->h2);
    if (T->gst) cudaStreamDestroy(T->gst);
}

}  // namespace wec
