// Pointwise steps of the right-hand side (Eqs. 5-11, 26; Secs. 2.2, 3.3) as device bodies over an
// index range. Each body processes indices lo + threadIdx.x, lo + threadIdx.x + stride, ... < hi
// of one grid: the single-grid kernels (rhs.cu) call it with a grid-stride range, the batched
// persistent kernels (batch.cu) with one tile of one grid at a time. Both run the same
// arithmetic, so a grid's results do not depend on what it is batched with.
#pragma once

#include "grid.h"
#include "thermo.cuh"

namespace hyp {

__device__ __forceinline__ void atomic_status(unsigned* st, unsigned bits) {
    if (bits) atomicOr(st, bits);
}

// Reciprocals of the freestream scales, computed once per thread by the caller of closure_point
// (the point loop multiplies by them).
struct ScaleInv {
    double iT_ref, imu_inf, ik_inf, ia_inf, iRe, iRePr, ip_ref, ia2, d_nd, wscale;
};

__device__ __forceinline__ ScaleInv scale_inv(const Scales& sc) {
    ScaleInv c;
    c.iT_ref = 1.0 / sc.T_ref;
    c.imu_inf = 1.0 / sc.mu_inf;
    c.ik_inf = 1.0 / sc.k_inf;
    c.ia_inf = 1.0 / sc.a_inf;
    c.iRe = 1.0 / sc.Re;
    c.iRePr = 1.0 / (sc.Re * sc.Pr);
    c.ip_ref = __ddiv_rn(__dmul_rn(c.ia_inf, c.ia_inf), sc.rho_inf);
    c.ia2 = __dmul_rn(c.ia_inf, c.ia_inf);
    c.d_nd = __dmul_rn(__dmul_rn(sc.rho_inf, c.imu_inf), c.iRe);   // D (SI) -> rho_inf D / (mu_inf Re)
    c.wscale = __ddiv_rn(__dmul_rn(sc.L_ref, c.ia_inf), sc.rho_inf);   // w (SI) -> nondimensional
    return c;
}

// (A) primitives and the closure at one cell centre (MIXED: binary32 transport, Sec. 2.2).
// LTE: the gas is in local thermodynamic equilibrium (its own instantiation, so that the other
// kinds' code keeps its registers); the species fields are passive and the closure ignores them.
// The point is a function of its own, not inlined: the single-grid kernel and the batched
// executor call this one compiled body, so a member's results do not depend on which of the
// two ran it (inlined into two different kernels, the compiler's fusion of multiplies and adds
// may differ between the copies by a rounding).
template <bool MIXED, bool LTE>
__device__ __noinline__ void closure_point(const GasDev& g, const Scales& sc, const ScaleInv& c,
                                           const GridView& v, const double* __restrict__ U,
                                           const Scratch& s, int idx) {
    const bool cpg = sc.kind == HYP_GAS_CPG;
    const bool tpg = sc.kind == HYP_GAS_TPG;
    const bool cneq = sc.kind == HYP_GAS_CNEQ;
    const double iT_ref = c.iT_ref, imu_inf = c.imu_inf, ik_inf = c.ik_inf, ia_inf = c.ia_inf;
    const double iRe = c.iRe, iRePr = c.iRePr, ip_ref = c.ip_ref, ia2 = c.ia2, d_nd = c.d_nd;
    const double wscale = c.wscale;
    {
        const double rho = U[v.off[0] + idx];
        const double irho = cl_rcp(rho);
        double Y[NSP];
        double rest = rho;
#pragma unroll
        for (int sp = 1; sp < NSP; ++sp) {
            const double r = U[v.off[sp] + idx];
            Y[sp] = r * irho;
            rest -= r;
        }
        Y[0] = rest * irho;
        const double rhoE = U[v.off[NSP] + idx];
        const double u = s.ru_c[idx] * irho;
        const double vv = s.rv_c[idx] * irho;
        const double e = rhoE * irho - 0.5 * (u * u + vv * vv);
        double T, p, mu, k, a;
        double h[NSP], wd[NSP], X[NSP], W[NSP], Wd[NSP];
        if constexpr (LTE) {
            ClosureOut o;
            double Yeq[NSP], kr;
            // the previous evaluation at this point seeds this one: the element potentials start
            // the first equilibrium solve, and the temperature starts a step (e - e_c) / c_v,eq
            // off the cached one (kept in the first species-energy cache arrays, which the
            // equilibrium closure does not otherwise use)
            const double e_si = e * sc.a_inf * sc.a_inf;
            double lam[2] = {NAN, NAN}, cv_eq = 0.0;
            double T0 = s.Tcache[idx];
            if (v.predict) {
                lam[0] = s.esc[0][idx];
                lam[1] = s.esc[1][idx];
                const double ec = s.esc[2][idx], cvc = s.esc[3][idx];
                if (cvc > 0.0 && isfinite(ec)) T0 += (e_si - ec) / cvc;
            }
            lte_closure<MIXED>(g, rho * sc.rho_inf, e_si, T0, Yeq, kr, o, lam, &cv_eq);
            atomic_status(v.status, o.status);
            s.Tcache[idx] = o.T;
            s.esc[0][idx] = lam[0];
            s.esc[1][idx] = lam[1];
            s.esc[2][idx] = e_si;
            s.esc[3][idx] = cv_eq;
            T = __dmul_rn(o.T, iT_ref);
            p = __dmul_rn(o.p, ip_ref);
            mu = __dmul_rn(o.mu, imu_inf);
            k = __dmul_rn(o.k, ik_inf);
            a = __dmul_rn(o.a, ia_inf);
#pragma unroll
            for (int sp = 0; sp < NSP; ++sp) {
                h[sp] = wd[sp] = W[sp] = Wd[sp] = 0.0;
                X[sp] = o.X[sp];
            }
        } else if (cpg) {
            T = sc.gamma_inf * e;
            p = rho * (sc.gamma_inf - 1.0) / sc.gamma_inf * T;
            const double Td = T * sc.T_ref;
            mu = SUTH_C1 * Td * sqrt(Td) / (Td + SUTH_TS) / sc.mu_inf;
            k = mu;
            a = sqrt(sc.gamma_inf * p / rho);
#pragma unroll
            for (int sp = 0; sp < NSP; ++sp) h[sp] = wd[sp] = X[sp] = W[sp] = Wd[sp] = 0.0;
        } else if (tpg) {
            // thermally perfect gas (Eqs. 22-25): Newton on e(T) from the cached temperature
            const TpgModel m{sc.tpg_cp0, (sc.gamma_inf - 1.0) / sc.gamma_inf, sc.tpg_theta, sc.R_inf};
            unsigned st = rho > 0.0 ? 0u : HYP_STATUS_NONPHYSICAL;
            const double T0 = v.predict ? s.Tcache[idx] : sc.gamma_inf * e * sc.T_ref;
            const double Tk = m.temperature(e * sc.a_inf * sc.a_inf, T0, st);
            atomic_status(v.status, st);
            s.Tcache[idx] = Tk;
            T = Tk / sc.T_ref;
            p = rho * (sc.gamma_inf - 1.0) / sc.gamma_inf * T;
            mu = SUTH_C1 * Tk * sqrt(Tk) / (Tk + SUTH_TS) / sc.mu_inf;
            k = keyes(Tk) / sc.k_inf;
            const double cp = m.cp(Tk);
            a = sqrt(cp / (cp - sc.R_inf) * p / rho);
#pragma unroll
            for (int sp = 0; sp < NSP; ++sp) h[sp] = wd[sp] = X[sp] = W[sp] = Wd[sp] = 0.0;
        } else {
            const double e_si = e * sc.a_inf * sc.a_inf;
            double T0 = s.Tcache[idx];
            if (v.predict) {
                // second-order step from the cached species state with the new composition:
                // e(Tc + d) ~ ec + cv d + cvp d^2 / 2 = e
                double ec = 0.0, cvc = 0.0, cvpc = 0.0;
#pragma unroll
                for (int sp = 0; sp < NSP; ++sp) {
                    ec += Y[sp] * s.esc[sp][idx];
                    cvc += Y[sp] * s.cvsc[sp][idx];
                    cvpc += Y[sp] * s.cvpc[sp][idx];
                }
                const double icv = cl_rcp(cvc);
                const double d1 = (e_si - ec) * icv;
                T0 += d1 - 0.5 * cvpc * d1 * d1 * icv;
            }
            ClosureOut o;
            closure_si_p<MIXED>(g, rho * sc.rho_inf, e_si, Y, T0, cneq, cneq && !v.sm, o);
            atomic_status(v.status, o.status);
            s.Tcache[idx] = o.T;
#pragma unroll
            for (int sp = 0; sp < NSP; ++sp) {
                s.esc[sp][idx] = o.es[sp];
                s.cvsc[sp][idx] = o.cvs[sp];
                s.cvpc[sp][idx] = o.cvps[sp];
            }
            T = __dmul_rn(o.T, iT_ref);
            p = __dmul_rn(o.p, ip_ref);
            mu = __dmul_rn(o.mu, imu_inf);
            k = __dmul_rn(o.k, ik_inf);
            a = __dmul_rn(o.a, ia_inf);
            double ym = 0.0;
#pragma unroll
            for (int sp = 0; sp < NSP; ++sp) ym += Y[sp] * g.invM[sp];
#pragma unroll
            for (int sp = 0; sp < NSP; ++sp) {
                h[sp] = __dmul_rn(o.h[sp], ia2);
                wd[sp] = __dmul_rn(o.wdot[sp], wscale);
                X[sp] = o.X[sp];
                // the electron's diffusive flux follows the ions (flux_point): no coefficient
                W[sp] = cneq && (!HAS_CHARGE || g.heavy[sp]) ? rho * g.M[sp] * ym : 0.0;
                Wd[sp] = cneq ? __dmul_rn(W[sp], __dmul_rn(o.D[sp], d_nd)) : 0.0;
            }
        }
        s.T[idx] = T;
        s.p[idx] = p;
        s.H[idx] = (rhoE + p) * irho;
        s.u_c[idx] = u;
        s.v_c[idx] = vv;
        s.e[idx] = e;
        s.a[idx] = a;
        s.mu_e[idx] = __dmul_rn(mu, iRe);
        s.K[idx] = __dmul_rn(k, iRePr);
        if (!v.ad) s.beta[idx] = 0.0;
#pragma unroll
        for (int sp = 0; sp < NSP; ++sp) {
            s.Y[sp][idx] = Y[sp];
            s.X[sp][idx] = X[sp];
            s.h[sp][idx] = h[sp];
            s.Wd[sp][idx] = Wd[sp];
            s.W[sp][idx] = W[sp];
            if (!v.ad) s.G[sp][idx] = Wd[sp];
        }
#pragma unroll
        for (int sp = 1; sp < NSP; ++sp) s.SRC[v.off[sp] + idx] = wd[sp];
    }
}

// (A) over an index range of one grid
template <bool MIXED, bool LTE = false>
__device__ __forceinline__ void closure_body(const GasDev& g, const Scales& sc, const GridView& v,
                                             const double* __restrict__ U, const Scratch& s,
                                             long long lo, long long hi, long long stride) {
    const ScaleInv c = scale_inv(sc);
    for (long long li = lo + threadIdx.x; li < hi; li += stride)
        closure_point<MIXED, LTE>(g, sc, c, v, U, s, (int)li);
}

// (B) face velocities and the face products of the normal momentum fluxes;
// index range: the x-faces, then the y-faces
__device__ __forceinline__ void face_vel_body(const GridView& v, const double* __restrict__ U,
                                              const Scratch& s, long long lo, long long hi,
                                              long long stride) {
    const int nxf = v.ny * (v.nx + 1);
    for (long long li = lo + threadIdx.x; li < hi; li += stride) {
        const int i = (int)li;
        if (i < nxf) {
            const double m = U[v.off[NSP + 1] + i];
            const double u = cl_div(m, s.rho_xf[i]);
            s.u_xf[i] = u;
            s.mux_f[i] = m * u;
        } else {
            const int j = i - nxf;
            const double m = U[v.off[NSP + 2] + j];
            const double vv = cl_div(m, s.rho_yf[j]);
            s.v_yf[j] = vv;
            s.mvy_f[j] = m * vv;
        }
    }
}

// (D) artificial diffusivity: strain-rate magnitude, dilatation, Ducros switch
__device__ __forceinline__ void ad_prep_body(const Scratch& s, long long lo, long long hi,
                                             long long stride) {
    for (long long li = lo + threadIdx.x; li < hi; li += stride) {
        const int i = (int)li;
        const double ux = s.dudx[i], vy = s.dvdy[i], uy = s.dudy_c[i], vx = s.dvdx_c[i];
        const double sxy = uy + vx;
        s.S[i] = cl_sqrt(ux * ux + vy * vy + 0.5 * sxy * sxy);
        const double dv = ux + vy;
        const double om = vx - uy;
        s.div[i] = dv;
        s.fsw[i] = dv < 0.0 ? cl_div(dv * dv, dv * dv + om * om + DUCROS_EPS) : 0.0;
    }
}

__device__ __forceinline__ double d4x(const double* f, int j, int i, int nx) {
    const int c = min(max(i, 2), nx - 3);
    const double* r = f + (long long)j * nx + c;
    return r[-2] - 4.0 * r[-1] + 6.0 * r[0] - 4.0 * r[1] + r[2];
}

__device__ __forceinline__ double d4y(const double* f, int j, int i, int nx, int ny) {
    const int c = min(max(j, 2), ny - 3);
    const double* r = f + (long long)c * nx + i;
    return r[-2 * nx] - 4.0 * r[-nx] + 6.0 * r[0] - 4.0 * r[nx] + r[2 * nx];
}

// Raw artificial diffusivities: a factor times |d4x wx + d4y wy|. Fourteen binary64 operations per
// point and field bound the plain form (110 us at 2048 x 256); here a thread takes four neighbours
// along x of one field, the fourth differences (weights 1, -4, 6, exact) on integers (fourth_run,
// fix64.cuh), and two products and a sum remain binary64: 80 us. (The same in three dimensions, forty
// inputs a run, was slower than the plain form there: jet right-hand side 9.77 against 9.61 ms.) Runs
// at the ends of a row and those that fourth_run does not take have the plain form.
// Runs of four per field along dir.
__host__ __device__ __forceinline__ int gauss_runs(int nx, int ny, int dir) {
    return dir == 0 ? ny * ((nx + RUN - 1) / RUN) : (ny + RUN - 1) / RUN * nx;
}

__device__ __forceinline__ void ad_raw_body(bool cneq, const GridView& v,
                                            const double* __restrict__ U, const Scratch& s,
                                            long long lo, long long hi, long long stride) {
    const int nx = v.nx, ny = v.ny, qx = (nx + RUN - 1) / RUN, n = ny * qx;
    hi = min(hi, (long long)AD_FIELDS * n);
    for (long long li = lo + threadIdx.x; li < hi; li += stride) {
        const int f = (int)((unsigned)li / (unsigned)n), q = (int)li - f * n;
        const int j = q / qx, i = (q - j * qx) * RUN;
        const long long row = (long long)j * nx;
        if (f >= 3 && !cneq) {
            for (int k = 0; k < RUN && i + k < nx; ++k) s.raw[f][row + i + k] = 0.0;
            continue;
        }
        const double* __restrict__ in = f == 0 ? s.S : (f == 1 ? s.div : (f == 2 ? s.e : s.Y[f - 3]));
        const double dx = cl_rcp(v.xi_c[i]), dy = cl_rcp(v.eta_c[j]);      // x is uniform
        const double wt[2] = {f < 2 ? dx * dx : dx, f < 2 ? dy * dy : dy};
        double sum[RUN];
        bool done = false;
        if (i >= 2 && i + RUN + 1 < nx && j >= 2 && j < ny - 2) {
            double w[RUN + 4], r[4][RUN];
#pragma unroll
            for (int k = 0; k < RUN + 4; ++k) w[k] = in[row + i - 2 + k];
#pragma unroll
            for (int k = 0; k < RUN; ++k) {
                r[0][k] = in[row + i + k - 2 * nx];
                r[1][k] = in[row + i + k - nx];
                r[2][k] = in[row + i + k + nx];
                r[3][k] = in[row + i + k + 2 * nx];
            }
            done = fourth_run(w, r, wt, sum);
        }
        if (!done)
            for (int k = 0; k < RUN; ++k)
                if (i + k < nx) {
                    const double t = d4x(in, j, i + k, nx) * wt[0] + d4y(in, j, i + k, nx, ny) * wt[1];
#pragma unroll
                    for (int o = 0; o < RUN; ++o) if (o == k) sum[o] = t;
                }
#pragma unroll
        for (int k = 0; k < RUN; ++k) {
            if (i + k >= nx) continue;
            const long long at = row + i + k;
            double c;
            if (f >= 3) c = v.C_D * s.a[at];
            else {
                c = (f == 0 ? v.C_mu : (f == 1 ? v.C_beta * s.fsw[at] : v.C_kappa * cl_div(s.a[at], s.T[at]))) *
                    U[v.off[0] + at];
            }
            s.raw[f][at] = c * fabs(sum[k]);
        }
    }
}

// Gaussian filter of the raw diffusivities along x (dir 0) or y (dir 1); indices clamp. Nine
// binary64 operations a point on a unit that takes 19 cycles each bound the plain form (80 us a
// pass at 2048 x 256). Here a thread filters four neighbours on 62-bit integers scaled by the
// largest of their twelve inputs, which share the conversions (gauss_fixed, fix64.cuh): 40 us
// (binary32 in the mixed path before: 37). Outputs that it does not give to binary64's precision
// take the plain form (without that check 36 us).
// in(i): input i of the line, indices clamped or wrapped by the caller; put(k, v): output pos + k
template <class In, class Put>
__device__ __forceinline__ void gauss_run(int pos, const In& in, const Put& put) {
    double x[RUN + 8], y[RUN];
#pragma unroll
    for (int k = 0; k < RUN + 8; ++k) x[k] = in(pos - 4 + k);
    const int plain = gauss_fixed(x, y);
#pragma unroll
    for (int o = 0; o < RUN; ++o)
        if (!(plain >> o & 1)) put(o, y[o]);
    for (int o = 0; plain >> o; ++o) {
        if (!(plain >> o & 1)) continue;
        double acc = c_gauss[0] * in(pos + o);
#pragma unroll
        for (int d = 1; d <= 4; ++d) acc += c_gauss[d] * (in(pos + o - d) + in(pos + o + d));
        put(o, acc);
    }
}

__device__ __forceinline__ void gauss_body(const GridView& v, const Scratch& s, int dir,
                                           long long lo, long long hi, long long stride) {
    const int n = gauss_runs(v.nx, v.ny, dir), qx = (v.nx + RUN - 1) / RUN;
    hi = min(hi, (long long)AD_FIELDS * n);
    for (long long li = lo + threadIdx.x; li < hi; li += stride) {
        const int f = (int)((unsigned)li / (unsigned)n), r = (int)li - f * n;
        if (dir == 0) {
            const int j = r / qx, i = (r - j * qx) * RUN;
            const double* __restrict__ in = s.raw[f] + (long long)j * v.nx;
            double* __restrict__ out = s.filt[f] + (long long)j * v.nx;
            gauss_run(i, [&](int k) { return in[min(max(k, 0), v.nx - 1)]; },
                      [&](int k, double y) { if (i + k < v.nx) out[i + k] = y; });
        } else {
            const int q = r / v.nx, i = r - q * v.nx, j = q * RUN;
            const double* __restrict__ in = s.filt[f] + i;
            double* __restrict__ out = s.raw[f] + i;
            gauss_run(j, [&](int k) { return in[(long long)min(max(k, 0), v.ny - 1) * v.nx]; },
                      [&](int k, double y) { if (j + k < v.ny) out[(long long)(j + k) * v.nx] = y; });
        }
    }
}

// (F, I) normal stresses and momentum fluxes at centres (Eqs. 5, 6, 9). AD: the filtered artificial
// diffusivities join the transport coefficients first: memory bounds both, and one pass instead of
// two (beta is no longer stored, beta and mu not read again) takes a launch off the chain too: the
// 32 x 16 right-hand side 166 -> 163 us with the single flux launch below, 515 x 131 411 -> 402.
template <bool AD>
__device__ __forceinline__ void stress_c_body(const Scratch& s, long long lo, long long hi,
                                              long long stride) {
    for (long long li = lo + threadIdx.x; li < hi; li += stride) {
        const int i = (int)li;
        const double ux = s.dudx[i], vy = s.dvdy[i];
        const double dv = ux + vy;
        double mu = s.mu_e[i], b;
        if constexpr (AD) {
            mu += s.raw[0][i];
            b = s.raw[1][i];
            s.mu_e[i] = mu;
            s.K[i] += s.raw[2][i];
#pragma unroll
            for (int sp = 0; sp < NSP; ++sp) s.G[sp][i] = s.Wd[sp][i] + s.W[sp][i] * s.raw[3 + sp][i];
        } else {
            b = s.beta[i];
        }
        const double txx = mu * (2.0 * ux - 2.0 / 3.0 * dv) + b * dv;
        const double tyy = mu * (2.0 * vy - 2.0 / 3.0 * dv) + b * dv;
        s.tau_xx[i] = txx;
        s.tau_yy[i] = tyy;
        // normal momentum fluxes: rho u u formed on the faces, interpolated to the centres
        s.Gxx[i] = s.mux_c[i] + s.p[i] - txx;
        s.Gyy[i] = s.mvy_c[i] + s.p[i] - tyy;
    }
}

// (F, I) shear stress and cross momentum flux at corners
__device__ __forceinline__ void stress_cn_body(const Scratch& s, long long lo, long long hi,
                                               long long stride) {
    for (long long li = lo + threadIdx.x; li < hi; li += stride) {
        const int i = (int)li;
        const double txy = s.mu_cn[i] * (s.dudy_cn[i] + s.dvdx_cn[i]);
        s.tau_xy[i] = txy;
        s.Gxy[i] = s.rho_cn[i] * s.u_cn[i] * s.v_cn[i] - txy;
    }
}

// (G, H) species and energy fluxes at the x-faces (dir 0) or y-faces (dir 1) of face index i;
// SMK: the kernel carries the Stefan-Maxwell solve (used by grids with v.sm)
template <bool SMK>
__device__ __forceinline__ void flux_point(const GasDev& gd, const Scales& sc, const GridView& v,
                                           const double* __restrict__ U, const Scratch& s, int dir,
                                           int i) {
    const double* __restrict__ mom = U + v.off[NSP + 1 + dir];
    double* const* Yf = dir == 0 ? s.Yx : s.Yy;
    double* const* Gf = dir == 0 ? s.Gx : s.Gy;
    double* const* hf = dir == 0 ? s.hx : s.hy;
    double* const* dX = dir == 0 ? s.dXdx : s.dXdy;
    double* const* Fs = dir == 0 ? s.Fsx : s.Fsy;
    const double* Hf = dir == 0 ? s.Hx : s.Hy;
    const double* Kf = dir == 0 ? s.Kx : s.Ky;
    const double* dT = dir == 0 ? s.dTdx : s.dTdy;
    const double* tn = dir == 0 ? s.txx_x : s.tyy_y;      // normal stress at the face
    const double* tsh = dir == 0 ? s.txy_x : s.txy_y;     // shear stress at the face
    const double* un = dir == 0 ? s.u_xf : s.v_yf;        // velocity normal to the face
    const double* ut = dir == 0 ? s.v_x : s.u_y;          // tangential velocity
    double* FE = dir == 0 ? s.FEx : s.FEy;
    const bool wallface = dir == 1 && v.wall && i < v.nx;
    double g[NSP], J[NSP], sum = 0.0;
#pragma unroll
    for (int sp = 0; sp < NSP; ++sp) {
        g[sp] = Gf[sp][i] * dX[sp][i];
        sum += g[sp];
    }
    double q = -Kf[i] * dT[i];
    const double m = mom[i];
    if (SMK && v.sm && !wallface) {
        // Stefan-Maxwell fluxes (Eq. 17); the algebraic part above carries only the artificial
        // diffusivity in this mode
        double Yl[NSP], dXl[NSP], Jsm[NSP];
#pragma unroll
        for (int sp = 0; sp < NSP; ++sp) {
            Yl[sp] = Yf[sp][i];
            dXl[sp] = dX[sp][i];
        }
        const double* Tf = dir == 0 ? s.Tx : s.Ty;
        const double* pf = dir == 0 ? s.px : s.py;
        const double* rf = dir == 0 ? s.rho_xf : s.rho_yf;
        stefan_maxwell_face(gd, Tf[i] * sc.T_ref, pf[i] * sc.rho_inf * sc.a_inf * sc.a_inf,
                            sc.mu_inf * sc.Re / sc.rho_inf, rf[i], Yl, dXl, Jsm);
#pragma unroll
        for (int sp = 0; sp < NSP; ++sp) J[sp] = Jsm[sp];
    } else {
#pragma unroll
        for (int sp = 0; sp < NSP; ++sp) J[sp] = 0.0;
    }
#pragma unroll
    for (int sp = 0; sp < NSP; ++sp) J[sp] = wallface ? 0.0 : J[sp] - (g[sp] - Yf[sp][i] * sum);
    if (HAS_CHARGE && gd.ie >= 0 && !wallface) {
        // zero conduction current: J_e = M_e sum_ions J_i / M_i; the omitted first species
        // takes J_0 = -sum_{s >= 1} J_s (the diffusive mass fluxes sum to zero)
        double acc = 0.0;
#pragma unroll
        for (int sp = 0; sp < NSP; ++sp)
            if (gd.charge[sp] > 0) acc += J[sp] / gd.M[sp];
        double tot = 0.0;
#pragma unroll
        for (int sp = 1; sp < NSP; ++sp) {
            if (sp == gd.ie) J[sp] = gd.M[sp] * acc;
            tot += J[sp];
        }
        J[0] = -tot;
    }
#pragma unroll
    for (int sp = 0; sp < NSP; ++sp) q += hf[sp][i] * J[sp];
#pragma unroll
    for (int sp = 1; sp < NSP; ++sp) Fs[sp][i] = m * Yf[sp][i] + J[sp];
    // tau . u normal component: x-face tau_xx u + tau_xy v; y-face tau_xy u + tau_yy v
    const double work = dir == 0 ? tn[i] * un[i] + tsh[i] * ut[i] : tsh[i] * ut[i] + tn[i] * un[i];
    FE[i] = m * Hf[i] + q - work;
}

// Index range: the x-faces, then the y-faces, in one launch: the two families are independent and
// a launch each left the chip idle between them (2048 x 256 step 5.46 -> 5.43 ms, 515 x 131
// right-hand side 407 -> 402 us).
template <bool SMK>
__device__ __forceinline__ void flux_body(const GasDev& gd, const Scales& sc, const GridView& v,
                                          const double* __restrict__ U, const Scratch& s,
                                          long long lo, long long hi, long long stride) {
    const int nxf = v.ny * (v.nx + 1);
    for (long long li = lo + threadIdx.x; li < hi; li += stride) {
        const int i = (int)li;
        if (i < nxf) flux_point<SMK>(gd, sc, v, U, s, 0, i);
        else flux_point<SMK>(gd, sc, v, U, s, 1, i - nxf);
    }
}

// (J) sum of divergences, sources and sponge; Dirichlet rows; optional RK stage update
// rk: 0 right-hand side only, 1 2N-storage stage (dQ <- A dQ + dt R, U <- U + B dQ),
// 2 TVD stage, 3 first TVD stage (also stores the start state)
struct AssembleArgs {
    const double *DX, *DY, *SRC, *sigma, *Uref;
    const uint8_t* mask;
    double *U, *out, *dQ;
    int rk;
    double A, B, dt;
};

__device__ __forceinline__ void assemble_body(const AssembleArgs& a, long long lo, long long hi,
                                              long long stride) {
    for (long long li = lo + threadIdx.x; li < hi; li += stride) {
        const long long i = li;
        const double u = a.U[i];
        double r = a.DX[i] + a.DY[i] + a.SRC[i] - a.sigma[i] * (u - a.Uref[i]);
        if (a.mask[i]) r = 0.0;
        if (a.rk >= 2) {
            // TVD RK3 stage: U <- A W + B (U + dt R) with W the step's start state, which the
            // first stage (rk == 3) stores in the second register
            const double w = a.rk == 3 ? u : a.dQ[i];
            if (a.rk == 3) a.dQ[i] = u;
            a.U[i] = a.A * w + a.B * (u + a.dt * r);
        } else if (a.rk) {
            const double q = a.A * a.dQ[i] + a.dt * r;
            a.dQ[i] = q;
            a.U[i] = u + a.B * q;
        } else {
            a.out[i] = r;
        }
    }
}

// Low-pass filter of the conserved state along x (dir 0) or y (dir 1) lines of every field:
// out_i = in_i - sigma (D_m in)_i with the binomial 2m-th difference of weights c_filter_w,
// m = min(5, distance to the nearer end of the line); end points copied.
// c_filter_w[m - 1][n + m] = (-1)^n C(2m, m + n) / 4^m (exact in binary64).
static __constant__ double c_filter_w[5][11] = {
    {-1.0 / 4, 2.0 / 4, -1.0 / 4},
    {1.0 / 16, -4.0 / 16, 6.0 / 16, -4.0 / 16, 1.0 / 16},
    {-1.0 / 64, 6.0 / 64, -15.0 / 64, 20.0 / 64, -15.0 / 64, 6.0 / 64, -1.0 / 64},
    {1.0 / 256, -8.0 / 256, 28.0 / 256, -56.0 / 256, 70.0 / 256, -56.0 / 256, 28.0 / 256,
     -8.0 / 256, 1.0 / 256},
    {-1.0 / 1024, 10.0 / 1024, -45.0 / 1024, 120.0 / 1024, -210.0 / 1024, 252.0 / 1024,
     -210.0 / 1024, 120.0 / 1024, -45.0 / 1024, 10.0 / 1024, -1.0 / 1024}};

// Runs of four entries along dir in the three sections of the state: the index range of filter_body.
__host__ __device__ __forceinline__ long long filter_runs(int nx, int ny, int dir) {
    if (dir == 0)
        return ((NSP + 1) * (long long)ny + ny + 1) * ((nx + RUN - 1) / RUN) + (long long)ny * ((nx + RUN) / RUN);
    return ((NSP + 1) * (long long)nx + nx + 1) * ((ny + RUN - 1) / RUN) + (long long)nx * ((ny + RUN) / RUN);
}

// The plain form took twelve binary64 operations an entry (96 us a pass at 2048 x 256). A thread
// takes four entries of a line: away from the ends the tenth difference is formed on integers, whose
// weights are exact (tenth_run, fix64.cuh: closer than the plain form's eleven roundings); one FMA with
// the entry itself (binary64) finishes: 47 us. Entries near the ends, and runs that tenth_run does not
// take, have the plain form.
__device__ __forceinline__ void filter_body(int nx, int ny, const double* __restrict__ in,
                                            double* __restrict__ out, int dir, double sigma,
                                            long long lo, long long hi, long long stride) {
    const int across = dir == 0 ? ny : nx, along = dir == 0 ? nx : ny;
    const long long q0 = (along + RUN - 1) / RUN, q1 = (along + RUN) / RUN;   // runs per line
    // sections: centres, the faces with one more entry across, the faces with one more along
    const long long nc = (long long)nx * ny, nxf = (long long)(nx + 1) * ny;
    const long long n0 = (NSP + 1) * (long long)across * q0, n1 = (across + 1) * q0;
    hi = min(hi, n0 + n1 + across * q1);
    for (long long idx = lo + threadIdx.x; idx < hi; idx += stride) {
        long long t = idx, base, q = q0;
        int pitch = nx, n = along;
        bool xf = false;
        if (idx < n0) {
            base = 0;
        } else if (idx < n0 + n1) {
            t = idx - n0;
            xf = dir == 1;                               // one more across: x-faces' columns
            base = (NSP + 1) * nc + (xf ? 0 : nxf);
        } else {
            t = idx - n0 - n1;
            q = q1;
            n = along + 1;
            xf = dir == 0;
            base = (NSP + 1) * nc + (xf ? 0 : nxf);
        }
        if (xf) pitch = nx + 1;
        // dir 0: line = row (of a field), run fastest; dir 1: column fastest, then run, then field
        long long first, st;
        int pos;
        if (dir == 0) {
            const long long line = t / q;
            pos = (int)(t - line * q) * RUN;
            first = base + line * pitch;
            st = 1;
        } else {
            const long long field = t / (q * pitch), r = t - field * q * pitch;
            const int run = (int)(r / pitch), col = (int)(r - (long long)run * pitch);
            pos = run * RUN;
            first = base + field * n * pitch + col;
            st = pitch;
        }
        const double* __restrict__ p = in + first;
        double x[RUN + 10], tenth[RUN];
#pragma unroll
        for (int k = 0; k < RUN + 10; ++k) x[k] = p[min(max(pos - 5 + k, 0), n - 1) * st];
        const bool fixed = tenth_run(x, tenth);
#pragma unroll
        for (int o = 0; o < RUN; ++o) {
            const int at = pos + o;
            if (at >= n) continue;
            const int m = min(min(at, n - 1 - at), 5);
            const double f = x[o + 5];
            double acc = 0.0;
            if (m == 5 && fixed) {
                acc = tenth[o];
            } else if (m > 0) {
                const double* w = c_filter_w[m - 1];
                const double* c = p + (at - m) * st;
                for (int k = 0; k <= 2 * m; ++k) acc = fma(w[k], c[k * st], acc);
            }
            out[first + at * st] = m == 0 ? f : fma(-sigma, acc, f);
        }
    }
}

}  // namespace hyp
