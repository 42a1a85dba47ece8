// Internal declarations of the GB300 library (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <string>
#include <vector>

#include "../../include/hyp.h"

// Species count the kernels are compiled for: the library is built once for five-species air
// (libhyp.so) and once for eleven-species air with ions and electrons (libhyp11.so).
#ifndef HYP_NSP
#define HYP_NSP 5
#endif
#define NSP HYP_NSP
#define MAXR 64                // elementary reactions
#define MAXG 24                // reaction groups sharing (n, T_a, net stoichiometry)
#define MAXLEV 6               // electronic levels per species
#define MAXEPS 16              // distinct Lennard-Jones well depths of species pairs
#define ETAB_N 64              // temperatures of the species-energy table (start of the T inversion)
#define LSEG 8                 // rows of a line per thread of the line-operator kernel
#define LINE_THREADS 288       // threads per block: fits lines of 2^k + 1 rows (k = 5 .. 11)
#define LINE_MAX_LINES 72      // lines per block, at most (a thread for each of 4 closure rows)
#define LINE_FALL_0 11         // bits that a segment's scale loses per segment of distance: at most
#define LINE_FALL_1 20         // log2 rho^-LSEG (interpolation, derivative)
#define LINE_MARGIN 40         // rows a chunk of a line starts early (rho^40 < 2^-63)
#define LINE_TAIL 64           // rows a line's start reaches into (rho^64 < 2^-101)

namespace hyp {

static_assert(NSP <= HYP_MAX_SPECIES, "species count above the C ABI's capacity");
// Only the eleven-species build accepts charged species (ions, the electron): in the five-species
// build the mixing rules, diffusion and fluxes compile without the charge handling.
constexpr bool HAS_CHARGE = NSP > 5;

void set_error(const std::string& msg);
int fail(int code, const std::string& msg);
int cuda_fail(cudaError_t err, const char* what);

#define HYP_CUDA(call)                                         \
    do {                                                       \
        cudaError_t _e = (call);                               \
        if (_e != cudaSuccess) return ::hyp::cuda_fail(_e, #call); \
    } while (0)

// Integer constants of the closure (closure_fix.cuh): a name ending in a number n is in units of
// 2^-n, a pair (_m, _e) is the number (m / 2^63) 2^e, m in [2^63, 2^64).
struct FixGas {
    int ok;                                      // the table fits the fixed-point ranges
    int lev_g[NSP][MAXLEV];                      // degeneracies
    int lev_e[NSP][MAXLEV], tv_e[NSP], r_e[NSP], iMq_e[NSP];
    int ta_e[MAXG], tb_e[MAXG], sgn[MAXG];       // sgn: bit 0 T_a < 0, bit 1 T_a - theta_d < 0
    int om_e[MAXEPS], oe_e[MAXEPS][3], dscale_e;
    unsigned long long lev_m[NSP][MAXLEV];       // theta_el
    unsigned long long tv_m[NSP];                // theta_v
    unsigned long long r_m[NSP];                 // A_tr (atoms), A_tr / (sigma theta_r) (molecules)
    unsigned long long iMq_m[NSP];               // M^(-1/4)
    long long bA63[NSP], bB61[NSP], bC57[NSP];   // Blottner
    unsigned long long wd64[NSP][NSP];           // wilke_d
    long long n59[MAXG];
    unsigned long long ta_m[MAXG], tb_m[MAXG];   // |T_a|, |T_a - theta_d|
    unsigned long long om_m[MAXEPS];             // A eps^B of the collision integral
    unsigned long long oe_m[MAXEPS][3];          // D / eps, F / eps, H / eps
    unsigned long long oc62[3], njaB64;          // C, E, G; B
    unsigned long long dinv63[NSP * (NSP - 1) / 2], dscale_m;   // pair_dinv / dscale
};

// Gas model as seen by the kernels: a plain struct passed by value as a kernel parameter.
struct GasDev {
    int kind;                    // hyp_gas_kind
    int nr, ngroup, neps, npair;
    // species thermodynamics (rigid rotor / harmonic oscillator, Sec. 2.2.1)
    double M[NSP], invM[NSP], Rs[NSP];
    double e0[NSP];              // (hf298 - H_sens(298.15)) / M, J/kg: internal energy at 0 K
    int linear[NSP];
    double theta_v[NSP];
    int nlev[NSP];               // electronic levels, ascending theta (ground level first)
    double lev_g[NSP][MAXLEV], lev_th[NSP][MAXLEV];
    double A_tr[NSP];            // (2 pi m k / h^2)^(3/2) / N_A: molar translational factor
    double inv_sr[NSP];          // 1 / (sigma theta_r) for linear molecules
    // transport
    double blA[NSP], blB[NSP], blC[NSP];
    double Mq[NSP], iMq[NSP];    // M_s^(1/4) and its reciprocal (Wilke's rule)
    double wilke_d[NSP][NSP];    // 1 / sqrt(8 (1 + M_s / M_r))
    // unordered species pairs grouped by their Lennard-Jones well depth
    int pstart[MAXEPS + 1];
    int pair_i[NSP * (NSP - 1) / 2], pair_r[NSP * (NSP - 1) / 2];
    double pair_dinv[NSP * (NSP - 1) / 2];   // pi sigma^2 / ((3/16) sqrt(2 pi k^3 / m_sr))
    double eps_inv[MAXEPS];      // 1 / sqrt(eps_s eps_r)
    double eps_powB[MAXEPS];     // sqrt(eps_s eps_r)^B of the collision-integral fit
    // binary32 copies of the transport constants for the mixed-precision closure (HYP_MIXED)
    float f_blA[NSP], f_blB[NSP], f_blC[NSP], f_Mq[NSP], f_iMq[NSP], f_Rs[NSP];
    float f_wilke_d[NSP][NSP];
    float f_pair_dinv[NSP * (NSP - 1) / 2];
    float f_eps_inv[MAXEPS], f_eps_powB[MAXEPS];
    // species energies e_s and heat capacities c_v,s (J/kg, J/(kg K)) at ETAB_N temperatures
    // spaced evenly in ln T from 50 K to 1e5 K: a starting temperature for the inversion when no
    // earlier temperature is known. A device array [e | c_v][species][ETAB_N] in global memory
    // (the bisection reads it at a different temperature in every lane, which the constant cache
    // would serialise); null until an evaluation that needs it (hyp_thermo_eval, hyp_lte_eval).
    double etab_lnT0, etab_dlnT;
    const double* etab;
    // kinetics (Eqs. 13-15): elementary reactions with explicit colliders, sorted by group
    int gstart[MAXG + 1];        // reactions of group k: [gstart[k], gstart[k+1])
    double C[MAXR];              // SI pre-exponential factor
    int spec[MAXR];              // species on both sides of the reaction (collider), -1 if none
    signed char g_rf[MAXG][NSP], g_rb[MAXG][NSP];   // group reactants / products without collider
    double g_n[MAXG], g_Ta[MAXG];
    double g_theta_d[MAXG];      // sum_s nu_s E0_s / R_u (K): 0 K reaction energy of the group
    signed char g_nu[MAXG][NSP]; // net stoichiometry nu'' - nu' of the group
    double g_nud[MAXG][NSP];     // the same, as doubles
    // nondimensionalisation (Eqs. 7, 11)
    double rho_inf, a_inf, T_inf, p_inf, mu_inf, k_inf, cp_inf, gamma_inf, R_inf, T_ref, L_ref,
        Re, Pr;
    double prandtl_cpg;
    double mach;
    double Y_inf[NSP];
    double tpg_cp0, tpg_theta;   // thermally perfect gas (Eq. 23): c_p0 (J/(kg K)) and Theta (K)
    // local thermodynamic equilibrium (HYP_GAS_LTE): atoms of N and O per particle, element
    // content of the freestream air (mol/kg), and the partition-function constants of
    // c_s = exp(a_s . lambda - theta0_s / T + ln r_s)
    // charged species (eleven-species build): charge per species, 1 for the species in the mixing
    // rules and binary pairs (all but the electron), the factor on the averaged diffusion
    // coefficient (2: ambipolar ions, 1 neutrals, 0 the electron), the electron's index or -1
    int charge[NSP], heavy[NSP];
    double dfac[NSP];
    int ie;
    double atoms[NSP][2];
    double elem_b[2];
    double lnA_tr[NSP];          // ln A_tr
    double ln_isr[NSP];          // ln(1 / (sigma theta_r)) for linear molecules
    double theta0[NSP];          // E0_s / R_u (K): ground-state energy incl. formation
    double e_lo[NSP], e_hi[NSP]; // species energies at the ends of the inversion's range
    FixGas fix;
};

}  // namespace hyp

struct hyp_gas {
    hyp::GasDev dev;
    std::vector<std::string> names;
    std::vector<double> etab_host;   // the table behind GasDev::etab
    double* etab_dev = nullptr;      // its device copy, made on first use (gas.cu)
    std::mutex etab_mu;
};

namespace hyp {

// What the unknown start of q adds to the first rows of a line (lines.cu): row k of the interior gets
// h_k Q, h_k = (-rho)^(k+1) (1 - rho^(2 (n - k))) / (1 - rho^2), Q = kappa (y_left + rho y_first).
struct LineTail {
    long long h[LINE_TAIL], kappa;               // in units of 2^-64 2^-up, 2^-63
    int up[LINE_TAIL / LSEG];                    // per segment of rows of the line: its h below 1/2
    double hd[LINE_TAIL], kappa_d;
};

// One compact line operator (Sec. 3.1): tridiagonal (alpha, 1, alpha) on the interior rows, explicit
// closure rows at the ends.
struct LineOp {
    int m, n_in;                 // output and input points along the line
    int dir;                     // 0 centre->face, 1 face->centre
    int kind;                    // 0 interpolation, 1 first derivative
    int wall;                    // 1: known value at position 0 enters the closure rows
    int periodic;                // every row interior, indices modulo m
    int margin;                  // rows a chunk (or an extended periodic line) starts early
    int first_interior, last_interior;
    const LineTail* tail;        // device; null for periodic lines
    int ncl;                     // closure rows (<= 4)
    int crow[4], cstart[4], cnum[4];
    double cw[4][5];
    double gw[4];                // weight of the wall value
};

struct LineJob {
    const LineOp* op;            // device pointer
    const double* in;            // input field, or an element offset into the state when in_state
    int in_state;
    double* out;
    long long in_ls, in_es, out_ls, out_es;
    int nlines;
    // plan_line: lines per block (and 2^20 over it), segments per line (or chunk), output rows per
    // chunk, chunks, blocks per chunk and in all
    int nl, inv_nl, nseg, cstep, nchunk, groups, blocks;
    double wall_value;
    double scale;                // factor on the results (sign, and 1 / spacing along z)
    const double* metric;        // per output element along the line, nullable
    // three-dimensional grids: lines grouped by plane, line L starting at
    // (L / lpp) * plane stride + (L % lpp) * line stride (lpp = 0: one group)
    int lpp;
    long long in_ps, out_ps;
    const double* wall_arr;      // per-line wall values (line index), replacing wall_value
};

// Fill in how a job's lines are spread over thread blocks (a function of the operator and the line
// count alone).
void plan_line(const LineOp& op, LineJob& j);

cudaError_t launch_lines(const LineJob* d_jobs, int njobs, int max_blocks, const double* U,
                         cudaStream_t s);

}  // namespace hyp
