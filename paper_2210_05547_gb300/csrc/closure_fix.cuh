// The thermochemistry closure of Sec. 2.2 with its bulk on 64-bit integers (fix64.cuh): species
// modal sums, Newton iteration for T, rate groups, transport and diffusion coefficients, the same
// formulas as thermo.cuh's binary64 closure.
//
// What bounds it: GB300's one binary64 unit per SM (19 cycles per warp instruction). The binary64
// form spends ~1450 of those per point. Here the quantities that are bounded and positive
// (Boltzmann factors, level moments, mole fractions, viscosity ratios, collision integrals) are
// fixed-point numbers, the partition functions, rate constants and their products xf (64-bit
// mantissa and exponent), and only the sums over species and the scaling of the results stay
// binary64, so the two kinds of pipes run at the same time. Every fixed-point quantity keeps at
// least 54 bits below its largest term, against the 53 significant bits and ~1e-15 accumulated
// rounding of the binary64 form; the sum behind D_s of a species among traces, which has no term of
// that size, is formed in binary64 (trace_diffusion: 1,000,003 states of nitrogen with 1e-8 of the
// others 4.33 -> 1.45 ms against handing the whole state to the binary64 closure).
//
// Units below: a name ending in a number n is an integer in units of 2^-n.
//
// Measured (GB300): 4,000,037 independent states 14.4 -> 6.30 ms, 300,007
// eleven-species states in mixed precision 2.66 -> 1.30 ms, the 2048 x 256 RK3 step 8.16 ->
// 6.69 ms, 1200 states 104 -> 59 us (a binary64 chain costs 64 cycles a link, an
// integer product about ten).
//
// Valid for gases whose tables fit the fixed-point ranges (GasDev::fix.ok, checked when the gas
// is loaded) and states with rho, p in [2^-300, 2^300] and |X_s| < 2; any other (non-physical
// compositions, NaN, infinities) takes thermo.cuh's binary64 closure.
#pragma once

#include "fix64.cuh"
#include "internal.h"

namespace hyp {

struct FixState {
    double e[NSP], cv[NSP], cvp[NSP];   // J/kg, J/(kg K), J/(kg K^2)
    xf qv[NSP];                         // q_el / (1 - e^(-theta_v / T)) (atoms: q_el)
    u64 s57[NSP];                       // d ln qv / d ln T
};

// c t (two xf numbers) in units of 2^-58 when it is below 64.
FX bool fix_product58(u64 cm, int ce, xf t, u64& out) {
    const u64 p = mulhi64(cm, t.m);              // 2^-62 2^(ce + te)
    const int d = 4 - ce - t.e;
    if (d < -1 || (d < 0 && (i64)p < 0)) return false;
    out = d < 0 ? p + p : (d < 64 ? p >> d : 0);
    return true;
}

// Species state at T in [50, 1e5] K (it = 1 / T). Per excited electronic level: x = theta / T,
// w = e^-x, and the moments w x, w x^2, w x^3 (each at most 1.4).
FX void species_state_fix(const GasDev& g, double T, xf it, FixState& s) {
    const double invT = f64_of_xf(it);
#pragma unroll
    for (int i = 0; i < NSP; ++i) {
        u64 q57 = (u64)g.fix.lev_g[i][0] << 57, a1 = 0, a2 = 0, a3 = 0;
        for (int l = 1; l < g.nlev[i]; ++l) {
            u64 x58;
            if (!fix_product58(g.fix.lev_m[i][l], g.fix.lev_e[i][l], it, x58) ||
                x58 > ((u64)45 << 58))
                break;                           // LEVEL_CUT: below 1e-19 of the ground level
            const xf b = exp_fixed<57>(-(i64)(x58 >> 1));
            // small w (x > 14, x > 28) raised by 2^k while its moments are formed
            const int sh = -b.e, k = sh > 40 ? 24 : (sh > 20 ? 10 : 0);
            const u64 w63 = b.m >> (sh - k);
            const u64 v1 = mulhi64(w63, x58);            // 2^-57
            const u64 v2 = mulhi64(v1 << 6, x58);
            const u64 v3 = mulhi64(v2 << 6, x58);
            const u32 gl = (u32)g.fix.lev_g[i][l];
            q57 += gl * (w63 >> (6 + k));
            a1 += gl * (v1 >> k);
            a2 += gl * (v2 >> k);
            a3 += gl * (v3 >> k);
        }
        const int z = clz64(q57);                        // q in [1, 64): z in 1..6
        xf qv{q57 << z, 6 - z};
        u64 m1 = 0;
        i64 var54 = 0, cvp54 = 0;
        if (a1 != 0) {
            const u64 r = rcp64(q57 << z);
            m1 = mulhi64(a1, r) >> (6 - z);
            const u64 m2 = mulhi64(a2, r) >> (6 - z), m3 = mulhi64(a3, r) >> (6 - z);
            var54 = (i64)(m2 >> 3) - (i64)mulhi64(m1 << 2, m1 << 2);
            // T d(var)/dT terms: (m3 - m1 m2) - 2 m1 var - 2 var
            cvp54 = (i64)(m3 >> 3) - (i64)(mulhi64(m1 << 2, m2 << 1) << 1) -
                    (mulhi64su(var54 << 4, m1 << 2) << 2) - 2 * var54;
        }
        u64 eo57 = ((u64)3 << 56) + m1;                  // e / (R_s T) above the ground state
        i64 cvo54 = ((i64)3 << 53) + var54;
        u64 s57 = m1;
        if (g.linear[i]) {
            eo57 += (u64)1 << 57;
            cvo54 += (i64)1 << 54;
            u64 x58;
            if (fix_product58(g.fix.tv_m[i], g.fix.tv_e[i], it, x58)) {
                // u = e^-x, v = 1 / (1 - u), E = x u v = x / (e^x - 1), C = E (x + E)
                const xf b = exp_fixed<57>(-(i64)(x58 >> 1));
                const u64 u63 = -b.e < 64 ? b.m >> -b.e : 0;
                const u64 om = ((u64)1 << 63) - u63;
                const int zv = clz64(om);
                const u64 r = rcp64(om << zv);
                const u64 E57 = mulhi64(mulhi64(x58 << (zv > 1 ? zv - 1 : 0), u63), r) << 1;
                const u64 C57 = mulhi64(E57 << 6, (x58 >> 1) + E57) << 1;
                eo57 += E57;
                s57 += E57;
                cvo54 += (i64)(C57 >> 3);
                // T d/dT of C: -C (2 - x - 2 E)
                const i64 h57 = ((i64)1 << 58) - (i64)(x58 >> 1) - (i64)(2 * E57);
                cvp54 -= mulhi64su(h57, C57 << 6) >> 2;
                qv = xf_mul(qv, xf{r, zv - 1});
            }
        }
        const double RT = g.Rs[i] * T, RiT = g.Rs[i] * invT;
        s.e[i] = fma(RT, f64_of_fixed(eo57, 57), g.e0[i]);
        s.cv[i] = g.Rs[i] * f64_of_fixed((u64)cvo54, 54);
        s.cvp[i] = RiT * f64_of_signed(cvp54, 54);
        s.qv[i] = qv;
        s.s57[i] = s57;
    }
}

// First-order shift of the state from T to T + dT, |dT| <= 1e-8 T (the neglected second order is
// below 1e-16 relative).
FX void species_shift_fix(double invT, double dT, FixState& s) {
    const double d = dT * invT;
    const u64 u = bits_of(d);
    const int sh = 1023 - 27 - (int)((u >> 52) & 0x7ff);       // |d| < 2^-26: sh >= 0
    const u64 d90 = sh < 64 ? ((u << 11) | 0x8000000000000000ull) >> sh : 0;
#pragma unroll
    for (int i = 0; i < NSP; ++i) {
        s.e[i] = fma(s.cv[i], dT, s.e[i]);
        s.cv[i] = fma(s.cvp[i], dT, s.cv[i]);
        const u64 c = mulhi64(s.qv[i].m, mulhi64(s.s57[i], d90)) >> 19;
        u64 m = s.qv[i].m;
        int e = s.qv[i].e;
        if ((i64)u < 0) {
            m -= c;
            if (!(m >> 63)) {
                m += m;
                --e;
            }
        } else {
            m += c;
            if (m < c) {                                       // carried past 2^64
                m = (m >> 1) | 0x8000000000000000ull;
                ++e;
            }
        }
        s.qv[i] = xf{m, e};
    }
}

// The safeguarded Newton iteration of temperature_from_energy on species_state_fix.
FX double temperature_from_energy_fix(const GasDev& g, double e, const double* Y, double T0,
                                      unsigned& status, FixState& s) {
    double T = fmin(fmax(T0, T_LO), T_HI);
    double lo = T_LO, hi = T_HI;
    for (int it = 0; it < NEWTON_MAXIT; ++it) {
        const xf iT = xf_rcp(xf_of(T));
        species_state_fix(g, T, iT, s);
        double f = -e, cv = 0.0;
#pragma unroll
        for (int i = 0; i < NSP; ++i) {
            f += Y[i] * s.e[i];
            cv += Y[i] * s.cv[i];
        }
        if (f > 0.0) hi = T; else lo = T;
        double Tn = T - cl_div(f, cv);
        if (fabs(Tn - T) <= NEWTON_RTOL * T) {
            species_shift_fix(f64_of_xf(iT), Tn - T, s);
            return Tn;
        }
        if (!(Tn > lo && Tn < hi)) Tn = 0.5 * (lo + hi);
        T = Tn;
    }
    T = temperature_not_found(g, e, Y, T, status);
    species_state_fix(g, T, xf_rcp(xf_of(T)), s);
    return T;
}

// |X| < 2 as a signed fixed-point number (NaN and larger values: false).
FX bool fix_signed62(double x, i64& out) {
    const u64 u = bits_of(x);
    const int ex = (int)((u >> 52) & 0x7ff) - 1023;
    const u64 m = (u << 11) | 0x8000000000000000ull;
    const int sh = 1 - ex;
    const i64 v = sh < 64 ? (i64)(m >> (sh > 0 ? sh : 1)) : 0;
    out = (i64)u < 0 ? -v : v;
    return ex <= 0;
}

// e^(n ln T - theta / T), theta given by sign and xf; zero for theta / T > 900. F32: in binary32
// (the exponent rounded to binary32, a subnormal result zero), above binary32's range in 64 bits.
template <bool F32>
FX xf rate_exp(i64 n59, i64 L58, int neg, u64 tm, int te, xf iT) {
    const u64 p = mulhi64(tm, iT.m);             // theta / T in units of 2^-62 2^(te + ie)
    const int d = 9 - te - iT.e;                 // to units of 2^-53
    u64 t53;
    if (d >= 0) t53 = d < 64 ? p >> d : 0;
    else t53 = ~(u64)0;
    if (t53 > ((u64)900 << 53)) return xf{0, 0};
    const i64 a = mulhi64su(n59, (u64)L58) + (neg ? (i64)t53 : -(i64)t53);
    if (F32 && a < ((i64)88 << 53)) {
        const u32 u = bits_of_float(expf((float)a * (1.0f / 9007199254740992.0f)));
        const int ex = (int)(u >> 23);
        return ex == 0 ? xf{0, 0} : xf{(u64)((u & 0x7fffffu) | 0x800000u) << 40, ex - 127};
    }
    return exp_fixed<53>(a);
}

// Production rates (Eqs. 14, 15). With z_s = conc_s / r_s (r_s the molar partition function per
// unit volume): R = (sum_r C_r [M_r]) prod r^rf (E_f prod z^rf - E_b prod z^rb). MIXED: E_f in
// binary32.
template <bool MIXED>
FX void kinetics_fix(const GasDev& g, double T, i64 L58, xf iT, const FixState& s,
                     const double* conc, double* wdot) {
    const xf t15 = exp_fixed<58>(L58 + (L58 >> 1));          // T^(3/2): below e^17.3
    const xf t25 = xf_mul(t15, xf_of(T));
    xf r[NSP], z[NSP];
    unsigned neg = 0;
    double molar[NSP];
#pragma unroll
    for (int i = 0; i < NSP; ++i) {
        molar[i] = 0.0;
        r[i] = xf_mul(xf{g.fix.r_m[i], g.fix.r_e[i]}, xf_mul(g.linear[i] ? t25 : t15, s.qv[i]));
        const u64 u = bits_of(conc[i]);
        xf c = xf_of(conc[i]);
        if (((u >> 52) & 0x7ff) == 0) c.m = 0;
        z[i] = xf_mul(c, xf_rcp(r[i]));
        neg |= (unsigned)(u >> 63) << i;
    }
    for (int k = 0; k < g.ngroup; ++k) {
        const xf one{0x8000000000000000ull, 0};
        xf f = rate_exp<MIXED>(g.fix.n59[k], L58, g.fix.sgn[k] & 1, g.fix.ta_m[k], g.fix.ta_e[k], iT);
        xf b = rate_exp<false>(g.fix.n59[k], L58, g.fix.sgn[k] >> 1, g.fix.tb_m[k], g.fix.tb_e[k], iT);
        xf rr = one;
        unsigned nf = 0, nb = 0;
#pragma unroll
        for (int i = 0; i < NSP; ++i) {
            const int rf = g.g_rf[k][i], rb = g.g_rb[k][i];
            for (int q = 0; q < rf; ++q) {
                rr = xf_mul(rr, r[i]);
                f = xf_mul(f, z[i]);
                nf ^= neg >> i;
            }
            for (int q = 0; q < rb; ++q) {
                b = xf_mul(b, z[i]);
                nb ^= neg >> i;
            }
        }
        double Rf = f64_of_xf_any(xf_mul(f, rr)), Rb = f64_of_xf_any(xf_mul(b, rr));
        if (nf & 1) Rf = -Rf;
        if (nb & 1) Rb = -Rb;
        double w = 0.0;
        for (int rx = g.gstart[k]; rx < g.gstart[k + 1]; ++rx)
            w += g.C[rx] * (g.spec[rx] >= 0 ? conc[g.spec[rx]] : 1.0);
        const double Rg = w * (Rf - Rb);
#pragma unroll
        for (int i = 0; i < NSP; ++i)
            if (g.g_nu[k][i] != 0) molar[i] += g.g_nud[k][i] * Rg;   // the group's species only
    }
#pragma unroll
    for (int i = 0; i < NSP; ++i) wdot[i] = g.M[i] * molar[i];
}

// D_i of one species in binary64, where the other species are traces (or cancel): their sum keeps
// its own exponent. Out of line, and only the well depths of the species' own pairs: a mixture has one
// such species.
#ifdef __CUDACC__
__host__ __device__ __noinline__
#endif
static double trace_diffusion(const GasDev& g, double T, double lnT, double p, const double* X, int i) {
    const double TmB = cl_exp(-NJA_B * lnT), rT = cl_rsqrt(T), c = p * (rT * (rT * rT));
    double den = 0.0;
    for (int q = 0; q < g.neps; ++q) {
        double sum = 0.0;
        for (int pr = g.pstart[q]; pr < g.pstart[q + 1]; ++pr) {
            if (g.pair_i[pr] == i) sum += X[g.pair_r[pr]] * g.pair_dinv[pr];
            if (g.pair_r[pr] == i) sum += X[g.pair_i[pr]] * g.pair_dinv[pr];
        }
        if (sum == 0.0) continue;
        const double ts = T * g.eps_inv[q];
        double om = NJA_A * TmB * g.eps_powB[q];
        if (NJA_D * ts < OMEGA_CUT) om += NJA_C * cl_exp(-NJA_D * ts);
        if (NJA_F * ts < OMEGA_CUT) om += NJA_E * cl_exp(-NJA_F * ts);
        if (NJA_H * ts < OMEGA_CUT) om += NJA_G * cl_exp(-NJA_H * ts);
        den += c * om * sum;
    }
    return den != 0.0 ? cl_div(1.0 - X[i], den) : 0.0;
}

// Transport (Blottner, Eucken, Wilke) and the averaged diffusion coefficients (Eq. 19); false
// when a mixture sum leaves the fixed-point range.
// Wilke: with a_s = sqrt(mu_s) M_s^(-1/4), phi_i = X_i + sum_{r != i} (X_r / a_r^2) d_ir (a_i +
// a_r)^2, the square shared by the pair; a scaled so that the largest is in [1, 2).
FX bool transport_fix(const GasDev& g, double T, i64 L58, double p, const double* cv, const double* X,
                      const i64* X62, bool diffusion, double& mu, double& kk, double* D) {
    const u64 L60 = (u64)L58 << 2;
    xf m_s[NSP];
    u64 a62[NSP];
    i64 W58[NSP];
    i64 phi54[NSP];
    int E = -100000;
    xf a[NSP];
#pragma unroll
    for (int i = 0; i < NSP; ++i) {
        phi54[i] = 0;
        if (HAS_CHARGE && !g.heavy[i]) continue;
        const i64 v61 = (mulhi64su(g.fix.bA63[i], L60) << 2) + g.fix.bB61[i];
        const i64 arg57 = mulhi64su(v61, L60) + g.fix.bC57[i];
        const xf h = exp_fixed<58>(arg57);                     // e^(arg / 2)
        m_s[i] = xf_mul(h, h);                                 // 10 mu_s
        a[i] = xf_mul(h, xf{g.fix.iMq_m[i], g.fix.iMq_e[i]});
        E = a[i].e > E ? a[i].e : E;
    }
#pragma unroll
    for (int i = 0; i < NSP; ++i) {
        if (HAS_CHARGE && !g.heavy[i]) continue;
        const int d = E - a[i].e;                              // a_max < 4 a_min: d <= 2
        a62[i] = a[i].m >> (1 + d);
        const u64 b = rcp64(a[i].m);                           // 2^E / a: (b 2^-64) 2^d
        W58[i] = mulhi64su(X62[i], mulhi64(b, b) >> 4 << (2 * d));   // X (2^E / a)^2
    }
#pragma unroll
    for (int i = 0; i < NSP; ++i) {
        if (HAS_CHARGE && !g.heavy[i]) continue;
        phi54[i] += X62[i] >> 8;
#pragma unroll
        for (int r = i + 1; r < NSP; ++r) {
            if (HAS_CHARGE && !g.heavy[r]) continue;
            const u64 sum = a62[i] + a62[r];
            const u64 sq = mulhi64(sum, sum);                  // 2^-60
            phi54[i] += mulhi64su_rn(W58[r], mulhi64(sq, g.fix.wd64[i][r]));
            phi54[r] += mulhi64su_rn(W58[i], mulhi64(sq, g.fix.wd64[r][i]));
        }
    }
    double sm = 0.0, sk = 0.0;
    bool ok = true;
#pragma unroll
    for (int i = 0; i < NSP; ++i) {
        if (HAS_CHARGE && !g.heavy[i]) continue;
        if (phi54[i] < ((i64)1 << 44)) {
            ok = false;
            continue;
        }
        const double t = X[i] * f64_of_xf(xf_mul(m_s[i], xf_rcp(xf_fixed((u64)phi54[i], 54))));
        sm += t;
        sk = fma(t, cv[i] + 2.25 * g.Rs[i], sk);
    }
    if (!ok) return false;
    mu = 0.1 * sm;
    kk = 0.1 * sk;
    if (!diffusion) return true;

    i64 den56[NSP];
#pragma unroll
    for (int i = 0; i < NSP; ++i) den56[i] = 0;
    const xf t = xf_of(T);
    const xf tmB = exp_fixed<58>(-(i64)mulhi64((u64)L58, g.fix.njaB64));
    for (int q = 0; q < g.neps; ++q) {
        // Omega(T / eps) in units of 2^-60
        const u64 pw = mulhi64(g.fix.om_m[q], tmB.m);
        const int dq = 2 - g.fix.om_e[q] - tmB.e;
        u64 om60 = dq >= 0 ? pw >> dq : pw << -dq;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            u64 x58;
            if (fix_product58(g.fix.oe_m[q][k], g.fix.oe_e[q][k], t, x58) && x58 < ((u64)40 << 58)) {
                const xf b = exp_fixed<57>(-(i64)(x58 >> 1));
                om60 += mulhi64(b.m >> (1 - b.e < 64 ? 1 - b.e : 63), g.fix.oc62[k]);
            }
        }
        for (int pr = g.pstart[q]; pr < g.pstart[q + 1]; ++pr) {
            const int i = g.pair_i[pr], r = g.pair_r[pr];
            const u64 inv58 = mulhi64(om60, g.fix.dinv63[pr]) >> 1;
            // rounded: a nearly pure mixture's den is a sum of traces
            den56[i] += mulhi64su_rn(X62[r], inv58);
            den56[r] += mulhi64su_rn(X62[i], inv58);
        }
    }
    // 1 / D_ir = (p / T^(3/2)) Omega dinv_ir
    const xf t15 = exp_fixed<58>(L58 + (L58 >> 1));
    const xf K = xf_mul(t15, xf_rcp(xf_mul(xf_of(p), xf{g.fix.dscale_m, g.fix.dscale_e})));
#pragma unroll
    for (int i = 0; i < NSP; ++i) {
        const i64 d = den56[i];
        const u64 ad = (u64)(d < 0 ? -d : d);
        // below 2^-7 (units of 2^-56) the sum's roundings, at most (ns - 1) / 2 units, would pass 2^-48 of
        // it; above, the rounding of X_s in 1 - X_s is the larger one. (With the line at 2^-4, one lane in
        // a hundred of mixed states: 4,000,037 of them 5.24 -> 11.96 ms.)
        if (ad >= (u64)1 << 49) {
            const double v = f64_of_xf(xf_mul(K, xf_rcp(xf_fixed(ad, 56))));
            D[i] = (1.0 - X[i]) * (d < 0 ? -v : v);
        } else if (!HAS_CHARGE || g.heavy[i]) {
            double x[NSP];
#pragma unroll
            for (int r = 0; r < NSP; ++r) x[r] = X[r];
            D[i] = trace_diffusion(g, T, f64_of_fixed((u64)L58, 58), p, x, i);
        } else {
            D[i] = 0.0;
        }
        if (HAS_CHARGE) D[i] *= g.dfac[i];       // ambipolar ions, no electron coefficient
    }
    return true;
}

}  // namespace hyp
