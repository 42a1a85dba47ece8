// Batched compact staggered line operators (Sec. 3.1): y = A^{-1} (B x) along grid lines, on
// 64-bit fixed-point numbers.
//
// What bounds it: a tridiagonal solve costs about seven binary64 operations per point, and GB300
// has one binary64 unit per SM (19 cycles per warp instruction), so the binary64 sweeps this file
// held before ran at 125 cycles per 32 points with that unit 60-85% busy and the lines' length
// (latency) behind it. The operators are linear with constant coefficients and neighbouring values
// share a scale, so the solve runs on integers: a product with a constant takes three 32-bit
// integer products (3 cycles), a sum less than one.
//
// Scales: a thread's LSEG = 8 rows have one, the power of two above the largest of their inputs, to
// which the inputs are taken to 62 bits (exact for values down to 2^-9 of it). What the neighbours
// add carries their own scale; a segment whose neighbours' share needs more is shifted down to it.
// A neighbour's scale counts in full one segment away and LINE_FALL bits less (2^11, 2^20; rho^8 is
// 2^-12.7, 2^-22) for each segment more, so an entry's error is a few units of 2^-60 of the largest
// value within sixteen rows, and of farther ones by how much their influence has decayed: fields that
// fall by decades along a line keep binary64's precision at their small end. (With one scale per
// line, as before, a fall over twelve decades left 2e-7 there.) End values reach eight segments on
// (rho^64 < 2^-101); chunks and extended periodic lines start LINE_MARGIN rows early
// (rho^40 < 2^-63).
//
// One thread solves its rows in registers; the threads of a line sit
// in one block and exchange end values, so nothing is stored between the forward and
// the backward recurrence (the earlier sweeps wrote and read it, and re-ran 26-40 warm-up rows per
// segment). With rho / (1 + rho^2) = alpha the interior rows factor into
//     q_r = (1 + rho^2) rhs_r - rho q_{r-1},     y_r = q_r - rho y_{r+1}
// with the same rho (1/3, 0.148) on every row. A thread runs both from zero; what enters from its
// neighbours follows from their own end values, q_in = e_{-1} + rho^8 e_{-2} + ... (eight terms),
// likewise y_in, and their effect on row k, a_k q_in + b_k y_in, is added. The row
// before the first interior row is an explicit closure row, as is the row after the last: the
// latter starts the backward recurrence, the former fixes q's unknown start Q, whose effect h_k Q
// is added to the first rows. Periodic lines wrap the exchange around (or, when 8 does not divide
// the period, extend the line by LINE_MARGIN rows each way); lines of more than LINE_THREADS threads
// are cut into chunks with such margins.
//
// Inputs and, for lines along x (unit stride), results pass through shared memory, 9 words per
// thread of 8 so that neither the threads' rows nor the coalesced copies meet bank conflicts;
// neighbouring threads hold neighbouring lines, which keeps the few threads with closure rows in
// one or two warps.
//
// Lines with NaN, infinities or magnitudes above 2^899 run the same steps in binary64 (the whole
// block), so that such values spread as far as a binary64 solve lets them.
//
// Measured (GB300): the 50 operators of the face phase at 1024 x 256 take 197 us (189 with one scale
// per line; the binary64 sweeps 234, those in pairs of binary32 words 201), a phase of one or two
// operators 19-21 us (38-46). When the solver came in, with one scale per line: the step of the
// 2048 x 256 shock case 6.69 -> 5.96 ms, of the 256 x 64 boundary layer 0.85 -> 0.57, the
// 256 x 128 x 64 jet's right-hand side 12.2 -> 10.5; sixteen rows a thread (three blocks of 288 threads
// per SM instead of four) 6.5 ms, converting the results and adding the corrections on the binary64
// pipe 7.5. The scales per segment cost 1.5-2% of a step; ten neighbours read one by one instead of
// the three exchanges cost 10%. About 310 integer instructions per 32 rows at 2.2 per clock and SM
// bound it.
#include "fix64.cuh"
#include "internal.h"
#include "line_table.h"

namespace hyp {
namespace {

struct LineConst {
    int h, l;
    double d;
};
enum { C_8 = 16, C_16, C_32, C_WA, C_WB, C_G, C_A };
// per kind: rho^1 .. rho^16, (rho^8 2^LINE_FALL)^1, ^2 and ^4, the right-hand side's weights,
// rho^2 / (1 - rho^2), and |response| of a segment's rows to what enters its forward recurrence,
// rho^(k+1) (1 - rho^(2 (LSEG - k))) / (1 - rho^2), the sign (-1)^(k+1)
__constant__ LineConst c_line[2][C_A + LSEG] = {LINE_TABLE_BODY};

// y >> s, all sign bits for s > 63.
__device__ __forceinline__ i64 shift_right(i64 y, int s) {
    i64 v;
    asm("shr.s64 %0, %1, %2;" : "=l"(v) : "l"(y), "r"(s));   // PTX clamps the shift amount
    return v;
}

struct Fix {                                     // y is held as y / 4
    typedef i64 T;
    static constexpr bool scaled = true;
    int E;                                       // the segment's scale: inputs below 2^E
    __device__ __forceinline__ T input(double x) const { return to_scale(x, E, 62); }
    __device__ __forceinline__ T closure(double x) const { return to_scale(x, E, 60); }
    __device__ __forceinline__ double value(T y, unsigned sign) const { return from_scale(y, E, 60, sign); }
    static __device__ __forceinline__ T flip(T a, int kind) { return kind ? -a : a; }
    static __device__ __forceinline__ T shift(T a, int s) { return shift_right(a, s); }
    static __device__ __forceinline__ T mul(T a, const LineConst& c) { return mul_const(a, c.h, c.l); }
    static __device__ __forceinline__ T mul(T a, const LineTail& t, int k) { return __mul64hi(a, t.h[k]); }
    static __device__ __forceinline__ T start(T a, const LineTail& t) { return __mul64hi(a, t.kappa) << 1; }
};

struct Dbl {
    typedef double T;
    static constexpr bool scaled = false;
    int E;                                       // unused
    static __device__ __forceinline__ T input(double x) { return x; }
    static __device__ __forceinline__ T closure(double x) { return x; }
    static __device__ __forceinline__ double value(T y, unsigned sign) { return sign ? -y : y; }
    static __device__ __forceinline__ T flip(T a, int kind) { return kind ? -a : a; }
    static __device__ __forceinline__ T shift(T a, int) { return a; }
    static __device__ __forceinline__ T mul(T a, const LineConst& c) { return a * c.d; }
    static __device__ __forceinline__ T mul(T a, const LineTail& t, int k) { return a * t.hd[k]; }
    static __device__ __forceinline__ T start(T a, const LineTail& t) { return a * t.kappa_d; }
};

// Closure row c of a line.
__device__ __forceinline__ double closure_rhs(const LineOp& op, const double* __restrict__ in,
                                              long long ies, int c, double wall) {
    const double* p = in + (long long)op.cstart[c] * ies;
    const int n = op.cnum[c];
    double x[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) x[k] = k < n ? p[(long long)k * ies] : 0.0;
    double v = op.gw[c] * wall;
#pragma unroll
    for (int k = 0; k < 5; ++k)
        if (k < n) v += op.cw[c][k] * x[k];
    return v;
}

constexpr int SLOT = LSEG + 1;                   // words of shared memory per thread

struct Shared {
    double stage[LINE_THREADS * SLOT];           // inputs, then results of x lines
    u64 ends[2][LINE_THREADS];                   // what the segments exchange (by turns)
    int scale[2][LINE_THREADS];                  // and its scales
    u64 start[LINE_MAX_LINES];                   // Q
    double clos[LINE_MAX_LINES][4];              // the closure rows' values, in the operator's order
};

// The thread's place: rows r0 .. r0 + LSEG - 1 of a line, segment `seg` of `nseg`; the line's next
// segment is `nl` threads on.
struct Place {
    int r0, seg, nseg, nl, line, lo, hi;
    bool active, wrap;
};

template <class T>
__device__ __forceinline__ u64 raw(T v) {
    u64 u;
    memcpy(&u, &v, 8);
    return u;
}

template <class T>
__device__ __forceinline__ T cooked(u64 u) {
    T v;
    memcpy(&v, &u, 8);
    return v;
}

// What enters a segment from the eight before it (way -1) or after it (way 1): the sum of their end
// values times rho^(8 (i - 1)), gathered in three exchanges (two, four, eight segments). The
// segment's numbers q go over to the scale of that sum.
template <class N>
__device__ __forceinline__ typename N::T carried(Shared& sh, int buf, typename N::T end, const Place& P,
                                                 int way, int kind, const LineConst* C, N& num,
                                                 typename N::T (&q)[LSEG]) {
    typedef typename N::T T;
    const int tid = threadIdx.x, fall = kind ? LINE_FALL_1 : LINE_FALL_0;
    auto thread = [&](int i) {                           // of the segment i on, -1 past the line's ends
        int s = P.seg + way * i;
        if (P.wrap) {
            s %= P.nseg;
            s += s < 0 ? P.nseg : 0;
        }
        return (unsigned)s < (unsigned)P.nseg ? tid + (s - P.seg) * P.nl : -1;
    };
    auto publish = [&](T v, int E) {
        sh.ends[buf][tid] = raw(v);
        if (N::scaled) sh.scale[buf][tid] = E;
        __syncthreads();
    };
    auto scale = [&](int at, int down) { return N::scaled && at >= 0 ? sh.scale[buf][at] - down : -(1 << 20); };
    auto value = [&](int at, int by, int c) {
        T e = at >= 0 ? cooked<T>(sh.ends[buf][at]) : T(0);
        if (c >= 0) e = N::mul(e, C[c]);
        return N::shift(e, by);
    };
    publish(end, num.E);
    const int a1 = thread(1), a2 = thread(2);
    const int s1 = scale(a1, 0), s2 = scale(a2, fall);
    int E = max(num.E, max(s1, s2));
    T v = value(a1, E - s1, -1) + value(a2, E - s2, C_8);
#pragma unroll
    for (int i = 2; i <= 4; i += 2) {
        buf ^= 1;
        publish(v, E);
        const int at = thread(i), s = scale(at, fall * i), E0 = E;
        E = max(E, s);
        v = N::shift(v, E - E0) + value(at, E - s, i == 2 ? C_16 : C_32);
    }
    if (N::scaled && E != num.E) {
#pragma unroll
        for (int k = 0; k < LSEG; ++k) q[k] = N::shift(q[k], E - num.E);
        num.E = E;
    }
    return v;
}

// The solve and its output, once the inputs are in shared memory.
template <class N>
__device__ __forceinline__ void solve(N num, const LineJob& J, const LineOp& op, const Place& P,
                                      Shared& sh, double* __restrict__ out) {
    typedef typename N::T T;
    const int kind = op.kind, fi = op.first_interior, li = op.last_interior, tid = threadIdx.x;
    const LineConst* C = c_line[kind];
    const bool left = !op.periodic && P.lo == 0;         // uniform per block
    const bool first = left && P.active && P.seg == 0;
    const int rr = P.active ? li + 1 - P.r0 : LSEG;      // the right closure row, if in this segment
    const double* own = sh.stage + tid * SLOT;
    const int next = P.seg + 1 < P.nseg ? tid + P.nl : (P.wrap ? tid - (P.nseg - 1) * P.nl : tid);
    const double* nxt = sh.stage + (P.active ? next : tid) * SLOT;
    if constexpr (N::scaled) {
        unsigned top = 0;
#pragma unroll
        for (int k = 0; k < LSEG + 3; ++k) top = larger(top, magnitude(k < LSEG ? own[k] : nxt[k - LSEG]));
        if (first) top = larger(top, magnitude(sh.clos[P.line][fi - 1]));
        if (rr >= 0 && rr < LSEG) top = larger(top, magnitude(sh.clos[P.line][fi]));
        num.E = scale_of(top);
    }
    // forward: f0 f1 f2 f3 at offsets -3/2 .. +3/2 of row r; g the same, negated for a derivative
    T q[LSEG];
    T g0 = N::flip(num.input(own[0]), kind), g1 = N::flip(num.input(own[1]), kind);
    T f2 = num.input(own[2]), p = 0;
#pragma unroll
    for (int k = 0; k < LSEG; ++k) {
        const T f3 = num.input(k + 3 < LSEG ? own[k + 3] : nxt[k + 3 - LSEG]);
        p = N::mul(f2 + g1, C[C_WA]) + N::mul(f3 + g0, C[C_WB]) - N::mul(p, C[0]);
        if (k < 2 && first && k < fi) p = 0;             // q starts after the left closure rows
        q[k] = p;
        g0 = g1;
        g1 = N::flip(f2, kind);
        f2 = f3;
    }
    if (rr < LSEG) {                                     // the line ends here
        const T yr = num.closure(rr >= 0 ? sh.clos[P.line][fi] : 0.0);
#pragma unroll
        for (int k = 0; k < LSEG; ++k)
            if (k >= rr) q[k] = k == rr ? yr : 0;
    }
    // backward
    T y = 0;
#pragma unroll
    for (int k = LSEG - 1; k >= 0; --k) {
        y = q[k] - N::mul(y, C[0]);
        q[k] = y;
    }
    const T qin = carried(sh, 0, p, P, -1, kind, C, num, q);
    if (rr >= LSEG) {
#pragma unroll
        for (int k = 0; k < LSEG; ++k) {
            const T c = N::mul(qin, C[C_A + k]);
            q[k] = (k & 1) ? q[k] + c : q[k] - c;
        }
    } else {                                             // rows from rr on do not respond
        const T qe = qin + N::mul(qin, C[C_G]);
#pragma unroll
        for (int k = 0; k < LSEG; ++k) {
            if (k >= rr) continue;
            const T c = N::mul(qe, C[k]) - N::mul(qe, C[2 * rr - k]);
            q[k] = (k & 1) ? q[k] + c : q[k] - c;
        }
    }
    const T yin = carried(sh, 1, q[0], P, 1, kind, C, num, q);
#pragma unroll
    for (int k = 0; k < LSEG; ++k) {
        const T c = N::mul(yin, C[LSEG - 1 - k]);
        q[k] = ((LSEG - k) & 1) ? q[k] - c : q[k] + c;
    }
    if (left) {
        if (first) {
            const T Yl = num.closure(sh.clos[P.line][fi - 1]);
            sh.start[P.line] = raw(N::start(Yl + N::mul(fi == 1 ? q[1] : q[2], C[0]), op.tail[0]));
            if (N::scaled) sh.scale[0][tid] = num.E;     // (the last exchange used the other)
        }
        __syncthreads();
        constexpr int tail = N::scaled ? LINE_TAIL : LINE_MARGIN;
        if (P.active && P.seg < tail / LSEG) {
            const T Q = cooked<T>(sh.start[P.line]);
            // the share of Q in this segment's scale; it outgrows that by less than its headroom
            const int down = N::scaled ? num.E + op.tail->up[P.seg] - sh.scale[0][P.line] : 0;
            if (down < 63) {
#pragma unroll
                for (int k = 0; k < LSEG; ++k) {
                    const int i = P.r0 + k - fi;
                    if (i < 0 || i >= tail) continue;
                    T v = N::mul(Q, op.tail[0], i);
                    if constexpr (N::scaled) v = down < 0 ? v << -down : N::shift(v, down);
                    q[k] += v;
                }
            }
        }
    }
    // output: sign and constant factor, then the metric
    const double scale = J.scale;
    const unsigned sign = (unsigned)__double2hiint(scale) & 0x80000000u;
    const bool scaled = ((unsigned)__double2hiint(scale) & 0x7fffffffu) != 0x3ff00000u || __double2loint(scale);
    const double* __restrict__ met = J.metric;
    const bool edge = P.r0 < fi || rr < LSEG || P.r0 < P.lo || P.r0 + LSEG > P.hi;
    double* st = sh.stage + tid * SLOT;
    double* __restrict__ o = out + (long long)P.r0 * J.out_es;
    const bool xl = J.in_es == 1;
#pragma unroll
    for (int k = 0; k < LSEG; ++k) {
        double v = num.value(q[k], sign);
        bool put = P.active;
        if (edge) {
            const int r = P.r0 + k;
            put = put && r >= P.lo && r < P.hi;
            if (put && (r < fi || r > li)) {
                v = sh.clos[P.line][r < fi ? r : fi + r - li - 1];
                if (sign) v = -v;
            }
        }
        if (scaled) v *= fabs(scale);
        if (xl) {
            st[k] = v;
        } else if (put) {
            if (met) v *= met[P.r0 + k];
            *o = v;
        }
        o += J.out_es;
    }
    if (xl) {
        __syncthreads();
        if (P.active) {
            const int row0 = P.r0 - P.seg * LSEG;
            for (unsigned j = P.seg; j < (unsigned)(P.nseg * LSEG); j += P.nseg) {
                const int r = row0 + (int)j;
                if (r < P.lo || r >= P.hi) continue;
                double v = sh.stage[((j / LSEG) * P.nl + P.line) * SLOT + (j % LSEG)];
                if (met) v *= met[r];
                out[r] = v;
            }
        }
    }
}

// The rare binary64 form, out of line.
__device__ __noinline__ void solve_wild(const LineJob& J, const LineOp& op, const Place& P, Shared& sh,
                                        double* __restrict__ out) {
    solve<Dbl>(Dbl(), J, op, P, sh, out);
}

__global__ void __launch_bounds__(LINE_THREADS, 4) k_lines(const LineJob* __restrict__ jobs,
                                                           const double* __restrict__ U) {
    __shared__ Shared sh;
    const LineJob& J = jobs[blockIdx.y];
    const LineOp& op = *J.op;
    const int nl = J.nl, nseg = J.nseg, tid = threadIdx.x;
    const int chunk = J.nchunk == 1 ? 0 : blockIdx.x / J.groups;
    const int group = blockIdx.x - chunk * J.groups;
    if (group >= J.groups) return;
    Place P;
    P.lo = chunk * J.cstep;                              // output rows [lo, hi)
    if (P.lo >= op.m) return;
    P.hi = min(op.m, P.lo + J.cstep);
    P.nseg = nseg;
    P.nl = nl;
    P.seg = (tid * J.inv_nl) >> 20;                      // tid / nl
    P.line = tid - P.seg * nl;
    P.wrap = op.periodic && !op.margin;
    const int line = group * nl + P.line;
    P.active = P.seg < nseg && line < J.nlines;
    const int row0 = P.lo - (P.lo > 0 || op.periodic ? op.margin : 0);
    P.r0 = row0 + P.seg * LSEG;
    auto offset = [&](int l, long long ls, long long ps) {
        if (!J.lpp) return (long long)l * ls;
        const int k = l / J.lpp;
        return k * ps + (long long)(l - k * J.lpp) * ls;
    };
    const double* __restrict__ base_in = J.in_state ? U + (size_t)J.in : J.in;
    const double* __restrict__ in = base_in + (P.active ? offset(line, J.in_ls, J.in_ps) : 0);
    double* __restrict__ out = J.out + (P.active ? offset(line, J.out_ls, J.out_ps) : 0);
    const double wall = (J.wall_arr && P.active) ? J.wall_arr[line] : J.wall_value;

    // inputs: row r reads r + base .. r + base + 3
    const int base = op.dir == 0 ? -2 : -1, n_in = op.n_in;
    unsigned top = op.wall ? magnitude(wall) : 0u;
    double* st = sh.stage + tid * SLOT;
    if (!P.active) {
#pragma unroll
        for (int k = 0; k < LSEG; ++k) st[k] = 0.0;
    } else if (J.in_es == 1) {
        const int j0 = row0 + base;
        for (unsigned j = P.seg; j < (unsigned)(nseg * LSEG); j += nseg) {
            const int i = j0 + (int)j;
            const double v = (unsigned)i < (unsigned)n_in ? in[i] : 0.0;
            sh.stage[((j / LSEG) * nl + P.line) * SLOT + (j % LSEG)] = v;
            top = max(top, magnitude(v));
        }
    } else {
        const long long ies = J.in_es;
        int j = P.r0 + base;
        if (op.periodic) {
            j %= n_in;
            j += j < 0 ? n_in : 0;
#pragma unroll
            for (int k = 0; k < LSEG; ++k) {
                const double v = in[j * ies];
                st[k] = v;
                top = max(top, magnitude(v));
                j = j + 1 == n_in ? 0 : j + 1;
            }
        } else {
            const double* __restrict__ p = in + j * ies;
#pragma unroll
            for (int k = 0; k < LSEG; ++k) {
                const double v = (unsigned)(j + k) < (unsigned)n_in ? *p : 0.0;
                st[k] = v;
                top = max(top, magnitude(v));
                p += ies;
            }
        }
    }
    // the closure rows, one per thread from the block's end
    if (!op.periodic && LINE_THREADS - 1 - tid < nl * op.ncl) {
        const int i = LINE_THREADS - 1 - tid, c = (i * J.inv_nl) >> 20, l = i - c * nl;
        const int ln = group * nl + l;
        if (ln < J.nlines)
            sh.clos[l][c] = closure_rhs(op, base_in + offset(ln, J.in_ls, J.in_ps), J.in_es, c,
                                        J.wall_arr ? J.wall_arr[ln] : J.wall_value);
    }
    if (__syncthreads_or(P.active && scale_wild(top))) {
        solve_wild(J, op, P, sh, out);
        return;
    }
    solve<Fix>(Fix(), J, op, P, sh, out);
}

}  // namespace

void plan_line(const LineOp& op, LineJob& j) {
    // two rows more than the line has: the last interior row's inputs then lie in the line's own
    // segments
    const int segs = op.periodic ? (op.m + LSEG - 1) / LSEG : (op.m + 2) / LSEG + 1;
    const int extra = op.margin ? 2 * (op.margin / LSEG) : 0;
    if (segs + (op.periodic ? extra : 0) <= LINE_THREADS) {
        j.nseg = segs + (op.periodic ? extra : 0);
        j.cstep = op.m;
        j.nchunk = 1;
    } else {
        j.nseg = LINE_THREADS;
        j.cstep = (LINE_THREADS - extra) * LSEG;
        j.nchunk = (op.m + j.cstep - 1) / j.cstep;
    }
    j.nl = LINE_THREADS / j.nseg;
    if (j.nl > LINE_MAX_LINES) j.nl = LINE_MAX_LINES;
    j.inv_nl = (1 << 20) / j.nl + 1;
    j.groups = (j.nlines + j.nl - 1) / j.nl;
    j.blocks = j.groups * j.nchunk;
}

cudaError_t launch_lines(const LineJob* d_jobs, int njobs, int max_blocks, const double* U,
                         cudaStream_t s) {
    if (njobs == 0) return cudaSuccess;
    k_lines<<<dim3(max_blocks, njobs), LINE_THREADS, 0, s>>>(d_jobs, U);
    return cudaGetLastError();
}

}  // namespace hyp
