// Refinement of approximate manifold intersections (Sec. 7, Eqs. tosolve and
// dampedNewtonEquation): from each seed x = (theta_u, s_u, theta_s, s_s) the
// damped Newton iteration x <- x - alpha Df^{-1} f on
// f = W_A(theta_u, s_u) - W_B(theta_s, s_s), with W_A, W_B the closed-form
// sheet pair of tms_surface_pair and Df their exact partials, all in FP64.
//
// Layout: four lanes per seed, lane c owning coordinate c of every 4-vector
// (W, its partials, the normal frame, one row of Df).  The four sines/cosines
// and two exponentials an iteration needs are spread over the four lanes and
// exchanged by shuffles; dot products are summed over the quad four at a time; the
// 4x4 solve is a partial-pivot elimination whose rows live in the lanes.  Every stop
// decision is taken on the quad's first lane and broadcast, so the four lanes always
// agree.  A warp loops while any of its eight seeds is still iterating; the loop is
// bounded by max_iter + 1 evaluations per seed.
//
// What bounds it: the FP64 pipe, which takes one warp instruction an SM every 19 clocks
// (measured).  So scalars that all four lanes would compute alike are computed by one of
// them and shuffled, comparisons and sign changes are integer, and a block is one warp,
// so that 1500 warps (12,000 seeds) load the 152 SMs evenly (blocks of four put twelve
// on some and eight on others): 12,000 seeds 1476 -> 866 us, 12,000 branches of 50 steps
// 31.5 -> 17.9 ms, the results the same but for roundings in a few of 10,000.
#include <cuda_runtime.h>
#include <math.h>

#include <cstddef>
#include <string>

#include "tms_common.cuh"

namespace {

constexpr int kH = TMS_SURF_MAX_HARMONICS;
constexpr int kF = TMS_SURF_MAX_FOLDS;
constexpr int kThreads = 32;           // 8 seeds per block
constexpr int kSeedsPerBlock = kThreads / 4;
constexpr unsigned kFull = 0xffffffffu;
constexpr double kPi = 3.141592653589793;
constexpr double kTwoPi = 6.283185307179586;

struct RefineArgs {
    tms_surface_pair sp;
    tms_refine_params p;
    const double *x0;
    long long ld;
    long long n;
    double *x;
    double *fnorm;
    double *rho;
    int *iters;
    int *status;
};

struct ContArgs {
    tms_surface_pair sp;
    tms_continue_params p;
    const double *alphas;   // nSteps values after the start
    int steps;              // nSteps
    const double *x0;
    long long ld;
    long long n;
    double *x;
    int *status;
    int *iters;
    double *rho;
    double *fnorm;
};

// Per-block tables, coordinate fastest (lane c reads column c).  With
// a_k = ca_k + alpha dca_k, b_k likewise:
//   T   = sum (a_k/k) cos + (b_k/k) sin     T' = sum b_k cos + (-a_k) sin
//   T'' = sum (-k a_k) cos + (-k b_k) sin
// so every harmonic term is two fused multiply-adds.  W_A's sheet is taken at
// alpha_u, B's underlying sheet at alpha_s, the normal frame at alpha_ref.
struct Coef {
    double uak[kH][4], ubk[kH][4], una[kH][4], ub[kH][4];     // at alpha_u
    double sak[kH][4], sbk[kH][4], sna[kH][4], sb[kH][4];     // at alpha_s
    double ark[kH][4], brk[kH][4], nar[kH][4], br[kH][4];     // at alpha_ref
    double kar[kH][4], kbr[kH][4];                            // at alpha_ref, T''
    // continuation: the walking sheet's tables above are taken at parameter 0 and
    // these hold their derivatives, so a branch at its own alpha uses
    // fma(alpha, d, table) -- the coefficients are affine in the parameter
    double dak[kH][4], dbk[kH][4], dna[kH][4], db[kH][4];
    double fd[kF][4];               // fold_amp * fold_dir
    double root[kF][3];             // fold roots
    double v1[4], v2[4];
    double qpi, hreg;               // Q pi and reg / 2
};

// Fills the tables for (alpha_u, alpha_s) and, for a walking sheet (walk != 0),
// the derivative tables; called by the threads of the block before a barrier.
__device__ void build_tables(Coef &cf, const tms_surface_pair &sp, double au, double as, int walk,
                             int t, int nt) {
    for (int q = t; q < kH * 4; q += nt) {
        const int h = q >> 2, c = q & 3;
        const double k = (double)(h + 1);
        const double a = sp.ca[h][c] + au * sp.dca[h][c];
        const double b = sp.cb[h][c] + au * sp.dcb[h][c];
        const double a2 = sp.ca[h][c] + as * sp.dca[h][c];
        const double b2 = sp.cb[h][c] + as * sp.dcb[h][c];
        const double ar = sp.ca[h][c] + sp.alpha_ref * sp.dca[h][c];
        const double br = sp.cb[h][c] + sp.alpha_ref * sp.dcb[h][c];
        cf.uak[h][c] = a / k;
        cf.ubk[h][c] = b / k;
        cf.una[h][c] = -a;
        cf.ub[h][c] = b;
        cf.sak[h][c] = a2 / k;
        cf.sbk[h][c] = b2 / k;
        cf.sna[h][c] = -a2;
        cf.sb[h][c] = b2;
        cf.ark[h][c] = ar / k;
        cf.brk[h][c] = br / k;
        cf.nar[h][c] = -ar;
        cf.br[h][c] = br;
        cf.kar[h][c] = -k * ar;
        cf.kbr[h][c] = -k * br;
        if (walk) {
            cf.dak[h][c] = sp.dca[h][c] / k;
            cf.dbk[h][c] = sp.dcb[h][c] / k;
            cf.dna[h][c] = -sp.dca[h][c];
            cf.db[h][c] = sp.dcb[h][c];
        }
    }
    if (t < kF * 4) cf.fd[t >> 2][t & 3] = sp.fold_amp[t >> 2] * sp.fold_dir[t >> 2][t & 3];
    if (t < kF * 3) cf.root[t / 3][t % 3] = sp.fold_root[t / 3][t % 3];
    if (t < 4) {
        cf.v1[t] = sp.v1[t];
        cf.v2[t] = sp.v2[t];
    }
    if (t == 0) {
        cf.qpi = sp.Q * kPi;
        cf.hreg = sp.reg * 0.5;
    }
}

// One seed's Newton solve, held identically by the quad's four lanes.
struct Solve {
    double x0, x1, x2, x3;   // iterate (angles unwrapped)
    int code;                // -1 while iterating, else TMS_REFINE_*
    int iters;               // updates made when the solve stopped
    int k;                   // updates made so far
    double fn, rh, rc2;      // ||f||^2, det Df, prod ||Df e_j||^2 at the last evaluation
};

__device__ __forceinline__ double quad_sum(double v) {
    v += __shfl_xor_sync(kFull, v, 1);
    v += __shfl_xor_sync(kFull, v, 2);
    return v;
}

// the quad's sums of four values: lane c holds that of the c-th, added in the order
// quad_sum adds (three additions instead of eight)
__device__ __forceinline__ double quad_sum4(double v0, double v1, double v2, double v3, int c) {
    const bool b0 = c & 1, b1 = c & 2;
    const double u = (b0 ? v1 : v0) + __shfl_xor_sync(kFull, b0 ? v0 : v1, 1);
    const double w = (b0 ? v3 : v2) + __shfl_xor_sync(kFull, b0 ? v2 : v3, 1);
    return (b1 ? w : u) + __shfl_xor_sync(kFull, b1 ? u : w, 2);
}

__device__ __forceinline__ double lane_val(double v, int base, int j) {
    return __shfl_sync(kFull, v, base + j);
}

// |v|'s bits (ordered as |v|, NaN above everything), and v negated when neg
__device__ __forceinline__ long long abs_bits(double v) {
    return __double_as_longlong(v) & 0x7fffffffffffffffLL;
}
__device__ __forceinline__ double flip(double v, bool neg) {
    return __longlong_as_double(__double_as_longlong(v) ^ (neg ? (long long)(1ULL << 63) : 0LL));
}
__device__ __forceinline__ int exponent(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// the corrector's thresholds: tol^2 and switch_below^2 (not negative) as their bits, the
// limits of s as ordered integers (a zero limit as the zero that no zero passes)
struct Stop {
    long long tol2, sw2, lo, hi;
};

__device__ __forceinline__ Stop make_stop(const tms_refine_params &pr) {
    Stop t;
    t.tol2 = __double_as_longlong(pr.tol * pr.tol);
    t.sw2 = __double_as_longlong(pr.switch_below * pr.switch_below);
    t.lo = tms::ord64(pr.s_lo == 0.0 ? -0.0 : pr.s_lo);
    t.hi = tms::ord64(pr.s_hi == 0.0 ? 0.0 : pr.s_hi);
    return t;
}

// p = (s - r0)(s - r1)(s - r2) and its first two derivatives.
__device__ __forceinline__ void cubic(double s, const double *r, double &p, double &p1,
                                      double &p2) {
    const double d0 = s - r[0], d1 = s - r[1], d2 = s - r[2];
    p = d0 * d1 * d2;
    p1 = d1 * d2 + d0 * d2 + d0 * d1;
    p2 = 2.0 * (d0 + d1 + d2);
}

// The quantities one damped-Newton iteration needs at the iterate (x0..x3): the
// stop checks, ||f||^2, the product of Df's squared column norms, det Df and the
// Newton step dx = Df^{-1} f.  Every lane of the warp calls it together (it
// exchanges values within the quad).  WALK = 1 or 2: the sheet of W_A or of B
// is taken at the quad's own parameter aw (continuation); 0: both at the
// tables' values.
struct Eval {
    int pre;       // stop decided before evaluating (non-finite or escaped iterate), or -1
    int fin;       // f and Df finite
    double r2, cn2, det, dx[4];
};

// The walking sheet's coefficients of each harmonic at a quad's own parameter (a, b over
// k; -a; b), lane fastest: filled when the quad starts a step, read by its iterations.
struct WalkCoef {
    double v[kH][4][32];
};

template <int WALK>
__device__ __forceinline__ void evaluate(const Coef &cf, const WalkCoef *wc, const tms_surface_pair &sp,
                                         const Stop &stop, double lnlam, double x0,
                                         double x1, double x2, double x3, int c,
                                         int base, Eval &E) {
    const int K = sp.n_harmonics;
    const int NF = sp.n_folds;
    const int lane = threadIdx.x & 31;
    // B's sheet at the frame's parameter: its sums are the frame's
    const bool same = WALK != 2 && sp.alpha_s == sp.alpha_ref;
    // ---- stop checks on the iterate (identical on the quad's lanes)
    int pre = -1;
    {
        const long long o1 = tms::ord64(x1), o3 = tms::ord64(x3);
        if (max(max(exponent(x0), exponent(x1)), max(exponent(x2), exponent(x3))) == 0x7ff)
            pre = TMS_REFINE_NON_FINITE;
        else if (o1 < stop.lo || o1 > stop.hi || o3 < stop.lo || o3 > stop.hi)
            pre = TMS_REFINE_ESCAPED;
    }

    // ---- sines/cosines and exponentials, one per lane: of x0, x2 + c0,
    //      P (x2 - theta0) and Q pi (x3 - s0)
    const double arg = (c == 2 ? sp.P : c == 3 ? cf.qpi : 1.0) *
                       ((c == 0 ? x0 : c == 3 ? x3 : x2) -
                        (c == 0 ? 0.0 : c == 1 ? -sp.c0 : c == 2 ? sp.theta0 : sp.s0));
    double sn, cs;
    sincos(arg, &sn, &cs);
    const double sA = lane_val(sn, base, 0), cA = lane_val(cs, base, 0);
    const double sB = lane_val(sn, base, 1), cB = lane_val(cs, base, 1);
    const double sh1 = lane_val(sn, base, 2), ch1 = lane_val(cs, base, 2);
    const double sh2 = lane_val(sn, base, 3), ch2 = lane_val(cs, base, 3);
    const double s1 = 1.0 - x3;   // s' of B's underlying sheet
    double gA, gA1, gB, gB1, gB2;
    if (sp.stretch) {
        const double e = exp(lnlam * (c == 0 ? x1 : s1));
        gA = lane_val(e, base, 0);
        gB = lane_val(e, base, 1);
        gA1 = lnlam * gA;
        gB1 = lnlam * gB;
        gB2 = lnlam * gB1;
    } else {
        gA = 1.0 + x1;
        gA1 = 1.0;
        gB = 1.0 + s1;
        gB1 = 1.0;
        gB2 = 0.0;
    }

    // ---- folds F(s) at s_u and at s': lane f evaluates fold f's cubics
    double FA = 0.0, FA1 = 0.0, FB = 0.0, FB1 = 0.0, FB2 = 0.0;
    if (NF > 0) {
        double p, p1, p2, q, q1, q2;
        const int fo = c < NF ? c : 0;
        cubic(x1, cf.root[fo], p, p1, p2);
        cubic(s1, cf.root[fo], q, q1, q2);
#pragma unroll
        for (int f = 0; f < kF; ++f) {
            if (f < NF) {
                const double w = cf.fd[f][c];
                FA = fma(w, lane_val(p, base, f), FA);
                FA1 = fma(w, lane_val(p1, base, f), FA1);
                FB = fma(w, lane_val(q, base, f), FB);
                FB1 = fma(w, lane_val(q1, base, f), FB1);
                FB2 = fma(w, lane_val(q2, base, f), FB2);
            }
        }
    }

    // ---- harmonic sums: T, T' at theta_u (alpha_u); T, T' at theta' (alpha_s);
    //      T, T', T'' at theta' (alpha_ref).  cos/sin of k theta by angle addition.
    double TA = 0.0, TAt = 0.0, TB = 0.0, TBt = 0.0, TR = 0.0, TRt = 0.0, TRtt = 0.0;
    double ckA = cA, skA = sA, ckB = cB, skB = sB;
    // lane c advances one of cos, sin of k theta_u, cos, sin of k theta'
    const double r1 = c == 0 ? cA : c == 1 ? sA : c == 2 ? cB : sB;
    const double r2 = c == 0 ? -sA : c == 1 ? cA : c == 2 ? -sB : cB;
#pragma unroll
    for (int h = 0; h < kH; ++h) {
        if (h < K) {
            double uak, ubk, una, ub, sak, sbk, sna, sb;
            if (WALK == 1) {
                uak = wc->v[h][0][lane];
                ubk = wc->v[h][1][lane];
                una = wc->v[h][2][lane];
                ub = wc->v[h][3][lane];
            } else {
                uak = cf.uak[h][c];
                ubk = cf.ubk[h][c];
                una = cf.una[h][c];
                ub = cf.ub[h][c];
            }
            if (WALK == 2) {
                sak = wc->v[h][0][lane];
                sbk = wc->v[h][1][lane];
                sna = wc->v[h][2][lane];
                sb = wc->v[h][3][lane];
            } else {
                sak = cf.sak[h][c];
                sbk = cf.sbk[h][c];
                sna = cf.sna[h][c];
                sb = cf.sb[h][c];
            }
            TA = fma(uak, ckA, fma(ubk, skA, TA));
            TAt = fma(ub, ckA, fma(una, skA, TAt));
            TB = fma(sak, ckB, fma(sbk, skB, TB));
            TBt = fma(sb, ckB, fma(sna, skB, TBt));
            if (!same) {
                TR = fma(cf.ark[h][c], ckB, fma(cf.brk[h][c], skB, TR));
                TRt = fma(cf.br[h][c], ckB, fma(cf.nar[h][c], skB, TRt));
            }
            TRtt = fma(cf.kar[h][c], ckB, fma(cf.kbr[h][c], skB, TRtt));
            if (h + 1 < K) {
                // cos: ck c1 - sk s1;  sin: sk c1 + ck s1
                const double ck = c & 2 ? ckB : ckA, sk = c & 2 ? skB : skA;
                const double v = fma(ck, r1, sk * r2);
                ckA = lane_val(v, base, 0);
                skA = lane_val(v, base, 1);
                ckB = lane_val(v, base, 2);
                skB = lane_val(v, base, 3);
            }
        }
    }
    if (same) {
        TR = TB;
        TRt = TBt;
    }

    // ---- W_A and its partials; B's underlying sheet; the frame sheet
    const double WA = gA * TA + FA, WAt = gA * TAt, WAs = gA1 * TA + FA1;
    const double SB = gB * TB + FB, SBt = gB * TBt, SBs = gB1 * TB + FB1;
    const double t1 = gB * TRt, t2 = gB1 * TR + FB1;
    const double Wtt = gB * TRtt, Wts = gB1 * TRt, Wss = gB2 * TR + FB2;
    const double v1 = cf.v1[c], v2 = cf.v2[c];

    // ---- normal frame (n1, n2) and its theta- and s-partials.  G = J^T J + eps I; lane c
    //      solves for frame vector r = c & 1 and its derivative in theta (d = 0) or s
    //      (d = 1), where d t1 = Wtt, d t2 = Wts or d t1 = -Wts, d t2 = -Wss
    const int r = c & 1, d = c >> 1;
    const double q1 = quad_sum4(t1 * t1, t1 * t2, t2 * t2, t2 * Wts, c);
    const double q2 = quad_sum4(t1 * v1, t1 * v2, t2 * v1, t2 * v2, c);
    const double q3 = quad_sum4(t1 * Wtt, t1 * Wts, Wtt * t2, t1 * Wss, c);
    const double q4 = quad_sum4(Wtt * v1, Wtt * v2, Wts * v1, Wts * v2, c);
    const double q5 = quad_sum4(Wss * v1, Wss * v2, t2 * Wss, 0.0, c);
    const double g11 = lane_val(q1, base, 0), g12 = lane_val(q1, base, 1), g22 = lane_val(q1, base, 2);
    const double eps = cf.hreg * (g11 + g22);
    const double G11 = g11 + eps, G12 = g12, G22 = g22 + eps;
    const double idet = 1.0 / (G11 * G22 - G12 * G12);
    double yv[4];
    {
        const double P4 = lane_val(q1, base, 3), P6 = lane_val(q5, base, 2), P3 = lane_val(q3, base, 2);
        const double j1 = lane_val(q2, base, r), j2 = lane_val(q2, base, 2 + r);
        const double Ls = lane_val(q4, base, 2 + r), Ss = lane_val(q5, base, r);
        const double e11 = flip(2.0 * lane_val(q3, base, d), d);
        const double e12 = flip(lane_val(q3, base, 1 + 2 * d) + (d ? P4 : P3), d);
        const double e22 = flip(2.0 * (d ? P6 : P4), d);
        const double te = cf.hreg * (e11 + e22);
        const double E11 = e11 + te, E22 = e22 + te;
        const double y1 = (G22 * j1 - G12 * j2) * idet, y2 = (G11 * j2 - G12 * j1) * idet;
        const double a1 = flip(lane_val(q4, base, r + 2 * d), d) - (E11 * y1 + e12 * y2);
        const double a2 = flip(d ? Ss : Ls, d) - (e12 * y1 + E22 * y2);
        yv[0] = y1;
        yv[1] = y2;
        yv[2] = (G22 * a1 - G12 * a2) * idet;
        yv[3] = (G11 * a2 - G12 * a1) * idet;
    }
    double n[2], nt[2], ns[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const double v = r == 0 ? v1 : v2;
        const double y1 = lane_val(yv[0], base, r), y2 = lane_val(yv[1], base, r);
        const double dt1 = lane_val(yv[2], base, r), dt2 = lane_val(yv[3], base, r);
        const double ds1 = lane_val(yv[2], base, 2 + r), ds2 = lane_val(yv[3], base, 2 + r);
        n[r] = v - t1 * y1 - t2 * y2;
        nt[r] = -(Wtt * y1 + Wts * y2) - (t1 * dt1 + t2 * dt2);
        ns[r] = (Wts * y1 + Wss * y2) - (t1 * ds1 + t2 * ds2);
    }

    // ---- W_B, f and the row of Df this lane owns
    const double h = sp.h_amp;
    const double H = h * (sh1 * n[0] + sh2 * n[1]);
    const double Ht = h * (sp.P * ch1 * n[0] + sh1 * nt[0] + sh2 * nt[1]);
    const double Hs = h * (sh1 * ns[0] + cf.qpi * ch2 * n[1] + sh2 * ns[1]);
    const double fc = WA - (SB + H);
    double m[4] = {WAt, WAs, -(SBt + Ht), -(-SBs + Hs)};

    const double f2 = quad_sum(fc * fc);
    // product of the squared column norms
    const double qn = quad_sum4(m[0] * m[0], m[1] * m[1], m[2] * m[2], m[3] * m[3], c);
    const double cn2 = lane_val(qn, base, 0) * lane_val(qn, base, 1) * lane_val(qn, base, 2) * lane_val(qn, base, 3);
    int fin = max(max(exponent(fc), exponent(m[0])), max(exponent(m[1]), max(exponent(m[2]), exponent(m[3])))) < 0x7ff;
    fin &= __shfl_xor_sync(kFull, fin, 1);
    fin &= __shfl_xor_sync(kFull, fin, 2);

    // ---- Df dx = f by partial-pivot elimination over the quad's rows
    double rr = fc, det = 1.0, ip[4];
    int used = 0, pl[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        long long cand = ((used >> c) & 1) ? -1LL : abs_bits(m[j]);
        int bl = c;
#pragma unroll
        for (int off = 1; off <= 2; off <<= 1) {
            const long long oc = __shfl_xor_sync(kFull, cand, off);
            const int ol = __shfl_xor_sync(kFull, bl, off);
            if (oc > cand || (oc == cand && ol < bl)) {
                cand = oc;
                bl = ol;
            }
        }
        used |= 1 << bl;
        pl[j] = bl;
        double pj[4];
#pragma unroll
        for (int q = j; q < 4; ++q) pj[q] = lane_val(m[q], base, bl);
        const double prr = lane_val(rr, base, bl);
        det *= pj[j];
        ip[j] = cand != 0 ? 1.0 / pj[j] : 0.0;
        if (j < 3 && !((used >> c) & 1)) {
            const double fct = m[j] * ip[j];
#pragma unroll
            for (int q = j + 1; q < 4; ++q) m[q] -= fct * pj[q];
            rr -= fct * prr;
        }
    }
    bool odd = false;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int w = u + 1; w < 4; ++w) odd ^= pl[u] > pl[w];
    det = flip(det, odd);
    double dx[4];
#pragma unroll
    for (int j = 3; j >= 0; --j) {
        double v = rr;
#pragma unroll
        for (int q = j + 1; q < 4; ++q) v -= m[q] * dx[q];
        dx[j] = lane_val(v * ip[j], base, pl[j]);
    }

    E.pre = pre;
    E.fin = fin;
    E.r2 = f2;
    E.cn2 = cn2;
    E.det = det;
#pragma unroll
    for (int q = 0; q < 4; ++q) E.dx[q] = dx[q];
}

// |det| >= rho_min sqrt(cn2), out of line: only near the threshold
__device__ __noinline__ bool above_rho_min(double det, double rho_min, double cn2) {
    return fabs(det) >= rho_min * sqrt(cn2);
}

// The decision of Eq. (dampedNewtonEquation)'s iteration k from an evaluation:
// -1 to update, else the stop status (taken on the quad's first lane).
__device__ __forceinline__ int decide(const Eval &E, const tms_refine_params &pr, const Stop &stop, int k,
                                      int base) {
    // ||f|| <= tol as ||f||^2 <= tol^2; |det| / prod ||col|| >= rho_min as
    // |det| >= rho_min sqrt(prod ||col||^2), decided by the exponents alone (|det| >=
    // 2^(ed - 1023), rho_min < 2^(er - 1022), cn2 < 2^(ec - 1022)) where they do
    int dec = E.pre;
    if (dec < 0) {
        const int ed = exponent(E.det), er = exponent(pr.rho_min), ec = exponent(E.cn2);
        const bool clear = ed > 0 && ed < 0x7ff && er < 0x7ff && ec < 0x7ff && 2 * ed + 1020 >= 2 * er + ec;
        if (!E.fin) dec = TMS_REFINE_NON_FINITE;
        else if (__double_as_longlong(E.r2) <= stop.tol2) dec = TMS_REFINE_CONVERGED;
        else if (k == pr.max_iter) dec = TMS_REFINE_MAX_ITER;
        else if (!clear && !above_rho_min(E.det, pr.rho_min, E.cn2)) dec = TMS_REFINE_SINGULAR;
    }
    return __shfl_sync(kFull, dec, base);
}

// Applies a decision to a quad that is still iterating (every lane of the warp calls
// it: lane c updates x_c).
__device__ __forceinline__ void apply(const Eval &E, const tms_refine_params &pr, const Stop &stop, int dec,
                                      int k, Solve &S, int c, int base) {
    const double al = __double_as_longlong(E.r2) > stop.sw2 ? pr.alpha0 : pr.alpha1;
    const double own = c == 0 ? S.x0 : c == 1 ? S.x1 : c == 2 ? S.x2 : S.x3;
    const double nx = own - al * (c == 0 ? E.dx[0] : c == 1 ? E.dx[1] : c == 2 ? E.dx[2] : E.dx[3]);
    const double n0 = lane_val(nx, base, 0), n1 = lane_val(nx, base, 1);
    const double n2 = lane_val(nx, base, 2), n3 = lane_val(nx, base, 3);
    if (S.code >= 0) return;
    if (E.pre < 0) {
        S.fn = E.r2;
        S.rh = E.det;
        S.rc2 = E.cn2;
    }
    if (dec >= 0) {
        S.code = dec;
        S.iters = k;
    } else {
        S.x0 = n0;
        S.x1 = n1;
        S.x2 = n2;
        S.x3 = n3;
        S.k = k + 1;
    }
}

// The whole solve for every quad of the warp at once (the refinement): the
// iteration counter is the warp's; at most max_iter + 1 evaluations each.
__device__ __forceinline__ void newton_solve(const Coef &cf, const tms_surface_pair &sp,
                                             const tms_refine_params &pr, Solve &S, int c,
                                             int base) {
    const double lnlam = sp.stretch ? log(sp.lam) : 0.0;
    const Stop stop = make_stop(pr);
    for (int k = 0; __any_sync(kFull, S.code < 0); ++k) {
        Eval E;
        evaluate<0>(cf, nullptr, sp, stop, lnlam, S.x0, S.x1, S.x2, S.x3, c, base, E);
        apply(E, pr, stop, decide(E, pr, stop, k, base), k, S, c, base);
    }
}

// One iteration for each quad at its own count S.k (the continuation).
template <int WALK>
__device__ __forceinline__ void newton_iter(const Coef &cf, const WalkCoef *wc, const tms_surface_pair &sp,
                                            const tms_refine_params &pr, const Stop &stop, double lnlam,
                                            Solve &S, int c, int base) {
    Eval E;
    evaluate<WALK>(cf, wc, sp, stop, lnlam, S.x0, S.x1, S.x2, S.x3, c, base, E);
    apply(E, pr, stop, decide(E, pr, stop, S.k, base), S.k, S, c, base);
}

// the walking sheet's coefficients at the quad's parameter (lane c its column c)
template <int WALK>
__device__ __forceinline__ void fill_walk(const Coef &cf, WalkCoef &wc, int K, double aw, int c) {
    const int lane = threadIdx.x & 31;
    for (int h = 0; h < K; ++h) {
        wc.v[h][0][lane] = fma(aw, cf.dak[h][c], WALK == 1 ? cf.uak[h][c] : cf.sak[h][c]);
        wc.v[h][1][lane] = fma(aw, cf.dbk[h][c], WALK == 1 ? cf.ubk[h][c] : cf.sbk[h][c]);
        wc.v[h][2][lane] = fma(aw, cf.dna[h][c], WALK == 1 ? cf.una[h][c] : cf.sna[h][c]);
        wc.v[h][3][lane] = fma(aw, cf.db[h][c], WALK == 1 ? cf.ub[h][c] : cf.sb[h][c]);
    }
}

__device__ __noinline__ double wrap_far(double v) { return fmod(v, kTwoPi); }

// v modulo 2 pi in [0, 2 pi] (fmod, which leaves |v| < 2 pi as it is)
__device__ __forceinline__ double wrap_angle(double v) {
    double w = v;
    if (abs_bits(v) >= __double_as_longlong(kTwoPi)) w = wrap_far(v);
    const long long b = __double_as_longlong(w);
    if (b == (long long)(1ULL << 63)) w = 0.0;   // +0 for a -0 remainder
    else if (b < 0) w += kTwoPi;
    return w;
}

__device__ __forceinline__ double nan_value() { return __longlong_as_double(0x7ff8000000000000LL); }

__global__ void __launch_bounds__(kThreads) k_refine(const __grid_constant__ RefineArgs a) {
    __shared__ Coef cf;
    const tms_surface_pair &sp = a.sp;
    const int t = threadIdx.x;
    build_tables(cf, sp, sp.alpha_u, sp.alpha_s, 0, t, kThreads);
    __syncthreads();

    const int lane = t & 31;
    const int c = lane & 3;
    const int base = lane & ~3;
    const long long i = (long long)blockIdx.x * kSeedsPerBlock + (t >> 2);
    const bool live = i < a.n;
    Solve S;
    S.x0 = 0.0;
    S.x1 = 0.5;
    S.x2 = 0.0;
    S.x3 = 0.5;
    if (live) {
        const double *s = a.x0 + i * a.ld;
        S.x0 = s[0];
        S.x1 = s[1];
        S.x2 = s[2];
        S.x3 = s[3];
    }
    S.code = live ? -1 : TMS_REFINE_CONVERGED;
    S.iters = 0;
    S.k = 0;
    S.fn = nan_value();
    S.rh = S.fn;
    S.rc2 = 1.0;
    newton_solve(cf, sp, a.p, S, c, base);

    if (live) {
        double xc = c == 0 ? S.x0 : c == 1 ? S.x1 : c == 2 ? S.x2 : S.x3;
        if (c == 0 || c == 2) xc = wrap_angle(xc);
        a.x[i * 4 + c] = xc;
        if (c == 0) {
            if (a.fnorm) a.fnorm[i] = sqrt(S.fn);
            if (a.rho) a.rho[i] = S.rh / sqrt(S.rc2);
            if (a.iters) a.iters[i] = S.iters;
            if (a.status) a.status[i] = S.code;
        }
    }
}

// Continuation (Sec. 8): one quad per branch walks the parameter values
// alpha_0 (the pair's own), alphas[0..steps) of the walking sheet (WALK = 1:
// W_A's alpha_u, 2: B's alpha_s).  The branches of a warp do not wait for one
// another between steps: each quad evaluates its sheet at its own current
// parameter (the coefficients are affine in it), and when its corrector stops
// it records the step and, unless the branch stopped, predicts the next step
// and goes on in the same warp-wide iteration loop, which ends when all of the
// warp's branches have.
template <int WALK>
__global__ void __launch_bounds__(kThreads) k_continue(const __grid_constant__ ContArgs a) {
    __shared__ Coef cf;
    __shared__ WalkCoef wc;
    const tms_surface_pair &sp = a.sp;
    const tms_continue_params &cp = a.p;
    const int t = threadIdx.x;
    build_tables(cf, sp, WALK == 1 ? 0.0 : sp.alpha_u, WALK == 2 ? 0.0 : sp.alpha_s, WALK, t,
                 kThreads);
    __syncthreads();
    const int lane = t & 31;
    const int c = lane & 3;
    const int base = lane & ~3;
    const long long i = (long long)blockIdx.x * kSeedsPerBlock + (t >> 2);
    const bool live = i < a.n;
    const bool angle = !(c & 1);
    double g = angle ? 0.0 : 0.5;         // lane c's coordinate of the current step's start
    if (live) g = a.x0[i * a.ld + c];
    double p1 = 0.0, p2 = 0.0;            // of x_{j-1}, x_{j-2}
    bool alive = live;
    int j = 0;
    double rho_prev = nan_value();
    const double a0 = WALK == 1 ? sp.alpha_u : sp.alpha_s;
    double aj = a0, am1 = a0, am2 = a0;   // alpha_j, alpha_{j-1}, alpha_{j-2}
    const long long K1 = (long long)a.steps + 1;
    Solve S;
    S.x0 = lane_val(g, base, 0);
    S.x1 = lane_val(g, base, 1);
    S.x2 = lane_val(g, base, 2);
    S.x3 = lane_val(g, base, 3);
    S.code = alive ? -1 : TMS_REFINE_CONVERGED;
    S.iters = 0;
    S.k = 0;
    S.fn = nan_value();
    S.rh = S.fn;
    S.rc2 = 1.0;
    const double lnlam = sp.stretch ? log(sp.lam) : 0.0;
    const Stop stop = make_stop(cp.corrector);
    fill_walk<WALK>(cf, wc, sp.n_harmonics, aj, c);
    while (__any_sync(kFull, alive)) {
        newton_iter<WALK>(cf, &wc, sp, cp.corrector, stop, lnlam, S, c, base);
        if (!(alive && S.code >= 0)) continue;
        // ---- step j is done: of one quad, as a rule, with the warp's others waiting, so
        // lane c takes coordinate c, and the square roots and quotients are taken by
        // different lanes at once (all of them on every lane: 19.4 ms for 12,000 branches
        // of 50 steps; so 17.9)
        const unsigned quad = 0xFu << base;
        const double own = c == 0 ? S.x0 : c == 1 ? S.x1 : c == 2 ? S.x2 : S.x3;
        const double xs = angle ? wrap_angle(own) : own;
        const double root = sqrt(c == 3 ? S.rc2 : S.fn);
        double moved = fabs(xs - g);
        const double q1 = (c == 3 ? S.rh : moved) / (c == 3 ? root : kTwoPi);
        const double rho = __shfl_sync(quad, q1, base + 3);
        if (angle) moved = fabs(moved - kTwoPi * rint(q1));
        long long jump = abs_bits(moved);
        jump = max(jump, __shfl_xor_sync(quad, jump, 1));
        jump = max(jump, __shfl_xor_sync(quad, jump, 2));
        int st = S.code;
        if (st == TMS_REFINE_CONVERGED) {
            // (the thresholds are not negative, so their bits are ordered as they are)
            const long long size = abs_bits(rho), inf = 0x7ff0000000000000LL;
            const bool up = __double_as_longlong(rho) > 0, was_up = __double_as_longlong(rho_prev) > 0;
            if (jump > __double_as_longlong(cp.max_jump)) st = TMS_CONT_JUMPED;
            else if (size > inf || size < __double_as_longlong(cp.rho_turn)) st = TMS_CONT_TURNING;
            else if (j > 0 && up != was_up) st = TMS_CONT_TURNING;
        }
        const long long o = i * K1 + j;
        a.x[o * 4 + c] = xs;
        if (c == 0) {
            a.status[o] = st;
            if (a.iters) a.iters[o] = S.iters;
            if (a.rho) a.rho[o] = rho;
            if (a.fnorm) a.fnorm[o] = root;
        }
        p2 = p1;
        p1 = xs;
        rho_prev = rho;
        if (st != TMS_REFINE_CONVERGED || j == a.steps) {
            alive = false;
            for (long long r = j + 1; r <= a.steps; ++r) {
                const long long oo = i * K1 + r;
                a.x[oo * 4 + c] = nan_value();
                if (c == 0) {
                    a.status[oo] = TMS_CONT_STOPPED;
                    if (a.iters) a.iters[oo] = 0;
                    if (a.rho) a.rho[oo] = nan_value();
                    if (a.fnorm) a.fnorm[oo] = nan_value();
                }
            }
            continue;
        }
        // ---- next step: predictor, Eq. (predictor); angle differences on the circle
        ++j;
        am2 = am1;
        am1 = aj;
        aj = a.alphas[j - 1];
        fill_walk<WALK>(cf, wc, sp.n_harmonics, aj, c);
        g = p1;
        if (j > 1) {
            double d = p1 - p2;
            const double q2 = (c == 1 ? aj - am1 : d) / (c == 1 ? am1 - am2 : kTwoPi);
            const double ratio = __shfl_sync(quad, q2, base + 1);
            if (angle) d -= kTwoPi * rint(q2);
            g = p1 + ratio * d;
        }
        S.x0 = __shfl_sync(quad, g, base);
        S.x1 = __shfl_sync(quad, g, base + 1);
        S.x2 = __shfl_sync(quad, g, base + 2);
        S.x3 = __shfl_sync(quad, g, base + 3);
        S.code = -1;
        S.iters = 0;
        S.k = 0;
        S.fn = nan_value();
        S.rh = S.fn;
        S.rc2 = 1.0;
    }
}

bool all_finite(const double *v, size_t n) {
    for (size_t j = 0; j < n; ++j)
        if (!isfinite(v[j])) return false;
    return true;
}

bool is_device_ptr(const void *p) {
    cudaPointerAttributes at;
    cudaError_t e = cudaPointerGetAttributes(&at, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

tms_status arg_error(const char *msg) {
    tms::set_last_error(msg);
    return TMS_ERR_ARG;
}


tms_status check_surface(const tms_surface_pair &s, const char *who) {
    const std::string w(who);
    if (s.n_harmonics < 1 || s.n_harmonics > TMS_SURF_MAX_HARMONICS)
        return arg_error((w + ": n_harmonics outside 1..8").c_str());
    if (s.n_folds < 0 || s.n_folds > TMS_SURF_MAX_FOLDS)
        return arg_error((w + ": n_folds outside 0..4").c_str());
    if (s.stretch != 0 && s.stretch != 1) return arg_error((w + ": stretch must be 0 or 1").c_str());
    if (s.stretch == 1 && !(s.lam > 0.0)) return arg_error((w + ": lam must be > 0").c_str());
    bool fin = true;
    for (int h = 0; h < s.n_harmonics; ++h)
        fin = fin && all_finite(s.ca[h], 4) && all_finite(s.cb[h], 4) && all_finite(s.dca[h], 4) &&
              all_finite(s.dcb[h], 4);
    for (int f = 0; f < s.n_folds; ++f)
        fin = fin && isfinite(s.fold_amp[f]) && all_finite(s.fold_root[f], 3) &&
              all_finite(s.fold_dir[f], 4);
    const size_t ns = (sizeof(tms_surface_pair) - offsetof(tms_surface_pair, c0)) / sizeof(double);
    fin = fin && isfinite(s.alpha_u) && isfinite(s.alpha_s) && isfinite(s.alpha_ref) &&
          (s.stretch == 0 || isfinite(s.lam)) && all_finite(&s.c0, ns);
    if (!fin) return arg_error((w + ": non-finite surface value").c_str());
    if (!(s.reg >= 0.0)) return arg_error((w + ": reg must be >= 0").c_str());
    return TMS_OK;
}

tms_status check_corrector(const tms_refine_params &p, const char *who) {
    const std::string w(who);
    if (!(p.alpha0 > 0.0 && p.alpha0 <= 1.0 && p.alpha1 > 0.0 && p.alpha1 <= 1.0))
        return arg_error((w + ": alpha0 and alpha1 must lie in (0, 1]").c_str());
    if (!(p.tol >= 0.0) || !(p.switch_below >= 0.0) || !(p.rho_min >= 0.0))
        return arg_error((w + ": tol, switch_below and rho_min must be >= 0").c_str());
    if (!(p.s_lo < p.s_hi)) return arg_error((w + ": need s_lo < s_hi").c_str());
    if (p.max_iter < 0 || p.max_iter > 1000000)
        return arg_error((w + ": max_iter outside 0..1000000").c_str());
    return TMS_OK;
}

}  // namespace

extern "C" void tms_refine_params_default(tms_refine_params *p) {
    if (!p) return;
    p->alpha0 = 0.5;
    p->alpha1 = 0.5;
    p->switch_below = 0.0;
    p->tol = 1e-10;
    p->s_lo = -0.5;
    p->s_hi = 1.5;
    p->rho_min = 1e-14;
    p->max_iter = 200;
    p->pad = 0;
}

extern "C" tms_status tms_refine(const tms_surface_pair *surf, const tms_refine_params *params,
                                 const double *dX0, long long ldx0, long long n, double *dX,
                                 double *dFnorm, double *dRho, int32_t *dIters, int32_t *dStatus,
                                 void *stream) {
    if (!surf) return arg_error("tms_refine: surface is NULL");
    if (n < 0) return arg_error("tms_refine: n < 0");
    tms_refine_params p;
    if (params) p = *params;
    else tms_refine_params_default(&p);
    tms_status st = check_surface(*surf, "tms_refine");
    if (st == TMS_OK) st = check_corrector(p, "tms_refine");
    if (st != TMS_OK) return st;
    if (n == 0) return TMS_OK;
    if (ldx0 < 4) return arg_error("tms_refine: ldx0 < 4");
    if (!dX0 || !dX || !is_device_ptr(dX0) || !is_device_ptr(dX))
        return arg_error("tms_refine: seeds and output must be device pointers");
    if (dX == dX0 && ldx0 != 4) return arg_error("tms_refine: in place needs ldx0 == 4");
    RefineArgs a;
    a.sp = *surf;
    a.p = p;
    a.x0 = dX0;
    a.ld = ldx0;
    a.n = n;
    a.x = dX;
    a.fnorm = dFnorm;
    a.rho = dRho;
    a.iters = dIters;
    a.status = dStatus;
    const long long blocks = (n + kSeedsPerBlock - 1) / kSeedsPerBlock;
    if (blocks > 0x7fffffffLL) return arg_error("tms_refine: too many seeds");
    k_refine<<<(unsigned)blocks, kThreads, 0, (cudaStream_t)stream>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        tms::set_last_error(std::string("tms_refine launch: ") + cudaGetErrorString(e));
        return TMS_ERR_CUDA;
    }
    return TMS_OK;
}

extern "C" void tms_continue_params_default(tms_continue_params *p) {
    if (!p) return;
    tms_refine_params_default(&p->corrector);
    p->rho_turn = 1e-8;
    p->max_jump = 0.25;
    p->param = 0;
    p->pad = 0;
}

extern "C" tms_status tms_continue(const tms_surface_pair *surf, const tms_continue_params *params,
                                   const double *dAlphas, int nSteps, const double *dX0,
                                   long long ldx0, long long n, double *dX, int32_t *dStatus,
                                   int32_t *dIters, double *dRho, double *dFnorm, void *stream) {
    if (!surf) return arg_error("tms_continue: surface is NULL");
    if (n < 0) return arg_error("tms_continue: n < 0");
    if (nSteps < 0) return arg_error("tms_continue: nSteps < 0");
    tms_continue_params p;
    if (params) p = *params;
    else tms_continue_params_default(&p);
    tms_status st = check_surface(*surf, "tms_continue");
    if (st == TMS_OK) st = check_corrector(p.corrector, "tms_continue");
    if (st != TMS_OK) return st;
    if (p.param != 0 && p.param != 1) return arg_error("tms_continue: param must be 0 or 1");
    if (!(p.rho_turn >= 0.0)) return arg_error("tms_continue: rho_turn must be >= 0");
    if (!(p.max_jump > 0.0)) return arg_error("tms_continue: max_jump must be > 0");
    if (n == 0) return TMS_OK;
    if (ldx0 < 4) return arg_error("tms_continue: ldx0 < 4");
    if (!dX0 || !dX || !dStatus || !is_device_ptr(dX0) || !is_device_ptr(dX) ||
        !is_device_ptr(dStatus))
        return arg_error("tms_continue: seeds, dX and dStatus must be device pointers");
    if (nSteps > 0 && (!dAlphas || !is_device_ptr(dAlphas)))
        return arg_error("tms_continue: dAlphas must be a device pointer");
    ContArgs a;
    a.sp = *surf;
    a.p = p;
    a.alphas = dAlphas;
    a.steps = nSteps;
    a.x0 = dX0;
    a.ld = ldx0;
    a.n = n;
    a.x = dX;
    a.status = dStatus;
    a.iters = dIters;
    a.rho = dRho;
    a.fnorm = dFnorm;
    const long long blocks = (n + kSeedsPerBlock - 1) / kSeedsPerBlock;
    if (blocks > 0x7fffffffLL) return arg_error("tms_continue: too many branches");
    if (p.param == 0) k_continue<1><<<(unsigned)blocks, kThreads, 0, (cudaStream_t)stream>>>(a);
    else k_continue<2><<<(unsigned)blocks, kThreads, 0, (cudaStream_t)stream>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        tms::set_last_error(std::string("tms_continue launch: ") + cudaGetErrorString(e));
        return TMS_ERR_CUDA;
    }
    return TMS_OK;
}
