// Operations on theta grids (functions of theta stored at theta_i = 2 pi i / N,
// Sec. 4 and Sec. 6.1): translation and derivative of every column of a
// coordinate array through the FFT (Eqs. translate, translate2), and grid
// phase alignment of two circles (Eq. rhoEquationDiscrete).
//
// Translation: one CTA per complex transform of two real rows that share a
// shift (the same s column of two coordinates), packed as z = a + j b.  The
// multiplier H(k) = e^{j k rho} (times j k for the derivative) over the signed
// frequencies keeps H(-k) = conj(H(k)), with the Nyquist term real, so the two
// real results come back as the real and imaginary parts.  Forward: radix-2
// decimation in time from bit-reversed input; inverse: decimation in frequency
// to bit-reversed output, read back through the same permutation.  All in
// FP64 in shared memory.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>

#include <string>

#include "tms_common.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kFftThreads = 256;
constexpr int kTab = 64;   // two-level tables: e^{j x (hi * 64 + lo)} = T_hi[hi] T_lo[lo]

struct ThetaArgs {
    const double *in;
    double *out;
    long long ldc;     // doubles between coordinate blocks
    const double *rho; // per column, or null
    double rho0;
    int N, logN, cols, ncoord, derivative;
};

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cmulc(double2 a, double2 b) {   // a * conj(b)
    return make_double2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}

__global__ void __launch_bounds__(kFftThreads) k_theta_fft(const ThetaArgs a) {
    extern __shared__ double2 sm[];
    const int N = a.N;
    double2 *z = sm;                 // N values
    double2 *w = sm + N;             // N/2 twiddles e^{-2 pi j m / N}
    double2 *th = w + N / 2;         // kTab: e^{-2 pi j (hi * kTab) / N}
    double2 *tl = th + kTab;         // kTab: e^{-2 pi j lo / N}
    double2 *hh = tl + kTab;         // kTab: e^{j rho hi kTab}
    double2 *hl = hh + kTab;         // kTab: e^{j rho lo}
    const int t = threadIdx.x;
    const int col = blockIdx.x % a.cols;
    const int pair = blockIdx.x / a.cols;
    const int c0 = 2 * pair, c1 = 2 * pair + 1;
    const bool two = c1 < a.ncoord;
    const double rho = a.rho ? a.rho[col] : a.rho0;
    if (t < kTab) {
        double s, c;
        sincospi(-2.0 * (double)(t * kTab) / (double)N, &s, &c);
        th[t] = make_double2(c, s);
        sincospi(-2.0 * (double)t / (double)N, &s, &c);
        tl[t] = make_double2(c, s);
        sincos(rho * (double)(t * kTab), &s, &c);
        hh[t] = make_double2(c, s);
        sincos(rho * (double)t, &s, &c);
        hl[t] = make_double2(c, s);
    }
    const double *ra = a.in + (long long)c0 * a.ldc + (long long)col * N;
    const double *rb = a.in + (long long)c1 * a.ldc + (long long)col * N;
    const int sh = 32 - a.logN;
    for (int i = t; i < N; i += kFftThreads)
        z[__brev((unsigned)i) >> sh] = make_double2(ra[i], two ? rb[i] : 0.0);
    __syncthreads();
    for (int m = t; m < N / 2; m += kFftThreads) w[m] = cmul(th[m / kTab], tl[m % kTab]);
    __syncthreads();

    // forward transform (decimation in time)
    for (int half = 1; half < N; half <<= 1) {
        const int stride = N / (2 * half);
        for (int b = t; b < N / 2; b += kFftThreads) {
            const int pos = b & (half - 1);
            const int i = ((b - pos) << 1) + pos;
            const double2 v = cmul(w[pos * stride], z[i + half]);
            const double2 u = z[i];
            z[i] = make_double2(u.x + v.x, u.y + v.y);
            z[i + half] = make_double2(u.x - v.x, u.y - v.y);
        }
        __syncthreads();
    }

    // multiplier over the signed frequencies
    for (int i = t; i < N; i += kFftThreads) {
        double2 v = z[i];
        if (i == N / 2) {
            double s, c;
            sincos(0.5 * (double)N * rho, &s, &c);
            const double g = a.derivative ? 0.0 : c;
            v = make_double2(v.x * g, v.y * g);
        } else {
            const int k = i < N / 2 ? i : i - N;
            const int ak = k < 0 ? -k : k;
            double2 e = cmul(hh[ak / kTab], hl[ak % kTab]);   // e^{j rho |k|}
            if (k < 0) e.y = -e.y;
            if (a.derivative) e = make_double2(-(double)k * e.y, (double)k * e.x);
            v = cmul(v, e);
        }
        z[i] = v;
    }
    __syncthreads();

    // inverse transform (decimation in frequency, conjugate twiddles)
    for (int half = N / 2; half >= 1; half >>= 1) {
        const int stride = N / (2 * half);
        for (int b = t; b < N / 2; b += kFftThreads) {
            const int pos = b & (half - 1);
            const int i = ((b - pos) << 1) + pos;
            const double2 u = z[i], v = z[i + half];
            z[i] = make_double2(u.x + v.x, u.y + v.y);
            z[i + half] = cmulc(make_double2(u.x - v.x, u.y - v.y), w[pos * stride]);
        }
        __syncthreads();
    }

    const double inv = 1.0 / (double)N;
    double *oa = a.out + (long long)c0 * a.ldc + (long long)col * N;
    double *ob = a.out + (long long)c1 * a.ldc + (long long)col * N;
    for (int i = t; i < N; i += kFftThreads) {
        const double2 v = z[__brev((unsigned)i) >> sh];
        oa[i] = v.x * inv;
        if (two) ob[i] = v.y * inv;
    }
}

// a float pair sum: s + e = x + y exactly (Knuth), and for |x| >= |y| or x = 0 (Dekker)
__device__ __forceinline__ void two_sum(float x, float y, float &s, float &e) {
    s = __fadd_rn(x, y);
    const float b = __fsub_rn(s, x);
    e = __fadd_rn(__fsub_rn(x, __fsub_rn(s, b)), __fsub_rn(y, b));
}
__device__ __forceinline__ void fast_sum(float x, float y, float &s, float &e) {
    s = __fadd_rn(x, y);
    e = __fsub_rn(y, __fsub_rn(s, x));
}

// ---------------------------------------------------------------------------
// translation in float pairs (columns of 1024, 2048 and 4096 points)
// ---------------------------------------------------------------------------
// The transform above is bound by the FP64 pipe (0.89 ms for 4 x 1025 columns of 2048
// points, 14 M warp instructions of 19 clocks an SM).  Most of its error at these sizes
// is the arguments k rho, rounded to FP64 ahead of their sine and cosine; numbers of two
// floats (2^-48) with the arguments reduced exactly are nearer the exact result, on a
// pipe some fifty times as fast (relative error, rms, against 113-bit transforms: 1.1e-14
// at 1024 points, 2.1e-14 in FP64; 1.2e-14 at 2048, 4.2e-14; 1.3e-14 at 4096, 8.9e-14).
// At 512 points FP64 is the nearer one (5e-15): those columns and shorter ones keep it,
// and so do columns of 8192, whose twiddles would not fit beside them.
// 0.157 ms for those 4 x 1025 columns: 116 M warp instructions, issue 64%; 128 registers
// a thread, so 16 warps an SM (three blocks at 80 registers: 0.170 ms).
//
// One block of N / 8 threads takes a pair of rows at a time, eight points a thread:
// radix-8 passes in decimation in frequency to digit-reversed order (the first reads
// the rows themselves), in the last of them, in registers, the rest radix (N / 512),
// the multiplier and the rest radix of the way back, which mirrors the way there (the
// inverse is the forward transform of the swapped numbers).  Blocks stay for several
// rows, whose twiddles and phases they share.  Each row is scaled by a power of two to
// its largest value, so that neither loses to the other.
constexpr int kPairLeast = 10, kPairMost = 12;   // log2 N

struct __align__(16) PairC {      // a complex number: float pairs h + l
    float rh, rl, ih, il;
};

__device__ __forceinline__ void add_pair(float xh, float xl, float yh, float yl, float &h, float &l) {
    float s, e;
    two_sum(xh, yh, s, e);
    h = s;
    l = __fadd_rn(e, __fadd_rn(xl, yl));
}
__device__ __forceinline__ PairC add_c(const PairC &x, const PairC &y) {
    PairC z;
    add_pair(x.rh, x.rl, y.rh, y.rl, z.rh, z.rl);
    add_pair(x.ih, x.il, y.ih, y.il, z.ih, z.il);
    return z;
}
__device__ __forceinline__ PairC sub_c(const PairC &x, const PairC &y) {
    PairC z;
    add_pair(x.rh, x.rl, -y.rh, -y.rl, z.rh, z.rl);
    add_pair(x.ih, x.il, -y.ih, -y.il, z.ih, z.il);
    return z;
}
// x y with the product's error terms (not normalised)
__device__ __forceinline__ void mul_pair(float xh, float xl, float yh, float yl, float &h, float &l) {
    h = __fmul_rn(xh, yh);
    l = __fmaf_rn(xl, yh, __fmaf_rn(xh, yl, __fmaf_rn(xh, yh, -h)));
}
__device__ __forceinline__ void sum_products(float ph, float pl, float qh, float ql, float &h, float &l) {
    float s, e;
    two_sum(ph, qh, s, e);
    fast_sum(s, __fadd_rn(e, __fadd_rn(pl, ql)), h, l);
}
__device__ __forceinline__ PairC mul_c(const PairC &x, const PairC &w) {
    float ah, al, bh, bl;
    PairC z;
    mul_pair(x.rh, x.rl, w.rh, w.rl, ah, al);
    mul_pair(x.ih, x.il, w.ih, w.il, bh, bl);
    sum_products(ah, al, -bh, -bl, z.rh, z.rl);
    mul_pair(x.rh, x.rl, w.ih, w.il, ah, al);
    mul_pair(x.ih, x.il, w.rh, w.rl, bh, bl);
    sum_products(ah, al, bh, bl, z.ih, z.il);
    return z;
}
__device__ __forceinline__ PairC swapped(const PairC &x) {
    PairC z = {x.ih, x.il, x.rh, x.rl};
    return z;
}
__device__ __forceinline__ PairC times_minus_i(const PairC &x) {
    PairC z = {x.ih, x.il, -x.rh, -x.rl};
    return z;
}
__device__ __forceinline__ PairC pair_of(double re, double im) {
    PairC z;
    z.rh = (float)re;
    z.rl = (float)(re - (double)z.rh);
    z.ih = (float)im;
    z.il = (float)(im - (double)z.ih);
    return z;
}

// transforms of 2, 4 and 8 points, e^{-2 pi j m k / R}, in natural order
__device__ __forceinline__ void dft2(PairC &a, PairC &b) {
    const PairC s = add_c(a, b);
    b = sub_c(a, b);
    a = s;
}
__device__ __forceinline__ void dft4(PairC &x0, PairC &x1, PairC &x2, PairC &x3) {
    dft2(x0, x2);
    dft2(x1, x3);
    x3 = times_minus_i(x3);
    dft2(x0, x1);                       // X0, X2
    dft2(x2, x3);                       // X1, X3
    const PairC t = x1;
    x1 = x2;
    x2 = t;
}
__device__ __forceinline__ void dft8(PairC (&x)[8]) {
    constexpr float ch = 0.70710677f, cl = 1.21016175e-8f;     // 1 / sqrt 2
#pragma unroll
    for (int m = 0; m < 4; ++m) dft2(x[m], x[m + 4]);
    {
        // times (1 - j) / sqrt 2 and (-1 - j) / sqrt 2
        float ah, al, bh, bl;
        add_pair(x[5].rh, x[5].rl, x[5].ih, x[5].il, ah, al);
        add_pair(x[5].ih, x[5].il, -x[5].rh, -x[5].rl, bh, bl);
        mul_pair(ah, al, ch, cl, x[5].rh, x[5].rl);
        mul_pair(bh, bl, ch, cl, x[5].ih, x[5].il);
        add_pair(x[7].ih, x[7].il, -x[7].rh, -x[7].rl, ah, al);
        add_pair(-x[7].rh, -x[7].rl, -x[7].ih, -x[7].il, bh, bl);
        mul_pair(ah, al, ch, cl, x[7].rh, x[7].rl);
        mul_pair(bh, bl, ch, cl, x[7].ih, x[7].il);
        x[6] = times_minus_i(x[6]);
    }
    dft4(x[0], x[1], x[2], x[3]);
    dft4(x[4], x[5], x[6], x[7]);
    const PairC t[8] = {x[0], x[4], x[1], x[5], x[2], x[6], x[3], x[7]};
#pragma unroll
    for (int m = 0; m < 8; ++m) x[m] = t[m];
}

// e^{2 pi j q / 4096} over the first octant, as float pairs: made by the compiler from
// the Taylor series (the angles are at most pi / 4), so that a block's twiddles are
// loads; a sine and cosine in FP64 for each took 40 us of the kernel's 0.2 ms
constexpr int kRootBits = kPairMost, kRoots = 1 << kRootBits, kOctant = kRoots / 8;
struct Roots {
    float ch[kOctant + 1], cl[kOctant + 1], sh[kOctant + 1], sl[kOctant + 1];
};
constexpr Roots octant_roots() {
    Roots r = {};
    for (int q = 0; q <= kOctant; ++q) {
        // cos and sin by Horner from the 20th and 21st powers
        const double x = 6.283185307179586476925 * q / kRoots, x2 = x * x;
        double c = 1.0, s = 1.0;
        for (int k = 20; k >= 2; k -= 2) {
            c = 1.0 - c * x2 / (k * (k - 1));
            s = 1.0 - s * x2 / (k * (k + 1));
        }
        s *= x;
        r.ch[q] = (float)c;
        r.cl[q] = (float)(c - (double)r.ch[q]);
        r.sh[q] = (float)s;
        r.sl[q] = (float)(s - (double)r.sh[q]);
    }
    return r;
}
__device__ const Roots g_roots = octant_roots();

// e^{-2 pi j q / 4096}, 0 <= q < 4096
__device__ __forceinline__ PairC root(int q) {
    const int r = q & (kRoots / 4 - 1), quarter = q >> (kRootBits - 2);
    const bool upper = r > kOctant;
    const int i = upper ? kRoots / 4 - r : r;
    const float ch = g_roots.ch[i], cl = g_roots.cl[i], sh = g_roots.sh[i], sl = g_roots.sl[i];
    const PairC e = upper ? PairC{sh, sl, -ch, -cl} : PairC{ch, cl, -sh, -sl};
    // times (-j)^quarter
    const PairC f = quarter & 1 ? times_minus_i(e) : e;
    return quarter & 2 ? PairC{-f.rh, -f.rl, -f.ih, -f.il} : f;
}

// x 2^-e as a float pair, for |x| < 2^(e + 1) (truncated, then the rest); values below
// 2^-126 of that vanish
__device__ __forceinline__ void scaled_pair(double x, int e, float &h, float &l) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int field = (int)((hi >> 20) & 0x7ffu);
    const int e32 = field ? field - 1023 - e + 127 : 0;
    const unsigned sign = hi & 0x80000000u;
    const unsigned mant = __funnelshift_l(lo, hi & 0xfffffu, 3);
    const float r = __uint2float_rn(lo & 0x1fffffffu) * __uint_as_float((unsigned)max(e32 - 52, 0) << 23);
    const float a = __uint_as_float(((unsigned)max(e32, 0) << 23) | mant);
    h = e32 > 0 ? __uint_as_float(__float_as_uint(a) | sign) : 0.0f;
    l = e32 > 52 ? __uint_as_float(__float_as_uint(r) | sign) : 0.0f;
}
// rare cases out of line, or the compiler runs their FP64 instructions every time
// under a predicate (half of the kernel's time went to them)
__device__ __noinline__ double lifted(double x) { return x * 0x1p300; }
__device__ __noinline__ double unscaled_any(float h, float l, int e) { return ldexp((double)h + (double)l, e); }
// (h + l) 2^e in FP64
__device__ __forceinline__ double unscaled(float h, float l, int e) {
    float H, L;
    fast_sum(h, l, H, L);
    const unsigned b = __float_as_uint(H);
    const int e32 = (int)((b >> 23) & 0xffu);
    // H as a 53-bit integer, L in its last places
    const float f = __uint_as_float((unsigned)min(306 - e32, 254) << 23);
    int place = e32 >= 52 ? __float2int_rn(L * f) : 0;
    if ((int)b < 0) place = -place;
    long long m = ((long long)(0x800000u | (b & 0x7fffffu)) << 29) + place;
    int ex = e32 - 127 + 1023 + e;
    if (m < (1LL << 52)) { m <<= 1; --ex; }
    if (e32 == 0 || ex < 1 || ex > 2046) return unscaled_any(H, L, e);
    m = (m & 0xFFFFFFFFFFFFFLL) | ((long long)ex << 52);
    return __longlong_as_double(m | (long long)((unsigned long long)(b & 0x80000000u) << 32));
}

// padded so that eight neighbouring points a thread, or any run of points, fall on
// different banks
__device__ __forceinline__ int padded(int p) { return p + (p >> 3); }

// e^{j x n} for the phase tables: x n as an exact sum of two doubles less the nearest
// multiple of 2 pi (in three parts), so that its sine and cosine are good to FP64
__device__ __forceinline__ PairC phase(double x, int n) {
    constexpr double p1 = 6.283185307179586, p2 = 2.4492935982947064e-16, p3 = -5.989539619436679e-33;
    const double a = x * n, al = fma(x, (double)n, -a);
    double sn, cs;
    if (!(fabs(a) < 1e15)) {            // no multiple of 2 pi that is exact enough
        sincos(a, &sn, &cs);
        return pair_of(cs, sn);
    }
    const double q = rint(a * 0.15915494309189535);
    double r = fma(-q, p1, a);          // exact: a and q p1 are close
    const double t = q * p2, tl = fma(q, p2, -t);
    const double s = r - t;
    const double sl = ((r - s) - t) - tl + al - q * p3;
    r = s + sl;
    sincos(r, &sn, &cs);
    const double low = (s - r) + sl;    // what r lost: a first-order term
    return pair_of(cs - sn * low, sn + cs * low);
}

template <int LOG>
struct PairPlan {
    static constexpr int N = 1 << LOG, T = N / 8, mid = N / 512;
    static constexpr int lo_bits = LOG / 2, lo = 1 << lo_bits, hi = N / 2 / lo + 1;
    // twiddles of the three radix-8 passes, e^{-2 pi j n m / Lp} at [m - 1][n]
    static constexpr int tw = 7 * (N / 8 + N / 64 + N / 512);
    static constexpr int data = N + N / 8;
    static constexpr size_t smem = sizeof(PairC) * (size_t)(data + tw + lo + hi) + 64 * sizeof(unsigned);
};

template <int LOG>
__global__ void __launch_bounds__(PairPlan<LOG>::T) k_theta_pairs(const ThetaArgs a, int items) {
    typedef PairPlan<LOG> P;
    constexpr int N = P::N, T = P::T;
    extern __shared__ __align__(16) PairC pc[];
    PairC *z = pc;
    PairC *tw = z + P::data;
    PairC *plo = tw + P::tw, *phi = plo + P::lo;
    unsigned *top = reinterpret_cast<unsigned *>(phi + P::hi);     // [2][32]
    const int t = threadIdx.x;
    {
        PairC *w = tw;
        for (int len = N; len >= N / 64; len /= 8) {
            const int s = len / 8;
            for (int q = t; q < 7 * s; q += T) {
                const int m = q / s + 1, n = q % s;
                w[q] = root(m * n * (kRoots / len));
            }
            w += 7 * s;
        }
    }
    const int first = (int)((long long)items * blockIdx.x / gridDim.x);
    const int last = (int)((long long)items * (blockIdx.x + 1) / gridDim.x);
    const int pairs = (a.ncoord + 1) / 2;
    int have = -1;                                     // the column of the phase tables
    for (int item = first; item < last; ++item) {
        const int col = item / pairs, c0 = 2 * (item % pairs);
        const bool two = c0 + 1 < a.ncoord;
        const double *ra = a.in + (long long)c0 * a.ldc + (long long)col * N;
        const double *rb = ra + a.ldc;
        double xa[8], xb[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            xa[m] = ra[t + m * T];
            xb[m] = two ? rb[t + m * T] : 0.0;
        }
        unsigned ma = 0, mb = 0;
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            ma = max(ma, (unsigned)__double2hiint(xa[m]) & 0x7fffffffu);
            mb = max(mb, (unsigned)__double2hiint(xb[m]) & 0x7fffffffu);
        }
        ma = __reduce_max_sync(0xffffffffu, ma);
        mb = __reduce_max_sync(0xffffffffu, mb);
        if ((t & 31) == 0) {
            top[t >> 5] = ma;
            top[32 + (t >> 5)] = mb;
        }
        if (col != have) {
            const double rho = a.rho ? a.rho[col] : a.rho0;
            for (int q = t; q < P::lo + P::hi; q += T) {
                if (q < P::lo) plo[q] = phase(rho, q);
                else phi[q - P::lo] = phase(rho, (q - P::lo) * P::lo);
            }
            have = col;
        }
        __syncthreads();
        ma = mb = 0;
#pragma unroll 4
        for (int w = 0; w < T / 32; ++w) {
            ma = max(ma, top[w]);
            mb = max(mb, top[32 + w]);
        }
        int ea = (int)(ma >> 20) - 1023, eb = (int)(mb >> 20) - 1023;
        // rows of (nearly) subnormal numbers are lifted first
        int la = 0, lb = 0;
        if (min(ma, mb) < (200u << 20)) {
            if (ma < (200u << 20)) { la = 300; ++ea; }
            if (mb < (200u << 20)) { lb = 300; ++eb; }
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                if (la) xa[m] = lifted(xa[m]);
                if (lb) xb[m] = lifted(xb[m]);
            }
        }
        PairC x[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            scaled_pair(xa[m], ea + la, x[m].rh, x[m].rl);
            scaled_pair(xb[m], eb + lb, x[m].ih, x[m].il);
        }
        // ---- there
        dft8(x);
#pragma unroll
        for (int m = 0; m < 8; ++m) z[padded(t + m * T)] = m ? mul_c(x[m], tw[(m - 1) * T + t]) : x[0];
        __syncthreads();
        const PairC *w = tw + 7 * T;
#pragma unroll 1
        for (int len = N / 8; len > P::mid; len /= 8) {
            const int s = len / 8, n = t % s, p = (t / s) * len + n;
#pragma unroll
            for (int m = 0; m < 8; ++m) x[m] = z[padded(p + m * s)];
            dft8(x);
#pragma unroll
            for (int m = 0; m < 8; ++m) z[padded(p + m * s)] = m ? mul_c(x[m], w[(m - 1) * s + n]) : x[0];
            w += 7 * s;
            __syncthreads();
        }
        // ---- the middle: eight neighbouring points, 8 / mid groups
#pragma unroll
        for (int m = 0; m < 8; ++m) x[m] = z[padded(8 * t + m)];
        auto rest = [&]() {
            if (P::mid == 8) dft8(x);
            else if (P::mid == 4) { dft4(x[0], x[1], x[2], x[3]); dft4(x[4], x[5], x[6], x[7]); }
            else {
#pragma unroll
                for (int m = 0; m < 8; m += 2) dft2(x[m], x[m + 1]);
            }
        };
        rest();
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            // the digits of the group, most significant first: k = d1 + 8 d2 + 64 d3 + 512 d4
            const int g = (8 * t + m) / P::mid, d4 = m % P::mid;
            const int k = (g >> 6) + ((g >> 3) & 7) * 8 + (g & 7) * 64 + 512 * d4;
            const int sk = k < N / 2 ? k : k - N, ak = sk < 0 ? -sk : sk;
            PairC e = mul_c(phi[ak >> P::lo_bits], plo[ak & (P::lo - 1)]);       // e^{j rho |k|}
            if (sk < 0) { e.ih = -e.ih; e.il = -e.il; }
            if (k == N / 2) { e.ih = e.il = 0.0f; }
            if (a.derivative) {
                // times j k (0 for the Nyquist frequency)
                const float f = k == N / 2 ? 0.0f : (float)sk;
                const float rh = __fmul_rn(f, e.rh), rl = __fmaf_rn(f, e.rl, __fmaf_rn(f, e.rh, -rh));
                const float ih = __fmul_rn(-f, e.ih), il = __fmaf_rn(-f, e.il, __fmaf_rn(-f, e.ih, -ih));
                e.rh = ih; e.rl = il; e.ih = rh; e.il = rl;
            }
            x[m] = swapped(mul_c(x[m], e));
        }
        // ---- and back
        rest();
        // the eight points are this thread's own: no wait before they are replaced
#pragma unroll
        for (int m = 0; m < 8; ++m) z[padded(8 * t + m)] = x[m];
        __syncthreads();
#pragma unroll 1
        for (int len = P::mid * 8; len < N; len *= 8) {
            const int s = len / 8, n = t % s, p = (t / s) * len + n;
            w -= 7 * s;
#pragma unroll
            for (int m = 0; m < 8; ++m) x[m] = m ? mul_c(z[padded(p + m * s)], w[(m - 1) * s + n]) : z[padded(p)];
            dft8(x);
#pragma unroll
            for (int m = 0; m < 8; ++m) z[padded(p + m * s)] = x[m];
            __syncthreads();
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) x[m] = m ? mul_c(z[padded(t + m * T)], tw[(m - 1) * T + t]) : z[padded(t)];
        dft8(x);
        // (the next rows' first pass writes z after a barrier behind these reads)
        double *oa = a.out + (long long)c0 * a.ldc + (long long)col * N;
        double *ob = oa + a.ldc;
        // a row with an infinity or a NaN leaves nothing of either; a row of zeros stays one
        const bool broken = ma >= 0x7ff00000u || mb >= 0x7ff00000u;
        const double nan = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const double va = unscaled(x[m].ih, x[m].il, ea - LOG), vb = unscaled(x[m].rh, x[m].rl, eb - LOG);
            oa[t + m * T] = broken ? nan : ma ? va : 0.0;
            if (two) ob[t + m * T] = broken ? nan : mb ? vb : 0.0;
        }
    }
}

template <int LOG>
cudaError_t launch_theta_pairs(const ThetaArgs &a, int items, cudaStream_t st) {
    typedef PairPlan<LOG> P;
    cudaError_t e = cudaFuncSetAttribute(k_theta_pairs<LOG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P::smem);
    if (e != cudaSuccess) return e;
    int device = 0, sms = 0, resident = 0;
    if ((e = cudaGetDevice(&device)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, k_theta_pairs<LOG>, P::T, P::smem)) != cudaSuccess)
        return e;
    const int grid = items < sms * resident ? items : sms * resident;
    k_theta_pairs<LOG><<<grid, P::T, P::smem, st>>>(a, items);
    return cudaGetLastError();
}

// Phase alignment cost.  N^2 distances of C coordinates, each C subtractions, C
// multiply-adds, a square root and an addition: in FP64 about 19 instructions of a
// pipe that takes 19 clocks an SM for each of a warp's (9.6 ms for 16 alignments of
// 4 x 4096 circles), so here the distances are computed on the FP32 pipe, whose rate
// is some fifty times that, in numbers of two or three floats:
//   digits      every coordinate, scaled by the alignment's power of two to |y| <= 1,
//               as y = x1 + x2 + x3 with x1 a multiple of 2^-22, x2 of 2^-45, and x3
//               the rest rounded to FP32 (2^-70); the differences of the first two
//               digits are exact FP32 numbers;
//   distance    the difference as a float pair, its square with the product's error
//               term, the sum over the coordinates with every addition's error, the
//               root with one correction: about 2^-47 relative, without bias;
//   sum         four distances as a pair, then FP64 (two additions every four
//               distances, which the FP64 pipe takes beside the rest).
// 1.27 ms for those 16 alignments (1.05 G warp instructions, issue 79%).
// A distance's error, 3e-15 rms, averages out over the sum, whose own FP64 roundings
// are a quarter as many as in order of i: against 113-bit costs the relative error is
// 3.6e-16 rms at N = 200 (4.1e-16 in FP64 in order of i), 1.6e-16 at 1000 (7.4e-16),
// 1.9e-16 at 4096 (1.8e-15).  The two meet near N = 160: shorter circles, whose time
// is launches, take the FP64 loop, and so does an alignment whose largest value's
// exponent leaves no room for the scaling, or that is not finite.
// Split: a cluster of eight blocks takes 512 shifts, each block an eighth of the i
// (the same split for every shift and number of alignments: equal terms give equal
// costs), each thread two neighbouring shifts, whose windows overlap; the even and
// odd entries of the window are apart in shared memory, so that a warp's loads of
// every second entry are consecutive.
constexpr int kPhThreads = 256;
constexpr int kPhShifts = 2 * kPhThreads;
constexpr int kPhTile = 128;            // i per shared tile (a multiple of 4)
constexpr int kPhSplit = 8;             // blocks of a cluster, each an eighth of the i
constexpr int kPhWin = kPhTile + kPhShifts;
constexpr int kPhWide = 0x7fffffff;     // no scale: the FP64 loop
constexpr int kPhLeast = 192;           // shorter circles take the FP64 loop

struct PhaseArgs {
    const double *wr;
    const double *wp;
    double *cost;
    int *scale;                         // per alignment: the exponent e, |values| < 2^e
    int N, ncoord, nalign;
};

// The scale of each alignment, left in the shift output, which the minimum's kernel
// writes last.
__global__ void __launch_bounds__(1024) k_phase_scale(const PhaseArgs a) {
    __shared__ unsigned top[32];
    const long long n = (long long)a.ncoord * a.N, base = n * blockIdx.x;
    unsigned m = 0;                     // high words of |x|: the largest holds the largest exponent
    for (long long q = threadIdx.x; q < n; q += 1024) {
        m = max(m, (unsigned)__double2hiint(a.wr[base + q]) & 0x7fffffffu);
        m = max(m, (unsigned)__double2hiint(a.wp[base + q]) & 0x7fffffffu);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) top[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = __reduce_max_sync(0xffffffffu, top[threadIdx.x]);
        const int e = (int)(m >> 20);
        if (threadIdx.x == 0) a.scale[blockIdx.x] = a.N < kPhLeast || e < 100 || e > 1900 ? kPhWide : e - 1022;
    }
}

__device__ __forceinline__ double power_of_two(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// the distance between two points given by their digits, as a float pair; what the
// pair has no room for (the low halves' squares, the root's second-order terms: 2^-50
// of the distance, but of one sign) goes to `rest`
template <int C>
__device__ __forceinline__ void pair_distance(const float (&x)[3][C], const float (&y)[3][C], float &g, float &lo,
                                              float &rest) {
    float S = 0.0f, T = 0.0f, L2 = 0.0f;   // the squares' sum, and the low halves'
#pragma unroll
    for (int c = 0; c < C; ++c) {
        float h, e, H, L;
        // the first two differences are exact; the second is at most 2^-22, the least
        // nonzero value of the first
        fast_sum(__fsub_rn(x[0][c], y[0][c]), __fsub_rn(x[1][c], y[1][c]), h, e);
        fast_sum(h, __fadd_rn(e, __fsub_rn(x[2][c], y[2][c])), H, L);
        const float p = __fmul_rn(H, H);
        float q = __fmaf_rn(H, H, -p);
        q = __fmaf_rn(H, __fadd_rn(L, L), q);
        L2 = __fmaf_rn(L, L, L2);
        if (c == 0) {
            S = p;
            T = q;
        } else {
            float s, r;
            two_sum(S, p, s, r);
            S = s;
            T = __fadd_rn(T, __fadd_rn(r, q));
        }
    }
    // sqrt(S + T): g the root of S to a rounding, then one correction by the residual
    // (0 for S = 0, where the reciprocal root stays finite)
    const float r = rsqrtf(fmaxf(S, 1e-37f));
    const float hr = __fmul_rn(0.5f, r), g0 = __fmul_rn(S, r);
    g = __fmaf_rn(__fmaf_rn(-g0, g0, S), hr, g0);
    lo = __fmul_rn(__fadd_rn(__fmaf_rn(-g, g, S), T), hr);
    // with d = sqrt(S) - g and t = T hr: lo = d - d^2 hr + t and sqrt(S + T) =
    // g + d + t - t^2 hr + ..., so d^2 - t^2 = lo (lo - 2 t) is missing
    rest = __fmaf_rn(__fmaf_rn(lo, __fmaf_rn(-T, r, lo), L2), hr, rest);
}

// the digits of a value scaled to |y| <= 1
__device__ __forceinline__ void digits(double y, float &x1, float &x2, float &x3) {
    constexpr double m1 = 1.5 * (double)(1 << 30), m2 = 1.5 * (double)(1 << 7);
    const double t1 = __dsub_rn(__dadd_rn(y, m1), m1);      // to a multiple of 2^-22
    const double r1 = __dsub_rn(y, t1);
    const double t2 = __dsub_rn(__dadd_rn(r1, m2), m2);     // to a multiple of 2^-45
    x1 = (float)t1;
    x2 = (float)t2;
    x3 = (float)__dsub_rn(r1, t2);
}

template <int C>
__global__ void __cluster_dims__(kPhSplit, 1, 1) __launch_bounds__(kPhThreads) k_phase_cost(const PhaseArgs a) {
    extern __shared__ __align__(16) float ps[];
    float(*prev)[3][C] = reinterpret_cast<float(*)[3][C]>(ps);            // [kPhTile], by i
    float *win = ps + kPhTile * 3 * C;                                    // [odd][digit][C][kPhWin / 2]
    constexpr int kHalf = kPhWin / 2;
    double *part = reinterpret_cast<double *>(win + 3 * C * kPhWin);      // [kPhShifts]
    const int N = a.N, al = blockIdx.y, t = threadIdx.x;
    const int rank = blockIdx.x % kPhSplit;
    const int m0 = (int)(blockIdx.x / kPhSplit) * kPhShifts;
    const double *Wr = a.wr + (long long)al * C * N;
    const double *Wp = a.wp + (long long)al * C * N;
    const int e = a.scale[al];
    double acc[2] = {0.0, 0.0};
    float rest[2] = {0.0f, 0.0f};
    if (e == kPhWide) {
        if (rank == 0)
            for (int k = 0; k < 2; ++k) {
                const int m = m0 + 2 * t + k;
                if (m >= N) continue;
                for (int i = 0; i < N; ++i) {
                    const int w = i + m < N ? i + m : i + m - N;
                    double d2 = 0.0;
                    for (int c = 0; c < C; ++c) {
                        const double d = Wr[(long long)c * N + w] - Wp[(long long)c * N + i];
                        d2 = fma(d, d, d2);
                    }
                    acc[k] += sqrt(d2);
                }
                a.cost[(long long)al * N + m] = acc[k];
            }
        return;                         // the whole cluster: e is the alignment's
    }
    const double down = power_of_two(-e);
    const int per = ((N + 4 * kPhSplit - 1) / (4 * kPhSplit)) * 4;
    const int i_end = (int)min((long long)N, (long long)(rank + 1) * per);
    for (long long i0 = (long long)rank * per; i0 < i_end; i0 += kPhTile) {
        const int ti = (int)min((long long)kPhTile, i_end - i0);
        __syncthreads();                // the previous tile is read
        for (int q = t; q < C * kPhTile; q += kPhThreads) {
            const int c = q / kPhTile, u = q % kPhTile;
            if (u < ti) digits(Wp[(long long)c * N + i0 + u] * down, prev[u][0][c], prev[u][1][c], prev[u][2][c]);
        }
        const int w0 = (int)((i0 + m0) % N);
        const int wn = min(kPhWin, ti + kPhShifts + 4);
        for (int c = 0; c < C; ++c)
            for (int u = t; u < wn; u += kPhThreads) {
                float x1, x2, x3;
                digits(Wr[(long long)c * N + ((unsigned)w0 + (unsigned)u) % (unsigned)N] * down, x1, x2, x3);
                float *o = win + ((u & 1) * 3 * C + c) * kHalf + (u >> 1);
                o[0] = x1;
                o[C * kHalf] = x2;
                o[2 * C * kHalf] = x3;
            }
        __syncthreads();
        if (m0 + 2 * t >= N) continue;
        for (int u = 0; u < ti; u += 4) {
            // window entries u + 2t + j, j = 0..4: shift k at i0 + u + v reads entry v + k
            float x[2][3][C];
            auto load = [&](int j, float (&w)[3][C]) {
                const float *p = win + (j & 1) * 3 * C * kHalf + (u >> 1) + t + (j >> 1);
#pragma unroll
                for (int d = 0; d < 3; ++d)
#pragma unroll
                    for (int c = 0; c < C; ++c) w[d][c] = p[(d * C + c) * kHalf];
            };
            load(0, x[0]);
            float G[2] = {0.0f, 0.0f}, E[2] = {0.0f, 0.0f};
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                load(v + 1, x[(v + 1) & 1]);
                if (u + v < ti) {
                    float y[3][C];
#pragma unroll
                    for (int d = 0; d < 3; ++d)
#pragma unroll
                        for (int c = 0; c < C; ++c) y[d][c] = prev[u + v][d][c];
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        float g, lo, s, r;
                        pair_distance<C>(x[(v + k) & 1], y, g, lo, rest[k]);
                        two_sum(G[k], g, s, r);
                        G[k] = s;
                        E[k] = __fadd_rn(E[k], __fadd_rn(r, lo));
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                acc[k] += (double)G[k];
                acc[k] += (double)E[k];
            }
        }
    }
    // the eight parts, added in order of i by the cluster's first block
    part[2 * t] = acc[0] + (double)rest[0];
    part[2 * t + 1] = acc[1] + (double)rest[1];
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    if (rank == 0) {
        for (int q = t; q < kPhShifts; q += kPhThreads) {
            double s = part[q];
            for (int r = 1; r < kPhSplit; ++r) s += cluster.map_shared_rank(part, r)[q];
            if (m0 + q < N) a.cost[(long long)al * N + m0 + q] = s * power_of_two(e);
        }
    }
    cluster.sync();                     // the parts are read before their blocks end
}

template <int C>
cudaError_t launch_phase_cost(const PhaseArgs &a, cudaStream_t st) {
    constexpr size_t smem = (size_t)(kPhTile + kPhWin) * 3 * C * sizeof(float) + kPhShifts * sizeof(double);
    const cudaError_t e = cudaFuncSetAttribute(k_phase_cost<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((a.N + kPhShifts - 1) / kPhShifts) * kPhSplit, (unsigned)a.nalign);
    k_phase_cost<C><<<grid, kPhThreads, smem, st>>>(a);
    return cudaGetLastError();
}

// Smallest cost per alignment, ties to the smallest shift.
__global__ void __launch_bounds__(256) k_phase_argmin(const double *cost, int N, int *shift) {
    __shared__ double bv[256];
    __shared__ int bi[256];
    const double *c = cost + (long long)blockIdx.x * N;
    double best = INFINITY;
    int idx = N;
    for (int m = threadIdx.x; m < N; m += 256) {
        const double v = c[m];
        if (v < best || (v == best && m < idx)) {
            best = v;
            idx = m;
        }
    }
    bv[threadIdx.x] = best;
    bi[threadIdx.x] = idx;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            const double ov = bv[threadIdx.x + s];
            const int oi = bi[threadIdx.x + s];
            if (ov < bv[threadIdx.x] || (ov == bv[threadIdx.x] && oi < bi[threadIdx.x])) {
                bv[threadIdx.x] = ov;
                bi[threadIdx.x] = oi;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) shift[blockIdx.x] = bi[0] < N ? bi[0] : 0;
}

bool device_ptr(const void *p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

tms_status fail(tms_status st, const std::string &msg) {
    tms::set_last_error(msg);
    return st;
}

}  // namespace

extern "C" tms_status tms_theta_translate(const double *dIn, double *dOut, int N, int nCols,
                                          int nCoord, long long ldc, const double *dRho,
                                          double rho0, int derivative, void *stream) {
    if (N < 8 || N > 8192 || (N & (N - 1)))
        return fail(TMS_ERR_ARG, "tms_theta_translate: N must be a power of two in 8..8192");
    if (nCols < 0 || nCoord < 1 || (derivative != 0 && derivative != 1))
        return fail(TMS_ERR_ARG, "tms_theta_translate: bad nCols, nCoord or derivative");
    if (!dRho && !isfinite(rho0)) return fail(TMS_ERR_ARG, "tms_theta_translate: rho0 not finite");
    if (nCols == 0) return TMS_OK;
    if (ldc < (long long)nCols * N) return fail(TMS_ERR_ARG, "tms_theta_translate: ldc < nCols * N");
    if (!dIn || !dOut || !device_ptr(dIn) || !device_ptr(dOut) || (dRho && !device_ptr(dRho)))
        return fail(TMS_ERR_ARG, "tms_theta_translate: arrays must be device pointers");
    int logN = 0;
    while ((1 << logN) < N) ++logN;
    ThetaArgs a;
    a.in = dIn;
    a.out = dOut;
    a.ldc = ldc;
    a.rho = dRho;
    a.rho0 = rho0;
    a.N = N;
    a.logN = logN;
    a.cols = nCols;
    a.ncoord = nCoord;
    a.derivative = derivative;
    const long long blocks = (long long)nCols * ((nCoord + 1) / 2);
    if (blocks > 0x7fffffffLL) return fail(TMS_ERR_ARG, "tms_theta_translate: too many columns");
    cudaError_t e;
    // a common shift so small that its arguments lose little (about 1.2e-17 |rho| N of the
    // result, against 1.2e-14 in float pairs) is the nearer one in FP64
    const bool small_shift = !dRho && fabs(rho0) * N < 1000.0;
    if (logN >= kPairLeast && logN <= kPairMost && !small_shift) {
        cudaStream_t st = (cudaStream_t)stream;
        e = logN == 10 ? launch_theta_pairs<10>(a, (int)blocks, st)
            : logN == 11 ? launch_theta_pairs<11>(a, (int)blocks, st) : launch_theta_pairs<12>(a, (int)blocks, st);
    } else {
        const size_t smem = (size_t)(N + N / 2 + 4 * kTab) * sizeof(double2);
        e = cudaFuncSetAttribute(k_theta_fft, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return fail(TMS_ERR_CUDA, cudaGetErrorString(e));
        k_theta_fft<<<(unsigned)blocks, kFftThreads, smem, (cudaStream_t)stream>>>(a);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return fail(TMS_ERR_CUDA, std::string("tms_theta_translate: ") +
                                                        cudaGetErrorString(e));
    return TMS_OK;
}

extern "C" tms_status tms_phase_align(const double *dWr, const double *dWprev, int N, int nCoord,
                                      int nAlign, double *dCost, int32_t *dShift, void *stream) {
    if (N < 1 || nCoord < 1 || nCoord > 8 || nAlign < 0)
        return fail(TMS_ERR_ARG, "tms_phase_align: need N >= 1, 1 <= nCoord <= 8, nAlign >= 0");
    if (nAlign == 0) return TMS_OK;
    if (!dWr || !dWprev || !dCost || !dShift || !device_ptr(dWr) || !device_ptr(dWprev) ||
        !device_ptr(dCost) || !device_ptr(dShift))
        return fail(TMS_ERR_ARG, "tms_phase_align: arrays must be device pointers");
    if (nAlign > 65535) return fail(TMS_ERR_ARG, "tms_phase_align: nAlign > 65535");
    PhaseArgs a;
    a.wr = dWr;
    a.wp = dWprev;
    a.cost = dCost;
    a.scale = dShift;
    a.N = N;
    a.ncoord = nCoord;
    a.nalign = nAlign;
    k_phase_scale<<<nAlign, 1024, 0, (cudaStream_t)stream>>>(a);
    cudaError_t (*const launch[8])(const PhaseArgs &, cudaStream_t) = {
        launch_phase_cost<1>, launch_phase_cost<2>, launch_phase_cost<3>, launch_phase_cost<4>,
        launch_phase_cost<5>, launch_phase_cost<6>, launch_phase_cost<7>, launch_phase_cost<8>};
    cudaError_t e = launch[nCoord - 1](a, (cudaStream_t)stream);
    if (e != cudaSuccess) return fail(TMS_ERR_CUDA, std::string("tms_phase_align: ") + cudaGetErrorString(e));
    k_phase_argmin<<<nAlign, 256, 0, (cudaStream_t)stream>>>(dCost, N, dShift);
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(TMS_ERR_CUDA, std::string("tms_phase_align: ") +
                                                        cudaGetErrorString(e));
    return TMS_OK;
}
