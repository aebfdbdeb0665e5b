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
// FP64 in shared memory, the arguments k rho reduced modulo 2 pi as exact
// numbers: rounded to FP64 ahead of their sine and cosine they were most of the
// error on rows with high frequencies.  What bounds it: the FP64 pipe (0.89 ms for
// 4 x 1025 columns of 2048 points, 14 M warp instructions of 19 clocks an SM).  A
// transform in pairs of floats took 0.16 ms, but holds 2^-48: 8e-15 of a smooth
// row against 6e-16 here, and 2e-12 of a derivative against 6e-14.
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

__device__ __forceinline__ int exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// e^{j x n}: x n as an exact sum of two doubles less the nearest multiple of 2 pi (in
// three parts), so that its sine and cosine are good to FP64
__device__ __forceinline__ double2 phase(double x, int n) {
    constexpr double p1 = 6.283185307179586, p2 = 2.4492935982947064e-16, p3 = -5.989539619436679e-33;
    const double a = x * n, al = fma(x, (double)n, -a);
    const double q = rint(a * 0.15915494309189535);
    double r = fma(-q, p1, a);          // exact: a and q p1 are close
    const double t = q * p2, tl = fma(q, p2, -t);
    const double s = r - t;
    const double sl = ((r - s) - t) - tl + al - q * p3;
    r = s + sl;
    double low = (s - r) + sl;          // what r lost: a first-order term
    if (exponent(a) >= 1023 + 49) {     // no multiple of 2 pi that is exact enough
        r = a;
        low = 0.0;
    }
    double sn, cs;
    sincos(r, &sn, &cs);
    return make_double2(cs - sn * low, sn + cs * low);
}

// The high word of |x|, with its last bit set for a rest below it: a row's largest tells
// its size (0: a row of zeros), and the exponent of that size.
__device__ __forceinline__ unsigned size_word(double x) {
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) | (__double2loint(x) != 0 ? 1u : 0u);
}
__device__ __forceinline__ int size_exponent(unsigned m) {
    return (m >> 20) ? (int)(m >> 20) - 1023 : 31 - __clz(m) - 1042;
}
// 2^e, -1022 <= e <= 1023
__device__ __forceinline__ double power_of_two(int e) { return __hiloint2double((1023 + e) << 20, 0); }
// x 2^e, the power of two in halves, which are in range (out of line: the compiler would run
// it for every value, under a predicate)
__device__ __noinline__ double scaled(double x, int e) {
    return x * power_of_two(e / 2) * power_of_two(e - e / 2);
}

__global__ void __launch_bounds__(kFftThreads, 6) k_theta_fft(const ThetaArgs a) {
    extern __shared__ double2 sm[];
    __shared__ unsigned top[2][kFftThreads / 32];
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
    // the four tables side by side, as far as they are used
    static_assert(kFftThreads == 4 * kTab, "64 threads a table");
    {
        const int table = t / kTab, e = t % kTab, n = table & 1 ? e : e * kTab;
        if (n < N / 2) {
            if (table < 2) {
                double s, c;
                sincospi(-2.0 * (double)n / (double)N, &s, &c);
                (table ? tl : th)[e] = make_double2(c, s);
            } else {
                (table == 3 ? hl : hh)[e] = phase(rho, n);
            }
        }
    }
    const double *ra = a.in + (long long)c0 * a.ldc + (long long)col * N;
    const double *rb = a.in + (long long)c1 * a.ldc + (long long)col * N;
    const int sh = 32 - a.logN;
    unsigned ma = 0, mb = 0;
    for (int i = t; i < N; i += kFftThreads) {
        const double2 v = make_double2(ra[i], two ? rb[i] : 0.0);
        z[__brev((unsigned)i) >> sh] = v;
        ma = max(ma, size_word(v.x));
        mb = max(mb, size_word(v.y));
    }
    ma = __reduce_max_sync(0xffffffffu, ma);
    mb = __reduce_max_sync(0xffffffffu, mb);
    if ((t & 31) == 0) {
        top[0][t >> 5] = ma;
        top[1][t >> 5] = mb;
    }
    __syncthreads();
    for (int m = t; m < N / 2; m += kFftThreads) w[m] = cmul(th[m / kTab], tl[m % kTab]);
#pragma unroll
    for (int k = 0; k < kFftThreads / 32; ++k) {
        ma = max(ma, top[0][k]);
        mb = max(mb, top[1][k]);
    }
    // rows of unlike size, whose larger one's rounding would be the smaller one's error, or
    // of extreme size are brought to about 1 (powers of two: the same digits)
    int ea = 0, eb = 0;
    if (max(ma, mb) < 0x7ff00000u) {
        ea = ma ? size_exponent(ma) : mb ? size_exponent(mb) : 0;
        eb = mb ? size_exponent(mb) : ea;
        if (abs(ea - eb) <= 2 && abs(ea) < 900) ea = eb = 0;
    }
    if (ea | eb) {
        for (int i = t; i < N; i += kFftThreads) {
            double2 &v = z[__brev((unsigned)i) >> sh];
            v = make_double2(scaled(v.x, -ea), scaled(v.y, -eb));
        }
    }
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
            const double2 h = cmul(hh[N / 4 / kTab], hl[N / 4 % kTab]);   // e^{j rho N / 4}
            const double g = a.derivative ? 0.0 : (h.x - h.y) * (h.x + h.y);
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
        double2 v = z[__brev((unsigned)i) >> sh];
        v.x *= inv;
        v.y *= inv;
        if (ea | eb) v = make_double2(scaled(v.x, ea), scaled(v.y, eb));
        // (a row of zeros stays one)
        oa[i] = ma == 0 ? 0.0 : v.x;
        if (two) ob[i] = mb == 0 ? 0.0 : v.y;
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

// Phase alignment cost.  N^2 distances of C coordinates, each C subtractions, C
// multiply-adds, a square root and an addition: in FP64 about 19 instructions of a
// pipe that takes 19 clocks an SM for each of a warp's (9.6 ms for 16 alignments of
// 4 x 4096 circles), so here the distances are computed on the FP32 pipe, whose rate
// is some fifty times that, in numbers of two or three floats:
//   digits      every coordinate, scaled by the alignment's power of two to |y| <= 1
//               (times 2^40, so that no square of a difference is subnormal), as
//               y = x1 + x2 + x3 with x1 a multiple of 2^-22, x2 of 2^-45, and x3 the
//               rest rounded to FP32 (2^-70); the differences of the first two digits
//               are exact FP32 numbers;
//   distance    the difference as a float pair, its square with the product's error
//               term, the sum over the coordinates with every addition's error, the
//               root with one correction: about 2^-47 relative, without bias;
//   sum         four distances as a pair, then FP64 (two additions every four
//               distances, which the FP64 pipe takes beside the rest).
// 1.26 ms for those 16 alignments (1.08 G warp instructions, issue 79%).
// A distance's error, 3e-15 rms, averages out over the sum, whose own FP64 roundings
// are a quarter as many as in order of i: against 113-bit costs the relative error is
// 3.6e-16 rms at N = 200 (4.1e-16 in FP64 in order of i), 1.6e-16 at 1000 (7.4e-16),
// 1.9e-16 at 4096 (1.8e-15).  The two meet near N = 160: shorter circles take FP64
// sums, and so does an alignment whose largest value's exponent leaves no room for the
// scaling, or that is not finite.
// A value of at least 2^-16 of the alignment's largest is the sum of its digits exactly;
// each of the others is off by 2^-70 at most, and so is a difference with it by its
// rounding.  Every value is in one distance of each shift, so `lost` such values cost a
// shift lost 2^-69: where that could be more than 2^-51 of its cost (a large coordinate
// that cancels leaves a cost of that size) the shift's cost is made again in FP64.
// So is one that few distances make, whose errors do not average out: 2.4e-15 of the root of
// the distances' squares is more than the 1.9e-17 N^(1/2) of the cost that a sum in FP64
// loses where those squares are more than N / 16384 of the cost's (evenly spread: N < 130).
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
constexpr int kPhWide = 0x7fffffff;     // no scale: FP64 sums
constexpr int kPhLeast = 192;           // shorter circles take FP64 sums
constexpr int kPhUp = 40;               // the digits' unit is 2^-40 of the scale
constexpr double kPhFew = 16384.0;      // N / kPhFew: the share of the squares that few distances pass

struct PhaseArgs {
    const double *wr;
    const double *wp;
    double *cost;
    int *scale;                         // per alignment (NULL: all kPhWide): the exponent e,
                                        // |values| < 2^e, + 1024, and from bit 12 l, 2^(l - 1)
                                        // at least its lost values (l = 0: none)
    int N, ncoord, nalign;
};

// The scale of each alignment, left in the shift output, which the minimum's kernel
// writes last.
__global__ void __launch_bounds__(1024) k_phase_scale(const PhaseArgs a) {
    __shared__ unsigned top[32], lost[32];
    const long long n = (long long)a.ncoord * a.N, base = n * blockIdx.x;
    const int t = threadIdx.x;
    unsigned m = 0;                     // high words of |x|: the largest holds the largest exponent
    for (long long q = t; q < n; q += 1024) {
        m = max(m, (unsigned)__double2hiint(a.wr[base + q]) & 0x7fffffffu);
        m = max(m, (unsigned)__double2hiint(a.wp[base + q]) & 0x7fffffffu);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((t & 31) == 0) top[t >> 5] = m;
    __syncthreads();
    m = __reduce_max_sync(0xffffffffu, top[t & 31]);
    const int field = (int)(m >> 20);   // 2^(field - 1022) = 2^e
    if (field < 100 || field > 1900) {
        if (t == 0) a.scale[blockIdx.x] = kPhWide;
        return;
    }
    // values below 2^(e - 16) with a bit below 2^(e - 69)
    unsigned count = 0;
    const unsigned small = (unsigned)(field - 15) << 20;
    auto look = [&](double x) {
        const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu;
        if (h < small && (h | (unsigned)__double2loint(x)) != 0u) {
            const int last = __ffs(__double2loint(x)), bit = last ? last - 1 : 31 + __ffs((int)(h | 0x100000u));
            count += max((int)(h >> 20), 1) - 1075 + bit < field - 1022 - 69;
        }
    };
    for (long long q = t; q < n; q += 1024) {
        look(a.wr[base + q]);
        look(a.wp[base + q]);
    }
    count = __reduce_add_sync(0xffffffffu, count);
    if ((t & 31) == 0) lost[t >> 5] = count;
    __syncthreads();
    count = __reduce_add_sync(0xffffffffu, lost[t & 31]);
    const int l = count ? 33 - __clz(count - 1) : 0;
    int word = (field - 1022 + 1024) | (l << 12);
    if (4 * (long long)count >= a.N) {
        // a coordinate's worth of them: where no distance can be large enough (the large
        // coordinates vary too little), FP64 for all, without the float pairs' sums first.
        // Ranges from the high words, as integers of the values' order.
        __shared__ int lo[8], hi[8];
        if (t < 8) {
            lo[t] = 0x7fffffff;
            hi[t] = (int)0x80000000;
        }
        __syncthreads();
        for (int c = 0; c < a.ncoord; ++c) {
            int least = 0x7fffffff, most = (int)0x80000000;
            for (int i = t; i < a.N; i += 1024) {
                const long long q = base + (long long)c * a.N + i;
                const int r = __double2hiint(a.wr[q]), p = __double2hiint(a.wp[q]);
                const int ro = r ^ ((r >> 31) & 0x7fffffff), po = p ^ ((p >> 31) & 0x7fffffff);
                least = min(least, min(ro, po));
                most = max(most, max(ro, po));
            }
            least = __reduce_min_sync(0xffffffffu, least);
            most = __reduce_max_sync(0xffffffffu, most);
            if ((t & 31) == 0) {
                atomicMin(&lo[c], least);
                atomicMax(&hi[c], most);
            }
        }
        __syncthreads();
        if (t == 0) {
            // (the last bits of a high word: outward)
            double d2 = 0.0;
            for (int c = 0; c < a.ncoord; ++c) {
                const int h = hi[c] ^ ((hi[c] >> 31) & 0x7fffffff), g = lo[c] ^ ((lo[c] >> 31) & 0x7fffffff);
                const double d = (__hiloint2double(h, h < 0 ? 0 : -1) - __hiloint2double(g, g < 0 ? -1 : 0)) *
                                 power_of_two(1022 - field);
                d2 = fma(d, d, d2);
            }
            if (a.N * sqrt(d2) < power_of_two(51 - 69 + l - 1)) word = kPhWide;
        }
    }
    if (t == 0) a.scale[blockIdx.x] = word;
}

// the part of shift m's cost at i = first, first + step, ..., in FP64
template <int C>
__device__ __forceinline__ double cost_part(const double *Wr, const double *Wp, int N, int m, int first, int step) {
    double s = 0.0;
#pragma unroll 1                        // (the float pairs' loop has the registers)
    for (long long i = first; i < N; i += step) {
        const long long w = i + m < N ? i + m : i + m - N;
        double d2 = 0.0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const double d = Wr[(long long)c * N + w] - Wp[(long long)c * N + i];
            d2 = fma(d, d, d2);
        }
        s += sqrt(d2);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    return s;
}

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

// the digits of a value scaled to |y| <= 2^kPhUp
__device__ __forceinline__ void digits(double y, float &x1, float &x2, float &x3) {
    constexpr double unit = 1LL << kPhUp, m1 = 1.5 * (1 << 30) * unit, m2 = 1.5 * (1 << 7) * unit;
    const double t1 = __dsub_rn(__dadd_rn(y, m1), m1);      // to a multiple of 2^(kPhUp - 22)
    const double r1 = __dsub_rn(y, t1);
    const double t2 = __dsub_rn(__dadd_rn(r1, m2), m2);     // to a multiple of 2^(kPhUp - 45)
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
    float *sq = reinterpret_cast<float *>(part + kPhShifts);              // [kPhShifts]
    const int N = a.N, al = blockIdx.y, t = threadIdx.x;
    const int rank = blockIdx.x % kPhSplit;
    const int m0 = (int)(blockIdx.x / kPhSplit) * kPhShifts;
    const double *Wr = a.wr + (long long)al * C * N;
    const double *Wp = a.wp + (long long)al * C * N;
    const int word = a.scale ? a.scale[al] : kPhWide;
    if (word == kPhWide) {              // (the whole cluster: it is the alignment's)
        // a shift a warp, 64 of them at once in the cluster
        const int last = min(kPhShifts, N - m0);
        for (int q = rank * (kPhThreads / 32) + (t >> 5); q < last; q += kPhSplit * (kPhThreads / 32)) {
            const double s = cost_part<C>(Wr, Wp, N, m0 + q, t & 31, 32);
            if ((t & 31) == 0) a.cost[(long long)al * N + m0 + q] = s;
        }
        return;
    }
    const int e = (word & 0xfff) - 1024, lost = word >> 12;
    double acc[2] = {0.0, 0.0};
    float rest[2] = {0.0f, 0.0f}, squares[2] = {0.0f, 0.0f};
    const double down = power_of_two(kPhUp - e);
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
                        squares[k] = __fmaf_rn(g, g, squares[k]);
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
    sq[2 * t] = squares[0];
    sq[2 * t + 1] = squares[1];
    cg::cluster_group cluster = cg::this_cluster();
    // shifts to be made again (the first block's), costs below which they are
    __shared__ unsigned short again[kPhShifts];
    __shared__ int n_again;
    if (t == 0) n_again = 0;
    const double least = lost ? power_of_two(kPhUp - 69 + 51 + lost - 1) : 0.0;
    cluster.sync();
    if (rank == 0) {
        for (int q = t; q < kPhShifts; q += kPhThreads) {
            double s = part[q];
            float d2 = sq[q];
            for (int r = 1; r < kPhSplit; ++r) {
                s += cluster.map_shared_rank(part, r)[q];
                d2 += cluster.map_shared_rank(sq, r)[q];
            }
            if (m0 + q >= N) continue;
            if (s < least || kPhFew * (double)d2 > N * (s * s)) again[atomicAdd(&n_again, 1)] = (unsigned short)q;
            else a.cost[(long long)al * N + m0 + q] = s * power_of_two(e - kPhUp);
        }
    }
    cluster.sync();                     // the parts are read before their blocks end
    const int n = *cluster.map_shared_rank(&n_again, 0);
    for (int k = rank; k < n; k += kPhSplit) {
        const int m = m0 + cluster.map_shared_rank(again, 0)[k];
        const double s = cost_part<C>(Wr, Wp, N, m, t, kPhThreads);
        __syncthreads();                // (the previous shift's sums are read)
        if ((t & 31) == 0) part[t >> 5] = s;
        __syncthreads();
        if (t == 0) {
            double sum = part[0];
            for (int w = 1; w < kPhThreads / 32; ++w) sum += part[w];
            a.cost[(long long)al * N + m] = sum;
        }
    }
    cluster.sync();                     // the list is read before the first block ends
}

template <int C>
cudaError_t launch_phase_cost(const PhaseArgs &a, cudaStream_t st) {
    constexpr size_t smem = (size_t)(kPhTile + kPhWin) * 3 * C * sizeof(float) + kPhShifts * (sizeof(double) + sizeof(float));
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
    const size_t smem = (size_t)(N + N / 2 + 4 * kTab) * sizeof(double2);
    cudaError_t e = cudaFuncSetAttribute(k_theta_fft, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return fail(TMS_ERR_CUDA, cudaGetErrorString(e));
    k_theta_fft<<<(unsigned)blocks, kFftThreads, smem, (cudaStream_t)stream>>>(a);
    e = cudaGetLastError();
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
    a.scale = N < kPhLeast ? nullptr : dShift;
    a.N = N;
    a.ncoord = nCoord;
    a.nalign = nAlign;
    if (a.scale) k_phase_scale<<<nAlign, 1024, 0, (cudaStream_t)stream>>>(a);
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
