// Narrow phase, merging of duplicate hits, output, and the adjoint.
//
// Narrow phase (arXiv 2109.14814, Sec. 6.2.4, Eq. (precise)): for triangles
// (x1, x2, x3) and (y1, y2, y3), the unknowns (a, b, c, d) solve the 4x4 system
//   [x1-x2 | x3-x2 | y2-y1 | y2-y3] (a, b, c, d)^T = y2 - x2,
// and the triangles meet iff a, b, c, d >= 0, a + b <= 1, c + d <= 1; the common
// point is x2 + a(x1-x2) + b(x3-x2).  The paper ran this on the CPU; here it is
// four lanes per triangle pair in FP64 (Gaussian elimination with partial
// pivoting).  Readings of the paper fixed by this library: the inequalities are
// closed with tolerance tau (margin = min(a, b, c, d, 1-a-b, 1-c-d) >= -tau),
// and a singular system (a zero pivot) is not a hit.  The (theta, s) estimates
// are the interpolation formulas that follow Eq. (precise).
//
// Mixed precision (optional): a verified FP32 solve first.  The system is formed
// in FP32 from the rounded entries of the FP64 system, with a bound on every
// entry's error.  Gaussian elimination on [A | I | r] gives z~
// and an approximate inverse C; with alpha >= |I - C A|_inf (computed with its
// rounding and input-error terms), A is nonsingular when alpha < 1 and
//   |z - z~|_inf <= | |C| |r - A z~| |_inf / (1 - alpha),
// the residual again bounded with its rounding and input errors.  A pair is
// rejected in FP32 only when the resulting upper bound of the margin is below
// -2 tau minus an allowance for the FP64 solve's own rounding (so an FP64 solve
// of the same system could not call it a hit); all other pairs, and every
// pair whose certificate fails, get the FP64 solve.
#include <cuda_runtime.h>
#include <stdint.h>

#include "tms_common.cuh"

namespace tms {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr double kTwoPi = 6.283185307179586476925286766559;

// ---------------------------------------------------------------------------
// FP64 Gaussian elimination with partial pivoting, fully unrolled in registers
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ bool solve4_gepp(T A[4][4], T r[4], T z[4], T &det) {
    T sign = 1;
    T inv[4];
    bool ok = true;
#pragma unroll
    for (int col = 0; col < 4; ++col) {
        int p = col;
        T best = fabs(A[col][col]);
#pragma unroll
        for (int row = col + 1; row < 4; ++row) {
            T v = fabs(A[row][col]);
            if (v > best) { best = v; p = row; }
        }
        ok &= best != T(0);
#pragma unroll
        for (int row = col + 1; row < 4; ++row) {
            const bool sw = (p == row);     // branch-free select keeps A in registers
#pragma unroll
            for (int j = col; j < 4; ++j) {
                const T lo = A[col][j], hi = A[row][j];
                A[col][j] = sw ? hi : lo;
                A[row][j] = sw ? lo : hi;
            }
            const T rl = r[col], rh = r[row];
            r[col] = sw ? rh : rl;
            r[row] = sw ? rl : rh;
            sign = sw ? -sign : sign;
        }
        inv[col] = T(1) / A[col][col];
#pragma unroll
        for (int row = col + 1; row < 4; ++row) {
            T f = A[row][col] * inv[col];
#pragma unroll
            for (int j = col + 1; j < 4; ++j) A[row][j] = A[row][j] - f * A[col][j];
            r[row] = r[row] - f * r[col];
        }
    }
#pragma unroll
    for (int row = 3; row >= 0; --row) {
        T acc = r[row];
#pragma unroll
        for (int j = row + 1; j < 4; ++j) acc = acc - A[row][j] * z[j];
        z[row] = acc * inv[row];
    }
    det = sign * A[0][0] * A[1][1] * A[2][2] * A[3][3];
    return ok;
}

__device__ __forceinline__ void gather_tri(const MeshDev &m, uint32_t t, double v[3][4]) {
    int ii[3], kk[3];
    tri_ij(m, t, ii, kk);
#pragma unroll
    for (int j = 0; j < 3; ++j) load_vertex(m, ii[j], kk[j], v[j]);
}

__device__ __forceinline__ float comp(const float4 &v, int c) {
    return c == 0 ? v.x : (c == 1 ? v.y : (c == 2 ? v.z : v.w));
}

// (i, k) of quad q = k N + i
__device__ __forceinline__ void quad_ik(const MeshDev &m, uint32_t q, int &i, int &k) {
    const uint32_t kk = (uint32_t)__umul64hi((unsigned long long)q, m.nmagic);
    k = (int)kk;
    i = (int)(q - kk * (uint32_t)m.N);
}

// the quad's vertices (i,k), (i+1,k), (i,k+1), (i+1,k+1), each coordinate rounded
// down to FP32
__device__ __forceinline__ void gather_quad_lo(const MeshDev &m, uint32_t q, float4 v[4]) {
    int i, k;
    quad_ik(m, q, i, k);
    const int ip = (i + 1 == m.N) ? 0 : i + 1;
    const size_t idx[4] = {(size_t)k * m.N + i, (size_t)k * m.N + ip, (size_t)(k + 1) * m.N + i,
                           (size_t)(k + 1) * m.N + ip};
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = __ldg(m.vlo + idx[j]);
}

// a face's vertices for the quad-level test: a quad's, or a triangle's x2, x1, x3, x3
template <int FACE>
__device__ __forceinline__ void gather_face_lo(const MeshDev &m, uint32_t face, float4 v[4]) {
    if (FACE == 1) {
        gather_quad_lo(m, face, v);
    } else {
        int ii[3], kk[3];
        tri_ij(m, face, ii, kk);
        v[1] = __ldg(m.vlo + (size_t)kk[0] * m.N + ii[0]);
        v[0] = __ldg(m.vlo + (size_t)kk[1] * m.N + ii[1]);
        v[2] = v[3] = __ldg(m.vlo + (size_t)kk[2] * m.N + ii[2]);
    }
}

// The FP32 system of a triangle pair: A and r as the FP64 solve forms them, rounded
// to nearest, so every entry is within kEntry |entry| + kTiny of the FP64 one (2^-126
// below the FP32 normal range; the FP64 entry's own rounding is inside the margin).
constexpr float kEntry = 1.001f * 5.9604645e-08f, kTiny = 1.2e-38f;

// true when the verified FP32 solve proves margin < -2 tau (not a hit)
__device__ __forceinline__ bool fp32_verified_reject(const float (&A)[4][4], const float (&r)[4], float tau) {
    const float u = 5.9604645e-08f;
    // Gaussian elimination with partial pivoting on [A | I | r]
    float M[4][9];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int j = 0; j < 4; ++j) { M[i][j] = A[i][j]; M[i][4 + j] = (i == j) ? 1.0f : 0.0f; }
        M[i][8] = r[i];
    }
#pragma unroll
    for (int col = 0; col < 4; ++col) {
        int p = col;
        float best = fabsf(M[col][col]);
#pragma unroll
        for (int row = col + 1; row < 4; ++row) {
            float v = fabsf(M[row][col]);
            if (v > best) { best = v; p = row; }
        }
        if (!(best > 0.0f)) return false;
#pragma unroll
        for (int row = col + 1; row < 4; ++row) {
            const bool sw = (p == row);
#pragma unroll
            for (int j = col; j < 9; ++j) {
                const float lo = M[col][j], hi = M[row][j];
                M[col][j] = sw ? hi : lo;
                M[row][j] = sw ? lo : hi;
            }
        }
        const float inv = 1.0f / M[col][col];
#pragma unroll
        for (int row = col + 1; row < 4; ++row) {
            const float f = M[row][col] * inv;
#pragma unroll
            for (int j = col + 1; j < 9; ++j) M[row][j] = fmaf(-f, M[col][j], M[row][j]);
        }
        M[col][col] = inv;   // keep the reciprocal pivot for the back substitution
    }
    // back substitution for the 5 right-hand sides: columns 4..7 give C, 8 gives z
    float C[4][4], z[4];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        float x[4];
#pragma unroll
        for (int row = 3; row >= 0; --row) {
            float acc = M[row][4 + k];
#pragma unroll
            for (int j = row + 1; j < 4; ++j) acc = fmaf(-M[row][j], x[j], acc);
            x[row] = acc * M[row][row];
        }
#pragma unroll
        for (int row = 0; row < 4; ++row) {
            if (k < 4) C[row][k] = x[row];
            else z[row] = x[row];
        }
    }
    // alpha >= |I - C A_exact|_inf: computed I - C A, its rounding (6u (1 + |C||A|))
    // and the input error |C| E, the last two as one product |C| W with
    // W = (6u + kEntry) |A| + kTiny
    float W[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) W[k][j] = fmaf(6.0f * u + kEntry, fabsf(A[k][j]), kTiny);
    float alpha = 0.0f, cnorm = 0.0f, anorm = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float row = 0.0f, crow = 0.0f, arow = 0.0f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float e = (i == j) ? 1.0f : 0.0f, cw = 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                e = fmaf(-C[i][k], A[k][j], e);
                cw = fmaf(fabsf(C[i][k]), W[k][j], cw);
            }
            row += fabsf(e) + 6.0f * u * ((i == j) ? 1.0f : 0.0f) + cw;
            crow += fabsf(C[i][j]);
            arow += fabsf(A[i][j]);
        }
        alpha = fmaxf(alpha, row);
        cnorm = fmaxf(cnorm, crow);
        anorm = fmaxf(anorm, arow);
    }
    alpha *= 1.0001f;
    if (!(alpha < 0.5f)) return false;
    // |r_exact - A_exact z~| componentwise
    const float zsum = (fabsf(z[0]) + fabsf(z[1])) + (fabsf(z[2]) + fabsf(z[3]));
    float res[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float acc = r[i], mag = fabsf(r[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            acc = fmaf(-A[i][j], z[j], acc);
            mag = fmaf(fabsf(A[i][j]), fabsf(z[j]), mag);
        }
        res[i] = (fabsf(acc) + (6.0f * u + kEntry) * mag + kTiny * (1.0f + zsum)) * 1.0001f;
    }
    float err = 0.0f, zmax = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float d = 0.0f;
#pragma unroll
        for (int j = 0; j < 4; ++j) d = fmaf(fabsf(C[i][j]), res[j], d);
        err = fmaxf(err, d);
        zmax = fmaxf(zmax, fabsf(z[i]));
    }
    err = err / (1.0f - alpha) * 1.001f;
    const float slack = 4.0f * u;
    float m = fminf(fminf(z[0], z[1]), fminf(z[2], z[3])) + err;
    m = fminf(m, 1.0f - z[0] - z[1] + 2.0f * err + slack * (1.0f + fabsf(z[0]) + fabsf(z[1])));
    m = fminf(m, 1.0f - z[2] - z[3] + 2.0f * err + slack * (1.0f + fabsf(z[2]) + fabsf(z[3])));
    // allowance for an FP64 solve of the same system (its own rounding)
    const float kappa = cnorm * anorm;
    const float allow = 2.0f * tau + 32.0f * 1.1102230e-16f * kappa * (1.0f + zmax);
    return isfinite(m) && isfinite(err) && (m < -allow);
}

// ---------------------------------------------------------------------------
// Separating-axis prefilter: a certificate of non-intersection cheaper than the
// verified solve, which it precedes.
//
// Lemma.  For any direction w let I_X = [min_i w.x_i, max_i w.x_i] (length D_X)
// and I_Y likewise.  A point of a triangle widened to weights >= -t projects
// within 3 t D_X of I_X (weights w_i = (1 + 3t) l_i - t with l on the simplex).
// If the FP64 solve reports a hit, its weights are >= -tau' and the two points
// it describes lie within fp64_reach of each other (backward error, below), so
// a gap g > 3 tau' (D_X + D_Y) + |w|_1 reach between I_X and I_Y proves that
// it reports none -- with no condition on the system, so near-parallel
// triangle planes are cleared too.
// Directions: for each triangle the two longest of the four vectors orthogonal
// to its plane (the duals of e1 ^ e2 ^ axis_k, read off the plane's Plucker
// coordinates m_ij = e1_i e2_j - e1_j e2_i); any direction is valid, these
// make the triangle's own interval almost a point.  det A is the pairing of
// the two planes' Plucker coordinates.  Every FP32 value carries a bound on its
// rounding and on the error of its input, so the test is rigorous for the FP64
// vertices.
// ---------------------------------------------------------------------------
struct SplitVec {
    float v[4];
    float E;       // |v_c - exact_c| <= E for every c
    float M;       // max_c |v_c|
};

// column j of the FP32 system, or its negative
__device__ __forceinline__ SplitVec column_vec(const float (&A)[4][4], int j, float sign) {
    SplitVec r;
    r.M = 0.0f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        r.v[c] = sign * A[c][j];
        r.M = fmaxf(r.M, fabsf(A[c][j]));
    }
    r.E = kEntry * r.M + kTiny;
    return r;
}

// a + b of two vectors with bounds
__device__ __forceinline__ SplitVec add_vec(const SplitVec &a, const SplitVec &b) {
    const float u = 5.9604645e-08f;
    SplitVec r;
    float vm = 0.0f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        r.v[c] = a.v[c] + b.v[c];
        vm = fmaxf(vm, fabsf(r.v[c]));
    }
    r.E = (a.E + b.E + u * vm) * 1.001f;
    r.M = vm;
    return r;
}

// the dual direction k (orthogonal to the plane and to axis k) from its
// Plucker coordinates m = (01, 02, 03, 12, 13, 23)
__device__ __forceinline__ void dual_dir(const float m[6], int k, float w[4]) {
    w[0] = k == 0 ? 0.0f : (k == 1 ? -m[5] : (k == 2 ? m[4] : -m[3]));
    w[1] = k == 1 ? 0.0f : (k == 0 ? m[5] : (k == 2 ? -m[2] : m[1]));
    w[2] = k == 2 ? 0.0f : (k == 0 ? -m[4] : (k == 1 ? m[2] : -m[0]));
    w[3] = k == 3 ? 0.0f : (k == 0 ? m[3] : (k == 1 ? -m[1] : m[0]));
}

// indices of the two longest duals
__device__ __forceinline__ void top2_duals(const float m[6], int &k1, int &k2) {
    const float s01 = m[0] * m[0], s02 = m[1] * m[1], s03 = m[2] * m[2];
    const float s12 = m[3] * m[3], s13 = m[4] * m[4], s23 = m[5] * m[5];
    const float n[4] = {s12 + s13 + s23, s02 + s03 + s23, s01 + s03 + s13, s01 + s02 + s12};
    k1 = 0;
#pragma unroll
    for (int k = 1; k < 4; ++k) k1 = n[k] > n[k1] ? k : k1;
    k2 = k1 == 0 ? 1 : 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) k2 = (k != k1 && n[k] > n[k2]) ? k : k2;
}

// What the relative bounds of the gap tests leave out: below 2^-126 an operation is off by up
// to 2^-150, and a bound that is a product may vanish.  A projection is three or four
// factors of an edge's size, so edges of 1e-11 come there; a test has some forty such
// operations, 700 times fewer than this.
constexpr float kUnder = 1e-42f;

__device__ __forceinline__ float dot4(const float w[4], const SplitVec &v) {
    return fmaf(w[3], v.v[3], fmaf(w[2], v.v[2], fmaf(w[1], v.v[1], w[0] * v.v[0])));
}

// fp64_reach and widen3 (the FP64 solve's backward error and the widening of
// a triangle's projection) are in tms_common.cuh: the patch-pair test uses them too.

// the gap test along w for X = {0, e1, e2} and Y = {r, s1, s3} (all relative to x2):
// the widened projections apart by more than |w|_1 reach
__device__ __forceinline__ bool separated(const float w[4], const SplitVec &e1, const SplitVec &e2,
                                          const SplitVec &r, const SplitVec &s1, const SplitVec &s3,
                                          float tp, float reach) {
    const float u = 5.9604645e-08f;
    const float w1 = fabsf(w[0]) + fabsf(w[1]) + fabsf(w[2]) + fabsf(w[3]);
    // |fl(w.v) - w.v_exact| <= |w|_1 (4.01 u M_v + E_v)
    const float a1 = dot4(w, e1), a3 = dot4(w, e2);
    const float b2 = dot4(w, r), b1 = dot4(w, s1), b3 = dot4(w, s3);
    const float ex = w1 * fmaxf(fmaf(4.01f * u, e1.M, e1.E), fmaf(4.01f * u, e2.M, e2.E));
    const float ey = w1 * fmaxf(fmaxf(fmaf(4.01f * u, r.M, r.E), fmaf(4.01f * u, s1.M, s1.E)),
                                fmaf(4.01f * u, s3.M, s3.E));
    const float xl = fminf(0.0f, fminf(a1, a3)), xh = fmaxf(0.0f, fmaxf(a1, a3));
    const float yl = fminf(b2, fminf(b1, b3)), yh = fmaxf(b2, fmaxf(b1, b3));
    const float DX = (xh - xl) + 2.0f * ex, DY = (yh - yl) + 2.0f * ey;
    const float need = fmaf(tp * (DX + DY) + w1 * reach + ex + ey, 1.001f, kUnder);
    const float gap = fmaxf(yl - xh, xl - yh) * (1.0f - 4.0f * u);
    return gap > need;
}

// Quad-level form of the separating-axis test: no one of the four triangle pairs of the
// quad candidate can be an FP64 hit (fp64_reach).  A triangle's vertices are among its
// quad's, so its projected interval lies inside the quad's, and its widening (3 tau' times
// its length) is at most the quad's.  Every triangle's edges are differences of the quad's
// vertices (|A_ij| <= 2 max of the edge vectors below), and every offset y2 - x2 is r0 plus
// at most the vectors to each quad's far vertex.
// (With triangle faces the fourth vertex repeats the third.)
//
// Edge vectors of both quads from their first vertices and the vector between those, from
// the vertices rounded down to FP32 alone: fp = f32_rd(p) has |p - fp| <= 2u |fp| + 2^-126
// (one FP32 place; 2^-126 below the normal range), so t = fl(fp - fq) has |t - (p - q)| <=
// u |t| / (1 - u) + 2u (|fp| + |fq|) + 2^-125.  One bound for all: with the largest |t|
// among the edges, M, and in r, R, and the largest |fp| of the eight vertices, H; the test
// is bound by instruction issue, and bounds for each vector of its own were a third of it.
// Looser than the FP64 difference rounded to FP32 by about H / M, which the test absorbs
// except for near-misses far below a face's size.
struct QuadPair {
    float a[3][4], b[3][4], r[4];
    float ka, kb;       // error of a projection of A's vectors, and of B's and r, over |w|_1
    float tp, reach;
};

__device__ __forceinline__ void quad_pair(const float4 QA[4], const float4 QB[4], float tau, QuadPair &q) {
    const float u = 5.9604645e-08f;
    float M = 0.0f, R = 0.0f, H = 0.0f, A3 = 0.0f, B3 = 0.0f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float a0 = comp(QA[0], c), b0 = comp(QB[0], c);
        H = fmaxf(H, fmaxf(fabsf(a0), fabsf(b0)));
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float ak = comp(QA[k + 1], c), bk = comp(QB[k + 1], c);
            q.a[k][c] = ak - a0;
            q.b[k][c] = bk - b0;
            H = fmaxf(H, fmaxf(fabsf(ak), fabsf(bk)));
        }
        M = fmaxf(M, fmaxf(fmaxf(fabsf(q.a[0][c]), fabsf(q.a[1][c])), fmaxf(fabsf(q.b[0][c]), fabsf(q.b[1][c]))));
        A3 = fmaxf(A3, fabsf(q.a[2][c]));
        B3 = fmaxf(B3, fabsf(q.b[2][c]));
        q.r[c] = b0 - a0;
        R = fmaxf(R, fabsf(q.r[c]));
    }
    M = fmaxf(M, fmaxf(A3, B3));
    // (a coordinate of 2^128 or more is rounded down to FLT_MAX or -inf, which says nothing
    // about it)
    const float inf = __int_as_float(0x7f800000);
    const float h = H < 1.7e38f ? (4.003f * u) * H + 3e-38f : inf;
    const float E = fmaf(1.002f * u, M, h), Er = fmaf(1.002f * u, R, h);
    q.ka = fmaf(4.01f * u, M, E) * 1.0001f;
    q.kb = q.ka + fmaf(4.01f * u, R, Er) * 1.0001f;
    q.reach = fp64_reach(2.0f * (M + E) * 1.001f, ((R + Er) + (A3 + E) + (B3 + E)) * 1.001f, tau);
    q.tp = widen3(tau);
}

// One axis of the quad-level test: A's vertices at 0, a1, a2, a3 and B's at r, r + b1,
// r + b2, r + b3 (all relative to A's v0) projected on w, each with its rounding and input
// error (|fl(w.v) - w.v_exact| <= |w|_1 (4.01 u M_v + E_v)); true when the widened intervals
// are further apart than |w|_1 reach.
__device__ __forceinline__ float dotv(const float w[4], const float v[4]) {
    return fmaf(w[3], v[3], fmaf(w[2], v[2], fmaf(w[1], v[1], w[0] * v[0])));
}
__device__ __forceinline__ bool quad_gap(const float w[4], const QuadPair &q) {
    const float u = 5.9604645e-08f;
    const float w1 = fabsf(w[0]) + fabsf(w[1]) + fabsf(w[2]) + fabsf(w[3]);
    const float p1 = dotv(w, q.a[0]), p2 = dotv(w, q.a[1]), p3 = dotv(w, q.a[2]);
    const float q0 = dotv(w, q.r);
    const float s1 = q0 + dotv(w, q.b[0]), s2 = q0 + dotv(w, q.b[1]), s3 = q0 + dotv(w, q.b[2]);
    const float xl = fminf(fminf(0.0f, p1), fminf(p2, p3)), xh = fmaxf(fmaxf(0.0f, p1), fmaxf(p2, p3));
    const float yl = fminf(fminf(q0, s1), fminf(s2, s3)), yh = fmaxf(fmaxf(q0, s1), fmaxf(s2, s3));
    // u |s| for the sums: at most u times the larger end
    const float err = fmaf(u, fmaxf(fabsf(yl), fabsf(yh)), w1 * (q.ka + q.kb));
    const float need = fmaf(q.tp * ((xh - xl) + (yh - yl) + 2.0f * err) + w1 * q.reach + err, 1.001f, kUnder);
    const float gap = fmaxf(yl - xh, xl - yh) * (1.0f - 4.0f * u);
    return gap > need;
}

// Plucker coordinates (01, 02, 03, 12, 13, 23) of the plane of a and b, and the vector
// orthogonal to that plane and to v (the cofactors of x in det(x, a, b, v))
__device__ __forceinline__ void minors(const float a[4], const float b[4], float m[6]) {
    const int I[6] = {0, 0, 0, 1, 1, 2}, J[6] = {1, 2, 3, 2, 3, 3};
#pragma unroll
    for (int k = 0; k < 6; ++k) m[k] = fmaf(a[I[k]], b[J[k]], -(a[J[k]] * b[I[k]]));
}
__device__ __forceinline__ void orthogonal(const float m[6], const float v[4], float w[4]) {
    w[0] = fmaf(v[3], m[3], fmaf(v[1], m[5], -(v[2] * m[4])));
    w[1] = fmaf(-v[3], m[1], fmaf(v[2], m[2], -(v[0] * m[5])));
    w[2] = fmaf(v[3], m[0], fmaf(v[0], m[4], -(v[1] * m[2])));
    w[3] = fmaf(-v[2], m[0], fmaf(v[1], m[1], -(v[0] * m[3])));
}

// Directions: FIRST: the mixed ones orthogonal to A's first-triangle edges a1, a2 and B's
// b1, and to a1, a2, b2; else those to b1, b2, a1 and to b1, b2, a2 (both quads are thin
// along each when their planes share a direction), then the two longest duals of each
// quad's first triangle.  Any direction serves (the bounds hold for the FP32 w as
// computed), so w is not normalised.  A candidate it cannot clear goes on to the tests of
// its triangle pairs.
template <bool FIRST>
__device__ __forceinline__ bool quad_reject(const float4 QA[4], const float4 QB[4], float tau) {
    QuadPair q;
    quad_pair(QA, QB, tau, q);
    float mA[6], mB[6], w[4];
    minors(q.a[0], q.a[1], mA);
    if (FIRST) {
        orthogonal(mA, q.b[0], w);
        if (quad_gap(w, q)) return true;
        orthogonal(mA, q.b[1], w);
        return quad_gap(w, q);
    }
    minors(q.b[0], q.b[1], mB);
    orthogonal(mB, q.a[0], w);
    if (quad_gap(w, q)) return true;
    orthogonal(mB, q.a[1], w);
    if (quad_gap(w, q)) return true;
    int kA1, kA2, kB1, kB2;
    top2_duals(mA, kA1, kA2);
    top2_duals(mB, kB1, kB2);
#pragma unroll 1
    for (int ax = 0; ax < 4; ++ax) {
        float m[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) m[k] = ax < 2 ? mA[k] : mB[k];
        dual_dir(m, ax == 0 ? kA1 : (ax == 1 ? kA2 : (ax == 2 ? kB1 : kB2)), w);
        if (quad_gap(w, q)) return true;
    }
    return false;
}

// true when the separating-axis test proves that the FP64 solve of the pair
// reports no hit (fp64_reach)
__device__ __forceinline__ bool fp32_sat_reject(const float (&A)[4][4], const float (&rhs)[4], float tau) {
    // vectors relative to x2: x1 - x2, x3 - x2, y1 - y2, y3 - y2, y2 - x2
    const SplitVec e1 = column_vec(A, 0, 1.0f), e2 = column_vec(A, 1, 1.0f);
    const SplitVec f1 = column_vec(A, 2, -1.0f), f2 = column_vec(A, 3, -1.0f);
    SplitVec r;
    r.M = 0.0f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        r.v[c] = rhs[c];
        r.M = fmaxf(r.M, fabsf(rhs[c]));
    }
    r.E = kEntry * r.M + kTiny;
    const SplitVec s1 = add_vec(r, f1), s3 = add_vec(r, f2);
    float mE[6], mF[6];
    minors(e1.v, e2.v, mE);
    minors(f1.v, f2.v, mF);
    const float amax = fmaxf(fmaxf(e1.M + e1.E, e2.M + e2.E), fmaxf(f1.M + f1.E, f2.M + f2.E));
    const float reach = fp64_reach(amax * 1.001f, (r.M + r.E) * 1.001f, tau);
    const float tp = widen3(tau);
    int kE1, kE2, kF1, kF2;
    top2_duals(mE, kE1, kE2);
    top2_duals(mF, kF1, kF2);
    // one loop over the four axes (a small kernel fetches its code faster);
    // the plane of each axis is chosen by selects, not by an indexed array
#pragma unroll 1
    for (int ax = 0; ax < 4; ++ax) {
        float m[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) m[k] = ax < 2 ? mE[k] : mF[k];
        float w[4];
        dual_dir(m, ax == 0 ? kE1 : (ax == 1 ? kE2 : (ax == 2 ? kF1 : kF2)), w);
        if (separated(w, e1, e2, r, s1, s3, tp, reach)) return true;
    }
    return false;
}

// ---------------------------------------------------------------------------
// FP64 solve (Eq. (precise)) by four lanes a triangle pair
// ---------------------------------------------------------------------------
// A warp's FP64 instruction holds its scheduler's part of the pipe for 64 clocks
// (measured, whatever its active lanes), so the solve's time is its count of FP64
// instructions: one lane a pair took 245 of them in a row (7.6 us), four lanes, lane c
// with row c of the system, take about 105.  Row operations, pivot choices (as
// integers) and results are those of one lane's elimination with partial pivoting.
__device__ __forceinline__ double quad_lane(double v, int base, int j) { return __shfl_sync(FULL, v, base + j); }

// the ordered bits of |v| (NaN above everything)
__device__ __forceinline__ unsigned long long abs64(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
}
// Triangles ta of ma and tb of mb (every lane of the warp calls it; dead quads solve
// whatever they are given): true on a quad's four lanes when the pair is a hit, whose
// record they then write to *out with pair index `pair`; `slot` gives the place.
template <typename Slot>
__device__ __forceinline__ void solve_pair(const MeshDev &ma, const MeshDev &mb, uint32_t ta, uint32_t tb,
                                           uint32_t pair, double tau, bool live, tms_hit *hits, const Slot &slot) {
    const int lane = threadIdx.x & 31, c = lane & 3, base = lane & ~3;
    double x1, A[4], r;
    {
        int ii[3], kk[3];
        const double *pa = ma.c[c], *pb = mb.c[c];
        tri_ij(ma, ta, ii, kk);
        const double x0 = __ldg(pa + (size_t)kk[0] * ma.N + ii[0]), x2 = __ldg(pa + (size_t)kk[2] * ma.N + ii[2]);
        x1 = __ldg(pa + (size_t)kk[1] * ma.N + ii[1]);
        tri_ij(mb, tb, ii, kk);
        const double y0 = __ldg(pb + (size_t)kk[0] * mb.N + ii[0]), y1 = __ldg(pb + (size_t)kk[1] * mb.N + ii[1]);
        const double y2 = __ldg(pb + (size_t)kk[2] * mb.N + ii[2]);
        A[0] = x0 - x1;
        A[1] = x2 - x1;
        A[2] = y1 - y0;
        A[3] = y1 - y2;
        r = y1 - x1;
    }
    const double col0 = A[0], col1 = A[1], col2 = A[2], col3 = A[3];
    // the row's place in the permuted system, and which lane holds each place
    int place = c, holder[4];
    bool ok = true, negative = false;
    double inv[4], diag[4];
#pragma unroll
    for (int col = 0; col < 4; ++col) {
        // the largest |A[.][col]| of the rows not used yet, the first in place among equals
        unsigned long long best = place >= col ? abs64(A[col]) : 0ULL;
        int bp = place >= col ? place : 4, bl = c;
#pragma unroll
        for (int off = 1; off <= 2; off <<= 1) {
            const unsigned long long ob = __shfl_xor_sync(FULL, best, off);
            const int op = __shfl_xor_sync(FULL, bp, off), ol = __shfl_xor_sync(FULL, bl, off);
            if (ob > best || (ob == best && op < bp)) { best = ob; bp = op; bl = ol; }
        }
        ok &= best != 0ULL;
        // swap places with the row at place col
        negative ^= bp != col;
        place = c == bl ? col : place == col ? bp : place;
        holder[col] = base + bl;
        double p[4];
#pragma unroll
        for (int j = col; j < 4; ++j) p[j] = __shfl_sync(FULL, A[j], holder[col]);
        const double pr = __shfl_sync(FULL, r, holder[col]);
        diag[col] = p[col];
        inv[col] = 1.0 / p[col];
        if (col < 3) {
            const double f = A[col] * inv[col];
            const bool below = place > col;
#pragma unroll
            for (int j = col + 1; j < 4; ++j) {
                const double v = A[j] - f * p[j];
                A[j] = below ? v : A[j];
            }
            const double v = r - f * pr;
            r = below ? v : r;
        }
    }
    double z[4];
#pragma unroll
    for (int row = 3; row >= 0; --row) {
        double acc = r;
#pragma unroll
        for (int j = row + 1; j < 4; ++j) acc = acc - A[j] * z[j];
        z[row] = __shfl_sync(FULL, acc * inv[row], holder[row]);
    }
    const double rest1 = 1.0 - z[0] - z[1], rest2 = 1.0 - z[2] - z[3];
    // the margin as an ordered integer
    long long mo = min(min(min(ord64(z[0]), ord64(z[1])), min(ord64(z[2]), ord64(z[3]))), min(ord64(rest1), ord64(rest2)));
    bool finite = true;
#pragma unroll
    for (int j = 0; j < 4; ++j) finite &= abs64(z[j]) < 0x7ff0000000000000ULL;
    bool hit = live && ok && finite && mo >= ord64(-tau);
    if (!__any_sync(FULL, hit)) return;
    const double det = (negative ? -1.0 : 1.0) * diag[0] * diag[1] * diag[2] * diag[3];
    // lane c takes column c's norm
    double n2 = 0.0;
    {
        const double cols[4] = {col0, col1, col2, col3};
        double e[4];
#pragma unroll
        for (int row = 0; row < 4; ++row) {
            double v = 0.0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const double o = __shfl_sync(FULL, cols[j], base + row);
                v = j == c ? o : v;
            }
            e[row] = v;
        }
        n2 = e[0] * e[0] + e[1] * e[1] + e[2] * e[2] + e[3] * e[3];
    }
    const double nc = sqrt(n2);
    const double norms = quad_lane(nc, base, 0) * quad_lane(nc, base, 1) * quad_lane(nc, base, 2) * quad_lane(nc, base, 3);
    const double rho = fabs(det) / norms;
    const double m = ord64_value(mo);
    hit &= rho > 0.0;
    // lane c's coordinate of the point, and its estimate: theta_u, s_u, theta_s, s_s
    // (formulas after Eq. (precise))
    const double P = x1 + z[0] * col0 + z[1] * col1;
    double est;
    {
        const MeshDev &me = c < 2 ? ma : mb;
        const uint32_t t = c < 2 ? ta : tb, q = t >> 1;
        const int k = (int)__umul64hi((unsigned long long)q, me.nmagic), i = (int)(q - (uint32_t)k * (uint32_t)me.N);
        double v0, v1;
        if (c & 1) {
            v0 = me.s[k];
            v1 = me.s[k + 1];
        } else {
            v0 = i * me.dtheta;
            v1 = v0 + me.dtheta;
        }
        const double w = c == 0 ? z[0] : c == 1 ? z[1] : c == 2 ? z[2] : z[3];
        // T2 measures its weights from the other corner
        const double w0 = t & 1 ? w : 1.0 - w, w1 = t & 1 ? 1.0 - w : w;
        est = w0 * v0 + w1 * v1;
        // theta: fmod(est, 2 pi); the weights of a hit lie in [-1, 2] (tau < 1) and dtheta
        // <= pi, so -2 pi < theta < 4 pi, where one subtraction is exact
        if (!(c & 1)) {
            if (est >= kTwoPi) est -= kTwoPi;
            if (est < 0) est += kTwoPi;
        }
    }
    const unsigned long long pos = slot(hit);
    if (!hit || pos == ~0ULL) return;
    double *o = reinterpret_cast<double *>(hits + pos);
    o[2 + c] = c == 0 ? z[0] : c == 1 ? z[1] : c == 2 ? z[2] : z[3];
    o[6 + c] = P;
    o[10 + c] = est;
    const unsigned band = rho < 1e-12 || fabs(m) < 1e-12 ? 1u : 0u;
    if (c == 0) reinterpret_cast<uint2 *>(o)[0] = make_uint2(ta, tb);
    else if (c == 1) reinterpret_cast<uint2 *>(o)[1] = make_uint2(pair, band);
    else if (c == 2) o[14] = rho;
    else o[15] = m;
}

// the place of a new raw hit (its key and bucket written), or ~0 past the capacity;
// every lane of the warp calls it, a quad's lanes with the same hit
__device__ __forceinline__ unsigned long long hit_place(const NarrowArgs &a, bool hit, uint32_t ta, uint32_t tb,
                                                        uint32_t pair) {
    const int lane = threadIdx.x & 31;
    unsigned long long pos = warp_append(&a.ctr->raw_hits, hit && (lane & 3) == 0, FULL);
    pos = __shfl_sync(FULL, pos, lane & ~3);
    if (!hit || pos >= a.hit_cap) return ~0ULL;
    if ((lane & 3) == 0) {
        const uint64_t key = ((uint64_t)pair << (2 * a.tri_bits)) | ((uint64_t)ta << a.tri_bits) | (uint64_t)tb;
        a.hit_key[pos] = key;
        if (a.tail) a.hit_slot[pos] = atomicAdd(a.tail + tail_bucket(key, a.tri_bits, a.bscale), 1u);
        else a.hit_val[pos] = (uint32_t)pos;
    }
    return pos;
}

// Stage 1a: the quad-level separating-axis test of every candidate (quads, or triangles)
// on its quads' vertices rounded down to FP32, the first mixed directions
// first; the candidates they leave gather in a per-warp queue, and every 32 of
// them take the other directions with all lanes busy, what is left of the block's queues
// at the end together; those still not cleared are listed for k_narrow_filter.  Bound by
// instruction issue and the gathers.  One wave of blocks: with four, a warp had one or two
// turns of 32 candidates and then a queue of about five to work off with 27 lanes idle
// (4096 x 512, 700,000 candidates: 41.6 us and 19.0 M instructions, so 26.2 and 11.7).
constexpr int kQuadWarps = 8;
template <int FACE>
__global__ void __launch_bounds__(32 * kQuadWarps, 3) k_quad_filter(NarrowArgs a) {
    __shared__ uint32_t s_q[kQuadWarps][64];
    __shared__ unsigned s_left[kQuadWarps];
    if (a.ctr->cand > a.cand_cap) return;
    const unsigned long long n = a.ctr->cand;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = lanemask_lt();
    const float tauf = __double2float_ru(a.tau);
    unsigned long long n_quad = 0;
    unsigned qn = 0;                                 // queued candidates (warp-uniform)
    // the other directions for cnt queued candidates
    auto drain = [&](const uint32_t *q, unsigned cnt) {
        bool keep = false;
        uint32_t g = 0;
        if ((unsigned)lane < cnt) {
            g = q[lane];
            const Cand cd = a.cand[g];
            const int2 pr = a.pairs[cd.pair];
            float4 QA[4], QB[4];
            gather_face_lo<FACE>(a.meshes[pr.x], cd.faceA, QA);
            gather_face_lo<FACE>(a.meshes[pr.y], cd.faceB, QB);
            keep = !quad_reject<false>(QA, QB, tauf);
        }
        const unsigned long long pos = warp_append(&a.ctr->qkeep, keep, FULL);
        if (keep && pos < a.qsurv_cap) a.qsurv[pos] = g;
    };
    for (unsigned long long g0 = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x - lane;
         g0 < n; g0 += stride) {
        const unsigned long long g = g0 + lane;
        const bool valid = g < n;
        bool need = false;
        if (valid) {
            const Cand cd = a.cand[g];
            const int2 pr = a.pairs[cd.pair];
            float4 QA[4], QB[4];
            gather_face_lo<FACE>(a.meshes[pr.x], cd.faceA, QA);
            gather_face_lo<FACE>(a.meshes[pr.y], cd.faceB, QB);
            need = !quad_reject<true>(QA, QB, tauf);
        }
        n_quad += __popc(__ballot_sync(FULL, valid));
        const uint32_t want = __ballot_sync(FULL, need);
        if (need) s_q[warp][qn + __popc(want & lt)] = (uint32_t)g;
        qn += __popc(want);
        __syncwarp();
        if (qn >= 32) {
            qn -= 32;
            drain(s_q[warp] + qn, 32);
            __syncwarp();
        }
    }
    // what the block's warps have left, together
    if (lane == 0) s_left[warp] = qn;
    __syncthreads();
    unsigned first = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kQuadWarps; ++w) {
        first += w < warp ? s_left[w] : 0u;
        total += s_left[w];
    }
    const uint32_t mine = (unsigned)lane < qn ? s_q[warp][lane] : 0u;
    __syncthreads();
    uint32_t *all = &s_q[0][0];
    if ((unsigned)lane < qn) all[first + lane] = mine;
    __syncthreads();
    for (unsigned k = 32 * warp; k < total; k += 32 * kQuadWarps) drain(all + k, min(32u, total - k));
    if (lane == 0 && n_quad) atomicAdd(&a.ctr->quad, n_quad);
}

// Stage 2: the triangle pairs of the candidates the quad-level test left, one a lane:
// the differences of the FP64 system, its FP32 rounding through the triangle-level
// separating axes and the verified solve, and the few pairs neither can reject, listed
// by block, through the FP64 solve, four lanes each.  One kernel, because each step waits
// on a chain of loads and dependent instructions and there is little work in any (54,000
// pairs, 12,050 solves at 4096 x 512; 740 and 157 at 1024 x 256): 35 us there against 27
// for a kernel of the FP32 tests and 21 for one of the solves, and the two launches' 33 us
// at 1024 x 256, with the quad-level test, became 22.  The FP32 system is the FP64
// differences rounded, not differences of two-part vertices: fewer conversions.  There is
// no test of the triangles' boxes; a pair that only they would clear takes the verified
// solve.
constexpr int kPairBlock = 128;
template <int FACE>
__global__ void __launch_bounds__(kPairBlock) k_narrow_filter(NarrowArgs a) {
    __shared__ uint4 s_pair[kPairBlock];
    __shared__ unsigned s_n;
    if (a.ctr->cand > a.cand_cap || a.ctr->qkeep > a.qsurv_cap) return;
    const unsigned long long ni = (FACE == 0 ? 1 : 4) * a.ctr->qkeep;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // tau rounded up: the FP32 tests only widen by it
    const float tauf = __double2float_ru(a.tau);
    for (unsigned long long i0 = blockIdx.x * (unsigned long long)kPairBlock; i0 < ni;
         i0 += gridDim.x * (unsigned long long)kPairBlock) {
        const unsigned long long it = i0 + threadIdx.x;
        const bool valid = it < ni;
        if (threadIdx.x == 0) s_n = 0;
        bool need = false, full = false;
        uint4 p = make_uint4(0u, 0u, 0u, 0u);
        if (valid) {
            const Cand cd = a.cand[a.qsurv[FACE == 0 ? it : it >> 2]];
            const int sub = FACE == 0 ? 0 : (int)(it & 3);
            const int2 pr = a.pairs[cd.pair];
            p = make_uint4(FACE == 0 ? cd.faceA : 2 * cd.faceA + (sub & 1),
                           FACE == 0 ? cd.faceB : 2 * cd.faceB + (sub >> 1), cd.pair, 0u);
            double x[3][4], y[3][4];
            gather_tri(a.meshes[pr.x], p.x, x);
            gather_tri(a.meshes[pr.y], p.y, y);
            float A[4][4], r[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                A[c][0] = f32_rn(x[0][c] - x[1][c]);
                A[c][1] = f32_rn(x[2][c] - x[1][c]);
                A[c][2] = f32_rn(y[1][c] - y[0][c]);
                A[c][3] = f32_rn(y[1][c] - y[2][c]);
                r[c] = f32_rn(y[1][c] - x[1][c]);
            }
            full = !fp32_sat_reject(A, r, tauf);
            need = full && !fp32_verified_reject(A, r, tauf);
        }
        const unsigned tested = __popc(__ballot_sync(FULL, valid)), solved = __popc(__ballot_sync(FULL, full));
        if (lane == 0) {
            if (tested) atomicAdd(&a.ctr->sat, (unsigned long long)tested);
            if (solved) atomicAdd(&a.ctr->fp32, (unsigned long long)solved);
        }
        __syncthreads();
        const uint32_t want = __ballot_sync(FULL, need);
        unsigned at = 0;
        if (lane == 0 && want) at = atomicAdd(&s_n, (unsigned)__popc(want));
        at = __shfl_sync(FULL, at, 0) + __popc(want & lanemask_lt());
        if (need) s_pair[at] = p;
        __syncthreads();
        const unsigned n = s_n;
        if (threadIdx.x == 0 && n) atomicAdd(&a.ctr->fp64, (unsigned long long)n);
        for (unsigned k0 = 8 * warp; k0 < n; k0 += kPairBlock / 4) {
            const unsigned k = k0 + (lane >> 2);
            const uint4 q = s_pair[k < n ? k : k0];
            const int2 pr = a.pairs[q.z];
            solve_pair(a.meshes[pr.x], a.meshes[pr.y], q.x, q.y, q.z, a.tau, k < n, a.hits,
                       [&](bool hit) { return hit_place(a, hit, q.x, q.y, q.z); });
        }
        __syncthreads();
    }
}

// The FP32 filters off: every triangle pair of every candidate through the FP64 solve
template <int FACE>
__global__ void __launch_bounds__(kPairBlock) k_narrow_all(NarrowArgs a) {
    if (a.ctr->cand > a.cand_cap) return;
    const unsigned long long n = (FACE == 0 ? 1 : 4) * a.ctr->cand;
    if (blockIdx.x == 0 && threadIdx.x == 0) a.ctr->fp64 = n;
    const int lane = threadIdx.x & 31;
    const unsigned long long gw = blockIdx.x * (unsigned long long)(kPairBlock / 32) + (threadIdx.x >> 5);
    const unsigned long long nw = gridDim.x * (unsigned long long)(kPairBlock / 32);
    for (unsigned long long k0 = 8 * gw; k0 < n; k0 += 8 * nw) {
        const unsigned long long k = k0 + (lane >> 2), kk = k < n ? k : k0;
        const Cand cd = a.cand[FACE == 0 ? kk : kk >> 2];
        const int sub = FACE == 0 ? 0 : (int)(kk & 3);
        const uint32_t ta = FACE == 0 ? cd.faceA : 2 * cd.faceA + (sub & 1);
        const uint32_t tb = FACE == 0 ? cd.faceB : 2 * cd.faceB + (sub >> 1);
        const int2 pr = a.pairs[cd.pair];
        solve_pair(a.meshes[pr.x], a.meshes[pr.y], ta, tb, cd.pair, a.tau, k < n, a.hits,
                   [&](bool hit) { return hit_place(a, hit, ta, tb, cd.pair); });
    }
}

// ---------------------------------------------------------------------------
// merging of duplicate hits (shared edges and vertices)
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool quad_ok(const MeshDev &m, int i, int k) {
    if (k < 0 || k >= m.nqk) return false;
    if (m.periodic) return true;
    return i >= 0 && i < m.nqi;
}
__device__ __forceinline__ int wrap_i(const MeshDev &m, int i) {
    if (!m.periodic) return i;
    return (i % m.N + m.N) % m.N;
}
__device__ __forceinline__ void add_tri(const MeshDev &m, int i, int k, int tau, uint32_t *inc,
                                        int &n) {
    int iw = wrap_i(m, i);
    if (quad_ok(m, iw, k)) inc[n++] = 2u * ((uint32_t)k * (uint32_t)m.N + (uint32_t)iw) + (uint32_t)tau;
}

// Feature of the point with weights (u, v) in triangle t, and the triangles
// incident to that feature.  Weights (w1, w2, w3) = (u, 1-u-v, v) on
// (x1, x2, x3); one weight below tau: the opposite edge; two: the vertex left.
// Codes: (0 << 30) | t, (1 << 30) | (3 * base_vertex + edge_type), (2 << 30) | vertex.
__device__ uint32_t feature_of(const MeshDev &m, uint32_t t, double u, double v, double tau,
                               uint32_t inc[6], int &ninc) {
    const double w[3] = {u, 1.0 - u - v, v};
    const bool s0 = fabs(w[0]) < tau, s1 = fabs(w[1]) < tau, s2 = fabs(w[2]) < tau;
    const int ns = (int)s0 + (int)s1 + (int)s2;
    ninc = 0;
    if (ns == 0) {
        inc[ninc++] = t;
        return t;
    }
    const uint32_t q = t >> 1;
    const int tau_t = t & 1;
    const int i = (int)(q % (uint32_t)m.N), k = (int)(q / (uint32_t)m.N);
    const int ip = (i + 1 == m.N) ? 0 : i + 1;
    if (ns == 1) {
        // edge opposite the small weight: 0 -> (x2,x3), 1 -> (x1,x3), 2 -> (x1,x2)
        const int opp = s0 ? 0 : (s1 ? 1 : 2);
        int bi, bk, type;
        if (opp == 1) { bi = i; bk = k; type = 2; }                      // diagonal of quad (i,k)
        else if (tau_t == 0) {
            if (opp == 2) { bi = i; bk = k; type = 0; }                 // T1 (x1,x2): theta edge at (i,k)
            else { bi = i; bk = k; type = 1; }                          // T1 (x2,x3): s edge at (i,k)
        } else {
            if (opp == 2) { bi = i; bk = k + 1; type = 0; }             // T2 (x1,x2): theta edge at (i,k+1)
            else { bi = ip; bk = k; type = 1; }                         // T2 (x2,x3): s edge at (i+1,k)
        }
        if (type == 0) { add_tri(m, bi, bk, 0, inc, ninc); add_tri(m, bi, bk - 1, 1, inc, ninc); }
        else if (type == 1) { add_tri(m, bi, bk, 0, inc, ninc); add_tri(m, bi - 1, bk, 1, inc, ninc); }
        else { add_tri(m, bi, bk, 0, inc, ninc); add_tri(m, bi, bk, 1, inc, ninc); }
        return (1u << 30) | (3u * ((uint32_t)bk * (uint32_t)m.N + (uint32_t)bi) + (uint32_t)type);
    }
    int j;
    if (ns == 2) j = !s0 ? 0 : (!s1 ? 1 : 2);
    else { j = 0; if (w[1] > w[j]) j = 1; if (w[2] > w[j]) j = 2; }
    int ii[3], kk[3];
    tri_ij(m, t, ii, kk);
    const int vi = ii[j], vk = kk[j];
    add_tri(m, vi, vk, 0, inc, ninc);
    add_tri(m, vi - 1, vk, 0, inc, ninc);
    add_tri(m, vi, vk - 1, 0, inc, ninc);
    add_tri(m, vi, vk - 1, 1, inc, ninc);
    add_tri(m, vi - 1, vk - 1, 1, inc, ninc);
    add_tri(m, vi - 1, vk, 1, inc, ninc);
    return (2u << 30) | ((uint32_t)vk * (uint32_t)m.N + (uint32_t)vi);
}

__global__ void k_dedup_flags(DedupArgs a) {
    const unsigned long long n = clamp_count(&a.ctr->raw_hits, a.raw_cap);
    // a sort whose look-back gave up leaves its output unordered and its value
    // slots possibly unwritten: keep nothing, and index nothing with them
    const bool sorted = (a.ctr->status & ST_TIMEOUT) == 0;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        if (!sorted) {
            a.keep[i] = 0;
            continue;
        }
        const uint64_t key = a.keys[i];
        const tms_hit &h = a.raw[a.vals[i]];
        const int2 pr = a.pairs[h.pair];
        const MeshDev ma = a.meshes[pr.x], mb = a.meshes[pr.y];
        uint32_t incA[6], incB[6];
        int nA, nB;
        const uint32_t fA = feature_of(ma, h.triA, h.a, h.b, a.tau, incA, nA);
        const uint32_t fB = feature_of(mb, h.triB, h.c, h.d, a.tau, incB, nB);
        uint32_t keep = 1;
        if ((fA >> 30) != 0 || (fB >> 30) != 0) {
            for (int p = 0; p < nA && keep; ++p) {
                for (int q = 0; q < nB && keep; ++q) {
                    const uint32_t ta = incA[p], tb = incB[q];
                    if (ta == h.triA && tb == h.triB) continue;
                    const uint64_t k2 = ((uint64_t)h.pair << (2 * a.tri_bits)) |
                                        ((uint64_t)ta << a.tri_bits) | (uint64_t)tb;
                    if (k2 >= key) continue;
                    unsigned long long lo = 0, hi = i;
                    while (lo < hi) {
                        unsigned long long mid = (lo + hi) >> 1;
                        if (a.keys[mid] < k2) lo = mid + 1; else hi = mid;
                    }
                    if (lo < i && a.keys[lo] == k2) {
                        const tms_hit &o = a.raw[a.vals[lo]];
                        uint32_t t1[6], t2[6];
                        int n1, n2;
                        const uint32_t gA = feature_of(ma, o.triA, o.a, o.b, a.tau, t1, n1);
                        const uint32_t gB = feature_of(mb, o.triB, o.c, o.d, a.tau, t2, n2);
                        if (gA == fA && gB == fB) keep = 0;
                    }
                }
            }
        }
        a.keep[i] = keep;
    }
}

__global__ void k_dedup_out(DedupArgs a) {
    const unsigned long long n = clamp_count(&a.ctr->raw_hits, a.raw_cap);
    if (a.ctr->status & ST_TIMEOUT) return;   // nothing was kept (k_dedup_flags)
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        if (!a.keep[i]) continue;
        const unsigned long long pos = a.keep_scan[i];
        tms_hit h = a.raw[a.vals[i]];
        const int2 pr = a.pairs[h.pair];
        uint32_t inc[6];
        int ninc;
        const uint32_t fA = feature_of(a.meshes[pr.x], h.triA, h.a, h.b, a.tau, inc, ninc);
        const uint32_t fB = feature_of(a.meshes[pr.y], h.triB, h.c, h.d, a.tau, inc, ninc);
        if ((fA >> 30) != 0 || (fB >> 30) != 0) h.flags |= 2u;
        a.out_keys[pos] = a.keys[i];
        if (pos < a.out_cap) a.out[pos] = h;
    }
}

__global__ void k_offsets(const uint64_t *out_keys, const unsigned long long *d_out,
                          unsigned long long raw_cap, int n_pairs, int tri_bits, long long *offsets) {
    const unsigned long long n = clamp_count(d_out, raw_cap);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p <= n_pairs; p += gridDim.x * blockDim.x) {
        if (p == n_pairs) { offsets[p] = (long long)n; continue; }
        const uint64_t k = (uint64_t)p << (2 * tri_bits);
        unsigned long long lo = 0, hi = n;
        while (lo < hi) {
            unsigned long long mid = (lo + hi) >> 1;
            if (out_keys[mid] < k) lo = mid + 1; else hi = mid;
        }
        offsets[p] = (long long)lo;
    }
}

// ---------------------------------------------------------------------------
// short merge: up to kTailMax raw hits
// ---------------------------------------------------------------------------
// Latency, not work, bounds the merge of a few thousand hits (a radix pass over
// six tiles is 7 us of loads, ranking and look-back, and the sort and merge took
// 15 launches), so it is one launch of one cluster, whose barrier takes the place of
// the launches between the steps: 16.5 us at 12,045 hits (three launches 10 + 7 + 7; a
// cluster of eight, with one record a turn, 28), and a search of 1024 x 256 vertices
// (157 hits) 112 -> 100 us.  The FP64 solve counts the hits into
// buckets of increasing key; each block scans the counts for itself (32 KB from L2) and
// lists its hits in their buckets; then compares a hit with its bucket (about one at
// 8192 buckets, at most kTailUneven) and decides whether it is a duplicate; then writes the
// records kept.  Hits that crowd a few buckets (a mesh of few triangles, a small pair of a
// batch beside large ones) go to the radix sort: a search with 14,000 hits of two triangles
// took 583 us here and takes 143 so; the two meet near a thousand in a bucket.
__device__ __forceinline__ bool tail_count(const TailArgs &a, unsigned &n) {
    const unsigned long long raw = a.ctr->raw_hits;
    n = (unsigned)raw;
    return raw <= a.raw_cap && raw <= kTailMax;
}

// The search's counters to the host, by one block of the last kernel: a copy of their 300
// bytes as a node of its own took the copy engine about 4 us.
__device__ __forceinline__ void tail_readback(const TailArgs &a) {
    for (int k = threadIdx.x; k < a.words; k += blockDim.x) a.readback[k] = __ldcg(a.result + k);
}

// what any block of the cluster wrote before is visible to all of them after
__device__ __forceinline__ void cluster_step() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// whether the point with weights (u, v) lies inside its triangle (feature_of's code 0)
__device__ __forceinline__ bool inside(double u, double v, double tau) {
    return !(fabs(u) < tau || fabs(1.0 - u - v) < tau || fabs(v) < tau);
}

// true when an earlier record of the sorted list finds the same point on the
// same features (k_dedup_flags' rule)
__device__ __noinline__ bool tail_duplicate(const TailArgs &a, const uint32_t *base, const tms_hit &h, uint64_t key) {
    const int2 pr = a.pairs[h.pair];
    const MeshDev &ma = a.meshes[pr.x], &mb = a.meshes[pr.y];
    uint32_t incA[6], incB[6], t1[6], t2[6];
    int nA, nB, n1, n2;
    const uint32_t fA = feature_of(ma, h.triA, h.a, h.b, a.tau, incA, nA);
    const uint32_t fB = feature_of(mb, h.triB, h.c, h.d, a.tau, incB, nB);
    for (int p = 0; p < nA; ++p) {
        for (int q = 0; q < nB; ++q) {
            const uint64_t k2 = ((uint64_t)h.pair << (2 * a.tri_bits)) | ((uint64_t)incA[p] << a.tri_bits) |
                                (uint64_t)incB[q];
            if (k2 >= key) continue;
            const unsigned b = tail_bucket(k2, a.tri_bits, a.bscale);
            for (uint32_t e = base[b]; e < base[b + 1]; ++e) {
                if (__ldcg(a.bkey + e) != k2) continue;
                const tms_hit &o = a.raw[__ldcg(a.bidx + e)];
                if (feature_of(ma, o.triA, o.a, o.b, a.tau, t1, n1) == fA &&
                    feature_of(mb, o.triB, o.c, o.d, a.tau, t2, n2) == fB)
                    return true;
            }
        }
    }
    return false;
}

constexpr int kTailBlock = 1024, kTailCluster = 16;
__global__ void __launch_bounds__(kTailBlock) k_tail(TailArgs a) {
    constexpr int kPer = kTailBuckets / kTailBlock;
    constexpr unsigned kThreads = kTailBlock * kTailCluster;
    static_assert(kPer == 8, "two 16-byte loads a thread");
    __shared__ uint32_t base[kTailBuckets + 1];     // each bucket's first place
    __shared__ uint32_t wsum[kTailBlock / 32];
    unsigned n;
    const unsigned t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (!tail_count(a, n)) {                        // (every block of the cluster alike)
        if (blockIdx.x == 0) tail_readback(a);
        return;
    }
    const unsigned tid = blockIdx.x * kTailBlock + t;
    {
        const uint4 lo = reinterpret_cast<const uint4 *>(a.tail)[2 * t], hi = reinterpret_cast<const uint4 *>(a.tail)[2 * t + 1];
        const uint32_t c[kPer] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        uint32_t sum = 0, most = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            sum += c[k];
            most = max(most, c[k]);
        }
        uint32_t incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, incl, off);
            if (lane >= off) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
        if (__syncthreads_or(most > kTailUneven)) {  // (every block of the cluster alike)
            if (blockIdx.x == 0) {
                if (t == 0) a.ctr->status |= ST_TAIL_UNEVEN;
                __syncthreads();
                tail_readback(a);
            }
            return;
        }
        uint32_t before = __reduce_add_sync(FULL, lane < warp ? wsum[lane] : 0u) + incl - sum;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            base[kPer * t + k] = before;
            before += c[k];
        }
        if (t == kTailBlock - 1) base[kTailBuckets] = before;
        __syncthreads();
    }
    for (unsigned i = tid; i < n; i += kThreads) {
        const uint64_t key = a.key[i];
        const unsigned pos = base[tail_bucket(key, a.tri_bits, a.bscale)] + a.slot[i];
        a.bkey[pos] = key;
        a.bidx[pos] = i;
    }
    cluster_step();
    for (unsigned e = tid; e < n; e += kThreads) {
        const uint64_t key = __ldcg(a.bkey + e);
        const uint32_t idx = __ldcg(a.bidx + e);
        const unsigned b = tail_bucket(key, a.tri_bits, a.bscale);
        const uint32_t lo = base[b], hi = base[b + 1];
        uint32_t rank = lo;
        for (uint32_t j = lo; j < hi; ++j) rank += __ldcg(a.bkey + j) < key;
        const tms_hit &h = a.raw[idx];
        const bool shared = !(inside(h.a, h.b, a.tau) && inside(h.c, h.d, a.tau));
        if (shared && tail_duplicate(a, base, h, key)) {
            atomicOr(a.tail + kTailBuckets + (rank >> 5), 1u << (rank & 31));
            atomicAdd(&a.ctr->dropped, 1u);
        }
        a.skey[rank] = key;
        a.order[rank] = idx | (shared ? 0x80000000u : 0u);
    }
    cluster_step();
    // eight lanes a record, 16 bytes each
    const uint32_t *drop = a.tail + kTailBuckets;
    const unsigned dropped = __ldcg(&a.ctr->dropped), l = tid & 7;
    // records dropped before rank r, counted by the record's eight lanes (every
    // lane of the warp calls it together)
    auto before = [&](unsigned r) {
        if (dropped == 0) return 0u;
        unsigned s = 0;
        for (unsigned w = l; w < (r >> 5); w += 8) s += __popc(__ldcg(drop + w));
        s += __shfl_xor_sync(FULL, s, 1);
        s += __shfl_xor_sync(FULL, s, 2);
        s += __shfl_xor_sync(FULL, s, 4);
        return s + ((r & 31) ? __popc(__ldcg(drop + (r >> 5)) & ((1u << (r & 31)) - 1u)) : 0);
    };
    if (dropped == 0) {
        // every record is kept, in its rank's place: four of them a turn
        const unsigned m = (unsigned)(n < a.out_cap ? n : a.out_cap);
        for (unsigned r0 = tid >> 3; r0 < m; r0 += kThreads / 2) {
            uint32_t o[4];
            uint4 v[4];
#pragma unroll
            for (unsigned k = 0; k < 4; ++k) {
                const unsigned r = r0 + k * (kThreads / 8);
                o[k] = r < m ? __ldcg(a.order + r) : 0u;
            }
#pragma unroll
            for (unsigned k = 0; k < 4; ++k)
                if (r0 + k * (kThreads / 8) < m) v[k] = reinterpret_cast<const uint4 *>(a.raw + (o[k] & 0x7FFFFFFFu))[l];
#pragma unroll
            for (unsigned k = 0; k < 4; ++k) {
                const unsigned r = r0 + k * (kThreads / 8);
                if (l == 0 && (o[k] >> 31)) v[k].w |= 2u;        // flags
                if (r < m) reinterpret_cast<uint4 *>(a.out + r)[l] = v[k];
            }
        }
    }
    for (unsigned g0 = tid & ~31u; dropped != 0 && g0 < 8 * n; g0 += kThreads) {
        const unsigned r = (g0 + lane) >> 3;
        const unsigned pos = r - before(r < n ? r : 0);
        if (r >= n || ((__ldcg(drop + (r >> 5)) >> (r & 31)) & 1u)) continue;
        const uint32_t o = __ldcg(a.order + r);
        uint4 v = reinterpret_cast<const uint4 *>(a.raw + (o & 0x7FFFFFFFu))[l];
        if (l == 0 && (o >> 31)) v.w |= 2u;        // flags
        if (pos < a.out_cap) reinterpret_cast<uint4 *>(a.out + pos)[l] = v;
    }
    if (blockIdx.x == 0) {
        if (t == 0) a.ctr->out = n - dropped;
        __syncthreads();
        tail_readback(a);
    }
    // offsets: the records kept of earlier pairs, one pair per eight lanes
    if (a.offsets) {
        for (unsigned g0 = tid & ~31u; g0 < 8u * (a.n_pairs + 1); g0 += kThreads) {
            const unsigned p = (g0 + lane) >> 3;
            const uint64_t k = (uint64_t)p << (2 * a.tri_bits);
            unsigned lo = 0, hi = n;
            if (p >= (unsigned)a.n_pairs) lo = n;
            while (lo < hi) {
                const unsigned mid = (lo + hi) >> 1;
                if (__ldcg(a.skey + mid) < k) lo = mid + 1; else hi = mid;
            }
            const unsigned d = before(lo);
            if (l == 0 && p <= (unsigned)a.n_pairs) a.offsets[p] = (long long)(lo - d);
        }
    }
}

// ---------------------------------------------------------------------------
// adjoint of the hit outputs
// ---------------------------------------------------------------------------
// Two lanes a hit: the first solves A z = r (the hit's weights) while the second
// solves A^T w = zbar, then the first takes mesh A's gradients and the second mesh
// B's.  A few hundred hits leave the chip nearly idle, so the time is one chain of
// loads and dependent FP64 instructions (16 cycles a warp on an SM's FP64 pipe, which
// eight warps of a 256-thread block shared): blocks of one warp put every warp on an
// SM of its own, and the two solves run side by side.
constexpr int kAdjointHits = 16;       // per block of one warp
__global__ void __launch_bounds__(2 * kAdjointHits) k_adjoint(const __grid_constant__ AdjointArgs a) {
    const int role = threadIdx.x & 1;
    const long long step = (long long)gridDim.x * kAdjointHits;
    for (long long h0 = (long long)blockIdx.x * kAdjointHits; h0 < a.n; h0 += step) {
        const long long h = h0 + (threadIdx.x >> 1);
        const bool live = h < a.n;
        const tms_hit *hit = a.hits + (live ? h : a.n - 1);
        const uint32_t triA = hit->triA, triB = hit->triB;
        double x[3][4], y[3][4];
        gather_tri(a.A, triA, x);
        gather_tri(a.B, triB, y);
        // this lane's mesh: vertex offsets, and the alpha derivatives, read ahead of
        // the solve
        const MeshDev &m = role ? a.B : a.A;
        const double *const *dv = role ? a.dB : a.dA;
        int ii[3], kk[3];
        tri_ij(m, role ? triB : triA, ii, kk);
        size_t off[3];
        double d[3][4];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            off[j] = (size_t)kk[j] * m.N + ii[j];
#pragma unroll
            for (int c = 0; c < 4; ++c) d[j][c] = dv[c] ? __ldg(dv[c] + off[j]) : 0.0;
        }
        double gP[4] = {0, 0, 0, 0}, zbar[4] = {0, 0, 0, 0};
        const long long hr = live ? h : a.n - 1;
        if (a.gP) for (int c = 0; c < 4; ++c) gP[c] = a.gP[4 * hr + c];
        if (a.gZ) for (int c = 0; c < 4; ++c) zbar[c] = a.gZ[4 * hr + c];
        double M[4][4], rhs[4];
        {
            double F[4][4], r[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                F[c][0] = x[0][c] - x[1][c];
                F[c][1] = x[2][c] - x[1][c];
                F[c][2] = y[1][c] - y[0][c];
                F[c][3] = y[1][c] - y[2][c];
                r[c] = y[1][c] - x[1][c];
                zbar[0] += F[c][0] * gP[c];
                zbar[1] += F[c][1] * gP[c];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
#pragma unroll
                for (int j = 0; j < 4; ++j) M[i][j] = role ? F[j][i] : F[i][j];
                rhs[i] = role ? zbar[i] : r[i];
            }
        }
        double s[4], det;
        bool ok = solve4_gepp<double>(M, rhs, s, det);
        ok &= __shfl_xor_sync(FULL, (int)ok, 1) != 0;
        double z[4], w[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const double o = __shfl_xor_sync(FULL, s[c], 1);
            z[c] = role ? o : s[c];
            w[c] = role ? s[c] : o;
        }
        // weights of this lane's triangle, and its share of the gradient
        const double u = role ? z[2] : z[0], v = role ? z[3] : z[1];
        const double wt[3] = {u, 1.0 - u - v, v};
        double *const *g = role ? a.gB : a.gA;
        double ga = 0.0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double gv = wt[j] * (role ? w[c] : gP[c] - w[c]);
                if (live && ok && g[c]) atomicAdd(g[c] + off[j], gv);
                ga += gv * d[j][c];
            }
        }
        ga += __shfl_xor_sync(FULL, ga, 1);
        if (a.galpha && live && role == 0) a.galpha[h] = ok ? ga : 0.0;
    }
}

}  // namespace

void launch_narrow(const NarrowArgs &a, int face_level, int sms, cudaStream_t st) {
    if (!a.fp32_filter) {
        if (face_level == 0) k_narrow_all<0><<<sms * 16, kPairBlock, 0, st>>>(a);
        else k_narrow_all<1><<<sms * 16, kPairBlock, 0, st>>>(a);
        return;
    }
    if (face_level == 0) {
        k_quad_filter<0><<<sms * 3, 32 * kQuadWarps, 0, st>>>(a);
        k_narrow_filter<0><<<sms * 8, kPairBlock, 0, st>>>(a);
    } else {
        k_quad_filter<1><<<sms * 3, 32 * kQuadWarps, 0, st>>>(a);
        k_narrow_filter<1><<<sms * 8, kPairBlock, 0, st>>>(a);
    }
}

void launch_dedup(const DedupArgs &a, int grid, cudaStream_t st) {
    k_dedup_flags<<<grid, 256, 0, st>>>(a);
    scan_u32(a.keep, a.keep_scan, &a.ctr->raw_hits, a.raw_cap, a.partials, &a.ctr->out, grid, st);
    k_dedup_out<<<grid, 256, 0, st>>>(a);
    if (a.offsets)
        k_offsets<<<(a.n_pairs + 256) / 256, 256, 0, st>>>(a.out_keys, &a.ctr->out, a.raw_cap,
                                                            a.n_pairs, a.tri_bits, a.offsets);
}

// (a cluster of sixteen is above the size that every device has to take)
cudaError_t configure_tail() {
    return cudaFuncSetAttribute(k_tail, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

cudaError_t launch_tail(const TailArgs &a, cudaStream_t st) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kTailCluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(kTailCluster);
    c.blockDim = dim3(kTailBlock);
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, k_tail, a);
}

void launch_adjoint(const AdjointArgs &a, cudaStream_t st) {
    if (a.n <= 0) return;
    const long long blocks = (a.n + kAdjointHits - 1) / kAdjointHits;
    k_adjoint<<<(unsigned)(blocks < (1 << 16) ? blocks : (1 << 16)), 2 * kAdjointHits, 0, st>>>(a);
}

}  // namespace tms
