// Face passes of the broad phase.
//
// Broad phase of arXiv 2109.14814, Sec. 6.2.1-6.2.2, re-designed for GB300:
//   bounds pass      (one read of every vertex) per-mesh world bounds, widest
//                    face extent per coordinate (the grid rule of Sec. 6.2.1:
//                    cell edge > widest face), a finiteness check of every
//                    vertex, the vertices rounded down to FP32, and the box of
//                    every face (Sec. 6.2.2; at the patch level the boxes of the
//                    patches and their quarters and the patches' frames instead,
//                    and no world bounds: tms_tree.cu takes the patch boxes on);
//   cell passes      (face level; one read of every face box) the cells each face
//                    covers:
//     MODE_MARK        occupancy bits of the cells covered by mesh A's faces;
//     MODE_PROBE_MARK  mesh B: one entry per face-cell incidence in a cell that
//                      mesh A occupies, and those cells marked "hot";
//     MODE_PROBE       mesh A: one entry per face-cell incidence in a hot cell;
//     MODE_EMIT_ALL    one entry per face-cell incidence (no filter).
// Cells that do not hold faces of both meshes are dropped, as the paper drops
// grid boxes whose quad list is empty on either side (Sec. 6.3); the occupancy
// bitmaps only decide this before any list is built.  A bitmap is a blocked
// Bloom filter over hash(pair, cell): a false positive only adds entries, never
// removes one, so every face pair sharing a cell still meets in the sort.
//
// Bounds pass tiling: a block owns a tile of TI quads along theta x TK quad
// rows.  All (TI+1) x (TK+1) vertices of the tile are loaded once, coalesced
// along theta, into shared memory (rounded down to FP32 in the mixed precision
// mode), then each thread builds the boxes of its quads' faces.  (At the patch level
// a patch row's vertices at a time.)
//
// Cell passes: one thread per face slot; a warp expands its 32 faces' cell
// ranges into one list of (face, cell) items and works through it 32 items at
// a time, so its loop runs ceil(sum of cells / 32) times instead of 32 x the
// largest count.  An entry is (key = pair << 32 | cell << 1 | role, face id).
#include <cuda_runtime.h>
#include <float.h>
#include <stdint.h>
#include <string.h>

#include <type_traits>

#include "tms_common.cuh"

namespace tms {

namespace {

constexpr unsigned FULL = 0xffffffffu;

// A vertex as the boxes need it: its coordinates rounded down to FP32 (mixed
// precision; every exact coordinate then lies in [v, f32_above(v)], so the box of a
// set of vertices is [min v, f32_above(max v)] and one value a coordinate does), or
// as integers of the doubles' order (plain; minima, maxima and comparisons of doubles
// run on the FP64 pipe: the bounds pass of 1019 x 253 and 771 x 331 meshes took 99 us
// of it, and 22 us as integers).
template <int PREC>
struct Num;
template <>
struct Num<1> {
    typedef float T;
    static __device__ __forceinline__ float of(double x) { return f32_rd(x); }
    static __device__ __forceinline__ float above(float v) { return f32_above(v); }
    static __device__ __forceinline__ float inf() { return __int_as_float(0x7f800000); }
};
template <>
struct Num<0> {
    typedef long long T;
    static __device__ __forceinline__ long long of(double x) { return ord64(x); }
    static __device__ __forceinline__ long long above(long long v) { return v; }
    static __device__ __forceinline__ long long inf() { return 0x7fffffffffffffffLL; }
};

template <int PREC>
struct __align__(16) Vtx {
    typename Num<PREC>::T v[4];
};

// lo: the least, hi: the largest vertex value (closed() makes it the box)
template <int PREC>
struct BoxT {
    typename Num<PREC>::T lo[4], hi[4];
};

template <int PREC>
__device__ __forceinline__ void box_init(BoxT<PREC> &b, const Vtx<PREC> &v) {
#pragma unroll
    for (int d = 0; d < 4; ++d) { b.lo[d] = v.v[d]; b.hi[d] = v.v[d]; }
}
template <int PREC>
__device__ __forceinline__ void box_add(BoxT<PREC> &b, const Vtx<PREC> &v) {
#pragma unroll
    for (int d = 0; d < 4; ++d) { b.lo[d] = min(b.lo[d], v.v[d]); b.hi[d] = max(b.hi[d], v.v[d]); }
}
template <int PREC>
__device__ __forceinline__ BoxT<PREC> closed(BoxT<PREC> b) {
#pragma unroll
    for (int d = 0; d < 4; ++d) b.hi[d] = Num<PREC>::above(b.hi[d]);
    return b;
}

// a vertex in the boxes' numbers; top takes high words of coordinates (shifted left by
// one), those of a coordinate that is not finite among them
static __device__ __noinline__ float4 rd_special4(double x, double y, double z, double w) {
    return make_float4(f32_rd(x), f32_rd(y), f32_rd(z), f32_rd(w));
}
__device__ __forceinline__ unsigned top_word(const double x[4]) {
    unsigned t = 0;
#pragma unroll
    for (int d = 0; d < 4; ++d) t = max(t, 2u * (unsigned)__double2hiint(x[d]));
    return t;
}
template <int PREC>
__device__ __forceinline__ Vtx<PREC> to_vtx(const double x[4], unsigned &top);
template <>
__device__ __forceinline__ Vtx<1> to_vtx<1>(const double x[4], unsigned &top) {
    Vtx<1> v;
    unsigned r = 0;
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        r = max(r, f32_range(x[d]));
        v.v[d] = f32_rd_normal(x[d]);
    }
    if (r >= kF32Range) {
        const float4 s = rd_special4(x[0], x[1], x[2], x[3]);
        v.v[0] = s.x; v.v[1] = s.y; v.v[2] = s.z; v.v[3] = s.w;
        top = max(top, top_word(x));
    }
    return v;
}
template <>
__device__ __forceinline__ Vtx<0> to_vtx<0>(const double x[4], unsigned &top) {
    Vtx<0> v;
#pragma unroll
    for (int d = 0; d < 4; ++d) v.v[d] = ord64(x[d]);
    top = max(top, top_word(x));
    return v;
}

// the rounded vertex, gathered later (MeshDev::vlo)
__device__ __forceinline__ void write_vlo(const MeshDev &m, size_t idx, const Vtx<1> &v) {
    m.vlo[idx] = make_float4(v.v[0], v.v[1], v.v[2], v.v[3]);
}
__device__ __forceinline__ void write_vlo(const MeshDev &m, size_t idx, const Vtx<0> &v) {
    if (m.vlo)
        m.vlo[idx] = make_float4(f32_rd(ord64_value(v.v[0])), f32_rd(ord64_value(v.v[1])),
                                 f32_rd(ord64_value(v.v[2])), f32_rd(ord64_value(v.v[3])));
}

template <int PREC>
struct GridView;
template <>
struct GridView<1> {
    float o[4], e[4], inv[4];
    int n[4];
    __device__ void load(const Grid &g) {
#pragma unroll
        for (int d = 0; d < 4; ++d) { o[d] = g.o32[d]; e[d] = g.e32[d]; inv[d] = g.inv32[d]; n[d] = g.n[d]; }
    }
    __device__ int cell(float v, int d) const { return cell_of(v, o[d], inv[d], n[d]); }
};
template <>
struct GridView<0> {
    double origin[4], inv[4];
    long long o[4], e[4];
    int n[4];
    __device__ void load(const Grid &g) {
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            origin[d] = g.o64[d]; o[d] = ord64(g.o64[d]); e[d] = ord64(g.e64[d]); inv[d] = g.inv64[d]; n[d] = g.n[d];
        }
    }
    __device__ int cell(long long v, int d) const { return cell_of(ord64_value(v), origin[d], inv[d], n[d]); }
};

// the (closed) box of a face or patch into slot `face` of a box array
template <int PREC>
__device__ __forceinline__ void write_box(void *arr, uint32_t face, const BoxT<PREC> &b);
template <>
__device__ __forceinline__ void write_box<1>(void *arr, uint32_t face, const BoxT<1> &b) {
    float4 *p = reinterpret_cast<float4 *>(arr) + 2 * (size_t)face;
    p[0] = make_float4(b.lo[0], b.lo[1], b.lo[2], b.lo[3]);
    p[1] = make_float4(b.hi[0], b.hi[1], b.hi[2], b.hi[3]);
}
template <>
__device__ __forceinline__ void write_box<0>(void *arr, uint32_t face, const BoxT<0> &b) {
    longlong2 *p = reinterpret_cast<longlong2 *>(arr) + 4 * (size_t)face;
    p[0] = make_longlong2(b.lo[0], b.lo[1]);
    p[1] = make_longlong2(b.lo[2], b.lo[3]);
    p[2] = make_longlong2(b.hi[0], b.hi[1]);
    p[3] = make_longlong2(b.hi[2], b.hi[3]);
}
// one side of a (closed) box: lo (side 0) or hi (side 1) of slot `face`
__device__ __forceinline__ void write_side(void *arr, uint32_t face, int side, const float v[4]) {
    reinterpret_cast<float4 *>(arr)[2 * (size_t)face + side] = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void write_side(void *arr, uint32_t face, int side, const long long v[4]) {
    longlong2 *p = reinterpret_cast<longlong2 *>(arr) + 4 * (size_t)face + 2 * side;
    p[0] = make_longlong2(v[0], v[1]);
    p[1] = make_longlong2(v[2], v[3]);
}
template <int PREC>
__device__ __forceinline__ void write_fbox(const MeshDev &m, uint32_t face, const BoxT<PREC> &b) {
    write_box<PREC>(m.fbox, face, closed<PREC>(b));
}

// The least and the negated largest of a vertex column's values over some rows (minima
// only, so that lanes can reduce either alike).
template <int PREC>
struct ColBox {
    typename Num<PREC>::T lo[4], nh[4];
    __device__ __forceinline__ void init() {
#pragma unroll
        for (int d = 0; d < 4; ++d) lo[d] = nh[d] = Num<PREC>::inf();
    }
    __device__ __forceinline__ void add(const Vtx<PREC> &v) {
#pragma unroll
        for (int d = 0; d < 4; ++d) { lo[d] = min(lo[d], v.v[d]); nh[d] = min(nh[d], -v.v[d]); }
    }
};

template <int PREC>
__device__ __forceinline__ void read_fbox(const MeshDev &m, uint32_t face, BoxT<PREC> &b);
template <>
__device__ __forceinline__ void read_fbox<1>(const MeshDev &m, uint32_t face, BoxT<1> &b) {
    const float4 *p = reinterpret_cast<const float4 *>(m.fbox) + 2 * (size_t)face;
    const float4 l = __ldg(p), h = __ldg(p + 1);
    b.lo[0] = l.x; b.lo[1] = l.y; b.lo[2] = l.z; b.lo[3] = l.w;
    b.hi[0] = h.x; b.hi[1] = h.y; b.hi[2] = h.z; b.hi[3] = h.w;
}
template <>
__device__ __forceinline__ void read_fbox<0>(const MeshDev &m, uint32_t face, BoxT<0> &b) {
    const longlong2 *p = reinterpret_cast<const longlong2 *>(m.fbox) + 4 * (size_t)face;
    const longlong2 x0 = __ldg(p), x1 = __ldg(p + 1), x2 = __ldg(p + 2), x3 = __ldg(p + 3);
    b.lo[0] = x0.x; b.lo[1] = x0.y; b.lo[2] = x1.x; b.lo[3] = x1.y;
    b.hi[0] = x2.x; b.hi[1] = x2.y; b.hi[2] = x3.x; b.hi[3] = x3.y;
}

__device__ __forceinline__ float extent(float lo, float hi) { return hi - lo; }
__device__ __forceinline__ long long extent(long long lo, long long hi) {
    return __double_as_longlong(ord64_value(hi) - ord64_value(lo));
}

// Per-thread accumulators of the bounds pass, in the boxes' numbers
template <int PREC>
struct BoundAcc {
    typename Num<PREC>::T lo[4], hi[4], w[4];   // w: extents (plain: the bits of doubles >= 0)
    unsigned seen;
    __device__ void init() {
#pragma unroll
        for (int d = 0; d < 4; ++d) { lo[d] = Num<PREC>::inf(); hi[d] = -lo[d]; w[d] = 0; }
        seen = 0;
    }
    __device__ void add(const BoxT<PREC> &raw) {
        const BoxT<PREC> b = closed<PREC>(raw);
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            lo[d] = min(lo[d], b.lo[d]);
            hi[d] = max(hi[d], b.hi[d]);
            w[d] = max(w[d], extent(b.lo[d], b.hi[d]));
        }
        seen = 1;
    }
};

// ord_enc of the value as a double: ordered integers directly; FP32 values through the
// exact float -> double conversion done on the bits (integer operations only)
__device__ __forceinline__ unsigned long long ord_enc_any(long long v) {
    return (unsigned long long)v ^ 0x8000000000000000ULL;
}
__device__ __forceinline__ unsigned long long ord_enc_any(float v) {
    const unsigned b = __float_as_uint(v);
    const unsigned long long sgn = (unsigned long long)(b >> 31) << 63;
    const unsigned e = (b >> 23) & 0xffu, m = b & 0x7fffffu;
    unsigned long long db;
    if (e == 255u) {
        db = sgn | (0x7ffULL << 52) | ((unsigned long long)m << 29);          // inf, NaN
    } else if (e == 0u) {
        if (m == 0u) {
            db = sgn;                                                         // +-0
        } else {
            // subnormal m 2^-149 = 1.f 2^(p - 149), p the top bit of m
            const int p = 31 - __clz(m);
            const unsigned long long frac = ((unsigned long long)m << (52 - p)) & 0xFFFFFFFFFFFFFULL;
            db = sgn | ((unsigned long long)(p - 149 + 1023) << 52) | frac;
        }
    } else {
        db = sgn | ((unsigned long long)(e + 896u) << 52) | ((unsigned long long)m << 29);
    }
    const long long bb = (long long)db;
    return (bb >= 0) ? (db | 0x8000000000000000ULL) : ~db;
}

// Maxima over a warp, as integers of the values' order: FP32 values by one instruction
// on their bits (negative ones with the magnitude's bits flipped), ordered 64-bit
// integers by shuffles.  A minimum is a maximum of the complements (negated).
__device__ __forceinline__ int ord32(float v) {
    const int b = __float_as_int(v);
    return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ long long warp_max(float v) { return __reduce_max_sync(FULL, ord32(v)); }
__device__ __forceinline__ long long warp_max(int v) { return __reduce_max_sync(FULL, v); }
__device__ __forceinline__ long long warp_max(long long v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = max(v, __shfl_xor_sync(FULL, v, off));
    return v;
}
__device__ __forceinline__ int negated(float v) { return ~ord32(v); }
__device__ __forceinline__ long long negated(long long v) { return ~v; }
// the Bounds encoding of a reduced value
template <int PREC>
__device__ __forceinline__ unsigned long long encoded(long long v) {
    if (PREC == 0) return ord_enc_any(v);
    const int b = (int)v;
    return ord_enc_any(__int_as_float(b ^ ((b >> 31) & 0x7fffffff)));
}

// the pass entry (mesh of a pass) holding global index x, by binary search
__device__ __forceinline__ int find_entry(const FacePassArgs &a, long long x, bool by_face) {
    int lo = 0, hi = a.n_entries - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        const long long b = by_face ? a.entries[mid].face_base : a.entries[mid].tile_base;
        if (b <= x) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------------------
// patch frames (mixed precision; the record and its bounds are described at
// kFrameF4).  The axes need not be orthonormal for the bounds to hold: the
// remainder r absorbs whatever the rounded axes fail to reproduce, and is
// bounded through the axes' Gram matrix.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float dot4f(const float a[4], const float b[4]) {
    return fmaf(a[3], b[3], fmaf(a[2], b[2], fmaf(a[1], b[1], a[0] * b[0])));
}
__device__ __forceinline__ float det3(float a0, float a1, float a2, float b0, float b1, float b2,
                                      float c0, float c1, float c2) {
    return a0 * (b1 * c2 - b2 * c1) - a1 * (b0 * c2 - b2 * c0) + a2 * (b0 * c1 - b1 * c0);
}
// the vector orthogonal to a, b and c in R^4 (cofactor expansion of the
// 4 x 4 determinant with rows (x, a, b, c))
__device__ __forceinline__ void cross4(const float a[4], const float b[4], const float c[4], float x[4]) {
    x[0] = det3(a[1], a[2], a[3], b[1], b[2], b[3], c[1], c[2], c[3]);
    x[1] = -det3(a[0], a[2], a[3], b[0], b[2], b[3], c[0], c[2], c[3]);
    x[2] = det3(a[0], a[1], a[3], b[0], b[1], b[3], c[0], c[1], c[3]);
    x[3] = -det3(a[0], a[1], a[2], b[0], b[1], b[2], c[0], c[1], c[2]);
}
// the maximum that keeps a NaN (fmaxf would drop it)
__device__ __forceinline__ float max_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// The frame of a patch, in three steps over the tile's patches: one thread a patch
// computes the axes (frame_axes), the patch's kPatchI lanes project its vertices on
// them (frame_extents), and one thread a patch closes the bounds and writes the record
// (frame_write).  What is the same for a whole patch runs on as many threads as there
// are patches (16 of a 128 x 4 tile): computed by all of a patch's lanes it was a third
// of the kernel's instructions (65.6 M and 87 us at 4096 x 512 then, 54.5 M and 72 us so).
// Axes: e_0, e_1 from the patch's two parameter directions (sums of opposite
// edges, one Gram-Schmidt step), e_2 orthogonal to e_0, e_1 and the coordinate
// axis farthest from their span, e_3 orthogonal to e_0, e_1, e_2.  A patch
// whose parameter directions are zero or unbounded gets a frame that
// separates nothing.
// Bounds, with u = 2^-24, the exact vertex V in its FP32 bounds [lo, hi] and
// d = V - c:
//   |d|_inf <= D = max_i max(pb.hi_i - c_i, c_i - pb.lo_i)   (all V in pb)
//   hi_i - lo_i <= 2^-23 L + 2^-149                           (adjacent floats)
//   d~ = fl(lo - c): |d_i - d~_i| <= (hi_i - lo_i) + u |d~_i|, |d~_i| <= D (1 + u)
//   a~_k = fl(e_k . d~) (4 FMAs, error <= gamma_4 sum_i |e_ki||d~_i|, gamma_4 <
//   4.0001 u), so |e_k . d - a~_k| <= n_k nu, nu = 2^-23 L + 5.001 u D (+ 2^-149)
//   and h_k = max |a~_k| + n_k nu (n_k >= |e_k|_1);
//   r = (I - E^T E) d, so |r|_inf <= g D with g >= ||I - E^T E||_inf, from
//   G~_ij = fl(delta_ij - sum_k e_ki e_kj) (4 FMAs, error <= gamma_4 (1 + 4 e_max^2)).
// Sums and products of non-negative terms are rounded up by a factor 1.0001
// (a handful of roundings of 2^-24 each); absolute terms cover underflow.
struct PatchScratch {         // of a patch of the tile
    float4 lo, hi;            // its (closed) box
    float4 axes[5];           // c, e_0..e_3
    float4 top;               // max |e_k . (V - c)|
    uint4 flags;              // x: no usable axes
};

__device__ __forceinline__ void patch_centre(const PatchScratch &P, float c[4], float &L, float &D) {
    const float lo[4] = {P.lo.x, P.lo.y, P.lo.z, P.lo.w}, hi[4] = {P.hi.x, P.hi.y, P.hi.z, P.hi.w};
    L = D = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        c[i] = 0.5f * (lo[i] + hi[i]);
        L = fmaxf(L, fmaxf(fabsf(lo[i]), fabsf(hi[i])));
        D = fmaxf(D, fmaxf(hi[i] - c[i], c[i] - lo[i]));
    }
    D *= 1.0001f;
}

// sv: the tile's vertices; p0, cq: the patch's first quad column in the tile and its
// columns, pr0, rq: its quad rows
__device__ __forceinline__ void frame_axes(const Vtx<1> *sv, int W, int p0, int cq, int pr0, int rq, PatchScratch &P) {
    const int pr1 = pr0 + rq;
    float c[4], L, D;
    patch_centre(P, c, L, D);
    float t1[4], t2[4];
    {
        const float4 v00 = *reinterpret_cast<const float4 *>(sv[pr0 * W + p0].v);
        const float4 v01 = *reinterpret_cast<const float4 *>(sv[pr0 * W + p0 + cq].v);
        const float4 v10 = *reinterpret_cast<const float4 *>(sv[pr1 * W + p0].v);
        const float4 v11 = *reinterpret_cast<const float4 *>(sv[pr1 * W + p0 + cq].v);
        t1[0] = (v01.x - v00.x) + (v11.x - v10.x); t2[0] = (v10.x - v00.x) + (v11.x - v01.x);
        t1[1] = (v01.y - v00.y) + (v11.y - v10.y); t2[1] = (v10.y - v00.y) + (v11.y - v01.y);
        t1[2] = (v01.z - v00.z) + (v11.z - v10.z); t2[2] = (v10.z - v00.z) + (v11.z - v01.z);
        t1[3] = (v01.w - v00.w) + (v11.w - v10.w); t2[3] = (v10.w - v00.w) + (v11.w - v01.w);
    }
    float E[4][4];
    const float n1 = dot4f(t1, t1);
    const float s1 = rsqrtf(n1);
#pragma unroll
    for (int i = 0; i < 4; ++i) E[0][i] = t1[i] * s1;
    const float pj = dot4f(t2, E[0]);
#pragma unroll
    for (int i = 0; i < 4; ++i) t2[i] = fmaf(-pj, E[0][i], t2[i]);
    const float n2 = dot4f(t2, t2);
    const float s2 = rsqrtf(n2);
#pragma unroll
    for (int i = 0; i < 4; ++i) E[1][i] = t2[i] * s2;
    // zero or unbounded parameter directions: no frame
    const bool bad = !(n1 > 1e-30f && n1 < 1e30f && n2 > 1e-30f && n2 < 1e30f);
    {
        // e_2 from the coordinate axis k farthest from span(e_0, e_1): the one
        // with the least e_0k^2 + e_1k^2 (|cross4(e_0, e_1, axis_k)|^2 is one minus
        // that for orthonormal e_0, e_1)
        int kb = 0;
        float best = __int_as_float(0x7f800000);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float sk = fmaf(E[0][k], E[0][k], E[1][k] * E[1][k]);
            if (sk < best) { best = sk; kb = k; }
        }
        float ax[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) ax[i] = i == kb ? 1.0f : 0.0f;
        float x[4];
        cross4(E[0], E[1], ax, x);
        const float s3 = rsqrtf(dot4f(x, x));
#pragma unroll
        for (int i = 0; i < 4; ++i) E[2][i] = x[i] * s3;
        cross4(E[0], E[1], E[2], x);
        const float s4 = rsqrtf(dot4f(x, x));
#pragma unroll
        for (int i = 0; i < 4; ++i) E[3][i] = x[i] * s4;
    }
    P.axes[0] = make_float4(c[0], c[1], c[2], c[3]);
#pragma unroll
    for (int k = 0; k < 4; ++k) P.axes[1 + k] = make_float4(E[k][0], E[k][1], E[k][2], E[k][3]);
    P.flags.x = bad;
}

// Lane l of a patch takes its vertex column l (its own vertices, rows 0..rq of the patch)
// and, for l <= rq, the vertex of the closing column in row l.  Every lane of the warp
// calls it (cq = 0: no patch).
__device__ __forceinline__ void frame_extents(const Vtx<1> *sv, const Vtx<1> *own, int W, int t, int cq, int pr0, int rq,
                                              PatchScratch &P) {
    const int l = t & (kPatchI - 1), p0 = t - l;
    float am[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (cq > 0) {
        const float4 c = P.axes[0], e0 = P.axes[1], e1 = P.axes[2], e2 = P.axes[3], e3 = P.axes[4];
        auto vertex = [&](const Vtx<1> &v) {
            const float4 x = *reinterpret_cast<const float4 *>(v.v);
            const float d[4] = {x.x - c.x, x.y - c.y, x.z - c.z, x.w - c.w};
            auto dot = [&](const float4 &e) {
                return fabsf(fmaf(e.w, d[3], fmaf(e.z, d[2], fmaf(e.y, d[1], e.x * d[0]))));
            };
            am[0] = max_nan(am[0], dot(e0));
            am[1] = max_nan(am[1], dot(e1));
            am[2] = max_nan(am[2], dot(e2));
            am[3] = max_nan(am[3], dot(e3));
        };
        if (l < cq) {
#pragma unroll
            for (int rr = 0; rr <= kPatchK; ++rr)
                if (rr <= rq) vertex(own[rr]);
        }
        if (l <= rq) vertex(sv[(pr0 + l) * W + p0 + cq]);
    }
#pragma unroll
    for (int off = 1; off < kPatchI; off <<= 1)
#pragma unroll
        for (int k = 0; k < 4; ++k) am[k] = max_nan(am[k], __shfl_xor_sync(0xffffffffu, am[k], off));
    if (cq > 0 && l == 0) P.top = make_float4(am[0], am[1], am[2], am[3]);
}

__device__ __forceinline__ void frame_write(const PatchScratch &P, float4 *out, uint32_t p) {
    const float u = 5.9604645e-08f;
    const float inf = __int_as_float(0x7f800000);
    float c[4], L, D;
    patch_centre(P, c, L, D);
    float E[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 e = P.axes[1 + k];
        E[k][0] = e.x; E[k][1] = e.y; E[k][2] = e.z; E[k][3] = e.w;
    }
    const float am[4] = {P.top.x, P.top.y, P.top.z, P.top.w};
    bool bad = P.flags.x != 0;
    float nk[4], emax = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        nk[k] = (fabsf(E[k][0]) + fabsf(E[k][1]) + fabsf(E[k][2]) + fabsf(E[k][3])) * 1.0001f;
        emax = fmaxf(emax, fmaxf(fmaxf(fabsf(E[k][0]), fabsf(E[k][1])), fmaxf(fabsf(E[k][2]), fabsf(E[k][3]))));
    }
    // |I - E^T E| (symmetric: ten entries)
    float G[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = i; j < 4; ++j) {
            float gij = i == j ? 1.0f : 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k) gij = fmaf(-E[k][i], E[k][j], gij);
            G[i][j] = G[j][i] = fabsf(gij);
        }
    float g = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) g = fmaxf(g, (G[i][0] + G[i][1]) + (G[i][2] + G[i][3]));
    g = fmaf((4.0f * 4.0001f) * u, fmaf(4.0f * emax, emax, 1.0f), g) * 1.0001f;
    const float nu = fmaf(5.001f * u, D, 1.1921e-7f * L) * 1.0001f + 1e-30f;
    float h[4], hs = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        h[k] = fmaf(nk[k], nu, am[k]) * 1.0001f + 1e-36f;
        hs += h[k];
        bad |= !(h[k] < inf);
    }
    // plus the rounding of fl(w . e_k) in the pair test: gamma_4 |w|_1 e_max
    // per unit of h_k
    float rho = fmaf((4.0001f * u) * emax, hs * 1.0001f, g * D * 1.0001f) * 1.0001f + 1e-36f;
    bad |= !(rho < inf) || !(fabsf(E[2][0] + E[2][1] + E[2][2] + E[2][3] + E[3][0] + E[3][1] + E[3][2] + E[3][3]) < inf);
    if (bad) {
        h[0] = h[1] = h[2] = h[3] = inf;
        rho = inf;
    }
    float4 *o = out + (size_t)p * kFrameF4;
#pragma unroll
    for (int k = 0; k < 5; ++k) o[k] = P.axes[k];
    o[5] = make_float4(h[0], h[1], h[2], h[3]);
    o[6] = make_float4(rho, L, nk[2], nk[3]);
}

// ---------------------------------------------------------------------------
// bounds pass
// ---------------------------------------------------------------------------
// Registers, mixed precision: 64 a thread for tiles of 4 rows (a few of the vertices in
// flight are spilled), 80 for those of 8: 64 pairs of meshes from 128 x 32 to 2048 x 512
// vertices took 960 us a search with the 100 that 4 rows would take, 840 with 80, 802 with
// 64; with 8 rows (a patch row at a time) the pass takes 398 us with 80, 411 with 64, and
// 449 with 128 and the next patch row's loads before the current one's boxes.
template <int PREC, int FACE, int TK>
__global__ void __launch_bounds__(256, PREC == 1 ? (TK == 4 ? 4 : 3) : 2) k_bounds_pass(FacePassArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Vtx<PREC> *sv = reinterpret_cast<Vtx<PREC> *>(smem_raw);
    const int TI = blockDim.x;
    const int W = TI + 1;
    PatchScratch *sp = reinterpret_cast<PatchScratch *>(sv + (TK + 1) * W);   // with frames: the tile's patches
    const long long tile = blockIdx.x;

    const PassEntry pe = a.entries[find_entry(a, tile, false)];
    const MeshDev m = a.meshes[pe.mesh];
    const long long lt = tile - pe.tile_base;
    const int ti = (int)(lt % pe.tiles_i), tk = (int)(lt / pe.tiles_i);
    const int i0 = ti * TI, kq0 = tk * TK;
    const int cols_q = min(TI, m.nqi - i0);
    const int rows_q = min(TK, m.nqk - kq0);

    // ---- load the tile's vertices: rows kq0..kq0+rows_q, columns i0..i0+cols_q
    // the largest high word of |x| tells whether any is not finite (a test of each value
    // beside its rounding becomes an FP64 comparison)
    unsigned top = 0;
    const int t = threadIdx.x;
    const bool col_valid = t < cols_q;
    const int i = i0 + t;
    // a vertex is written by the tile that owns it: rows below the tile's last
    // (the next tile's first) and the mesh's last row
    const bool last_rows = kq0 + rows_q == m.nqk;
    // this thread's vertex column over a patch row: rows r0..r0 + kPatchK of the tile (the
    // first of them, where r0 > 0, as the last of the patch row before)
    Vtx<PREC> own[kPatchK + 1];
    auto load_rows = [&](int r0, bool first) {
        double x[kPatchK + 1][4];
#pragma unroll
        for (int r = 0; r <= kPatchK; ++r) {
            if (r == 0 && !first) continue;
            if (col_valid && r0 + r <= rows_q) {
                const size_t off = (size_t)(kq0 + r0 + r) * m.N + i;
#pragma unroll
                for (int c = 0; c < 4; ++c) x[r][c] = __ldg(m.c[c] + off);
            }
        }
        if (!first) own[0] = own[kPatchK];
#pragma unroll
        for (int r = 0; r <= kPatchK; ++r) {
            if (r == 0 && !first) continue;
            if (col_valid && r0 + r <= rows_q) {
                own[r] = to_vtx<PREC>(x[r], top);
                sv[(r0 + r) * W + t] = own[r];
                if (r0 + r < rows_q || last_rows) write_vlo(m, (size_t)(kq0 + r0 + r) * m.N + i, own[r]);
            }
        }
    };
    load_rows(0, true);
    // the last vertex column of the tile (wraps to column 0 on a periodic mesh);
    // it belongs to the next tile, except an open mesh's last column
    if (t <= rows_q) {
        int vj = i0 + cols_q;
        if (vj == m.N) vj = 0;
        size_t off = (size_t)(kq0 + t) * m.N + vj;
        double y[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) y[c] = __ldg(m.c[c] + off);
        const Vtx<PREC> v = to_vtx<PREC>(y, top);
        sv[t * W + cols_q] = v;
        if (!m.periodic && vj == m.N - 1 && (t < rows_q || last_rows)) write_vlo(m, off, v);
    }
    if (!(FACE == 1 && a.patch)) {
#pragma unroll
        for (int r0 = kPatchK; r0 < TK; r0 += kPatchK) load_rows(r0, false);
    }
    __syncthreads();

    BoundAcc<PREC> acc;                // world bounds and widest face (face level)
    acc.init();

    if (FACE == 1 && a.patch) {
        // quad faces with patches.  A quarter (four columns by two rows of quads) is the
        // union of five vertex columns over three rows: each lane takes its own column,
        // the four lanes share out the closing column's rows, and exchange so that lane
        // j ends with one side (j & 1: lo, hi) of one of the two quarters (j & 2: upper,
        // lower), which it closes and writes; the patch is their union.  (Every lane of
        // the block takes part: the row loop and its shuffles are uniform.)  With a box
        // for each quad, every lane reducing whole boxes, and each coordinate's rounding
        // tested alone the kernel took 48.8 M instructions and 64 us at 4096 x 512; so
        // 38.4 M (with 64 registers, tiles of 4 rows) and 53 us.
        static_assert(kPatchI == 8 && kPatchK == 4 && TK % kPatchK == 0, "quarters of four columns by two rows");
        typedef typename Num<PREC>::T T;
        const int j = t & 3;
        // the patch exists when its first column is in the tile
        const bool patch_lane = (t & ~(kPatchI - 1)) < cols_q;
        const int close = min((t & ~3) + 4, cols_q);      // the quarter's closing column
#pragma unroll
        for (int pr = 0; pr < TK / kPatchK; ++pr) {
            const int pr0 = pr * kPatchK, rq = min(kPatchK, rows_q - pr0);
            if (rq <= 0) break;
            if (pr > 0) {
                load_rows(pr0, false);
                __syncthreads();
            }
            ColBox<PREC> upper, lower;
            upper.init();
            lower.init();
            if (col_valid) {
                upper.add(own[0]);
                upper.add(own[1]);
                if (rq > 1) upper.add(own[2]);
                if (rq > 2) {
                    lower.add(own[2]);
                    lower.add(own[3]);
                    if (rq > 3) lower.add(own[4]);
                }
            }
            if ((t & ~3) < cols_q) {
                if (j <= rq) {
                    const Vtx<PREC> v = sv[(pr0 + j) * W + close];
                    if (j <= 2) upper.add(v);
                    if (j >= 2 && rq > 2) lower.add(v);
                }
                if (j == 0 && rq > 3) lower.add(sv[(pr0 + 4) * W + close]);
            }
            T s[4];
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                const bool odd = t & 1, low = t & 2;
                const T u = min(odd ? upper.nh[d] : upper.lo[d],
                                __shfl_xor_sync(FULL, odd ? upper.lo[d] : upper.nh[d], 1));
                const T w = min(odd ? lower.nh[d] : lower.lo[d],
                                __shfl_xor_sync(FULL, odd ? lower.lo[d] : lower.nh[d], 1));
                s[d] = min(low ? w : u, __shfl_xor_sync(FULL, low ? u : w, 2));
            }
            const uint32_t p = (uint32_t)(kq0 / kPatchK + pr) * (uint32_t)m.npi + (uint32_t)(i / kPatchI);
            T out[4];
#pragma unroll
            for (int d = 0; d < 4; ++d) out[d] = t & 1 ? Num<PREC>::above(-s[d]) : s[d];
            if (patch_lane) write_side(m.qbox, 4 * p + (t & 2) + ((t >> 2) & 1), t & 1, out);
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                s[d] = min(s[d], __shfl_xor_sync(FULL, s[d], 2));
                s[d] = min(s[d], __shfl_xor_sync(FULL, s[d], 4));
                out[d] = t & 1 ? Num<PREC>::above(-s[d]) : s[d];
            }
            if (patch_lane && (t & (kPatchI - 2)) == 0) {
                write_side(m.pbox, p, t & 1, out);
                if constexpr (PREC == 1) {
                    PatchScratch &P = sp[pr * (TI / kPatchI) + t / kPatchI];
                    (t & 1 ? P.hi : P.lo) = make_float4(out[0], out[1], out[2], out[3]);
                }
            }
        }
        // the frames of the tile's patches
        if constexpr (PREC == 1) {
            if (a.frames) {
                const int across = TI / kPatchI, np = across * ((rows_q + kPatchK - 1) / kPatchK);
                __syncthreads();
                for (int q = t; q < np; q += TI) {
                    const int p0 = (q % across) * kPatchI, pr0 = (q / across) * kPatchK;
                    if (p0 < cols_q)
                        frame_axes(sv, W, p0, min(kPatchI, cols_q - p0), pr0, min(kPatchK, rows_q - pr0), sp[q]);
                }
                __syncthreads();
                const int cq = patch_lane ? min(kPatchI, cols_q - (t & ~(kPatchI - 1))) : 0;
                // (the last patch row's vertices are still the thread's own)
                for (int pr0 = (rows_q - 1) / kPatchK * kPatchK;; pr0 -= kPatchK) {
                    frame_extents(sv, own, W, t, cq, pr0, min(kPatchK, rows_q - pr0),
                                  sp[(pr0 / kPatchK) * across + t / kPatchI]);
                    if (pr0 == 0) break;
                    if (col_valid) {
#pragma unroll
                        for (int r = 0; r <= kPatchK; ++r) own[r] = sv[(pr0 - kPatchK + r) * W + t];
                    }
                }
                __syncthreads();
                for (int q = t; q < np; q += TI)
                    if ((q % across) * kPatchI < cols_q)
                        frame_write(sp[q], m.pframe,
                                    (uint32_t)(kq0 / kPatchK + q / across) * (uint32_t)m.npi +
                                        (uint32_t)(i0 / kPatchI + q % across));
            }
        }
    } else if (FACE == 1 && col_valid) {
        // quad faces: the extremes of the two vertex columns of each row once, each
        // quad box from two consecutive rows (exact: min and max only)
        BoxT<PREC> prev;
        box_init(prev, sv[t]);
        box_add(prev, sv[t + 1]);
        for (int r = 0; r < rows_q; ++r) {
            BoxT<PREC> next;
            box_init(next, sv[(r + 1) * W + t]);
            box_add(next, sv[(r + 1) * W + t + 1]);
            BoxT<PREC> bq;
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                bq.lo[d] = min(prev.lo[d], next.lo[d]);
                bq.hi[d] = max(prev.hi[d], next.hi[d]);
            }
            const uint32_t q = (uint32_t)(kq0 + r) * (uint32_t)m.N + (uint32_t)i;
            acc.add(bq);
            write_fbox<PREC>(m, q, bq);
            prev = next;
        }
    } else if (FACE == 0 && col_valid) {
        for (int r = 0; r < rows_q; ++r) {
            const int k = kq0 + r;
            const Vtx<PREC> va = sv[r * W + t];             // (i, k)
            const Vtx<PREC> vb = sv[r * W + t + 1];         // (i+1, k)
            const Vtx<PREC> vc = sv[(r + 1) * W + t];       // (i, k+1)
            const Vtx<PREC> vd = sv[(r + 1) * W + t + 1];   // (i+1, k+1)
            const uint32_t q = (uint32_t)k * (uint32_t)m.N + (uint32_t)i;
            BoxT<PREC> b1, b2;
            box_init(b1, vb); box_add(b1, va); box_add(b1, vc);   // T1: x1=(i+1,k) x2=(i,k) x3=(i,k+1)
            box_init(b2, vc); box_add(b2, vd); box_add(b2, vb);   // T2: x1=(i,k+1) x2=(i+1,k+1) x3=(i+1,k)
            acc.add(b1);
            acc.add(b2);
            write_fbox<PREC>(m, 2 * q, b1);
            write_fbox<PREC>(m, 2 * q + 1, b2);
        }
    }

    if (a.patch) {
        if (__any_sync(FULL, top >= 0xffe00000u) && (threadIdx.x & 31) == 0) atomicOr(a.nonfinite, 1u);
        return;
    }
    // block reduction, then one set of atomics per block, each of twelve lanes its own
    // (lo, hi, extent of every coordinate)
    __shared__ long long red[8][12];
    __shared__ unsigned redf[8][2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        const long long l = ~warp_max(negated(acc.lo[d])), h = warp_max(acc.hi[d]), w = warp_max(acc.w[d]);
        if (lane == 0) { red[warp][d] = l; red[warp][4 + d] = h; red[warp][8 + d] = w; }
    }
    const unsigned fl = __any_sync(FULL, top >= 0xffe00000u) ? 1u : 0u;
    const unsigned seen = __reduce_or_sync(FULL, acc.seen);
    if (lane == 0) {
        redf[warp][0] = fl;
        redf[warp][1] = seen;
    }
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        Bounds *B = a.bounds + pe.mesh;
        const unsigned f = __any_sync(FULL, lane < nw && redf[lane & 7][0]), s = __any_sync(FULL, lane < nw && redf[lane & 7][1]);
        if (s && lane < 12) {
            long long v = red[0][lane];
            for (int w = 1; w < nw; ++w) v = lane < 4 ? min(v, red[w][lane]) : max(v, red[w][lane]);
            const unsigned long long e = encoded<PREC>(v);
            if (lane < 4) atomicMin(&B->lo[lane], e);
            else if (lane < 8) atomicMax(&B->hi[lane - 4], e);
            else atomicMax(&B->w[lane - 8], e);
        }
        if (lane == 0) {
            if (s) atomicOr(&B->faces, 1u);
            if (f) {
                atomicOr(&B->flags, ST_NONFINITE);
                atomicOr(&a.ctr->status, ST_NONFINITE);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// cell passes
// ---------------------------------------------------------------------------
constexpr int kCellWarps = 8;

constexpr unsigned kEntryFlush = 224;   // entries per atomic on the entry counter

struct EntryRec {
    uint64_t key;
    uint32_t face;
    uint32_t pad;
};

// coordinate d of item r of a cell range (mixed radix over cnt[0..3]); counts
// of 1 and 2 (the usual case: a cell is wider than any face) take no division
__device__ __forceinline__ unsigned next_digit(unsigned &r, unsigned c) {
    unsigned q;
    if (c <= 2u) q = r >> (c - 1u);
    else q = r / c;
    const unsigned digit = r - q * c;
    r = q;
    return digit;
}

template <int PREC, int MODE>
__global__ void __launch_bounds__(32 * kCellWarps) k_cell_pass(FacePassArgs a, int face_level) {
    __shared__ uint32_t s_excl[kCellWarps][32];
    __shared__ uint2 s_lo[kCellWarps][32];
    __shared__ uint2 s_cnt[kCellWarps][32];
    __shared__ EntryRec s_out[kCellWarps][kEntryFlush + 32];   // staged entries
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long slot = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long wslot = slot - lane;           // the warp's first slot
    if (wslot >= a.total_faces) return;            // whole warps only
    // every mesh starts at a multiple of 32 slots: the warp lies in one mesh
    const PassEntry pe = a.entries[find_entry(a, wslot, true)];
    const Grid &gg = a.grids[pe.pair];
    if (gg.empty) return;
    GridView<PREC> g;
    g.load(gg);
    const MeshDev &mr = a.meshes[pe.mesh];
    const int N = mr.N, nqi = mr.nqi;
    const long long f = slot - pe.face_base;
    // a valid face: inside this mesh's slots, and not the unused last column of
    // an open mesh
    bool valid = f < pe.faces;
    const uint32_t face = (uint32_t)f;
    if (valid) {
        const uint32_t q = face >> (face_level == 0 ? 1 : 0);
        valid = (int)(q % (uint32_t)N) < nqi;
    }
    int clo[4] = {0, 0, 0, 0}, cnt[4] = {1, 1, 1, 1};
    unsigned count = 0;
    if (valid) {
        BoxT<PREC> b;
        read_fbox<PREC>(mr, face, b);
        bool out = false;
#pragma unroll
        for (int d = 0; d < 4; ++d) out |= (b.hi[d] < g.o[d]) || (b.lo[d] > g.e[d]);
        if (!out) {
            count = 1;
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                clo[d] = g.cell(b.lo[d], d);
                const int chi = g.cell(b.hi[d], d);
                cnt[d] = chi - clo[d] + 1;
                count *= (unsigned)cnt[d];
            }
        }
    }
    // warp-wide exclusive scan of the counts
    unsigned incl = count;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned v = __shfl_up_sync(FULL, incl, off);
        if (lane >= off) incl += v;
    }
    const unsigned total = __shfl_sync(FULL, incl, 31);
    s_excl[warp][lane] = incl - count;
    s_lo[warp][lane] = make_uint2((uint32_t)clo[0] | ((uint32_t)clo[1] << 16),
                                  (uint32_t)clo[2] | ((uint32_t)clo[3] << 16));
    s_cnt[warp][lane] = make_uint2((uint32_t)cnt[0] | ((uint32_t)cnt[1] << 16),
                                   (uint32_t)cnt[2] | ((uint32_t)cnt[3] << 16));
    __syncwarp();
    const uint64_t pair_hi = (uint64_t)(uint32_t)pe.pair << 32;
    const uint32_t n0 = (uint32_t)g.n[0], n1 = (uint32_t)g.n[1], n2 = (uint32_t)g.n[2];
    EntryRec *stage = s_out[warp];
    unsigned staged = 0;
    uint64_t *const ekey = a.ent_key;
    uint32_t *const eval = a.ent_val;
    const unsigned long long cap = a.ent_cap;
    auto store = [ekey, eval, cap](unsigned long long pos, const EntryRec &r) {
        if (pos < cap) {
            ekey[pos] = r.key;
            eval[pos] = r.face;
        }
    };
    for (unsigned base = 0; base < total; base += 32) {
        const unsigned j = base + lane;
        const bool act = j < total;
        uint32_t cell = 0;
        int owner = 0;
        if (act) {
            // the lane whose range holds item j: the last with excl <= j
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (s_excl[warp][owner + step] <= j) owner += step;
            unsigned r = j - s_excl[warp][owner];
            const uint2 lo = s_lo[warp][owner], cn = s_cnt[warp][owner];
            const uint32_t c0 = (lo.x & 0xFFFFu) + next_digit(r, cn.x & 0xFFFFu);
            const uint32_t c1 = (lo.x >> 16) + next_digit(r, cn.x >> 16);
            const uint32_t c2 = (lo.y & 0xFFFFu) + next_digit(r, cn.y & 0xFFFFu);
            const uint32_t c3 = (lo.y >> 16) + next_digit(r, cn.y >> 16);
            cell = ((c3 * n2 + c2) * n1 + c1) * n0 + c0;
        }
        const uint64_t h = mix64(pair_hi | cell);
        bool emit = false;
        if (MODE == MODE_MARK) {
            if (act) {
                // bits are only ever set during this pass, so a word that already
                // holds them needs no atomic (a stale read only costs an atomic)
                uint32_t w, m;
                bloom_slot(h, a.bmA_word_bits, w, m);
                if ((a.bmA[w] & m) != m) atomicOr(a.bmA + w, m);
            }
        } else if (MODE == MODE_PROBE_MARK) {
            if (act) {
                uint32_t w, m;
                bloom_slot(h, a.bmA_word_bits, w, m);
                if ((__ldg(a.bmA + w) & m) == m) {
                    emit = true;
                    uint32_t w2, m2;
                    bloom_slot(h, a.bmH_word_bits, w2, m2);
                    if ((a.bmH[w2] & m2) != m2) atomicOr(a.bmH + w2, m2);
                }
            }
        } else if (MODE == MODE_PROBE) {
            if (act) {
                uint32_t w2, m2;
                bloom_slot(h, a.bmH_word_bits, w2, m2);
                emit = (__ldg(a.bmH + w2) & m2) == m2;
            }
        } else {  // MODE_EMIT_ALL
            emit = act;
        }
        if (MODE != MODE_MARK) {
            EntryRec r;
            r.key = pair_hi | ((uint64_t)cell << 1) | (uint64_t)pe.role;
            r.face = (uint32_t)(wslot - pe.face_base) + (uint32_t)owner;
            stage_push<kEntryFlush>(stage, staged, emit, r, &a.ctr->entries, store);
        }
    }
    if (MODE != MODE_MARK) {
        __syncwarp();
        stage_flush<kEntryFlush>(stage, staged, &a.ctr->entries, store);
    }
}

// The start of a search, in one launch: counters zeroed, per-mesh bounds
// reset, and the two occupancy bitmaps cleared (n32a and n32h words, each a
// multiple of four).
__global__ void k_search_init(Bounds *b, int n, Counters *ctr, uint32_t *bmA,
                              unsigned long long n32a, uint32_t *bmH, unsigned long long n32h,
                              uint32_t *tail) {
    const unsigned long long tid = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    if (tid == 0) memset(ctr, 0, sizeof(Counters));
    if (tid < (unsigned long long)n) {
        Bounds &m = b[tid];
#pragma unroll
        for (int d = 0; d < 4; ++d) { m.lo[d] = ~0ULL; m.hi[d] = 0ULL; m.w[d] = 0ULL; }
        m.flags = 0;
        m.faces = 0;
    }
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    if (tail)
        for (unsigned long long i = tid; i < (kTailBuckets + kTailMax / 32) / 4; i += stride)
            reinterpret_cast<uint4 *>(tail)[i] = z;
    if (bmA)
        for (unsigned long long i = tid; i < n32a / 4; i += stride) reinterpret_cast<uint4 *>(bmA)[i] = z;
    if (bmH)
        for (unsigned long long i = tid; i < n32h / 4; i += stride) reinterpret_cast<uint4 *>(bmH)[i] = z;
}

// Trimmed world and uniform grid of each pair (Sec. 6.2.1 and its remark).
// World along coordinate d: the overlap of the two meshes' ranges; a face whose
// box misses it cannot meet any face of the other mesh.  Cell edge: cell_mult x
// the widest face extent of either mesh, so that a face spans at most two cells
// per coordinate; capped so that a pair's grid has fewer than 2^31 cells.
__global__ void k_grid_params(const Bounds *b, const int2 *pairs, int n_pairs, Grid *grids,
                              float cell_mult, const float *cm_pair) {
    // one warp per pair, lane d & 3 speaks for coordinate d: the FP64 chain of
    // one coordinate instead of four (FP64 arithmetic is slow on GB300)
    const int p = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (p >= n_pairs) return;                      // whole warps
    const int lane = threadIdx.x & 31, d = lane & 3;
    const Bounds &A = b[pairs[p].x];
    const Bounds &B = b[pairs[p].y];
    const double o = fmax(ord_dec(A.lo[d]), ord_dec(B.lo[d]));
    const double e = fmin(ord_dec(A.hi[d]), ord_dec(B.hi[d]));
    const int empty = (A.faces == 0 || B.faces == 0 || __any_sync(FULL, !(o <= e))) ? 1 : 0;
    const float cm = cm_pair ? cm_pair[p] : cell_mult;
    double step = (double)cm * fmax(ord_dec(A.w[d]), ord_dec(B.w[d]));
    const double range = empty ? 0.0 : e - o;
    int n;
    // (one cell where a face is unbounded: range / step is no number)
    if (!(range > 0.0) || !(step > 0.0) || step > DBL_MAX) {
        n = 1;
        step = 0.0;
    } else {
        if (range / step > (double)(kMaxCellsPerDim - 1)) step = range / (double)(kMaxCellsPerDim - 1);
        n = (int)floor(range / step) + 1;
        if (n > kMaxCellsPerDim) n = kMaxCellsPerDim;
    }
    const double cap = 2147483647.0;
    for (int iter = 0; iter < 64; ++iter) {
        double prod = (double)n;
        prod *= __shfl_xor_sync(FULL, prod, 1);
        prod *= __shfl_xor_sync(FULL, prod, 2);
        if (prod <= cap) break;                    // the same in every lane
        const double f = sqrt(sqrt(prod / cap)) * 1.001;
        if (n > 1) {
            step *= f;
            n = (int)floor(range / step) + 1;
            if (n < 1) n = 1;
        }
    }
    if (lane < 4) {
        Grid &G = grids[p];
        const double inv = (step > 0.0) ? 1.0 / step : 0.0;
        G.o64[d] = o;
        G.e64[d] = e;
        G.inv64[d] = inv;
        G.o32[d] = (float)o;
        G.e32[d] = (float)e;
        G.inv32[d] = (float)inv;
        G.n[d] = n;
        if (d == 0) {
            G.empty = empty;
            G.pad[0] = G.pad[1] = G.pad[2] = 0;
        }
    }
}

template <int PREC, int FACE, int TK>
void launch_one(const FacePassArgs &a, int block, cudaStream_t st) {
    size_t smem = (size_t)(TK + 1) * (block + 1) * sizeof(Vtx<PREC>);
    if (PREC == 1 && a.patch) smem += (size_t)(block / kPatchI) * (TK / kPatchK) * sizeof(PatchScratch);
    k_bounds_pass<PREC, FACE, TK><<<(unsigned)a.total_tiles, block, smem, st>>>(a);
}

template <int PREC, int FACE>
void launch_tk(const FacePassArgs &a, int block, cudaStream_t st) {
    if (a.tile_rows == 4) launch_one<PREC, FACE, 4>(a, block, st);
    else launch_one<PREC, FACE, 8>(a, block, st);
}

template <int PREC, int FACE, int TK>
cudaError_t configure_one() {
    return cudaFuncSetAttribute(k_bounds_pass<PREC, FACE, TK>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
}

template <int PREC>
void launch_cells_mode(const FacePassArgs &a, int face_level, cudaStream_t st) {
    const int B = 32 * kCellWarps;
    const unsigned grid = (unsigned)((a.total_faces + B - 1) / B);
    switch (a.mode) {
        case MODE_MARK: k_cell_pass<PREC, MODE_MARK><<<grid, B, 0, st>>>(a, face_level); break;
        case MODE_PROBE_MARK: k_cell_pass<PREC, MODE_PROBE_MARK><<<grid, B, 0, st>>>(a, face_level); break;
        case MODE_PROBE: k_cell_pass<PREC, MODE_PROBE><<<grid, B, 0, st>>>(a, face_level); break;
        default: k_cell_pass<PREC, MODE_EMIT_ALL><<<grid, B, 0, st>>>(a, face_level); break;
    }
}

}  // namespace

// Sets kernel attributes once, before any launch (and outside stream capture).
cudaError_t configure_face_pass() {
    cudaError_t e = cudaSuccess;
    cudaError_t r;
#define TMS_CFG(P, F, T) if ((r = configure_one<P, F, T>()) != cudaSuccess) e = r;
    TMS_CFG(0, 0, 4) TMS_CFG(0, 0, 8) TMS_CFG(0, 1, 4) TMS_CFG(0, 1, 8)
    TMS_CFG(1, 0, 4) TMS_CFG(1, 0, 8) TMS_CFG(1, 1, 4) TMS_CFG(1, 1, 8)
#undef TMS_CFG
    return e;
}

void launch_face_pass(const FacePassArgs &a, int precision, int face_level, int block,
                      cudaStream_t st) {
    if (a.mode == MODE_BOUNDS) {
        if (a.total_tiles <= 0) return;
        if (precision == 1) {
            if (face_level == 0) launch_tk<1, 0>(a, block, st); else launch_tk<1, 1>(a, block, st);
        } else {
            if (face_level == 0) launch_tk<0, 0>(a, block, st); else launch_tk<0, 1>(a, block, st);
        }
        return;
    }
    if (a.total_faces <= 0) return;
    if (precision == 1) launch_cells_mode<1>(a, face_level, st);
    else launch_cells_mode<0>(a, face_level, st);
}

void launch_search_init(Bounds *b, int n, Counters *ctr, uint32_t *bmA, unsigned long long n32a,
                        uint32_t *bmH, unsigned long long n32h, uint32_t *tail, int grid, cudaStream_t st) {
    k_search_init<<<grid, 256, 0, st>>>(b, n, ctr, bmA, n32a, bmH, n32h, tail);
}

void launch_grid_params(const Bounds *b, const int2 *pairs, int n_pairs, Grid *g,
                        float cell_mult, cudaStream_t st, const float *cm_pair) {
    k_grid_params<<<(n_pairs + 3) / 4, 128, 0, st>>>(b, pairs, n_pairs, g, cell_mult, cm_pair);
}

}  // namespace tms
