// Patch pairs of the broad phase (patch level): the pairs of patches, one of each
// mesh, whose boxes overlap.
//
// The paper bins quads in a uniform grid and tests the pairs of a box of the grid
// (Sec. 6.2.1).  A patch's neighbours on its own mesh are near it in space, so the
// mesh's own index grid is a hierarchy already: a node of level l + 1 is a block of
// 4 x 4 nodes of level l (level 0: the patches), its box the union of theirs.  Pairs
// of nodes with overlapping boxes are followed down from a level of few nodes; a pair
// of patches has one chain of ancestors, so each is found exactly once, with no cells,
// no table of them, no owner rule and nothing to sort or group:
//   k_tree_up     the boxes of two levels from the level below (one launch for up to
//                 32 x 16 x 16 x 16 quads a node), and the counters cleared;
//   k_tree_top    all pairs of nodes of the top level, in tiles of 32 x 32;
//   k_tree_down   per level, one warp a pair of nodes: 16 children a side, those of each
//                 side that meet the other's box first, then their pairs.
// The top level is the lowest that leaves at most kTreeTopPairs pairs to test, and at most
// kTreeTopNodes nodes of any mesh, which one block passes over (first_pair_empty): 65,536
// patches against 64 took 326 us a search without that limit and take 293, 8192 x 1024
// vertices against 16 x 8 1036 and 789; below 16,384 nodes the further level costs more.  On two
// 4096 x 512 meshes the grid's launches took 84 us (entries, hash table, three scans,
// scatter, tile tests); these take 47 (up 7, top 8, down 8 and 24: 31,000 node pairs,
// 1.4 M patch tests where the grid made 5.8 M), bound by the chain of loads a node pair
// waits for, and a search of two 64 x 32 meshes, all latency, loses seven launches.
#include <cuda_runtime.h>
#include <stdint.h>

#include "tms_common.cuh"

namespace tms {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr unsigned kPairFlush = 64;      // staged pairs per atomic

template <int PREC>
struct TBox;
template <>
struct __align__(16) TBox<1> {
    float lo[4], hi[4];
    __device__ void load(const void *arr, uint32_t i) {
        const float4 *p = reinterpret_cast<const float4 *>(arr) + 2 * (size_t)i;
        const float4 l = __ldg(p), h = __ldg(p + 1);
        lo[0] = l.x; lo[1] = l.y; lo[2] = l.z; lo[3] = l.w;
        hi[0] = h.x; hi[1] = h.y; hi[2] = h.z; hi[3] = h.w;
    }
    __device__ void store(void *arr, uint32_t i) const {
        float4 *p = reinterpret_cast<float4 *>(arr) + 2 * (size_t)i;
        p[0] = make_float4(lo[0], lo[1], lo[2], lo[3]);
        p[1] = make_float4(hi[0], hi[1], hi[2], hi[3]);
    }
    __device__ void set_empty() {
#pragma unroll
        for (int d = 0; d < 4; ++d) { lo[d] = __int_as_float(0x7f800000); hi[d] = -lo[d]; }
    }
};
template <>
struct __align__(16) TBox<0> {
    long long lo[4], hi[4];      // ordered integers (ord64)
    __device__ void load(const void *arr, uint32_t i) {
        const longlong2 *p = reinterpret_cast<const longlong2 *>(arr) + 4 * (size_t)i;
        const longlong2 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2), d = __ldg(p + 3);
        lo[0] = a.x; lo[1] = a.y; lo[2] = b.x; lo[3] = b.y;
        hi[0] = c.x; hi[1] = c.y; hi[2] = d.x; hi[3] = d.y;
    }
    __device__ void store(void *arr, uint32_t i) const {
        longlong2 *p = reinterpret_cast<longlong2 *>(arr) + 4 * (size_t)i;
        p[0] = make_longlong2(lo[0], lo[1]);
        p[1] = make_longlong2(lo[2], lo[3]);
        p[2] = make_longlong2(hi[0], hi[1]);
        p[3] = make_longlong2(hi[2], hi[3]);
    }
    __device__ void set_empty() {
#pragma unroll
        for (int d = 0; d < 4; ++d) { lo[d] = 0x7fffffffffffffffLL; hi[d] = -lo[d]; }
    }
};

template <int PREC>
__device__ __forceinline__ bool overlap(const TBox<PREC> &x, const TBox<PREC> &y) {
    bool ov = true;
#pragma unroll
    for (int d = 0; d < 4; ++d) ov &= !(x.hi[d] < y.lo[d]) & !(y.hi[d] < x.lo[d]);
    return ov;
}
// union over the aligned groups of `lanes` lanes (every lane gets it)
template <int PREC>
__device__ __forceinline__ void unite_lanes(TBox<PREC> &b, int lanes) {
#pragma unroll
    for (int off = 1; off < lanes; off <<= 1)
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            b.lo[d] = min(b.lo[d], __shfl_xor_sync(FULL, b.lo[d], off));
            b.hi[d] = max(b.hi[d], __shfl_xor_sync(FULL, b.hi[d], off));
        }
}

__device__ __forceinline__ void node_of(const TreeLevel &l, uint32_t id, int &i, int &k) {
    k = l.ni == 1 ? (int)id : (int)__umul64hi((unsigned long long)id, l.magic);
    i = (int)(id - (uint32_t)k * (uint32_t)l.ni);
}

// One block per node of level `from` + 2 of every mesh: 16 x 16 nodes of level `from`,
// a thread each.  The first launch also starts the search's counters.
template <int PREC>
__global__ void __launch_bounds__(256) k_tree_up(TreeArgs a, int from, bool start) {
    __shared__ TBox<PREC> mid[16];
    const int t = threadIdx.x;
    if (start) {
        const unsigned long long g = blockIdx.x * 256ULL + t, n = (kTailBuckets + kTailMax / 32) / 4;
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        for (unsigned long long q = g; q < n; q += gridDim.x * 256ULL) reinterpret_cast<uint4 *>(a.tail)[q] = z;
        if (blockIdx.x == 0 && t < (int)(sizeof(Counters) / 4)) reinterpret_cast<uint32_t *>(a.ctr)[t] = 0;
        if (blockIdx.x == 0) {
            __syncthreads();
            // the bounds pass, which runs before, leaves its finding here
            if (t == 0 && *a.nonfinite) {
                a.ctr->status = ST_NONFINITE;
                *a.nonfinite = 0;
            }
        }
    }
    if (a.top == 0) return;
    // the mesh holding this block's node
    int lo = 0, hi = a.n_meshes - 1;
    while (lo < hi) {
        const int m = (lo + hi + 1) >> 1;
        if (a.trees[m].up_base[from / 2] <= blockIdx.x) lo = m; else hi = m - 1;
    }
    const MeshTree &tr = a.trees[lo];
    const uint32_t id = blockIdx.x - tr.up_base[from / 2];
    const TreeLevel &l0 = tr.lev[from], &l1 = tr.lev[from + 1], &l2 = tr.lev[from + 2];
    if (id >= (uint32_t)(l2.ni * l2.nk)) return;   // past the last mesh's nodes (clearing only)
    int i2, k2;
    node_of(l2, id, i2, k2);
    const int n1 = t >> 4, c = t & 15;
    const int i1 = 4 * i2 + (n1 & 3), k1 = 4 * k2 + (n1 >> 2);
    const int i0 = 4 * i1 + (c & 3), k0 = 4 * k1 + (c >> 2);
    TBox<PREC> b;
    b.set_empty();
    if (i0 < l0.ni && k0 < l0.nk) b.load(l0.box, (uint32_t)k0 * (uint32_t)l0.ni + (uint32_t)i0);
    unite_lanes<PREC>(b, 16);
    if (c == 0) {
        if (i1 < l1.ni && k1 < l1.nk) b.store(l1.box, (uint32_t)k1 * (uint32_t)l1.ni + (uint32_t)i1);
        mid[n1] = b;
    }
    __syncthreads();
    if (t < 32) {
        b = mid[t & 15];
        unite_lanes<PREC>(b, 16);
        if (t == 0) b.store(l2.box, id);
    }
}

// the pair of top-level boxes of pair 0's meshes: whether their overlap is empty
template <int PREC>
__device__ void first_pair_empty(const TreeArgs &a) {
    __shared__ TBox<PREC> w[2][8];
    const int t = threadIdx.x;
    TBox<PREC> b[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const TreeLevel &l = a.trees[s ? a.pairs[0].y : a.pairs[0].x].lev[a.top];
        b[s].set_empty();
        for (int i = t; i < l.ni * l.nk; i += 256) {
            TBox<PREC> x;
            x.load(l.box, (uint32_t)i);
#pragma unroll
            for (int d = 0; d < 4; ++d) { b[s].lo[d] = min(b[s].lo[d], x.lo[d]); b[s].hi[d] = max(b[s].hi[d], x.hi[d]); }
        }
        unite_lanes<PREC>(b[s], 32);
        if ((t & 31) == 0) w[s][t >> 5] = b[s];
    }
    __syncthreads();
    if (t < 32) {
        for (int s = 0; s < 2; ++s) {
            b[s] = w[s][t & 7];
            unite_lanes<PREC>(b[s], 8);
        }
        if (t == 0) {
            Grid &g = *a.grid0;
            g.n[0] = g.n[1] = g.n[2] = g.n[3] = 0;
            g.empty = overlap(b[0], b[1]) ? 0 : 1;
        }
    }
}

__device__ __forceinline__ Cand node_pair(uint32_t x, uint32_t y, uint32_t pair) {
    Cand c;
    c.faceA = x;
    c.faceB = y;
    c.pair = pair;
    c.pad = 0;
    return c;
}

// A warp tests tiles of 32 x 32 nodes: a lane's node of B against every node of A.
template <int PREC>
__global__ void __launch_bounds__(256) k_tree_top(TreeArgs a) {
    __shared__ TBox<PREC> sA[8][32];
    __shared__ Cand sOut[8][kPairFlush + 32];
    if (blockIdx.x == 0) {             // beside the tests, which the other blocks take
        first_pair_empty<PREC>(a);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Cand *out = a.list[a.top & 1], *stage = sOut[warp];
    const unsigned long long cap = a.top ? a.cap : a.ppair_cap;
    unsigned long long *ctr = a.top ? &a.ctr->nodes[a.top] : &a.ctr->ppairs;
    if (a.top == 0) out = a.ppairs;
    auto store = [out, cap](unsigned long long pos, const Cand &r) {
        if (pos < cap) out[pos] = r;
    };
    unsigned staged = 0;
    const long long nw = (long long)(gridDim.x - 1) * 8;
    for (long long tile = (long long)(blockIdx.x - 1) * 8 + warp; tile < a.top_tiles; tile += nw) {
        int lo = 0, hi = a.n_pairs - 1;
        while (lo < hi) {
            const int m = (lo + hi + 1) >> 1;
            if (a.top_base[m] <= tile) lo = m; else hi = m - 1;
        }
        const int2 pr = a.pairs[lo];
        const TreeLevel &la = a.trees[pr.x].lev[a.top], &lb = a.trees[pr.y].lev[a.top];
        const int nA = la.ni * la.nk, nB = lb.ni * lb.nk, tB = (nB + 31) / 32;
        const int t = (int)(tile - a.top_base[lo]);
        const int a0 = t / tB * 32, b0 = t % tB * 32;
        const int rows = min(32, nA - a0);
        TBox<PREC> x, y;
        x.set_empty();
        y.set_empty();
        // (an unbounded box, of coordinates beyond FP32 on both sides, meets the empty one too)
        const bool inB = b0 + lane < nB;
        if (a0 + lane < nA) x.load(la.box, (uint32_t)(a0 + lane));
        if (inB) y.load(lb.box, (uint32_t)(b0 + lane));
        __syncwarp();
        sA[warp][lane] = x;
        __syncwarp();
        for (int j = 0; j < rows; ++j)
            stage_push<kPairFlush>(stage, staged, inB && overlap(sA[warp][j], y),
                                   node_pair((uint32_t)(a0 + j), (uint32_t)(b0 + lane), (uint32_t)lo), ctr, store);
    }
    __syncwarp();
    stage_flush<kPairFlush>(stage, staged, ctr, store);
}

// From the pairs of level `level` to those of level - 1 (level 1: the patch pairs).
// Lanes 0-15 hold the children of A's node, lanes 16-31 those of B's.
template <int PREC>
__global__ void __launch_bounds__(256) k_tree_down(TreeArgs a, int level) {
    __shared__ TBox<PREC> sBox[8][32];     // survivors' boxes, A's from 0, B's from 16
    __shared__ uint32_t sChild[8][32];     // and ids
    __shared__ Cand sOut[8][kPairFlush + 32];
    const unsigned long long n = clamp_count(&a.ctr->nodes[level], a.cap);
    if (256 * n > kMaxPairSlots) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&a.ctr->status, ST_PAIR_LIMIT);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = lane & 15;
    const Cand *in = a.list[level & 1];
    Cand *out = level == 1 ? a.ppairs : a.list[(level - 1) & 1];
    const unsigned long long cap = level == 1 ? a.ppair_cap : a.cap;
    unsigned long long *ctr = level == 1 ? &a.ctr->ppairs : &a.ctr->nodes[level - 1];
    Cand *stage = sOut[warp];
    auto store = [out, cap](unsigned long long pos, const Cand &r) {
        if (pos < cap) out[pos] = r;
    };
    unsigned staged = 0;
    unsigned long long tests = 0;
    const unsigned long long nw = (unsigned long long)gridDim.x * 8;
    // the pair's levels, looked up again only when the pair changes
    uint32_t cached = 0xFFFFFFFFu;
    TreeLevel up = {}, dn = {};
    const void *other = nullptr;
    unsigned long long q = blockIdx.x * 8ULL + warp;
    Cand next = node_pair(0, 0, 0);
    if (q < n) next = in[q];
    for (; q < n; q += nw) {
        const Cand np = next;
        if (q + nw < n) next = in[q + nw];
        if (np.pair != cached) {
            const int2 pr = a.pairs[np.pair];
            const MeshTree &tr = a.trees[lane < 16 ? pr.x : pr.y];
            up = tr.lev[level];
            dn = tr.lev[level - 1];
            other = a.trees[lane < 16 ? pr.y : pr.x].lev[level].box;
            cached = np.pair;
        }
        TBox<PREC> u;                   // the other node's box
        u.load(other, lane < 16 ? np.faceB : np.faceA);
        int i, k;
        node_of(up, lane < 16 ? np.faceA : np.faceB, i, k);
        i = 4 * i + (c & 3);
        k = 4 * k + (c >> 2);
        const uint32_t child = (uint32_t)k * (uint32_t)dn.ni + (uint32_t)i;
        TBox<PREC> b;
        b.set_empty();
        const bool real = i < dn.ni && k < dn.nk;       // (as in k_tree_top)
        if (real) b.load(dn.box, child);
        const uint32_t meet = __ballot_sync(FULL, real && overlap(b, u));
        const uint32_t mA = meet & 0xffffu, mB = meet >> 16;
        if (!mA || !mB) continue;
        const uint32_t nA = __popc(mA), nB = __popc(mB);
        __syncwarp();                   // the previous pair's boxes are read
        if ((meet >> lane) & 1u) {
            const int at = (lane & 16) + __popc(meet & (lane < 16 ? 0xffffu : 0xffff0000u) & lanemask_lt());
            sBox[warp][at] = b;
            sChild[warp][at] = child;
        }
        __syncwarp();
        tests += nA * nB;
        // the nA nB tests one a lane, B's children fastest; test t is child t / nB of A
        // (below 32 also past the last test) and t % nB of B, from FP32 reciprocals:
        // (x + 1/2) / nB lies at least 1/32 from an integer for x <= 32.  (Two of A's
        // children a step against B's sixteen: the leaf level of 64 uneven pairs 71 us, 64 so.)
        const float rB = __fdividef(1.0f, (float)nB);
        const uint32_t step_a = (uint32_t)(32.5f * rB), step_b = 32u - step_a * nB;
        uint32_t ia = (uint32_t)(((float)lane + 0.5f) * rB), ib = (uint32_t)lane - ia * nB;
        for (uint32_t base = 0; base < nA * nB; base += 32) {
            const bool ov = base + lane < nA * nB && overlap(sBox[warp][ia], sBox[warp][16 + ib]);
            stage_push<kPairFlush>(stage, staged, ov, node_pair(sChild[warp][ia], sChild[warp][16 + ib], np.pair), ctr, store);
            ia += step_a;
            ib += step_b;
            if (ib >= nB) {
                ib -= nB;
                ++ia;
            }
        }
    }
    __syncwarp();
    stage_flush<kPairFlush>(stage, staged, ctr, store);
    if (lane == 0 && tests && level == 1) atomicAdd(&a.ctr->pair_slots, tests);
}

int g_down_resident[2] = {};

template <int PREC>
int down_resident() {
    int &r = g_down_resident[PREC];
    if (r == 0) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_tree_down<PREC>, 256, 0) != cudaSuccess || nb < 1)
            nb = 1;
        r = nb;
    }
    return r;
}

template <int PREC>
void launch(const TreeArgs &a, int sms, cudaStream_t st) {
    // at least a few blocks: they also clear
    for (int from = 0; from == 0 || from < a.top; from += 2)
        k_tree_up<PREC><<<a.up_blocks[from / 2] > 8 ? a.up_blocks[from / 2] : 8, 256, 0, st>>>(a, from, from == 0);
    const long long top = (a.top_tiles + 7) / 8;
    k_tree_top<PREC><<<1 + (unsigned)(top < 8 * sms ? top : 8 * sms), 256, 0, st>>>(a);
    for (int level = a.top; level >= 1; --level)
        k_tree_down<PREC><<<sms * down_resident<PREC>(), 256, 0, st>>>(a, level);
}

}  // namespace

// kernel launches of launch_tree
int tree_launches(int top) { return (top < 2 ? 1 : (top + 1) / 2) + 1 + top; }

void configure_tree() {
    down_resident<0>();
    down_resident<1>();
}

void launch_tree(const TreeArgs &a, int precision, int sms, cudaStream_t st) {
    if (precision == 1) launch<1>(a, sms, st);
    else launch<0>(a, sms, st);
}

}  // namespace tms
