// sb_mst.cu -- randomized Kruskal trees (appendix, tree samplers: Kruskal's
// algorithm run on random edge weights drawn afresh for every tree), many
// trees at once.
//
// Tree t is the minimum spanning tree under the weights
//   w_t(u, v) = mix64(((u << 32) | v) ^ K_t),   u < v (graph-local ids),
// with K_t the tree key of the BFS sampler.  mix64 is a bijection, so the
// weights of one tree are distinct and the tree is unique: Kruskal's scan in
// weight order, Prim's growth and Boruvka's rounds all find it.  Kruskal's
// scan is sequential; Boruvka's rounds are not, so the GPU runs those:
//   1. every work item (a CSR row, or 256 entries of a longer one) finds its
//      lightest edge that leaves its vertex's component, and the component
//      keeps the lightest of those (64-bit atomicMin);
//   2. mix64 is a bijection, so that weight names the edge: every component
//      root inverts it and hooks below the component at the edge's far end;
//      two components that chose each other chose the same edge (the weights
//      are equal), and only the larger root hooks;
//   3. pointer jumping flattens the hooks; a pointer carries the parity of
//      the path to its target in its low bit, so each vertex ends with its
//      parity label relative to its component's root.
// From round 1 on one component of every tree, the largest as far as 32
// sampled edge ends tell, neither searches nor hooks: the others reach it.
// That costs no round (of x components, the x - 1 others each end up with
// another one, so x' - 1 <= (x - 1) / 2, and ceil(log2 n) + 1 rounds suffice),
// and once the largest component holds nearly all edges it spares going
// through all of them for its lightest outgoing one.
//
// What bounds it: hashing every (tree, edge) pair from both ends took 20 ms per
// round at 256 trees on the 2^20 R-MAT graph, and in a graph with a dense core
// most edges leave their components until the last rounds.  So round 0, which
// hashes every pair anyway, also records which edges are light (a fixed bound
// on the weight, about 3 edges per vertex), and the next rounds search those
// only, lane by lane: a component with a light edge leaving it finds its
// lightest edge among them, and one without waits.  Full rounds then join
// what is left, mostly vertices of low degree, to the largest component.  On
// that graph: 212-263 ms per 256 trees with full rounds only (and a separate
// record of every vertex's edge, now read back from the weight), 157 ms
// without the largest component's search, 84 ms with light rounds.
// A round after which nothing merged ends the loop early (its kernels return
// at once).
//
// Layout: [vertex][tree of the pass], trees innermost, so a warp holds 32
// trees of one vertex: it scans one CSR row in lockstep and its gathers of a
// neighbour's 32 root words are one coalesced 128-byte load.
#include <algorithm>

#include "sb_internal.cuh"

#define MST_THREADS 256
#define MST_BYTES_PER_SLOT 17            // P, R (4 B each), B (8 B), `done` bits
#define MST_PASS_BUDGET (32ull << 30)    // scratch bytes per pass of trees (at most half the free memory)

// Light rounds (k_mst_light).  2 m / n = 51 edges per vertex (2^20 R-MAT graph,
// 256 trees): 157 ms without them, 78 / 84 / 84 / 95 ms at 2 / 3 / 4 / 8 light
// edges per vertex; 60 edges per vertex of a uniform random graph (n = 100,000):
// 31.1 ms without, 17.8 / 15.4 ms at 2 / 3 (a smaller light degree leaves more
// of a uniform graph to the full rounds); 10 per vertex (n = 300,000): 35.7
// without, 31.4 ms at 3.  Below about 9 edges per vertex too few edges are left out.
#define MST_LIGHT_DEGREE 3.0             // light edges per vertex, on average
#define MST_LIGHT_MAX 0.35               // largest share of light edges worth separate rounds
#define MST_LIGHT_ROUNDS 8
// Fewest (CSR entry, tree) pairs worth the 9 further rounds of launches (a
// full round takes 5 us at most below that; ER(1000, 5000) with 64 trees:
// 0.54 ms with light rounds, 0.40 without).
#define MST_LIGHT_PAIRS (1ll << 26)
#define MST_ROUNDS_MAX 64
// Fewest vertices per graph for one component to sit out: finding it samples 32
// edge ends per (graph, tree) and round, as many as a graph of 32 vertices has
// rows (20,000 graphs of 9 vertices, 64 trees: 2.47 ms with, 1.34 without).
#define MST_BIG_VERTICES 32

struct MstArgs {
    int64_t n;
    int T;            // trees per pass (a multiple of 64)
    int64_t tb0;      // first tree of the pass, within the batch
    int64_t K;        // trees of the batch
    uint64_t S;       // seed key
    int64_t tree0;    // global index of batch tree 0
    const sb_bfs_item* items;  // rows, and chunks of long rows
    int64_t n_items;
    const int32_t* rowptr;
    const int32_t* col;
    const int32_t* vgid;   // graph of each vertex (batches), or null
    const int32_t* vgoff;  // first vertex of each vertex's graph (batches), or null
    const int32_t* voff;   // first vertex of each graph (batches), or null
    int64_t graphs;
    uint32_t* big;         // [graph][tree]: root of the component that sits the round out, or null
    uint32_t* P;
    uint32_t* R;
    uint64_t* B;
    uint32_t* done;        // [item][32 trees]: bit set when the item has nothing left to find
    uint32_t* light;       // [32 entries of a row][tree]: bit per entry lighter than `theta`
    uint32_t theta;        // bound on a light weight's upper half, 0 without light rounds
    int light_rounds;      // at most this many
    int32_t* mode;         // [r]: MST_DONE, MST_FULL or MST_LIGHT
    int32_t* merged;       // [r] = 1 when round r merged something
    const int2* edges;     // for in_tree (binary search of the pair)
    int64_t m;
    uint8_t* in_tree;      // K x m, or null
    uint32_t* err;
};

#define MST_DONE 0
#define MST_FULL 1   // every component searches all its edges
#define MST_LIGHT 2  // components search their light edges only

// Mode of round r, from the round before it.
__device__ __forceinline__ int mst_mode(const MstArgs& A, int r)
{
    if (r == 0) return MST_FULL;
    const int was = A.mode[r - 1], merged = A.merged[r - 1];
    if (r == 1) return !merged ? MST_DONE : A.theta ? MST_LIGHT : MST_FULL;
    if (was == MST_LIGHT) return merged && r <= A.light_rounds ? MST_LIGHT : MST_FULL;
    return was == MST_FULL && merged ? MST_FULL : MST_DONE;
}

// The (row, group of 32 trees) pairs of a kernel's warps: warp w takes w, w +
// warps, ..; the step is split into rows and groups once, so that no pair
// costs a division.
struct MstWalk {
    int64_t row, drow;
    int tg, dtg, TG;
    __device__ __forceinline__ explicit MstWalk(int T) : TG(T >> 5)
    {
        const int64_t w = ((int64_t)blockIdx.x * MST_THREADS + threadIdx.x) >> 5;
        const int64_t warps = (int64_t)gridDim.x * (MST_THREADS / 32);
        row = w / TG;
        tg = (int)(w - row * TG);
        drow = warps / TG;
        dtg = (int)(warps - drow * TG);
    }
    __device__ __forceinline__ void next()
    {
        row += drow;
        tg += dtg;
        if (tg >= TG) {
            tg -= TG;
            row++;
        }
    }
    __device__ __forceinline__ int tree() const { return 32 * tg + (int)(threadIdx.x & 31); }
};

// First block of 32 entries of row v (blocks of a row follow one another).
__device__ __forceinline__ int64_t mst_block(int64_t rowptr_v, int64_t v) { return (rowptr_v >> 5) + v; }

__device__ __forceinline__ uint32_t mst_ld(const uint32_t* p) { return __ldcg(p); }

// Inverse of an odd multiplier modulo 2^64 (Newton: each step doubles the
// correct low bits, 3 of them at the start).
__host__ __device__ constexpr uint64_t mst_inverse(uint64_t a)
{
    uint64_t x = a;
    for (int i = 0; i < 5; i++) x *= 2 - a * x;
    return x;
}

// The z with sb_mix64(z) = w.
__device__ __forceinline__ uint64_t mst_unmix64(uint64_t w)
{
    constexpr uint64_t i1 = mst_inverse(0xBF58476D1CE4E5B9ULL), i2 = mst_inverse(0x94D049BB133111EBULL);
    w ^= (w >> 31) ^ (w >> 62);
    w *= i2;
    w ^= (w >> 27) ^ (w >> 54);
    w *= i1;
    w ^= (w >> 30) ^ (w >> 60);
    return w;
}

// Start of a round: its mode, and per (graph, tree) the component that most of
// 32 edge ends, evenly spaced over the graph's CSR entries, lie in (one warp;
// any choice gives the same tree).
__global__ void __launch_bounds__(MST_THREADS) k_mst_big(MstArgs A, int r)
{
    const int mode = mst_mode(A, r);
    if (blockIdx.x == 0 && threadIdx.x == 0) A.mode[r] = mode;
    if (mode == MST_DONE || r == 0 || !A.big) return;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (MST_THREADS / 32);
    for (int64_t x = ((int64_t)blockIdx.x * MST_THREADS + threadIdx.x) >> 5; x < A.graphs * A.T; x += warps) {
        const int64_t g = x / A.T;
        const int tt = (int)(x - g * A.T);
        const int64_t v0 = A.voff ? A.voff[g] : 0, v1 = A.voff ? A.voff[g + 1] : A.n;
        const int64_t e0 = A.rowptr[v0], len = A.rowptr[v1] - e0;
        if (len == 0) continue;  // one vertex: nothing to search
        const int64_t v = (uint32_t)A.col[e0 + len * lane / 32] & SB_ID_MASK;
        const uint32_t c = A.R[v * A.T + tt] >> 1;
        const uint32_t same = __popc(__match_any_sync(0xffffffffu, c));
        const uint32_t most = __reduce_max_sync(0xffffffffu, same);
        const int first = __ffs((int)__ballot_sync(0xffffffffu, same == most)) - 1;
        if (lane == first) A.big[x] = c;
    }
}

__global__ void __launch_bounds__(MST_THREADS) k_mst_init(MstArgs A)
{
    for (MstWalk k(A.T); k.row < A.n; k.next()) {
        const int64_t i = k.row * A.T + k.tree();
        A.P[i] = (uint32_t)k.row << 1;
        A.R[i] = (uint32_t)k.row << 1;
        A.B[i] = ~0ull;
    }
    const int TG = A.T / 32;
    for (int64_t i = (int64_t)blockIdx.x * MST_THREADS + threadIdx.x; i < A.n_items * TG;
         i += (int64_t)gridDim.x * MST_THREADS) {
        const int64_t left = A.K - A.tb0 - 32 * (i % TG);  // trees of this word
        A.done[i] = left >= 32 ? 0u : left <= 0 ? ~0u : ~((1u << left) - 1u);
    }
}

// 1. lightest edge leaving the component, per (item, tree); component min.
// ROUND0: every vertex is alone, so every edge leaves and nothing is loaded.
// An edge whose ends share a component in all 32 trees is not hashed.
template <bool ROUND0>
__global__ void __launch_bounds__(MST_THREADS) k_mst_min(MstArgs A, int r)
{
    if (A.mode[r] != MST_FULL) return;
    const int lane = threadIdx.x & 31;
    for (MstWalk k(A.T); k.row < A.n_items; k.next()) {
        const int64_t item = k.row, x = item * k.TG + k.tg;
        uint32_t done = A.done[x];
        if (done == ~0u) continue;
        const int tt = k.tree();
        const int4 q = __ldg((const int4*)(A.items + item));
        const int32_t v = q.x;
        const uint32_t c = ROUND0 ? (uint32_t)v : A.R[(int64_t)v * A.T + tt] >> 1;
        bool act = !((done >> lane) & 1u);
        if (!ROUND0 && A.big) act = act && c != A.big[(A.vgid ? (int64_t)A.vgid[v] * A.T : 0) + tt];
        if (!__any_sync(0xffffffffu, act)) continue;
        const uint64_t kt = sb_tree_key(A.S, A.tree0 + A.tb0 + tt);
        const uint32_t base = A.vgoff ? (uint32_t)A.vgoff[v] : 0u;
        const uint32_t vl = (uint32_t)v - base;
        uint64_t best = ~0ull;
        bool found = false;
        const uint32_t* Rt = A.R + tt;
        for (int32_t p0 = q.y; p0 < q.z; p0 += 32) {
            const int cnt = min(32, q.z - p0);
            const uint32_t mycol = lane < cnt ? (uint32_t)__ldg(A.col + p0 + lane) & SB_ID_MASK : 0u;
            uint32_t lm = 0;
            for (int e0 = 0; e0 < cnt; e0 += 8) {
                uint32_t y[8], ry[8];
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    y[i] = __shfl_sync(0xffffffffu, mycol, (e0 + i) & 31);
                    // entries past the row count as inside
                    ry[i] = ROUND0 ? ~c : c << 1;
                    if (!ROUND0 && e0 + i < cnt) ry[i] = Rt[(int64_t)y[i] * A.T];
                }
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    if (ROUND0 && e0 + i >= cnt) break;
                    const bool leave = act && (ROUND0 || (ry[i] >> 1) != c);
                    if (!ROUND0 && !__any_sync(0xffffffffu, leave)) continue;
                    const uint32_t yl = y[i] - base;
                    const uint64_t w = sb_mix64((((uint64_t)min(vl, yl) << 32) | max(vl, yl)) ^ kt);
                    if (leave && w < best) best = w;
                    found |= leave;
                    if (ROUND0 && (uint32_t)(w >> 32) < A.theta) lm |= 1u << (e0 + i);
                }
            }
            if (ROUND0 && A.theta) {
                const int64_t rp = A.rowptr[v];
                A.light[(mst_block(rp, v) + ((p0 - rp) >> 5)) * A.T + tt] = lm;
            }
        }
        // a row with nothing outside keeps it so
        const uint32_t dead = done | __ballot_sync(0xffffffffu, act && !found);
        if (lane == 0) A.done[x] = dead;
        if (found) {
            uint64_t* b = A.B + (int64_t)c * A.T + tt;
            if (ROUND0 && q.w < 0) *b = best;
            else if (best < __ldcg(b)) atomicMin((unsigned long long*)b, (unsigned long long)best);
        }
    }
}

// 1'. the same over the light edges recorded in round 0, lane by lane.  A
// component with a light edge leaving it has its lightest edge among those;
// one without waits for the full rounds.  Entries found inside are dropped.
__global__ void __launch_bounds__(MST_THREADS) k_mst_light(MstArgs A, int r)
{
    if (A.mode[r] != MST_LIGHT) return;
    const int lane = threadIdx.x & 31;
    for (MstWalk k(A.T); k.row < A.n_items; k.next()) {
        const int64_t item = k.row, x = item * k.TG + k.tg;
        const uint32_t done = A.done[x];
        if (done == ~0u) continue;
        const int tt = k.tree();
        const int4 q = __ldg((const int4*)(A.items + item));
        const int32_t v = q.x;
        const uint32_t c = A.R[(int64_t)v * A.T + tt] >> 1;
        bool act = !((done >> lane) & 1u);
        if (A.big) act = act && c != A.big[(A.vgid ? (int64_t)A.vgid[v] * A.T : 0) + tt];
        if (!__any_sync(0xffffffffu, act)) continue;
        const uint64_t kt = sb_tree_key(A.S, A.tree0 + A.tb0 + tt);
        const uint32_t base = A.vgoff ? (uint32_t)A.vgoff[v] : 0u;
        const uint32_t vl = (uint32_t)v - base;
        const int64_t rp = A.rowptr[v];
        uint32_t* lmp = A.light + (mst_block(rp, v) + ((q.y - rp) >> 5)) * A.T + tt;
        uint64_t best = ~0ull;
        const uint32_t* Rt = A.R + tt;
        for (int32_t p0 = q.y; p0 < q.z; p0 += 32, lmp += A.T) {
            const uint32_t lm = act ? *lmp : 0u;
            int left = (int)__reduce_max_sync(0xffffffffu, (unsigned)__popc(lm));
            if (left == 0) continue;
            const uint32_t mycol = p0 + lane < q.z ? (uint32_t)__ldg(A.col + p0 + lane) & SB_ID_MASK : 0u;
            uint32_t m = lm, keep = lm;
            for (; left > 0; left -= 2) {  // two at a time
                uint32_t bit[2], y[2], ry[2];
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    bit[i] = m & (0u - m);
                    m ^= bit[i];
                    y[i] = __shfl_sync(0xffffffffu, mycol, __ffs((int)bit[i]) - 1);
                    ry[i] = c << 1;  // no entry left: counts as inside
                    if (bit[i]) ry[i] = Rt[(int64_t)y[i] * A.T];
                }
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    if ((ry[i] >> 1) == c) {
                        keep &= ~bit[i];
                        continue;
                    }
                    const uint32_t yl = y[i] - base;
                    const uint64_t w = sb_mix64((((uint64_t)min(vl, yl) << 32) | max(vl, yl)) ^ kt);
                    if (w < best) best = w;
                }
            }
            if (keep != lm) *lmp = keep;
        }
        if (best != ~0ull) {
            uint64_t* b = A.B + (int64_t)c * A.T + tt;
            if (best < __ldcg(b)) atomicMin((unsigned long long*)b, (unsigned long long)best);
        }
    }
}

// index of edge (a, b), a < b, in the sorted edge list
__device__ int64_t mst_edge_index(const int2* edges, int64_t m, uint32_t a, uint32_t b)
{
    int64_t lo = 0, hi = m;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        const int2 e = edges[mid];
        const uint32_t eu = (uint32_t)e.x, ev = (uint32_t)e.y & SB_ID_MASK;
        if (eu < a || (eu == a && ev < b)) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// sign bit of edge (a, b), from the shorter of its two rows
__device__ __forceinline__ uint32_t mst_edge_sign(const MstArgs& A, uint32_t a, uint32_t b)
{
    int32_t lo = A.rowptr[a], hi = A.rowptr[a + 1];
    const int32_t lo2 = A.rowptr[b], hi2 = A.rowptr[b + 1];
    uint32_t want = b;
    if (hi2 - lo2 < hi - lo) {
        lo = lo2;
        hi = hi2;
        want = a;
    }
    while (hi - lo > 1) {  // last entry not above `want`
        const int32_t mid = (lo + hi) >> 1;
        if (((uint32_t)A.col[mid] & SB_ID_MASK) <= want) lo = mid;
        else hi = mid;
    }
    return (uint32_t)A.col[lo] >> 31;
}

// 2. every root with an outgoing edge hooks below the far component
__global__ void __launch_bounds__(MST_THREADS) k_mst_hook(MstArgs A, int r)
{
    if (A.mode[r] == MST_DONE) return;
    bool hooked = false;
    for (MstWalk k(A.T); k.row < A.n; k.next()) {
        const int64_t c = k.row;
        const int tt = k.tree();
        const int64_t i = c * A.T + tt;
        const int64_t tb = A.tb0 + tt;
        if (tb >= A.K) continue;
        if ((int64_t)(A.R[i] >> 1) != c) continue;  // not a root
        const uint64_t w = A.B[i];
        if (w == ~0ull) continue;                    // sat this round out, or nothing leaves it
        const uint64_t pair = mst_unmix64(w) ^ sb_tree_key(A.S, A.tree0 + tb);
        const uint32_t base = A.vgoff ? (uint32_t)A.vgoff[c] : 0u;
        const uint32_t a = (uint32_t)(pair >> 32) + base, b = (uint32_t)pair + base;
        const uint32_t ra = A.R[(int64_t)a * A.T + tt], rb = A.R[(int64_t)b * A.T + tt];
        const uint32_t c2 = ((ra >> 1) == (uint32_t)c ? rb : ra) >> 1;
        // both chose this edge: the smaller root stays a root
        if ((uint32_t)c < c2 && A.B[(int64_t)c2 * A.T + tt] == w) continue;
        A.P[i] = (c2 << 1) | ((ra ^ rb ^ mst_edge_sign(A, a, b)) & 1u);
        hooked = true;
        if (A.in_tree) {
            const int64_t e = mst_edge_index(A.edges, A.m, a, b);
            if (e < A.m && (uint32_t)A.edges[e].x == a && ((uint32_t)A.edges[e].y & SB_ID_MASK) == b)
                A.in_tree[tb * A.m + e] = 1;
            else
                atomicOr(A.err, 4u);
        }
    }
    if (__syncthreads_or(hooked) && threadIdx.x == 0) A.merged[r] = 1;
}

// 3. pointer jumping to the roots; a pointer's low bit is the parity of the
// path to its target.  Roots do not move here, and every stored pointer names
// an ancestor, so a walk only climbs; it is bounded all the same.
__global__ void __launch_bounds__(MST_THREADS) k_mst_jump(MstArgs A, int r)
{
    if (A.mode[r] == MST_DONE || !A.merged[r]) return;
    for (MstWalk k(A.T); k.row < A.n; k.next()) {
        const int64_t v = k.row;
        const int tt = k.tree();
        if (A.tb0 + tt >= A.K) continue;
        const int64_t i = v * A.T + tt;
        uint32_t w = mst_ld(A.P + i);
        const uint32_t was = w;
        int64_t steps = 0;
        while (true) {
            const uint32_t a = w >> 1;
            const uint32_t wa = mst_ld(A.P + (int64_t)a * A.T + tt);
            if ((wa >> 1) == a) break;  // a is a root
            w = (wa & ~1u) | ((w ^ wa) & 1u);
            if (++steps > A.n) {
                atomicOr(A.err, 4u);
                break;
            }
        }
        if (w != was) A.P[i] = w;
        A.R[i] = w;
        if ((int64_t)(w >> 1) == v) A.B[i] = ~0ull;  // still a root: its next search starts afresh
    }
}

// raw labels (parity to the root) as 32-bit ballots, and the spanning check:
// every vertex must share its graph's first vertex's root
__global__ void __launch_bounds__(MST_THREADS) k_mst_pack(MstArgs A, uint32_t* lab32, int W, int w0)
{
    for (MstWalk k(A.T); k.row < A.n; k.next()) {  // a whole warp per vertex
        const int64_t v = k.row;
        const int tt = k.tree();
        const int64_t i = v * A.T + tt;
        const bool valid = A.tb0 + tt < A.K;
        const uint32_t rv = A.R[i];
        const unsigned bal = __ballot_sync(0xffffffffu, valid && (rv & 1u));
        // the last pass may hold words past W: they are not written
        if ((threadIdx.x & 31) == 0 && w0 + (tt >> 6) < W) lab32[(v * W + w0) * 2 + (tt >> 5)] = bal;
        if (valid) {
            const int64_t g0 = A.vgoff ? A.vgoff[v] : 0;
            if ((A.R[g0 * A.T + tt] >> 1) != (rv >> 1)) atomicOr(A.err, 4u);
        }
    }
}

static sb_status mst_scratch(sb_ctx* c, size_t slots, size_t done_words, size_t big, size_t light)
{
    if (c->mst_cap < slots) {
        sb_dfree(c, c->mst_P);
        sb_dfree(c, c->mst_R);
        sb_dfree(c, c->mst_B);
        c->mst_P = (uint32_t*)sb_dalloc(c, sizeof(uint32_t) * slots);
        c->mst_R = (uint32_t*)sb_dalloc(c, sizeof(uint32_t) * slots);
        c->mst_B = (uint64_t*)sb_dalloc(c, sizeof(uint64_t) * slots);
        c->mst_cap = c->mst_P && c->mst_R && c->mst_B ? slots : 0;
        if (!c->mst_cap) return sb_fail(c, SB_ERR_OOM, "Kruskal scratch (%zu slots)", slots);
    }
    SB_TRY(sb_ensure(c, (void**)&c->mst_done, &c->mst_done_cap, sizeof(uint32_t) * done_words));
    SB_TRY(sb_ensure(c, (void**)&c->mst_big, &c->mst_big_cap, sizeof(uint32_t) * big));
    if (light) SB_TRY(sb_ensure(c, (void**)&c->mst_light, &c->mst_light_cap, sizeof(uint32_t) * light));
    if (!c->mst_flags) c->mst_flags = (int32_t*)sb_dalloc(c, sizeof(int32_t) * 2 * MST_ROUNDS_MAX);
    return c->mst_flags ? SB_OK : sb_fail(c, SB_ERR_OOM, "Kruskal flags");
}

extern "C" sb_status sb_sample_trees_kruskal(sb_ctx* c, uint64_t seed, int64_t tree_begin, int64_t K,
                                             uint8_t* in_tree_out)
{
    if (!c) return SB_ERR_ARG;
    if (!c->has_graph) return sb_fail(c, SB_ERR_STATE, "no graph loaded");
    if (K < 1 || K > SB_TREES_MAX || tree_begin < 0)
        return sb_fail(c, SB_ERR_ARG, "K must be in [1, %d] and tree_begin >= 0", SB_TREES_MAX);
    if (in_tree_out && !sb_is_device_ptr(in_tree_out))
        return sb_fail(c, SB_ERR_ARG, "in_tree_out must be a device pointer");
    SB_CHECK_CUDA(c, cudaSetDevice(c->device));
    SB_TRY(sb_batch_begin(c, seed, tree_begin, K));
    const int64_t n = c->n;
    const int W = c->W;
    // words per pass: as many as the scratch budget holds (at most half the
    // free memory), at least one, and at most the SB_TUNE_MST_WORDS knob
    size_t free_b = 0, total_b = 0;
    SB_CHECK_CUDA(c, cudaMemGetInfo(&free_b, &total_b));
    const uint64_t budget = std::min<uint64_t>(MST_PASS_BUDGET, (uint64_t)free_b / 2);
    // light edges: a weight's upper half below theta, MST_LIGHT_DEGREE of them
    // per vertex on average; without a row long enough to spare, no such rounds
    const bool large = 2 * c->m * 64 * (int64_t)W >= MST_LIGHT_PAIRS;
    const double p_light = MST_LIGHT_DEGREE * (double)n / (2.0 * (double)std::max<int64_t>(c->m, 1));
    const uint32_t theta = large && p_light < MST_LIGHT_MAX ? (uint32_t)(p_light * 4294967296.0) : 0u;
    const int64_t blocks = (2 * c->m >> 5) + n;  // of 32 entries, see mst_block
    const int64_t per_word = 64 * (n * MST_BYTES_PER_SLOT + (theta ? blocks * (int64_t)sizeof(uint32_t) : 0));
    int Wp = (int)std::max<int64_t>(1, std::min<int64_t>(W, (int64_t)(budget / (uint64_t)per_word)));
    if (c->tune[SB_TUNE_MST_WORDS] > 0) Wp = std::min<int>(Wp, (int)c->tune[SB_TUNE_MST_WORDS]);
    const int T = 64 * Wp;
    const int64_t graphs = c->batch_G > 0 ? c->batch_G : 1;
    SB_TRY(mst_scratch(c, (size_t)n * T, (size_t)c->n_gl_items * (T / 32), (size_t)graphs * T, theta ? (size_t)blocks * T : 0));
    // rounds: ceil(log2(largest graph)) + 1
    int64_t nmax = n;
    if (c->batch_G > 0) {
        nmax = 1;
        for (int64_t g = 0; g < c->batch_G; g++) nmax = std::max<int64_t>(nmax, c->h_voff[g + 1] - c->h_voff[g]);
    }
    int rounds = 1 + (theta ? MST_LIGHT_ROUNDS + 1 : 0);
    const int more = rounds;
    while (((int64_t)1 << (rounds - more)) < nmax) rounds++;
    if (in_tree_out) SB_CHECK_CUDA(c, cudaMemsetAsync(in_tree_out, 0, (size_t)K * (size_t)c->m, c->stream));
    SB_CHECK_CUDA(c, cudaMemsetAsync(c->sync, 0, sizeof(uint32_t) * 16, c->stream));

    MstArgs A;
    A.n = n;
    A.T = T;
    A.K = K;
    A.S = sb_seed_key(seed);
    A.tree0 = tree_begin;
    A.items = c->gl_items;
    A.n_items = c->n_gl_items;
    A.rowptr = c->rowptr;
    A.col = c->col;
    A.vgid = c->batch_G > 0 ? c->vgid : nullptr;
    A.vgoff = c->batch_G > 0 ? c->vgoff : nullptr;
    A.voff = c->batch_G > 0 ? c->b_voff : nullptr;
    A.graphs = graphs;
    A.big = n >= MST_BIG_VERTICES * graphs ? c->mst_big : nullptr;
    A.P = c->mst_P;
    A.R = c->mst_R;
    A.B = c->mst_B;
    A.done = c->mst_done;
    A.light = c->mst_light;
    A.theta = theta;
    A.light_rounds = MST_LIGHT_ROUNDS;
    A.mode = c->mst_flags;
    A.merged = c->mst_flags + MST_ROUNDS_MAX;
    A.edges = c->edges;
    A.m = c->m;
    A.in_tree = in_tree_out;
    A.err = c->sync + 6;
    const unsigned grid = (unsigned)std::min<int64_t>(sb_cdiv(n * T, MST_THREADS), (int64_t)c->num_sms * 16);
    const unsigned grid_min =
        (unsigned)std::min<int64_t>(sb_cdiv(c->n_gl_items * T, MST_THREADS), (int64_t)c->num_sms * 16);
    const unsigned grid_big =
        A.big ? (unsigned)std::min<int64_t>(sb_cdiv(graphs * T * 32, MST_THREADS), (int64_t)c->num_sms * 16) : 1u;
    SbProf prof(c, SB_PROF_BFS);
    for (int w0 = 0; w0 < W; w0 += Wp) {
        A.tb0 = 64 * (int64_t)w0;
        SB_CHECK_CUDA(c, cudaMemsetAsync(c->mst_flags, 0, sizeof(int32_t) * 2 * MST_ROUNDS_MAX, c->stream));
        k_mst_init<<<grid, MST_THREADS, 0, c->stream>>>(A);
        SB_TRY(sb_after_launch(c, "k_mst_init"));
        for (int r = 0; r < rounds; r++) {
            k_mst_big<<<grid_big, MST_THREADS, 0, c->stream>>>(A, r);
            SB_TRY(sb_after_launch(c, "k_mst_big"));
            if (theta && r >= 1 && r <= MST_LIGHT_ROUNDS) {
                k_mst_light<<<grid_min, MST_THREADS, 0, c->stream>>>(A, r);
                SB_TRY(sb_after_launch(c, "k_mst_light"));
            }
            if (r == 0) k_mst_min<true><<<grid_min, MST_THREADS, 0, c->stream>>>(A, r);
            else if (!theta || r >= 2) k_mst_min<false><<<grid_min, MST_THREADS, 0, c->stream>>>(A, r);
            SB_TRY(sb_after_launch(c, "k_mst_min"));
            k_mst_hook<<<grid, MST_THREADS, 0, c->stream>>>(A, r);
            SB_TRY(sb_after_launch(c, "k_mst_hook"));
            k_mst_jump<<<grid, MST_THREADS, 0, c->stream>>>(A, r);
            SB_TRY(sb_after_launch(c, "k_mst_jump"));
        }
        k_mst_pack<<<grid, MST_THREADS, 0, c->stream>>>(A, (uint32_t*)c->labels, W, w0);
        SB_TRY(sb_after_launch(c, "k_mst_pack"));
    }
    return sb_batch_end(c);
}
