// sb_bpp.cu -- graphBpp hot path: batched randomized-BFS tree sampling with
// parity labelling (Algorithm 1 through the appendix graphB+ algorithm,
// restated with Harary's bipartition, Sec. 2), the state hash that keys the
// frustration cloud (the frustration scorer is in sb_score.cu).
//
// Data layout (vertex-major, 32 trees per half-word, 64 per uint64 word):
//   labels[v * W + w]  bit b = parity label of slot 64 w + b at vertex v
//   vis / frontier     [v * H + h] for the H half-words of one BFS launch
// A slot holds one tree of the batch (k_tree_order says which).
//
// A BFS launch grows up to 32 words (2048 trees) at once, level by level, in
// one cooperative persistent kernel: a group of G lanes owns one vertex (or one
// slice of 32 half-words of it), lane = half-word, gathers its neighbours'
// frontier rows with coalesced loads, and picks each newly reached tree's
// parent as the argmin of the packed key (fmix32((u ^ y_v) + a_t) << 32 | u).
// fmix32 is a bijection, so the hash alone orders the candidates of one (tree,
// vertex): comparing 32-bit hashes is the 64-bit packed argmin.  Rows longer
// than SB_BFS_CHUNK are split over several groups that merge with 64-bit
// atomicMin on the packed key.
//
// What bounds it: instructions of the hash loop (on the 2^20 R-MAT graph with
// 1024 trees 13.0 G warp instructions for 6.8 G candidates, 74 % of the issue
// slots, the ALU pipe 71 % busy; on the 2^24 graph also the frontier rows from
// DRAM).  A lane walks its own candidates, so what counts is that the lanes of
// a warp have about as many each.  One lane per half-word puts one vertex into
// a warp from 16 words on (one lane per 64-tree word made that two, whose
// neighbours differ), trees are dealt out over the
// half-words by depth, and warps take their work items as they get free instead
// of waiting for the slowest at every level.  With those shares so even, a
// queue that rebalances a tile's candidates over the group costs more than it
// gives in a whole warp (17.4 against 18.4 ms) and stays for narrower groups,
// whose vertices differ (45 against 62 ms on 512 uneven graphs).
#include <algorithm>

#include "sb_internal.cuh"

// Work items are sorted by degree.  Whole-warp groups: one round of items is
// dealt out in advance, the next BFS_SINGLE_PCT per cent of them are taken one
// by one and the rest, light by then, A.grab at a time.  All dealt out in
// advance (a round of one per group, the order reversing every round): 17.4 /
// 616 ms (2^20, 2^24 graph); half of them 16.8 / 571, a tenth 14.8 / 524; as
// here 13.9 / 506 (30 per cent one by one 14.2 / 523, everything 14.7 / 570: a
// ticket is an atomic on one counter).  Narrower groups: BFS_FIXED_PCT per cent
// in advance, the rest 4 per group and ticket (39.2 ms on 512 uneven graphs,
// 43.2 all in advance).  A launch of fewer rounds than BFS_TICKET_ROUNDS (whole
// warps) or BFS_TICKET_ROUNDS_NARROW deals everything out: there every warp draws
// a ticket at each level for hardly any work.  Uniform random graph of 100,000
// vertices and degree 10, one and 64 trees (1.5 rounds): 262 / 397 us with
// tickets, 126 / 184 without; grid of 300 x 300 (352 and 565 levels) 8.3 / 18.6
// against 4.0 / 7.8 ms.  Whole warps, R-MAT: 23,000 vertices (5 rounds), 250 trees
// 507 with tickets, 544 without; 85,000 (20 rounds), 500 trees 1.28 / 1.50 ms.
// Narrow: 100,000 vertices, 500 trees (12 rounds) 704 / 747 us.
#define BFS_SINGLE_PCT 10
#define BFS_FIXED_PCT 40
#define BFS_TICKET_ROUNDS 4
#define BFS_TICKET_ROUNDS_NARROW 8
#define BFS_THREADS 128
#define BFS_THREADS_PAR 128
// Candidate-queue entries per lane (more are hashed lane by lane).
#define BFS_QUEUE 16
// 28 warps, 72 registers: 588 ms per 4096 trees on the 2^24 graph, 627 with 6
// blocks (85 registers) and 602 with 8 (64); 16.6 / 16.7 / 16.7 ms per 1024
// trees on the 2^20 graph.
#define BFS_BLOCKS_PER_SM 7
// Batches on graphs of at least this many vertices fill the slots by the
// trees' expected depth: 589 -> 506 ms per 4096 trees on the 2^24 graph, 14.6 ->
// 13.9 ms per 1024 on the 2^20 graph, 1.45 -> 1.42 ms at 95,000 vertices, where
// bringing the labels back into tree order takes about as much.
#define BFS_ORDER_MIN (1 << 18)
// Threads per SM below which a launch spreads its half-words over more lanes.
#define BFS_SPREAD_THREADS 512
// Work items below which a graph of mean degree 16 and more with split rows does
// so too, up to 32 lanes per vertex.  Fewest lanes against 32, R-MAT, 1 / 64 /
// 250 trees: 14,000 vertices of degree 66 215 / 567 / 741 against 146 / 346 / 421
// us, 23,000 of degree 30 198 / 516 / 843 against 149 / 417 / 544, 85,000 of degree
// 34 450 / 970 / 995 against 433 / 789 / 1020; 180,000 of degree 23 (128 / 500
// trees) 1.19 / 1.87 against 1.57 / 2.06 ms.  Where degrees are alike (no split
// row) the vertices of a warp do not wait for one another, and few lanes are
// faster: uniform random graphs, 30,000 vertices of degree 60 112 / 169 / 300
// against 199 / 401 / 555 us, 100,000 of degree 60 185 / 311 / 927 against 510 /
// 1341 / 1666.
#define BFS_SPREAD_ITEMS (1 << 17)
#define SYNC_WORDS 48
// Shared-memory slots: rows of one owner thread's 32 trees (running minima,
// winner ids), 16-byte aligned, and of one half-word's tree salts.
#define BSLOT(o, t) ((o) * 36 + (t))
#define KSLOT(h, t) ((h) * 33 + (t))

struct BfsArgs {
    const sb_bfs_item* items;
    int64_t n_items;
    const int32_t* col;
    const int32_t* hub_vertex;
    int64_t n_hubs;
    uint32_t* lab;      // n x Ht half-words
    int Ht, h0;         // half-words of the batch; first one of this launch
    int H;              // half-words of this launch
    int slices;         // groups of 32 half-words, 1 or 2
    int64_t fixed_rounds;    // rounds of units dealt out in advance; the rest are taken as warps get free,
    int64_t single_tickets;  // that many times one unit per group, then
    int grab;                // `grab` units per group at a time
    int ls;             // 1 << ls lanes share a half-word, 32 >> ls trees each
    uint32_t* vis;      // n x H
    uint32_t* fr0;
    uint32_t* fr1;
    int32_t* done;      // n x slices: level at which every tree had the vertex, or -1
    uint32_t* hubnew;   // n_hubs x H
    uint64_t* hubbest;  // n_hubs x H x 32
    uint32_t* sync;
    int32_t* parents;   // K x n or null
    int64_t n;
    uint64_t S;            // seed key
    const int64_t* tree0;  // global index of batch tree 0 (device)
    const int32_t* perm;   // tree of each slot, or null (slot = tree)
    const int32_t* vgoff;  // first vertex of each vertex's graph (batches), or null
    long long wait;        // SM cycles a barrier wait may take before it reports a timeout
    unsigned bar_extra;    // arrivals a barrier expects beyond the launch's blocks (0; 1 tests the timeout path)
};

// ----------------------------------------------------------- grid barrier
// Cooperative launch makes every block resident; the wait is still bounded
// (`limit` SM cycles) and reports a timeout through sync[6] instead of
// hanging.  `nblocks` is the number of arrivals that open the barrier.
__device__ __forceinline__ void grid_barrier(uint32_t* sync, unsigned nblocks, long long limit)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile uint32_t* gen = sync + 5;
        uint32_t g = *gen;
        __threadfence();
        uint32_t arrived = atomicAdd(sync + 4, 1u);
        if (arrived == nblocks - 1) {
            atomicExch(sync + 4, 0u);
            __threadfence();
            atomicAdd(sync + 5, 1u);
        } else {
            long long t0 = clock64();
            while (*gen == g) {
                __nanosleep(40);
                if (clock64() - t0 > limit) {
                    atomicOr(sync + 6, 1u);
                    break;
                }
            }
        }
        __threadfence();
    }
    __syncthreads();
}

__device__ __forceinline__ unsigned group_mask(int G)
{
    if (G >= 32) return 0xffffffffu;
    unsigned base = (threadIdx.x & 31u) & ~(unsigned)(G - 1);
    return ((1u << G) - 1u) << base;
}

// Winner label bits: each lane keeps its trees' bits in a register while it
// hashes its own candidates; the queue path, where lanes write each other's
// trees, works on a copy in shared memory with atomic bit updates.
__device__ __forceinline__ void lbit_put_atomic(uint32_t* lbits, int o, int t, uint32_t v)
{
    const uint32_t m = 1u << t;
    if (v) atomicOr(lbits + o, m);
    else atomicAnd(lbits + o, ~m);
}

// Position of the highest set bit of a nonzero word.
__device__ __forceinline__ int bit_high(uint32_t x)
{
    uint32_t r;
    asm("bfind.u32 %0, %1;" : "=r"(r) : "r"(x));
    return (int)r;
}

// Group-wide exclusive prefix sum over the G lanes of one vertex.
template <int G>
__device__ __forceinline__ int group_excl_scan(int x, unsigned gmask, int gl, int& total)
{
    int incl = x;
#pragma unroll
    for (int d = 1; d < G; d <<= 1) {
        const int y = __shfl_up_sync(gmask, incl, d, G);
        if (gl >= d) incl += y;
    }
    total = __shfl_sync(gmask, incl, G - 1, G);
    return incl - x;
}

// Sum and maximum over the lanes of a group narrower than a warp.  By shuffles: a
// warp-wide reduction whose mask is a group's runs once per group of the warp
// (500,000 vertices of degree 10: 526 against 452 us for one tree, 804 / 681 for
// 64 trees in 16 groups per warp).
template <int G>
__device__ __forceinline__ unsigned group_sum(unsigned x, unsigned gmask)
{
#pragma unroll
    for (int d = 1; d < G; d <<= 1) x += __shfl_xor_sync(gmask, x, d);
    return x;
}
template <int G>
__device__ __forceinline__ unsigned group_max(unsigned x, unsigned gmask)
{
#pragma unroll
    for (int d = 1; d < G; d <<= 1) x = max(x, __shfl_xor_sync(gmask, x, d));
    return x;
}

// Hashes one lane's candidates m of neighbour u (label word lw), two at a time
// (the highest and the lowest: the same one when a single candidate is left,
// whose second update then repeats the first).
template <bool PAR>
__device__ __forceinline__ void hash_candidates(uint32_t m, uint32_t lw, uint32_t u, uint32_t y, const uint32_t* ak,
                                                uint32_t* bs, uint32_t& lbv, int32_t* bu)
{
    const uint32_t hx = u ^ y;
    while (m) {
        const int ia = bit_high(m);
        const int ib = __ffs((int)m) - 1;
        const uint32_t bita = 1u << ia, bitb = 1u << ib;
        m &= ~(bita | bitb);
        const uint32_t ha = sb_fmix32(hx + ak[ia]);
        const uint32_t hb = sb_fmix32(hx + ak[ib]);
        const uint32_t ba = bs[ia], bb = bs[ib];
        if (ha <= ba) {  // <=: the minima start at 0xFFFFFFFF
            bs[ia] = ha;
            lbv ^= (lbv ^ lw) & bita;  // the winner's label bit
            if (PAR) bu[ia] = (int32_t)u;
        }
        if (hb <= bb) {
            bs[ib] = hb;
            lbv ^= (lbv ^ lw) & bitb;
            if (PAR) bu[ib] = (int32_t)u;
        }
    }
}

// scan_row for a whole warp per vertex: its lanes look at the same neighbour
// and, with the trees dealt out evenly over the half-words, hold about as many
// candidates each, so every lane hashes its own.
template <bool PAR>
__device__ __forceinline__ void scan_row_warp(const int32_t* cp, int len, const uint32_t* cur, const uint32_t* lab, int H,
                                              int Ht, uint32_t mask, uint32_t y, uint32_t goff, const uint32_t* ak,
                                              uint32_t* bs, uint32_t& lbv, int32_t* bu, uint32_t& once, uint32_t& nhash)
{
    const int lane = threadIdx.x & 31;
    const bool any_mask = mask != 0;
    uint32_t cols = 0;
    for (int j = 0; j < len; j += 8) {
        uint32_t c[8], f[8];
        if ((j & 31) == 0) cols = j + lane < len ? (uint32_t)__ldg(cp + j + lane) : 0u;
#pragma unroll
        for (int k = 0; k < 8; k++) c[k] = __shfl_sync(0xffffffffu, cols, (j & 31) + k);
#pragma unroll
        for (int k = 0; k < 8; k++) f[k] = 0;
        if (any_mask) {
            if (j + 8 <= len) {
#pragma unroll
                for (int k = 0; k < 8; k++) f[k] = cur[(int64_t)(c[k] & SB_ID_MASK) * H];
            } else {
#pragma unroll
                for (int k = 0; k < 8; k++)
                    if (j + k < len) f[k] = cur[(int64_t)(c[k] & SB_ID_MASK) * H];
            }
        }
        uint32_t any = 0;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            f[k] &= mask;
            any |= f[k];
        }
        if (!__any_sync(0xffffffffu, any != 0)) continue;
        once |= any;
        uint32_t l[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            l[k] = 0;
            if (f[k]) l[k] = lab[(int64_t)(c[k] & SB_ID_MASK) * Ht];
        }
#pragma unroll
        for (int k = 0; k < 8; k++) {
            nhash += (uint32_t)__popc(f[k]);
            hash_candidates<PAR>(f[k], l[k] ^ (uint32_t)((int32_t)c[k] >> 31), (c[k] & SB_ID_MASK) - goff, y, ak, bs,
                                 lbv, bu);
        }
    }
}

// One pass over a CSR range for one vertex: lane gl of the group owns the
// trees in its `mask` of one half-word.  Neighbours are read 8 at a time so
// that 8 frontier gathers are in flight per lane.  It keeps the running argmin
// of the hashed parent key over the candidates: best (initialised to
// 0xFFFFFFFF) holds the smallest hash, lbv / bestu the winner's label bit /
// id; keys are distinct (the hash is a bijection in u), so `h <= best` accepts
// exactly the minimum.  `once` returns the trees that had a candidate.  For
// each tile of 8 neighbours the lanes hash their own candidates when their
// shares are even; otherwise the group's candidate bits are compacted into a
// shared queue (entry = neighbour, owner lane, tree, label bit) and hashed by
// all lanes in lockstep (atomicMin, then the entry equal to the minimum writes
// its label).
// `cur` and `lab` are rewritten between levels by other blocks, so they are
// read with plain (coherent) loads; the column array is read-only.
template <bool PAR, int G>
__device__ __forceinline__ void scan_row(const int32_t* cp, int len, const uint32_t* cur, const uint32_t* lab, int H,
                                         int Ht, int gl, int ls, uint32_t mask, uint32_t y, uint32_t goff,
                                         const uint32_t* akey, const uint32_t* ak, uint32_t* best, uint32_t* lbits,
                                         uint32_t& lbv, int32_t* bestu, uint16_t* queue, uint32_t* hxs, int tid,
                                         unsigned gmask, uint32_t& once, uint32_t& nhash)
{
    uint32_t* const bs = best + BSLOT(tid, 0);
    const int owner0 = tid - gl;  // thread index of the group's lane 0
    for (int j = 0; j < len; j += 8) {
        uint32_t c[8], f[8], l[8];
#pragma unroll
        for (int k = 0; k < 8; k++) c[k] = (j + k < len) ? (uint32_t)__ldg(cp + j + k) : 0u;
#pragma unroll
        for (int k = 0; k < 8; k++) f[k] = (j + k < len && mask) ? (cur[(int64_t)(c[k] & SB_ID_MASK) * H] & mask) : 0u;
#pragma unroll
        for (int k = 0; k < 8; k++)
            l[k] = f[k] ? (lab[(int64_t)(c[k] & SB_ID_MASK) * Ht] ^ (uint32_t)((int32_t)c[k] >> 31)) : 0u;
        int cnt = 0;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            once |= f[k];
            cnt += __popc(f[k]);
        }
        const unsigned Tsum = group_sum<G>((unsigned)cnt, gmask);
        if (Tsum == 0) continue;  // same for the whole group
        nhash += (uint32_t)cnt;
        const unsigned cmax = group_max<G>((unsigned)cnt, gmask);
        if (cmax * G <= 4 * Tsum + 2 * G || Tsum > BFS_QUEUE * G) {
            // the lanes' shares are even enough (or too many to queue): every
            // lane hashes its own candidates into its own slots, two at a
            // time, with no queue and no synchronisation
#pragma unroll
            for (int k = 0; k < 8; k++)
                hash_candidates<PAR>(f[k], l[k], (c[k] & SB_ID_MASK) - goff, y, ak, bs, lbv,
                                     PAR ? bestu + BSLOT(tid, 0) : nullptr);
            continue;
        }
        // the queue path updates other lanes' label bits: through shared memory
        lbits[tid] = lbv;
        int T;
        int pos = group_excl_scan<G>(cnt, gmask, gl, T);
#pragma unroll
        for (int k = 0; k < 8; k++) {
            // the group's table of the 8 neighbours' u ^ y (one writer per entry)
            if ((k & (G - 1)) == gl) hxs[k] = ((c[k] & SB_ID_MASK) - goff) ^ y;
            for (uint32_t b = f[k]; b;) {
                const int t = __ffs((int)b) - 1;
                b &= b - 1;
                queue[pos++] = (uint16_t)((k << 12) | (gl << 7) | (t << 1) | (int)((l[k] >> t) & 1u));
            }
        }
        __syncwarp(gmask);
        for (int i = gl; i < T; i += G) {
            const uint32_t e = queue[i];
            const int k = (int)(e >> 12), ow = (int)((e >> 7) & 31u), t = (int)((e >> 1) & 31u);
            atomicMin(&best[BSLOT(owner0 + ow, t)], sb_fmix32(hxs[k] + akey[KSLOT(ow >> ls, t)]));
        }
        __syncwarp(gmask);
        for (int i = gl; i < T; i += G) {
            const uint32_t e = queue[i];
            const int k = (int)(e >> 12), ow = (int)((e >> 7) & 31u), t = (int)((e >> 1) & 31u);
            const uint32_t hxk = hxs[k];
            const uint32_t h = sb_fmix32(hxk + akey[KSLOT(ow >> ls, t)]);
            const int o = owner0 + ow;
            if (best[BSLOT(o, t)] == h) {  // fmix32 is injective in u: one entry matches
                lbit_put_atomic(lbits, o, t, e & 1u);
                if (PAR) bestu[BSLOT(o, t)] = (int32_t)(hxk ^ y);
            }
        }
        __syncwarp(gmask);
        lbv = lbits[tid];
    }
}

// Phase B of one level for one split row: the merged minima of its chunks
// (a warp; lane = half-word, then lane = tree).
template <bool PAR>
__device__ __forceinline__ bool bfs_hub(const BfsArgs& A, int L, uint32_t* nxt, int64_t hi, int sl)
{
    const int lane = threadIdx.x & 31;
    const int32_t v = A.hub_vertex[hi];
    const int64_t dslot = (int64_t)v * A.slices + sl;
    const int32_t d = A.done[dslot];
    if (d >= 0 && L >= d + 3) return false;
    const int h = 32 * sl + lane;
    const bool act = h < A.H;
    uint32_t visw = ~0u, nw = 0, labw = 0;
    if (act) {
        visw = A.vis[(int64_t)v * A.H + h];
        nw = A.hubnew[hi * A.H + h] & ~visw;
        A.hubnew[hi * A.H + h] = 0;
    }
    for (uint32_t hs = __ballot_sync(0xffffffffu, nw != 0); hs; hs &= hs - 1) {
        const int hh = __ffs((int)hs) - 1;
        const uint32_t w = __shfl_sync(0xffffffffu, nw, hh);
        uint64_t key = 0;
        if ((w >> lane) & 1u) {
            uint64_t* hb = A.hubbest + (hi * A.H + 32 * sl + hh) * 32 + lane;
            key = *hb;
            *hb = ~0ull;
            if (PAR && A.parents) {
                const int64_t slot = 32 * (int64_t)(A.h0 + 32 * sl + hh) + lane;
                A.parents[(A.perm ? (int64_t)A.perm[slot] : slot) * A.n + v] = (int32_t)((key >> 1) & SB_ID_MASK);
            }
        }
        const uint32_t lb = __ballot_sync(0xffffffffu, (key & 1ull) != 0);
        if (lane == hh) labw = lb;
    }
    if (act) {
        if (nw) {
            if (labw) A.lab[(int64_t)v * A.Ht + A.h0 + h] |= labw;
            A.vis[(int64_t)v * A.H + h] = visw | nw;
        }
        nxt[(int64_t)v * A.H + h] = nw;
    }
    if (d < 0) {
        const bool all = __all_sync(0xffffffffu, (visw | nw) == ~0u);
        if (all && lane == 0) A.done[dslot] = L;
    }
    return nw != 0;
}

template <int G, bool PAR>
__global__ void __launch_bounds__(PAR ? BFS_THREADS_PAR : BFS_THREADS, PAR ? 2 : BFS_BLOCKS_PER_SM)
    k_bfs(BfsArgs A)
{
    constexpr int BD = PAR ? BFS_THREADS_PAR : BFS_THREADS;
    extern __shared__ __align__(16) uint32_t smem[];
    uint32_t* best = smem;                            // running minima, BSLOT(thread, tree)
    uint32_t* akey = best + BSLOT(BD, 0);             // tree salts, KSLOT(half-word, tree)
    uint32_t* lbits = akey + A.H * 33;                // winners' label bits (queue path)
    uint32_t* hx_tab = lbits + BD;                    // 8 neighbours' u ^ y per group
    int32_t* bestu = (int32_t*)(hx_tab + 8 * (BD / G));  // winners, BSLOT (PAR only)
    uint16_t* queues = (uint16_t*)(bestu + (PAR ? BSLOT(BD, 0) : 0));  // BFS_QUEUE x G entries per group
    __shared__ uint32_t s_any, s_stop;

    const int tid = threadIdx.x;
    const int gl = tid & (G - 1);
    const unsigned gmask = group_mask(G);
    const int64_t groups_total = (int64_t)gridDim.x * (BD / G);
    const int64_t group_id = (int64_t)blockIdx.x * (BD / G) + tid / G;
    const unsigned nblocks = gridDim.x + A.bar_extra;

    const int64_t tree0 = *A.tree0;
    for (int i = tid; i < A.H * 32; i += BD) {
        const int64_t slot = 32 * (int64_t)A.h0 + i;
        akey[KSLOT(i >> 5, i & 31)] = (uint32_t)sb_tree_key(A.S, tree0 + (A.perm ? (int64_t)A.perm[slot] : slot));
    }
    if (tid == 0) s_any = 0;
    __syncthreads();

    // this lane's trees within its half-word
    const int sub = gl & ((1 << A.ls) - 1), tpl = 32 >> A.ls;
    const uint32_t mine = A.ls ? ((1u << tpl) - 1u) << (sub * tpl) : ~0u;
    uint16_t* queue = queues + (tid / G) * (BFS_QUEUE * G);
    uint32_t* hxs = hx_tab + (tid / G) * 8;
    const int ss = A.slices - 1;  // 1 or 2 slices
    const int64_t units = A.n_items << ss;
    uint32_t n_scan = 0, n_hash = 0, n_hash_hub = 0;  // work counters
    // level 1 is built top-down before the launch (k_bfs_level1): every
    // neighbour of a root has that root as its only candidate
    int L = 2;
    while (true) {
        const uint32_t* cur = (L & 1) ? A.fr0 : A.fr1;
        uint32_t* nxt = (L & 1) ? A.fr1 : A.fr0;
        bool any_new = false;

        // ---- phase A: every work item (whole rows, and chunks of split rows)
        // (sorted by descending degree; see BFS_SINGLE_PCT for who takes which)
        auto unit = [&](int64_t x) {
            const int sl = (int)(x & ss);
            const int4 q = __ldg((const int4*)(A.items + (x >> ss)));  // vertex, CSR range, split row or -1
            const int32_t v = q.x;
            const int64_t dslot = (int64_t)v * A.slices + sl;
            const int32_t d = A.done[dslot];
            if (d >= 0 && L >= d + 3) return;
            const int h = 32 * sl + (gl >> A.ls);
            const bool act = h < A.H;
            const uint32_t vis_w = act ? A.vis[(int64_t)v * A.H + h] : ~0u;
            const uint32_t U = ~vis_w & mine;
            const int len = q.z - q.y;
            const bool hub = q.w >= 0;
            uint32_t once = 0, lbv = 0;
            // the pass below synchronises the group's lanes, so every lane of
            // the group enters it (a lane with nothing to do has mask 0)
            const uint32_t open = __ballot_sync(gmask, U != 0);
            if (open) {
                const uint32_t goff = A.vgoff ? (uint32_t)A.vgoff[v] : 0u;
                const uint32_t y = sb_child_salt(A.S, (uint32_t)v - goff);
                // neighbour entries per 64-tree word: the first open lane of
                // the word's lanes counts them
                const unsigned wl = 2u << A.ls;  // lanes of a word
                const unsigned first = (unsigned)(tid & 31) & ~(wl - 1u);
                if (U && (open & ((1u << (tid & 31)) - 1u) & ~((1u << first) - 1u)) == 0) n_scan += (uint32_t)len;
                uint4* b4 = (uint4*)(best + BSLOT(tid, 0));
#pragma unroll
                for (int i = 0; i < 8; i++) b4[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
                // one pass: every candidate of every open tree is hashed
                uint32_t& nh = hub ? n_hash_hub : n_hash;
                const uint32_t* ak = akey + KSLOT(act ? h : 0, 0);
                if constexpr (G == 32)
                    scan_row_warp<PAR>(A.col + q.y, len, cur + h, A.lab + A.h0 + h, A.H, A.Ht, U, y, goff, ak,
                                       best + BSLOT(tid, 0), lbv, PAR ? bestu + BSLOT(tid, 0) : nullptr, once, nh);
                else
                    scan_row<PAR, G>(A.col + q.y, len, cur + h, A.lab + A.h0 + h, A.H, A.Ht, gl, A.ls, U, y, goff,
                                     akey + KSLOT(32 * sl, 0), ak, best, lbits, lbv, bestu, queue, hxs, tid, gmask, once,
                                     nh);
                lbv &= once;
            }
            if (hub) {
                // chunk of a split row: publish the chunk minima, one atomic per tree
                if (once) {
                    uint64_t* hb = A.hubbest + ((int64_t)q.w * A.H + h) * 32;
                    for (uint32_t b = once; b;) {
                        const int t = __ffs((int)b) - 1;
                        b &= b - 1;
                        const unsigned long long key = ((unsigned long long)best[BSLOT(tid, t)] << 32) |
                                                       (PAR ? ((unsigned long long)(uint32_t)bestu[BSLOT(tid, t)] << 1) : 0ull) |
                                                       ((lbv >> t) & 1u);
                        atomicMin((unsigned long long*)(hb + t), key);
                    }
                    atomicOr(A.hubnew + (int64_t)q.w * A.H + h, once);
                }
                return;
            }
            if (PAR && A.parents) {
                for (uint32_t b = once; b;) {
                    const int t = __ffs((int)b) - 1;
                    b &= b - 1;
                    const int64_t slot = 32 * (int64_t)(A.h0 + h) + t;
                    A.parents[(A.perm ? (int64_t)A.perm[slot] : slot) * A.n + v] = bestu[BSLOT(tid, t)];
                }
            }
            // the lanes of one half-word put their trees together
            for (int s = 1; s < (1 << A.ls); s <<= 1) {
                once |= __shfl_xor_sync(gmask, once, s);
                lbv |= __shfl_xor_sync(gmask, lbv, s);
            }
            if (act && sub == 0) {
                if (once) {
                    if (lbv) A.lab[(int64_t)v * A.Ht + A.h0 + h] |= lbv;
                    A.vis[(int64_t)v * A.H + h] = vis_w | once;
                    any_new = true;
                }
                nxt[(int64_t)v * A.H + h] = once;
            }
            if (d < 0) {
                const bool all = __all_sync(gmask, (vis_w | once) == ~0u);
                if (all && gl == 0) A.done[dslot] = L;
            }
        };
        const int64_t fixed = A.fixed_rounds;
        for (int64_t r = 0; r < fixed; r++) {
            const int64_t x = r * groups_total + ((r & 1) ? groups_total - 1 - group_id : group_id);
            if (x < units) unit(x);
        }
        if (fixed * groups_total < units) {
            constexpr int GW = 32 / G;  // groups of a warp
            const int64_t first = fixed * groups_total, singles = A.single_tickets;
            uint32_t* ctr = A.sync + 36 + L % 3;
            auto ticket = [&]() { return (tid & 31) == 0 ? atomicAdd(ctr, 1u) : 0u; };
            unsigned nt = ticket();  // always one ahead
            while (true) {
                const int64_t t = __shfl_sync(0xffffffffu, nt, 0);
                const int64_t b = first + (t < singles ? t : singles + (t - singles) * A.grab) * GW;
                if (b >= units) break;
                nt = ticket();
                const int cnt = t < singles ? 1 : A.grab;
                for (int i = 0; i < cnt; i++) {
                    const int64_t x = b + i * GW + (tid & 31) / G;
                    if (x < units) unit(x);
                }
            }
        }

        // ---- phase B: resolve split rows, a warp each
        if (A.n_hubs > 0) {
            grid_barrier(A.sync, nblocks, A.wait);
            for (int64_t x = (int64_t)blockIdx.x * (BD / 32) + tid / 32; x < (A.n_hubs << ss);
                 x += (int64_t)gridDim.x * (BD / 32))
                any_new |= bfs_hub<PAR>(A, L, nxt, x >> ss, (int)(x & ss));
        }

        // ---- end of level: any tree grew?
        if (any_new) s_any = 1;
        __syncthreads();
        if (tid == 0) {
            if (s_any) atomicOr(A.sync + (L % 3), 1u);
            s_any = 0;
            if (blockIdx.x == 0) {
                A.sync[(L + 1) % 3] = 0;
                A.sync[36 + (L + 1) % 3] = 0;
            }
        }
        grid_barrier(A.sync, nblocks, A.wait);
        // one reader per block, so that every thread of a block leaves the
        // level loop at the same level
        if (tid == 0) {
            const uint32_t grew = *(volatile uint32_t*)(A.sync + (L % 3));
            const uint32_t err = *(volatile uint32_t*)(A.sync + 6);
            s_stop = (!grew || err) ? 1u : 0u;
        }
        __syncthreads();
        if (s_stop) break;
        if (++L > A.n + 1) {
            if (tid == 0 && blockIdx.x == 0) atomicOr(A.sync + 6, 2u);
            break;
        }
    }
    // work counters of the batch (sb_stats), one atomic per warp and counter
    unsigned long long* acc = (unsigned long long*)(A.sync + 16);
    if (tid == 0 && blockIdx.x == 0) {
        atomicMax(acc, (unsigned long long)L);
        atomicAdd(acc + 1, 1ull);
    }
    for (int d = 16; d; d >>= 1) {
        n_scan += __shfl_xor_sync(0xffffffffu, n_scan, d);
        n_hash += __shfl_xor_sync(0xffffffffu, n_hash, d);
        n_hash_hub += __shfl_xor_sync(0xffffffffu, n_hash_hub, d);
    }
    if ((tid & 31) == 0) {
        atomicAdd(acc + 2, (unsigned long long)n_scan);
        atomicAdd(acc + 3, (unsigned long long)n_hash);
        atomicAdd(acc + 5, (unsigned long long)n_hash_hub);
    }
}

// ------------------------------------------------------------ BFS set-up
// State of one BFS launch before its roots: visited bits, the level-1
// frontier, labels, split-row keys, level counters and barrier words.  (The
// other frontier buffer is written for every vertex at level 2, before its
// first read.  The error word sync[6] is cleared per batch, so that an error
// of an earlier launch stays.)
__global__ void k_bfs_init(int64_t n, int Wb, int Wt, int w0, int64_t K, uint64_t* vis, uint64_t* fr1, uint64_t* lab,
                           int32_t* done, int slices, int64_t nh, uint64_t* hubnew, uint64_t* hubbest, uint32_t* sync)
{
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    if (i0 < 6) sync[i0] = 0;
    if (i0 >= 36 && i0 < 39) sync[i0] = 0;
    const int64_t total = n * Wb;
    for (int64_t i = i0; i < total; i += step) {
        int64_t v = i / Wb;
        int w = (int)(i - v * Wb);
        int64_t trees = K - 64 * (int64_t)(w0 + w);  // trees of this word
        uint64_t active = trees >= 64 ? ~0ull : ((1ull << trees) - 1ull);
        vis[i] = ~active;
        fr1[i] = 0;
        lab[v * Wt + w0 + w] = 0;
        if (w < slices) done[v * slices + w] = -1;
    }
    for (int64_t i = i0; i < nh * Wb * 64; i += step) {
        hubbest[i] = ~0ull;
        if (i < nh * Wb) hubnew[i] = 0;
    }
}

// Roots and BFS level 1, top-down: a neighbour v of tree t's root r joins the
// tree at level 1 with r as its parent (the only vertex of level 0, so no hash
// decides), label lab(r) ^ neg(r, v) = neg(r, v).  One warp per (graph,
// tree of the launch); trees of one word may reach the same vertex, hence
// the atomics.  Frontier of level 1 -> fr1 (read as the current frontier of
// level 2).
__global__ void k_bfs_level1(const int32_t* perm, int64_t n, int Wb, int Wt, int w0, int64_t K, uint64_t S, const int64_t* tree0p,
                             const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, uint64_t* vis,
                             uint64_t* fr1, uint64_t* lab, int32_t* parents, const int32_t* voff, int64_t G)
{
    const int64_t per = 64 * (int64_t)Wb;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= per * G) return;
    const int64_t g = warp / per;
    const int64_t i = warp - g * per;         // tree within this launch
    if (64 * (int64_t)w0 + i >= K) return;
    const int64_t tb = perm ? perm[64 * w0 + i] : 64 * (int64_t)w0 + i;
    const uint64_t key = sb_tree_key(S, *tree0p + tb);
    const int64_t base = voff ? voff[g] : 0;
    const int64_t ng = voff ? voff[g + 1] - voff[g] : n;
    const int64_t r = base + sb_root(key, ng);
    const int w = (int)(i >> 6);
    const unsigned long long bit = 1ull << (i & 63);
    if (lane == 0) {
        atomicOr((unsigned long long*)(vis + r * Wb + w), bit);
        if (parents) parents[tb * n + r] = -1;
    }
    for (int32_t j = rowptr[r] + lane; j < rowptr[r + 1]; j += 32) {
        const uint32_t cv = (uint32_t)col[j];
        const int64_t v = cv & SB_ID_MASK;
        atomicOr((unsigned long long*)(vis + v * Wb + w), bit);
        atomicOr((unsigned long long*)(fr1 + v * Wb + w), bit);
        if (cv >> 31) atomicOr((unsigned long long*)(lab + v * Wt + w0 + w), bit);
        if (parents) parents[tb * n + v] = (int32_t)(r - base);
    }
}

// canonical flip per graph and word (the raw label of the graph's vertex 0),
// and the state-hash sums cleared for k_state_hash_tab; one thread per hash
__global__ void k_flip(const uint64_t* lab, int W, uint64_t* flipw, const int32_t* voff, int64_t G,
                       unsigned long long* H, unsigned long long* wsum)
{
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= 64 * (int64_t)W * G) return;
    H[x] = 0;
    if (x < G) wsum[x] = 0;
    if (x >= (int64_t)W * G) return;
    const int64_t g = x / W;
    const int w = (int)(x - g * W);
    flipw[x] = lab[(voff ? (int64_t)voff[g] : 0) * W + w];
}

// The same state hashes from subset-sum tables.  A block takes a contiguous
// range of 32-vertex groups.  For each group it tabulates, for each of the
// group's four runs of 8 vertices, the 256 subset sums of their weights; a
// warp then takes one 64-tree word at a time: lane k loads vertex k's label
// word, two 32 x 32 bit transposes across the warp give lane j the group's
// vertices labelled 1 in trees j and j + 32, and four table lookups per tree
// add their weights.  The sums are over raw labels (root labelled 0): the
// canonical flip of a tree is applied afterwards (k_state_hash_flip), as
// H = W_g - H_raw when the tree's vertex 0 is labelled 1, W_g = total weight
// of graph g (Sec. 2: the canonical state is the raw one switched at every
// vertex, so its 1-set is the complement).  A group with vertices of several
// graphs (batches) is taken once per graph, with the other graphs' weights
// left out of the tables.
#define HT_THREADS 256
#define HT_WARPS (HT_THREADS / 32)
#define HT_WPW 8  // words per warp: 64 words over 8 warps
// Fewest groups a block takes.  Groups of one block run one after the other,
// so a small graph wants many blocks; each block ends with one atomic per tree.
// 2 instead of 16: 25.9 -> 4.9 us at n = 1000, 64 trees, 50 -> 27 us at
// n = 95,000, 1000 trees; from 39,000 vertices on the grid is full either way.
#define HT_MIN_GROUPS 2

__global__ void __launch_bounds__(HT_THREADS, 4) k_state_hash_tab(const uint64_t* __restrict__ lab, int64_t n, int W,
                                                                  const uint64_t* __restrict__ weight,
                                                                  const int32_t* __restrict__ vgid, int64_t KP,
                                                                  int64_t groups_per_block,
                                                                  unsigned long long* __restrict__ Hraw,
                                                                  unsigned long long* __restrict__ wsum)
{
    // double-buffered, so that the tables of one group are built while no
    // thread can still be reading the buffer from two groups before
    __shared__ uint64_t tab[2][4][256];
    __shared__ uint64_t sw[2][32];
    const unsigned lane = threadIdx.x & 31u;
    const int warp = (int)(threadIdx.x >> 5);
    const int64_t ngroups = sb_cdiv(n, 32);
    const int64_t q0 = (int64_t)blockIdx.x * groups_per_block;
    const int64_t q1 = min(ngroups, q0 + groups_per_block);
    uint64_t accA[HT_WPW], accB[HT_WPW];
#pragma unroll
    for (int i = 0; i < HT_WPW; i++) accA[i] = accB[i] = 0;
    int64_t gcur = -1;
    int buf = 0;
    auto flush = [&]() {
        if (gcur < 0) return;
#pragma unroll
        for (int i = 0; i < HT_WPW; i++) {
            const int w = warp + HT_WARPS * i;
            if (w < W) {
                if (accA[i]) atomicAdd(Hraw + gcur * KP + 64 * w + lane, (unsigned long long)accA[i]);
                if (accB[i]) atomicAdd(Hraw + gcur * KP + 64 * w + 32 + lane, (unsigned long long)accB[i]);
            }
            accA[i] = accB[i] = 0;
        }
    };
    // table b, subsets s0 .. s0 + 3 of vertices 8 b .. 8 b + 7 of the group
    const int tb = (int)(threadIdx.x >> 6), s0 = (int)(threadIdx.x & 63u) << 2;
    for (int64_t q = q0; q < q1; q++) {
        const int64_t v0 = q * 32;
        const int64_t vk = v0 + lane;
        const int64_t vlast = min(n, v0 + 32) - 1;
        const int64_t ga = vgid ? vgid[v0] : 0, gb = vgid ? vgid[vlast] : 0;
        for (int64_t g = ga; g <= gb; g++) {  // the graphs present in the group (almost always one)
            if (g != gcur) {
                flush();
                gcur = g;
            }
            if (warp == 0) {  // the group's weights, and its share of the graph's total weight
                const uint64_t x = (vk < n && (!vgid || vgid[vk] == g)) ? weight[vk] : 0ull;
                sw[buf][lane] = x;
                uint64_t t = x;
#pragma unroll
                for (int dd = 16; dd; dd >>= 1) t += __shfl_xor_sync(0xffffffffu, t, dd);
                if (lane == 0 && t) atomicAdd(wsum + g, (unsigned long long)t);
            }
            __syncthreads();
            {
                const uint64_t* w8 = sw[buf] + 8 * tb;
                uint64_t base = 0;
#pragma unroll
                for (int i = 2; i < 8; i++)
                    if ((s0 >> i) & 1) base += w8[i];
                uint64_t* t4 = tab[buf][tb] + s0;
                t4[0] = base;
                t4[1] = base + w8[0];
                t4[2] = base + w8[1];
                t4[3] = base + w8[0] + w8[1];
            }
            __syncthreads();
            const uint64_t(*T)[256] = tab[buf];
#pragma unroll
            for (int i = 0; i < HT_WPW; i++) {
                const int w = warp + HT_WARPS * i;
                if (w >= W) break;
                const uint64_t L = vk < n ? lab[vk * W + w] : 0ull;
                const uint32_t MA = warp_transpose32((uint32_t)L, lane);
                const uint32_t MB = warp_transpose32((uint32_t)(L >> 32), lane);
                accA[i] += T[0][MA & 255u] + T[1][(MA >> 8) & 255u] + T[2][(MA >> 16) & 255u] + T[3][MA >> 24];
                accB[i] += T[0][MB & 255u] + T[1][(MB >> 8) & 255u] + T[2][(MB >> 16) & 255u] + T[3][MB >> 24];
            }
            buf ^= 1;
        }
    }
    flush();
}

// canonical flip of the raw sums: trees whose vertex 0 (of the tree's graph)
// is labelled 1 take the complement's weight.  Slot order in, tree order out.
__global__ void k_state_hash_flip(const unsigned long long* Hraw, unsigned long long* H, const unsigned long long* wsum,
                                  const uint64_t* flipw, const int32_t* perm, int W, int64_t KP, int64_t G)
{
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= KP * G) return;
    const int64_t g = x / KP;
    const int64_t t = x - g * KP;
    const unsigned long long h = Hraw[x];
    H[g * KP + (perm ? (int64_t)perm[t] : t)] = ((flipw[g * W + t / 64] >> (t % 64)) & 1ull) ? wsum[g] - h : h;
}

__global__ void k_canon_out(const uint64_t* __restrict__ lab, int64_t total, int W, int64_t K,
                            const uint64_t* __restrict__ flipw, const int32_t* __restrict__ vgid,
                            uint64_t* __restrict__ out)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = i / W;
        const int w = (int)(i - v * W);
        const int64_t g = vgid ? vgid[v] : 0;
        int64_t trees = K - 64 * (int64_t)w;
        uint64_t active = trees >= 64 ? ~0ull : ((1ull << trees) - 1ull);
        out[i] = (lab[i] ^ flipw[g * W + w]) & active;
    }
}

// The same for slots in another order than the trees (one graph).  A block
// stages the canonical rows of 32 vertices; a warp takes an output half-word
// at a time, whose 32 slots its lanes keep while they pick their bit of every
// vertex.
#define CO_THREADS 256
#define CO_ROWS 32
__global__ void __launch_bounds__(CO_THREADS) k_canon_out_order(const uint32_t* __restrict__ lab, int64_t n, int Ht,
                                                                int64_t K, const uint32_t* __restrict__ flip,
                                                                const int32_t* __restrict__ slot,
                                                                uint32_t* __restrict__ out)
{
    extern __shared__ uint32_t co[];
    uint32_t* rows = co;                   // CO_ROWS x Ht canonical rows, slot order
    uint32_t* res = co + CO_ROWS * Ht;     // the same, tree order
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t v0 = (int64_t)blockIdx.x * CO_ROWS; v0 < n; v0 += (int64_t)gridDim.x * CO_ROWS) {
        const int words = (int)min((int64_t)CO_ROWS, n - v0) * Ht;
        for (int i = threadIdx.x; i < words; i += CO_THREADS) rows[i] = lab[v0 * Ht + i] ^ flip[i % Ht];
        __syncthreads();
        for (int h = warp; h < Ht; h += CO_THREADS / 32) {
            const int s = slot[32 * h + lane];
            const uint32_t bit = 32 * (int64_t)h + lane < K ? 1u << (s & 31) : 0u;
            const uint32_t* src = rows + (s >> 5);
            uint32_t keep = 0;
#pragma unroll
            for (int r = 0; r < CO_ROWS; r++) {  // rows past n are read as they are and not written
                const uint32_t b = __ballot_sync(0xffffffffu, src[r * Ht] & bit);
                if (lane == r) keep = b;
            }
            res[lane * Ht + h] = keep;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < words; i += CO_THREADS) out[v0 * Ht + i] = res[i];
        __syncthreads();
    }
}

// --------------------------------------------------------------- host side
template <bool PAR>
static const void* bfs_kernel(int G)
{
    switch (G) {
    case 2: return (const void*)k_bfs<2, PAR>;
    case 4: return (const void*)k_bfs<4, PAR>;
    case 8: return (const void*)k_bfs<8, PAR>;
    case 16: return (const void*)k_bfs<16, PAR>;
    default: return (const void*)k_bfs<32, PAR>;
    }
}

static sb_status ensure_sync(sb_ctx* c)
{
    if (!c->sync) {
        c->sync = (uint32_t*)sb_dalloc(c, sizeof(uint32_t) * SYNC_WORDS);
        if (!c->sync) return sb_fail(c, SB_ERR_OOM, "sync words");
        SB_CHECK_CUDA(c, cudaMemsetAsync(c->sync, 0, sizeof(uint32_t) * SYNC_WORDS, c->stream));
    }
    return SB_OK;
}

static sb_status run_bfs(sb_ctx* c, int w0, int Wb, int32_t* parents)
{
    const bool par = parents != nullptr;
    const int BD = par ? BFS_THREADS_PAR : BFS_THREADS;
    const int H = 2 * Wb, slices = H > 32 ? 2 : 1;
    int G = 2;  // lanes of a vertex: one per half-word
    while (G < H && G < 32) G <<= 1;
    // A graph too small to fill the SMs that way spreads the trees of a
    // half-word over more lanes, which shortens every lane's run of hashes
    // (1000 vertices, 64 trees: 70 us with 2 lanes per vertex, 43 with 32).  The
    // knob asks for one lane per half-word or two; a width found for a launch of
    // more words is not taken over (64 trees on the 2^20 graph: 1.92 ms with 2
    // lanes, 3.02 with 4, 6.5 for the step with 32).
    int ls = 0;
    const int Gt = (int)c->tune[SB_TUNE_BFS_GROUP];
    const bool asked = Gt == G || Gt == 2 * G;
    if (asked && Gt > G) {
        G = Gt;
        ls = 1;
    }
    // and so does a dense one of uneven degrees that fills them a few times over
    // only: its rows take long, and whole warps hash without a queue
    const bool dense = c->n_items < BFS_SPREAD_ITEMS && 2 * c->m >= 16 * c->n && c->n_hubs > 0;
    while (!asked && G < 32 && (dense || c->n_items * slices * G < (int64_t)c->num_sms * BFS_SPREAD_THREADS)) {
        G <<= 1;
        ls++;
    }
    const void* fn = par ? bfs_kernel<true>(G) : bfs_kernel<false>(G);
    const size_t smem = sizeof(uint32_t) * ((size_t)BSLOT(BD, 0) * (par ? 2 : 1) + (size_t)H * 33 + BD + 8 * (BD / G)) +
                        sizeof(uint16_t) * BFS_QUEUE * BD;
    SB_CHECK_CUDA(c, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    SB_CHECK_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, BD, smem));
    if (per_sm < 1) return sb_fail(c, SB_ERR_CUDA, "BFS kernel does not fit on an SM");
    // one group per work unit at most: every further block would only lengthen
    // the grid barriers (1000 vertices, one word: 105 us with 8 blocks, 120
    // with 760, one lane per word)
    unsigned nblocks = (unsigned)std::max<int64_t>(
        1, std::min<int64_t>((int64_t)per_sm * c->num_sms, sb_cdiv(c->n_items * slices, BD / G)));
    const int64_t n = c->n;
    const int64_t ngraphs = c->batch_G > 0 ? c->batch_G : 1;
    const int32_t* perm = c->ordered ? c->order : nullptr;
    unsigned g = (unsigned)std::min<int64_t>(sb_cdiv(std::max(n, c->n_hubs * 64) * Wb, 256), (int64_t)c->num_sms * 16);
    k_bfs_init<<<g, 256, 0, c->stream>>>(n, Wb, c->W, w0, c->K, c->vis, c->fr1, c->labels, c->done, slices, c->n_hubs,
                                         c->hubnew, c->hubbest, c->sync);
    SB_TRY(sb_after_launch(c, "k_bfs_init"));
    {
        const int64_t warps = 64 * (int64_t)Wb * ngraphs;
        k_bfs_level1<<<(unsigned)sb_cdiv(warps * 32, 256), 256, 0, c->stream>>>(
            perm, n, Wb, c->W, w0, c->K, sb_seed_key(c->seed), sb_tree0_ptr(c->sync), c->rowptr, c->col, c->vis, c->fr1,
            c->labels, parents, c->batch_G > 0 ? c->b_voff : nullptr, ngraphs);
        SB_TRY(sb_after_launch(c, "k_bfs_level1"));
    }
    BfsArgs A;
    A.items = c->items;
    A.n_items = c->n_items;
    A.col = c->col;
    A.hub_vertex = c->hub_vertex;
    A.n_hubs = c->n_hubs;
    A.lab = (uint32_t*)c->labels;
    A.Ht = 2 * c->W;
    A.h0 = 2 * w0;
    A.H = H;
    A.slices = slices;
    A.ls = ls;
    {
        const int64_t units = c->n_items * slices, groups = (int64_t)nblocks * (BD / G), rounds = units / groups;
        const bool tickets = rounds >= (G == 32 ? BFS_TICKET_ROUNDS : BFS_TICKET_ROUNDS_NARROW);
        A.fixed_rounds = !tickets ? sb_cdiv(units, groups) : G == 32 ? 1 : std::max<int64_t>(1, rounds * BFS_FIXED_PCT / 100);
        A.single_tickets = G == 32 ? units * BFS_SINGLE_PCT / 100 : 0;
        A.grab = G == 32 && rounds >= 1000 ? 8 : 4;
    }
    A.vis = (uint32_t*)c->vis;
    A.fr0 = (uint32_t*)c->fr0;
    A.fr1 = (uint32_t*)c->fr1;
    A.done = c->done;
    A.hubnew = (uint32_t*)c->hubnew;
    A.hubbest = c->hubbest;
    A.sync = c->sync;
    A.parents = parents;
    A.n = n;
    A.S = sb_seed_key(c->seed);
    A.tree0 = sb_tree0_ptr(c->sync);
    A.perm = perm;
    A.vgoff = c->batch_G > 0 ? c->vgoff : nullptr;
    A.wait = sb_wait_cycles(c);
    A.bar_extra = c->tune[SB_TUNE_STALL_TEST] ? 1u : 0u;
    void* args[] = {&A};
    {
        // a cooperative launch (every block resident for the grid barrier),
        // issued through the launch-attribute form so that it can also be
        // captured into a CUDA graph
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeCooperative;
        attr.val.cooperative = 1;
        cfg.gridDim = dim3(nblocks);
        cfg.blockDim = dim3(BD);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = c->stream;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        SbProf prof(c, SB_PROF_BFS);
        SB_CHECK_CUDA(c, cudaLaunchKernelExC(&cfg, fn, args));
        return sb_after_launch(c, "k_bfs");
    }
}

// Expected depth of every tree of a single-graph batch, as the number of
// entries in the rows of its root's neighbours (most entries first: such a
// root reaches the bulk of the graph one level earlier).  One block per tree.
#define ORD_THREADS 128
__global__ void __launch_bounds__(ORD_THREADS) k_tree_keys(int64_t n, int64_t K, uint64_t S, const int64_t* tree0p,
                                                           const int32_t* __restrict__ rowptr,
                                                           const int32_t* __restrict__ col, uint64_t* __restrict__ keys)
{
    const int64_t t = blockIdx.x;
    const int64_t r = sb_root(sb_tree_key(S, *tree0p + t), n);
    unsigned sum = 0;  // at most 2 m < 2^31
    for (int32_t j = rowptr[r] + (int)threadIdx.x; j < rowptr[r + 1]; j += ORD_THREADS) {
        const int64_t u = (uint32_t)col[j] & SB_ID_MASK;
        sum += (unsigned)(rowptr[u + 1] - rowptr[u]);
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    __shared__ unsigned part[ORD_THREADS / 32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < ORD_THREADS / 32; i++) sum += part[i];
        keys[t] = ((uint64_t)(~sum) << 32) | (uint64_t)t;
    }
}

// order[slot] = tree, order[slots + tree] = slot.  The trees by ascending key
// (a tree's rank is the number of smaller keys, which are distinct; one warp
// counts them) are dealt out over the full half-words, so that each holds the
// same mix of depths: the lanes of a group then have about as many candidates
// each.  The last K % 32 trees and the slots past K come after them.
__global__ void __launch_bounds__(ORD_THREADS) k_tree_order(const uint64_t* __restrict__ keys, int64_t K, int64_t slots,
                                                            int32_t* __restrict__ order)
{
    const int64_t t = ((int64_t)blockIdx.x * ORD_THREADS + threadIdx.x) >> 5;
    if (t >= slots) return;
    unsigned rank = (unsigned)t;
    if (t < K) {
        const uint64_t key = keys[t];
        rank = 0;
        for (int64_t i = threadIdx.x & 31; i < K; i += 32) rank += keys[i] < key ? 1u : 0u;
        rank = __reduce_add_sync(0xffffffffu, rank);
        const unsigned full = (unsigned)(K >> 5);
        if (rank < 32 * full) rank = 32 * (rank % full) + rank / full;
    }
    if ((threadIdx.x & 31) == 0) {
        order[rank] = (int32_t)t;
        order[slots + t] = (int32_t)rank;
    }
}

// Start of a batch: work counters, error word and the device copy of the
// first tree.
__global__ void k_batch_begin(uint32_t* sync, int64_t tree0)
{
    if (threadIdx.x < 16) sync[16 + threadIdx.x] = 0;
    if (threadIdx.x == 16) sync[6] = 0;
    if (threadIdx.x == 17) *sb_tree0_ptr(sync) = tree0;
}

// moves the device copy of the first tree on
__global__ void k_add_i64(int64_t* p, int64_t add) { *p += add; }

// errors of one step kept across the steps of sb_batch_steps: BFS barrier
// (sync[6]) and scorer tile copies (sync[28]) into sync[34]
__global__ void k_latch_errors(uint32_t* sync)
{
    uint32_t e = 0;
    if (sync[6] & 1u) e |= 1u;
    if (sync[6] & ~1u) e |= 2u;
    if (sync[28]) e |= 1u;
    if (e) atomicOr(sync + 34, e);
}

__global__ void k_fold_min(int32_t* acc, const int32_t* x, int64_t n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        acc[i] = min(acc[i], x[i]);
}

__global__ void k_fill_i32(int32_t* p, int64_t n, int32_t v)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

sb_status sb_check_batch(sb_ctx* c, bool scored)
{
    uint32_t w[23] = {0};  // sync[6 .. 28]
    SB_CHECK_CUDA(c, cudaMemcpyAsync(w, c->sync + 6, sizeof(w), cudaMemcpyDeviceToHost, c->stream));
    SB_CHECK_CUDA(c, cudaStreamSynchronize(c->stream));
    const uint32_t err = w[0];
    if (err & 1u) return sb_fail(c, SB_ERR_TIMEOUT, "BFS grid barrier timed out");
    if (err & 2u) return sb_fail(c, SB_ERR_DEVICE_CHECK, "BFS exceeded n levels");
    if (err & 4u) return sb_fail(c, SB_ERR_DEVICE_CHECK, "Kruskal trees did not span their graph");
    if (scored && w[22]) return sb_fail(c, SB_ERR_TIMEOUT, "scorer tile copy timed out");
    return SB_OK;
}

sb_status sb_batch_begin(sb_ctx* c, uint64_t seed, int64_t tree_begin, int64_t K)
{
    SB_TRY(ensure_sync(c));
    const int64_t n = c->n;
    const int W = (int)sb_cdiv(K, 64);
    size_t lab_bytes = sizeof(uint64_t) * (size_t)n * W;
    if (c->labels_cap < lab_bytes) {
        sb_dfree(c, c->labels);
        c->labels = (uint64_t*)sb_dalloc(c, lab_bytes);
        c->labels_cap = c->labels ? lab_bytes : 0;
    }
    const int64_t G = c->batch_G > 0 ? c->batch_G : 1;  // per-graph results in a batch
    // kept while large enough, so that repeated calls allocate nothing
    sb_status st = sb_ensure(c, (void**)&c->flipw, &c->flipw_cap, sizeof(uint64_t) * W * G);
    if (st == SB_OK) st = sb_ensure(c, (void**)&c->hashes, &c->hashes_cap, sizeof(uint64_t) * 64 * W * G);
    if (st == SB_OK) st = sb_ensure(c, (void**)&c->hraw, &c->hraw_cap, sizeof(uint64_t) * 64 * W * G);
    if (st == SB_OK) st = sb_ensure(c, (void**)&c->counts, &c->counts_cap, sizeof(int32_t) * 64 * W * G);
    c->ordered = false;
    c->has_batch = false;
    if (st != SB_OK || !c->labels || !c->flipw || !c->hashes || !c->counts)
        return sb_fail(c, SB_ERR_OOM, "batch storage (n=%lld, K=%lld)", (long long)n, (long long)K);
    c->seed = seed;
    c->tree_begin = tree_begin;
    c->K = K;
    c->W = W;
    c->counts_valid = c->batch_checked = false;
    c->batch_in_cloud = false;
    k_batch_begin<<<1, 32, 0, c->stream>>>(c->sync, tree_begin);
    return sb_after_launch(c, "k_batch_begin");
}

sb_status sb_batch_end(sb_ctx* c)
{
    const int64_t n = c->n, G = c->batch_G > 0 ? c->batch_G : 1;
    const int W = c->W;
    SB_TRY(sb_ensure(c, (void**)&c->hwsum, &c->hwsum_cap, sizeof(uint64_t) * (size_t)G));
    k_flip<<<(unsigned)sb_cdiv(64 * (int64_t)W * G, 256), 256, 0, c->stream>>>(
        c->labels, W, c->flipw, c->batch_G > 0 ? c->b_voff : nullptr, G, (unsigned long long*)c->hraw,
        (unsigned long long*)c->hwsum);
    SB_TRY(sb_after_launch(c, "k_flip"));
    {
        SbProf prof(c, SB_PROF_HASH);
        const int64_t ngroups = sb_cdiv(n, 32);
        const int64_t nblk = std::max<int64_t>(1, std::min<int64_t>((int64_t)c->num_sms * 4, sb_cdiv(ngroups, HT_MIN_GROUPS)));
        const int64_t per = sb_cdiv(ngroups, nblk);
        k_state_hash_tab<<<(unsigned)sb_cdiv(ngroups, per), HT_THREADS, 0, c->stream>>>(
            c->labels, n, W, c->vweight, c->batch_G > 0 ? c->vgid : nullptr, 64 * (int64_t)W, per,
            (unsigned long long*)c->hraw, (unsigned long long*)c->hwsum);
        SB_TRY(sb_after_launch(c, "k_state_hash_tab"));
        k_state_hash_flip<<<(unsigned)sb_cdiv(64 * (int64_t)W * G, 256), 256, 0, c->stream>>>(
            (const unsigned long long*)c->hraw, (unsigned long long*)c->hashes, (const unsigned long long*)c->hwsum,
            c->flipw, c->ordered ? c->order : nullptr, W, 64 * (int64_t)W, G);
        SB_TRY(sb_after_launch(c, "k_state_hash_flip"));
    }
    c->has_batch = true;
    return SB_OK;
}

static int bfs_words_per_launch(const sb_ctx* c)
{
    return c->tune[SB_TUNE_BFS_WORDS] > 0 ? (int)c->tune[SB_TUNE_BFS_WORDS] : SB_WORDS_MAX;
}

// BFS scratch for the current batch (kept while large enough)
static sb_status bfs_alloc(sb_ctx* c)
{
    const int64_t n = c->n;
    const int W = c->W;
    const int WL = bfs_words_per_launch(c);
    const int Wb_max = W < WL ? W : WL;
    size_t words = (size_t)n * Wb_max;
    if (c->bfs_cap_words < words) {
        sb_dfree(c, c->vis);
        sb_dfree(c, c->fr0);
        sb_dfree(c, c->fr1);
        sb_dfree(c, c->hubnew);
        sb_dfree(c, c->hubbest);
        c->vis = (uint64_t*)sb_dalloc(c, sizeof(uint64_t) * words);
        c->fr0 = (uint64_t*)sb_dalloc(c, sizeof(uint64_t) * words);
        c->fr1 = (uint64_t*)sb_dalloc(c, sizeof(uint64_t) * words);
        const size_t hw = (size_t)(c->n_hubs > 0 ? c->n_hubs : 1) * Wb_max;
        c->hubnew = (uint64_t*)sb_dalloc(c, sizeof(uint64_t) * hw);
        c->hubbest = (uint64_t*)sb_dalloc(c, sizeof(uint64_t) * hw * 64);
        c->bfs_cap_words = (c->vis && c->fr0 && c->fr1 && c->hubnew && c->hubbest) ? words : 0;
    }
    if (!c->done) c->done = (int32_t*)sb_dalloc(c, sizeof(int32_t) * 2 * (size_t)n);  // two slices at most
    if (!c->bfs_cap_words || !c->done)
        return sb_fail(c, SB_ERR_OOM, "BFS batch storage (n=%lld, K=%lld)", (long long)n, (long long)c->K);
    return SB_OK;
}

// Fills the slots by the trees' expected depth (see BFS_ORDER_MIN).
static sb_status bfs_order(sb_ctx* c)
{
    if (c->batch_G > 0 || c->K <= 32 || c->n < BFS_ORDER_MIN) return SB_OK;
    const int64_t slots = 64 * (int64_t)c->W;
    SB_TRY(sb_ensure(c, (void**)&c->order, &c->order_cap, sizeof(int32_t) * 2 * (size_t)slots));
    SB_TRY(sb_ensure(c, (void**)&c->order_keys, &c->order_keys_cap, sizeof(uint64_t) * (size_t)slots));
    k_tree_keys<<<(unsigned)c->K, ORD_THREADS, 0, c->stream>>>(c->n, c->K, sb_seed_key(c->seed), sb_tree0_ptr(c->sync),
                                                               c->rowptr, c->col, c->order_keys);
    SB_TRY(sb_after_launch(c, "k_tree_keys"));
    k_tree_order<<<(unsigned)sb_cdiv(slots * 32, ORD_THREADS), ORD_THREADS, 0, c->stream>>>(c->order_keys, c->K, slots,
                                                                                          c->order);
    SB_TRY(sb_after_launch(c, "k_tree_order"));
    c->ordered = true;
    return SB_OK;
}

// the BFS launches of the current batch (no host synchronisation)
static sb_status bfs_enqueue(sb_ctx* c, int32_t* parents_out)
{
    const int W = c->W, WL = bfs_words_per_launch(c);
    for (int w0 = 0, Wb; w0 < W; w0 += Wb) {
        Wb = W - w0 < WL ? W - w0 : WL;
        // 17 to 23 words leave most lanes of the second slice idle: 16 words
        // and the rest apart take less (1100 trees on the 2^20 R-MAT graph 18.6
        // against 26.4 ms; 1536, 24 words, 27.0 against 28.2, but 2.9 against
        // 2.7 on 95,000 vertices).  Not so a graph of less than one round of
        // whole warps, whose levels take the same time however many words they
        // carry: 1100 trees, 1000 vertices 92 us in two launches, 57 in one, 3200
        // (R-MAT) 592 / 397, a path of 2000 22.0 / 16.7 ms; 10,000 vertices 276
        // / 329 us.
        if (Wb > 16 && Wb < 24 && c->n_items * 32 >= (int64_t)c->num_sms * BFS_BLOCKS_PER_SM * BFS_THREADS) Wb = 16;
        SB_TRY(run_bfs(c, w0, Wb, parents_out));
    }
    return SB_OK;
}

extern "C" sb_status sb_sample_trees(sb_ctx* c, uint64_t seed, int64_t tree_begin, int64_t K, int32_t* parents_out)
{
    if (!c) return SB_ERR_ARG;
    if (!c->has_graph) return sb_fail(c, SB_ERR_STATE, "no graph loaded");
    if (K < 1 || K > SB_TREES_MAX || tree_begin < 0)
        return sb_fail(c, SB_ERR_ARG, "K must be in [1, %d] and tree_begin >= 0", SB_TREES_MAX);
    if (parents_out && !sb_is_device_ptr(parents_out))
        return sb_fail(c, SB_ERR_ARG, "parents_out must be a device pointer");
    SB_CHECK_CUDA(c, cudaSetDevice(c->device));
    SB_TRY(sb_batch_begin(c, seed, tree_begin, K));
    SB_TRY(bfs_alloc(c));
    SB_TRY(bfs_order(c));
    const sb_status st = bfs_enqueue(c, parents_out);
    c->tune[SB_TUNE_STALL_TEST] = 0;  // a test of the timeout path covers one call
    SB_TRY(st);
    return sb_batch_end(c);
}

// One step of sb_batch_steps for the batch set up by sb_batch_begin: trees
// of the device's current range, counts, hashes and per-graph clouds, then
// the range moves on by K.  Enqueue only: no allocation, no host
// synchronisation, so that the step can be captured into a CUDA graph.
static sb_status batch_step_enqueue(sb_ctx* c)
{
    const int64_t G = c->batch_G;
    SB_TRY(bfs_enqueue(c, nullptr));
    SB_TRY(sb_batch_end(c));
    SB_TRY(sb_score_enqueue(c));
    k_latch_errors<<<1, 1, 0, c->stream>>>(c->sync);
    SB_TRY(sb_after_launch(c, "k_latch_errors"));
    SB_TRY(sb_batch_cloud_enqueue(c, c->bs_ns, c->bs_fm));
    k_fold_min<<<(unsigned)sb_cdiv(G, 256), 256, 0, c->stream>>>(c->bs_frmin, c->bs_fm, G);
    SB_TRY(sb_after_launch(c, "k_fold_min"));
    k_add_i64<<<1, 1, 0, c->stream>>>(sb_tree0_ptr(c->sync), c->K);
    return sb_after_launch(c, "k_add_i64");
}

// Captures one step into a CUDA graph (or reuses the captured one while its
// key matches) and launches it `reps` times on c->stream.
static sb_status batch_steps_graph(sb_ctx* c, const uint64_t* key, int reps)
{
    if (!(c->bs_exec && memcmp(key, c->bs_exec_key, sizeof(c->bs_exec_key)) == 0)) {
        if (c->bs_exec) cudaGraphExecDestroy(c->bs_exec);
        c->bs_exec = nullptr;
        cudaGraph_t graph = nullptr;
        SB_CHECK_CUDA(c, cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeRelaxed));
        c->capturing = true;
        const sb_status st = batch_step_enqueue(c);
        c->capturing = false;
        const cudaError_t ec = cudaStreamEndCapture(c->stream, &graph);
        if (st != SB_OK) {
            if (graph) cudaGraphDestroy(graph);
            return st;
        }
        if (ec != cudaSuccess) return sb_cuda_fail(c, ec, "cudaStreamEndCapture");
        const cudaError_t ei = cudaGraphInstantiate(&c->bs_exec, graph, 0);
        cudaGraphDestroy(graph);
        if (ei != cudaSuccess) {
            c->bs_exec = nullptr;
            return sb_cuda_fail(c, ei, "cudaGraphInstantiate");
        }
        memcpy(c->bs_exec_key, key, sizeof(c->bs_exec_key));
    }
    for (int r = 0; r < reps; r++) {
        SbProf prof(c, SB_PROF_BFS);  // a replay is timed as one step (the BFS dominates it)
        SB_CHECK_CUDA(c, cudaGraphLaunch(c->bs_exec, c->stream));
    }
    return SB_OK;
}

extern "C" sb_status sb_batch_steps(sb_ctx* c, uint64_t seed, int64_t tree_begin, int64_t K, int32_t steps,
                                    int32_t use_graph, int32_t* fr_min_out, int32_t* n_states_out)
{
    if (!c) return SB_ERR_ARG;
    if (!c->has_graph || c->batch_G <= 0) return sb_fail(c, SB_ERR_STATE, "no batch of graphs loaded");
    if (K < 1 || K > 1024 || steps < 1 || tree_begin < 0 || (use_graph != 0 && use_graph != 1))
        return sb_fail(c, SB_ERR_ARG, "K must be in [1, 1024], steps >= 1, tree_begin >= 0, use_graph 0 or 1");
    if ((fr_min_out && !sb_is_device_ptr(fr_min_out)) || (n_states_out && !sb_is_device_ptr(n_states_out)))
        return sb_fail(c, SB_ERR_ARG, "fr_min_out and n_states_out must be device pointers");
    SB_CHECK_CUDA(c, cudaSetDevice(c->device));
    const int64_t G = c->batch_G;
    SB_TRY(sb_batch_begin(c, seed, tree_begin, K));
    SB_TRY(bfs_alloc(c));
    if (c->bs_cap < (size_t)G) {
        sb_dfree(c, c->bs_frmin);
        sb_dfree(c, c->bs_fm);
        sb_dfree(c, c->bs_ns);
        c->bs_frmin = (int32_t*)sb_dalloc(c, sizeof(int32_t) * (size_t)G);
        c->bs_fm = (int32_t*)sb_dalloc(c, sizeof(int32_t) * (size_t)G);
        c->bs_ns = (int32_t*)sb_dalloc(c, sizeof(int32_t) * (size_t)G);
        c->bs_cap = (c->bs_frmin && c->bs_fm && c->bs_ns) ? (size_t)G : 0;
        if (!c->bs_cap) return sb_fail(c, SB_ERR_OOM, "batch step outputs");
    }
    SB_CHECK_CUDA(c, cudaMemsetAsync(c->sync + 34, 0, sizeof(uint32_t), c->stream));
    k_fill_i32<<<(unsigned)sb_cdiv(G, 256), 256, 0, c->stream>>>(c->bs_frmin, G, 0x7FFFFFFF);
    SB_TRY(sb_after_launch(c, "k_fill_i32"));
    // the first step runs directly (it also sizes every buffer the step uses)
    sb_status st = batch_step_enqueue(c);
    if (st == SB_OK && steps > 1) {
        if (use_graph) {
            // what the captured launches were made from: arguments, knobs, and the
            // buffers the step before this one left (any of them may have grown
            // since the capture, in a call with more trees)
            auto at = [](const void* p) { return (uint64_t)(uintptr_t)p; };
            const uint64_t key[SB_BS_KEY] = {seed, (uint64_t)K, (uint64_t)G, c->graph_gen, (uint64_t)bfs_words_per_launch(c),
                                             (uint64_t)c->tune[SB_TUNE_BFS_GROUP], (uint64_t)c->tune[SB_TUNE_SCORE_BLOCKS_SM],
                                             (uint64_t)c->tune[SB_TUNE_WAIT_US], (uint64_t)c->tune[SB_TUNE_STALL_TEST],
                                             at(c->labels), at(c->flipw), at(c->hraw), at(c->hwsum), at(c->hashes),
                                             at(c->counts), at(c->vis), at(c->fr0), at(c->fr1), at(c->done), at(c->hubnew),
                                             at(c->hubbest), at(c->sync), at(c->bs_frmin), at(c->bs_fm), at(c->bs_ns)};
            // capture and replay on a private stream ordered after / before
            // the context stream (the legacy default stream cannot be captured)
            if (!c->cap_stream) {
                SB_CHECK_CUDA(c, cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking));
                SB_CHECK_CUDA(c, cudaEventCreateWithFlags(&c->cap_in, cudaEventDisableTiming));
                SB_CHECK_CUDA(c, cudaEventCreateWithFlags(&c->cap_out, cudaEventDisableTiming));
            }
            cudaStream_t main_stream = c->stream;
            SB_CHECK_CUDA(c, cudaEventRecord(c->cap_in, main_stream));
            SB_CHECK_CUDA(c, cudaStreamWaitEvent(c->cap_stream, c->cap_in, 0));
            c->stream = c->cap_stream;
            st = batch_steps_graph(c, key, steps - 1);
            c->stream = main_stream;
            SB_CHECK_CUDA(c, cudaEventRecord(c->cap_out, c->cap_stream));
            SB_CHECK_CUDA(c, cudaStreamWaitEvent(main_stream, c->cap_out, 0));
        } else {
            for (int s = 1; s < steps && st == SB_OK; s++) st = batch_step_enqueue(c);
        }
    }
    c->tune[SB_TUNE_STALL_TEST] = 0;
    SB_TRY(st);
    if (fr_min_out)
        SB_CHECK_CUDA(c, cudaMemcpyAsync(fr_min_out, c->bs_frmin, sizeof(int32_t) * (size_t)G, cudaMemcpyDeviceToDevice,
                                         c->stream));
    if (n_states_out)
        SB_CHECK_CUDA(c, cudaMemcpyAsync(n_states_out, c->bs_ns, sizeof(int32_t) * (size_t)G, cudaMemcpyDeviceToDevice,
                                         c->stream));
    // the last step is the context's sampled batch (scored already)
    c->tree_begin = tree_begin + (int64_t)(steps - 1) * K;
    c->counts_valid = true;
    return SB_OK;
}

extern "C" sb_status sb_frustration(sb_ctx* c, int32_t* counts_out, uint64_t* hashes_out)
{
    if (!c) return SB_ERR_ARG;
    if (!c->has_batch) return sb_fail(c, SB_ERR_STATE, "no sampled batch");
    SB_CHECK_CUDA(c, cudaSetDevice(c->device));
    if (!c->counts_valid) SB_TRY(sb_score_enqueue(c));  // behind the sampler; one wait then covers both
    SB_TRY(sb_check_batch(c, c->m > 0));
    c->counts_valid = c->batch_checked = true;
    if (c->batch_G > 0) {
        // per graph: K entries, packed graph after graph
        const size_t KP = 64 * (size_t)c->W, K = (size_t)c->K, G = (size_t)c->batch_G;
        if (counts_out)
            SB_CHECK_CUDA(c, cudaMemcpy2DAsync(counts_out, K * sizeof(int32_t), c->counts, KP * sizeof(int32_t),
                                               K * sizeof(int32_t), G, cudaMemcpyDefault, c->stream));
        if (hashes_out)
            SB_CHECK_CUDA(c, cudaMemcpy2DAsync(hashes_out, K * sizeof(uint64_t), c->hashes, KP * sizeof(uint64_t),
                                               K * sizeof(uint64_t), G, cudaMemcpyDefault, c->stream));
        SB_CHECK_CUDA(c, cudaStreamSynchronize(c->stream));
        return SB_OK;
    }
    if (counts_out) SB_TRY(sb_copy_out(c, counts_out, c->counts, sizeof(int32_t) * c->K));
    if (hashes_out) SB_TRY(sb_copy_out(c, hashes_out, c->hashes, sizeof(uint64_t) * c->K));
    return SB_OK;
}

extern "C" sb_status sb_label(sb_ctx* c, uint64_t* labels_out)
{
    if (!c || !labels_out) return SB_ERR_ARG;
    if (!c->has_batch) return sb_fail(c, SB_ERR_STATE, "no sampled batch");
    SB_CHECK_CUDA(c, cudaSetDevice(c->device));
    SB_TRY(sb_check_batch(c, false));
    int64_t total = c->n * c->W;
    size_t bytes = sizeof(uint64_t) * (size_t)total;
    uint64_t* tmp = (uint64_t*)sb_dalloc(c, bytes);
    if (!tmp) return sb_fail(c, SB_ERR_OOM, "label export");
    if (c->ordered) {
        const int Ht = 2 * c->W;
        const size_t smem = sizeof(uint32_t) * 2 * CO_ROWS * (size_t)Ht;  // at most 32 KB
        const unsigned g = (unsigned)std::min<int64_t>(sb_cdiv(c->n, CO_ROWS), (int64_t)c->num_sms * 8);
        k_canon_out_order<<<g, CO_THREADS, smem, c->stream>>>((const uint32_t*)c->labels, c->n, Ht, c->K,
                                                              (const uint32_t*)c->flipw, c->order + 32 * Ht,
                                                              (uint32_t*)tmp);
    } else {
        unsigned g = (unsigned)std::min<int64_t>(sb_cdiv(total, 256), (int64_t)c->num_sms * 16);
        k_canon_out<<<g, 256, 0, c->stream>>>(c->labels, total, c->W, c->K, c->flipw,
                                              c->batch_G > 0 ? c->vgid : nullptr, tmp);
    }
    sb_status st = sb_after_launch(c, "k_canon_out");
    if (st == SB_OK) st = sb_copy_out(c, labels_out, tmp, bytes);
    cudaStreamSynchronize(c->stream);
    sb_dfree(c, tmp);
    return st;
}

extern "C" sb_status sb_stats(sb_ctx* c, int64_t* out, int32_t n)
{
    if (!c || !out || n < 0 || n > SB_STATS_N) return SB_ERR_ARG;
    if (!c->sync) {
        for (int i = 0; i < n; i++) out[i] = 0;
        return SB_OK;
    }
    SB_CHECK_CUDA(c, cudaSetDevice(c->device));
    unsigned long long acc[8];
    SB_CHECK_CUDA(c, cudaMemcpyAsync(acc, c->sync + 16, sizeof(acc), cudaMemcpyDeviceToHost, c->stream));
    SB_CHECK_CUDA(c, cudaStreamSynchronize(c->stream));
    for (int i = 0; i < n; i++) out[i] = (int64_t)acc[i];
    return SB_OK;
}
