// sb_score.cu -- the frustration count S_t of every tree of the last sample
// (Algorithm 1, Eq. 1): the number of edges whose sign differs between the
// graph and the tree's balanced state, lab[u] ^ lab[v] ^ neg summed per tree.
#include <algorithm>

#include "sb_count.cuh"
#include "sb_internal.cuh"

static int score_group_for(int Wb)
{
    int g = 1;
    while (g < Wb) g <<= 1;
    return g;
}

// ------------------------------------------------------------------ scorer
// S_t = sum over edges of bit t of lab[u] ^ lab[v] ^ neg.  The edge stream
// (each edge from its colder to its hotter endpoint, sorted by the colder
// one) moves through shared memory in tiles of SC_TILE edges, double-buffered
// with bulk copies; a group of G lanes takes one edge at a time, lane = word
// of 64 trees (two warps share an edge when there are more than 32 words),
// and gathers the two label words.  Every lane keeps 64 vertical counters as
// carry-save adders (ones, twos, fours) plus SC_PLANES ripple planes of
// eights, flushed into 32-bit counts before the planes can overflow.
#define SC_THREADS 256
#define SC_TILE 2048                     // edges per shared-memory tile (16 KB)
#define SC_FAST_BATCH 1                  // whole 8-edge batches without per-edge checks

struct ScoreArgs {
    const int2* edges;    // m edges + 2 of padding: (colder, hotter | neg << 31)
    int64_t m;
    const uint64_t* lab;  // n x Wt label words
    int Wt, w0, Wb;       // words [w0, w0 + Wb) of this launch, Wb <= 64
    const int32_t* vgid;  // graph of every vertex (batches of graphs) or null
    const int32_t* perm;  // tree of each slot, or null (slot = tree)
    int64_t KP;           // count slots per graph
    uint32_t* counts;     // [graph * KP + 64 * word + bit]
    uint32_t* err;        // bit 0 set when a tile copy did not arrive in time
    long long wait;       // SM cycles a tile wait may take before it reports a timeout
    long long drain;      // SM cycles the copies still in flight get before a failed block exits
};

template <int G, bool SEG>
__global__ void __launch_bounds__(SC_THREADS, SEG ? 3 : 4) k_score(ScoreArgs A)
{
    extern __shared__ __align__(128) unsigned char sc_smem[];
    int2* tiles = (int2*)sc_smem;                        // 2 x SC_TILE edges
    uint64_t* bar = (uint64_t*)(tiles + 2 * SC_TILE);    // 2 mbarriers
    uint32_t* scnt = (uint32_t*)(bar + 2);               // Wb x 64 block counts (single graph)
    __shared__ uint32_t s_fail;
    constexpr int NG = SC_THREADS / G;
    const int WS = (A.Wb + 31) >> 5;  // word slices of 32 (G == 32 when WS > 1)
    const int tid = threadIdx.x, gl = tid & (G - 1), grp = tid / G;
    const int slice = grp % WS, j = grp / WS, NGS = NG / WS;
    const int word = slice * 32 + gl;
    const bool act = word < A.Wb;
    if (!SEG)
        for (int i = tid; i < A.Wb * 64; i += SC_THREADS) scnt[i] = 0;
    if (tid == 0) {
        sb_mbar_init(&bar[0], 1);
        sb_mbar_init(&bar[1], 1);
        sb_mbar_init_fence();
        s_fail = 0;
    }
    __syncthreads();
    const int64_t ntiles = sb_cdiv(A.m, SC_TILE);
    const int64_t t0 = ntiles * blockIdx.x / gridDim.x, t1 = ntiles * (blockIdx.x + 1) / gridDim.x;
    // tile t -> buffer; the byte count is rounded up to 16 (the stream is padded)
    auto issue = [&](int64_t t, int buf) {
        const int64_t e0 = t * SC_TILE;
        const int64_t cnt = min((int64_t)SC_TILE, A.m - e0);
        sb_fence_proxy_async();
        sb_bulk_load(tiles + buf * SC_TILE, A.edges + e0, (uint32_t)(((cnt + 1) & ~1ll) * sizeof(int2)), &bar[buf]);
    };
    if (tid == 0 && t0 < t1) issue(t0, 0);
    const uint64_t* __restrict__ lw = A.lab + A.w0 + word;
    const int Wt = A.Wt;
    ScoreAcc acc;
    acc.reset();
    int64_t gcur = SEG ? -1 : 0;
    uint32_t* const dst0 = SEG ? A.counts + 64 * (int64_t)(A.w0 + word) : scnt + 64 * word;
    int64_t tf = -1;  // tile whose copy did not arrive
    for (int64_t t = t0; t < t1; t++) {
        const int buf = (int)((t - t0) & 1);
        if (tid == 0 && t + 1 < t1) issue(t + 1, buf ^ 1);  // read by nobody since the last barrier
        if (!sb_mbar_wait(&bar[buf], (uint32_t)(((t - t0) >> 1) & 1), A.wait)) atomicOr(&s_fail, 1u);
        __syncthreads();
        if (s_fail) {
            tf = t;
            break;
        }
        const int2* te = tiles + buf * SC_TILE;
        const int cnt = (int)min((int64_t)SC_TILE, A.m - t * SC_TILE);
        if (act) {
            int b = j;
            if (!SEG && SC_FAST_BATCH) {
                // whole batches of 8 edges: no per-edge checks
                for (; b + 7 * NGS < cnt; b += 8 * NGS) {
                    uint64_t x[8];
#pragma unroll
                    for (int k = 0; k < 8; k++) {
                        const int2 ed = te[b + k * NGS];
                        const uint64_t negm = (uint64_t)(int64_t)(ed.y >> 31);
                        x[k] = lw[(int64_t)ed.x * Wt] ^ lw[(int64_t)((uint32_t)ed.y & SB_ID_MASK) * Wt] ^ negm;
                    }
                    acc.add8(x);
                    if (acc.nb == SC_FLUSH) acc.flush(dst0);
                }
            }
            for (; b < cnt; b += 8 * NGS) {
                int2 ed[8];
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    const int i = b + k * NGS;
                    ed[k] = i < cnt ? te[i] : make_int2(-1, 0);
                }
                uint64_t x[8];
#pragma unroll
                for (int k = 0; k < 8; k++)
                    x[k] = ed[k].x >= 0 ? (lw[(int64_t)ed[k].x * Wt] ^ lw[(int64_t)((uint32_t)ed[k].y & SB_ID_MASK) * Wt] ^
                                           (ed[k].y < 0 ? ~0ull : 0ull))
                                        : 0ull;
                if (SEG) {
                    // edges are sorted by graph
                    int32_t gk[8];
                    uint32_t rem = 0;
#pragma unroll
                    for (int k = 0; k < 8; k++) {
                        gk[k] = ed[k].x >= 0 ? A.vgid[ed[k].x] : -1;
                        rem |= (ed[k].x >= 0 ? 1u : 0u) << k;
                    }
                    acc.add8_runs(x, gk, rem, gcur, dst0, A.KP);
                    continue;
                } else {
                    acc.add8(x);
                }
                if (acc.nb == SC_FLUSH) acc.flush(dst0 + gcur * A.KP);
            }
        }
        __syncthreads();  // the buffer is reloaded by the next issue
    }
    if (s_fail) {
        if (tid == 0) {
            atomicOr(A.err, 1u);
            // let the copies still in flight land (bounded) before the block exits
            for (int64_t t = tf; t < min(tf + 2, t1); t++)
                (void)sb_mbar_wait(&bar[(t - t0) & 1], (uint32_t)(((t - t0) >> 1) & 1), A.drain);
        }
        return;
    }
    if (SEG && act && gcur >= 0) acc.flush(dst0 + gcur * A.KP);
    if (!SEG) {
        acc.template flush_warp<G>(scnt + 64 * 32 * slice);
        __syncthreads();
        for (int i = tid; i < A.Wb * 64; i += SC_THREADS)
            if (scnt[i]) atomicAdd(A.counts + (A.perm ? A.perm[64 * A.w0 + i] : 64 * A.w0 + i), scnt[i]);
    }
}

template <bool SEG>
static const void* score_kernel(int G)
{
    switch (G) {
    case 1: return (const void*)k_score<1, SEG>;
    case 2: return (const void*)k_score<2, SEG>;
    case 4: return (const void*)k_score<4, SEG>;
    case 8: return (const void*)k_score<8, SEG>;
    case 16: return (const void*)k_score<16, SEG>;
    default: return (const void*)k_score<32, SEG>;
    }
}

__global__ void k_score_begin(uint32_t* counts, int64_t n, uint32_t* err)
{
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i0 == 0) *err = 0;
    for (int64_t i = i0; i < n; i += (int64_t)gridDim.x * blockDim.x) counts[i] = 0;
}

// counts of the current batch (into c->counts): the launches only (no host
// synchronisation); a tile copy that times out sets sync[28]
sb_status sb_score_enqueue(sb_ctx* c)
{
    const int64_t ngraphs = c->batch_G > 0 ? c->batch_G : 1;
    const int64_t nc = 64 * (int64_t)c->W * ngraphs;
    k_score_begin<<<(unsigned)std::min<int64_t>(sb_cdiv(nc, 256), (int64_t)c->num_sms * 16), 256, 0, c->stream>>>(
        (uint32_t*)c->counts, nc, c->sync + 28);
    SB_TRY(sb_after_launch(c, "k_score_begin"));
    if (c->m > 0) {
        const bool seg = c->batch_G > 0;
        const int Wb = c->W;
        const int G = Wb >= 32 ? 32 : score_group_for(Wb);
        const void* fn = seg ? score_kernel<true>(G) : score_kernel<false>(G);
        const size_t smem = 2 * SC_TILE * sizeof(int2) + 2 * sizeof(uint64_t) + (seg ? 0 : sizeof(uint32_t) * 64 * Wb);
        SB_CHECK_CUDA(c, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        int per_sm = 0;
        SB_CHECK_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, SC_THREADS, smem));
        if (c->tune[SB_TUNE_SCORE_BLOCKS_SM] > 0) per_sm = std::min<int>(per_sm, (int)c->tune[SB_TUNE_SCORE_BLOCKS_SM]);
        const int64_t ntiles = sb_cdiv(c->m, SC_TILE);
        const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((int64_t)c->num_sms * std::max(per_sm, 1), ntiles));
        ScoreArgs A;
        A.edges = c->sc_edges;
        A.m = c->m;
        A.lab = c->labels;
        A.Wt = c->W;
        A.w0 = 0;
        A.Wb = Wb;
        A.vgid = seg ? c->vgid : nullptr;
        A.perm = c->ordered ? c->order : nullptr;
        A.KP = 64 * (int64_t)c->W;
        A.counts = (uint32_t*)c->counts;
        A.err = c->sync + 28;
        A.wait = sb_wait_cycles(c);
        A.drain = std::max(A.wait, SB_WAIT_DEFAULT_US * (long long)c->clock_khz / 1000);
        void* args[] = {&A};
        SbProf prof(c, SB_PROF_SCORE);
        SB_CHECK_CUDA(c, cudaLaunchKernel(fn, dim3((unsigned)blocks), dim3(SC_THREADS), args, smem, c->stream));
        return sb_after_launch(c, "k_score");
    }
    return SB_OK;
}

// counts of the current batch, checked: waits for the launches and reports a
// sampler or a tile copy that gave up (no cloud takes such a batch)
sb_status sb_score_batch(sb_ctx* c)
{
    if (c->counts_valid && c->batch_checked) return SB_OK;
    if (!c->counts_valid) SB_TRY(sb_score_enqueue(c));
    SB_TRY(sb_check_batch(c, c->m > 0));
    c->counts_valid = c->batch_checked = true;
    return SB_OK;
}
