// sb_graphl.cu -- graphL (Sec. 4, Alg. 2): relaxed loss (Eq. 3), discrete
// loss (Eq. 2), the adjoint dL/dG_v = -1/2 sum_j e_vj G_j (Eq. 4), the descent
// update G <- G - alpha dL/dG, and the final rounding (Algorithm 2).
//
// Layout: G is n x R float32, row-major (the R starting points of one vertex
// are contiguous), so a neighbour gather reads a contiguous row segment.
// Determinism: the adjoint sums each CSR row in a fixed order (blocks of 32
// neighbours, then across blocks; rows longer than SB_GL_CHUNK are cut into
// chunks whose partial sums are added in chunk order by a second kernel).
// Integer counts and column maxima use order-free atomics; float sums never do.
#include <algorithm>

#include "sb_count.cuh"
#include "sb_internal.cuh"

#define GL_THREADS 256
// Blocks per SM the row kernel's registers must allow, and neighbour rows loaded
// before they are added.  Descent step on the 2^20 R-MAT graph, 256 columns:
// 3.12 / 2.92 / 2.94 ms at 4 / 5 / 6 blocks and 4 rows, 2.98 at 8 blocks and 2
// rows, 3.66 / 3.64 at 3 / 4 blocks and 8 rows.  The 5 blocks leave 48 registers,
// at which the step kernels spill 200 to 260 bytes per thread and the gradient's
// 50 to 90 (the four-piece strided step 100 to 170 at 64 registers); that costs
// less than the warps that more registers would take.
#define GL_ROWS_MIN_BLOCKS 5
#define GL_INFLIGHT 4

struct GlArgs {
    const sb_bfs_item* items;   // chunks of split rows first, then whole rows
    int64_t n_items;
    int64_t n_split_items;      // items [0, n_split_items) are chunks of split rows
    const int32_t* rowptr;
    const int32_t* col;
    const int32_t* hub_first;
    const float* gin;      // n x R input
    float* gout_rows;      // n x R output
    float* partial;        // partial sums of split rows
    const float* upstream; // GRAD: gout[G x R] (G = 1 for one graph)
    const float* scale;    // STEP: input scale per (graph, column), a power of two
    float half_alpha;      // STEP: alpha / 2
    uint32_t* signs;       // STEP: sign words of the output (see sign_col), nullable
    int sign_words;        // 32-bit sign words per vertex (even)
    bool vec_out;          // output (and upstream) rows are 16-byte aligned
    uint32_t* colmax;      // STEP: max |G_out| bits per (graph, column)
    const int32_t* vgid;   // graph of each vertex in a batch, or null (one graph)
    int64_t n;
    int R;
};

__device__ __forceinline__ float flip_sign(float x, uint32_t negbit) { return __uint_as_float(__float_as_uint(x) ^ negbit); }
// theta = -1 exactly when G < 0 (so -0.0 rounds to +1, as G >= 0 does)
__device__ __forceinline__ uint32_t is_neg(float x) { return __float_as_uint(x) > 0x80000000u ? 1u : 0u; }

// Sign words: bit of column r of G in word r / 32 of a vertex's sign words, 1
// for theta = -1.  When R is a multiple of 4 a lane of the row kernel holds
// four adjacent columns, so the word's bits are ordered by (r % 4, r / 4 % 8):
// byte k holds the lanes' k-th columns, one ballot each.  (Bits of columns past R
// are 0; a count over edges of such a bit means nothing.)
// column (of 32) at bit j
__device__ __forceinline__ int sign_col(int j, bool quad) { return quad ? 4 * (j & 7) + (j >> 3) : j; }
// adds a count of bit j of the 32-column block `blk` to its column
__device__ __forceinline__ void add_count(int32_t* F, int R, int blk, int j, uint32_t x)
{
    const int r = 32 * blk + sign_col(j, R % 4 == 0);
    if (x && r < R) atomicAdd(F + r, (int32_t)x);
}
// sign word of a warp whose lane c holds column c of 32
__device__ __forceinline__ uint32_t sign_word(bool neg, bool quad)
{
    const unsigned lane = threadIdx.x & 31u;
    return __ballot_sync(0xffffffffu, __shfl_sync(0xffffffffu, (int)neg, sign_col((int)lane, quad)));
}

// acc += s * x for two columns at once (s = +-1, so the product is exact and
// each sum is the rounded sum of the signed value)
__device__ __forceinline__ void add_signed2(uint64_t& acc, uint64_t x, uint64_t s)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(s), "l"(x));
}
__device__ __forceinline__ uint64_t pack2(float a, float b)
{
    return ((uint64_t)__float_as_uint(b) << 32) | __float_as_uint(a);
}
__device__ __forceinline__ float lo2(uint64_t x) { return __uint_as_float((uint32_t)x); }
__device__ __forceinline__ float hi2(uint64_t x) { return __uint_as_float((uint32_t)(x >> 32)); }

// Per-lane running column max of one graph; flushed into the block's shared
// accumulators (one graph) or into the per-(graph, column) global accumulators
// (a batch) when the graph changes.
template <int VEC>
struct GlCols {
    int64_t g = -1;
    uint32_t mx[VEC];
    __device__ __forceinline__ void reset(int64_t gg)
    {
        g = gg;
#pragma unroll
        for (int k = 0; k < VEC; k++) mx[k] = 0;
    }
    // columns r0, r0 + stride, ..
    __device__ __forceinline__ void flush(const GlArgs& A, int r0, int stride, uint32_t* smax)
    {
        if (g < 0) return;
#pragma unroll
        for (int k = 0; k < VEC; k++) {
            const int r = r0 + k * stride;
            if (r < A.R && mx[k]) atomicMax(A.vgid ? A.colmax + g * A.R + r : smax + r, mx[k]);
        }
    }
};

// epilogue shared by whole rows and by combined split rows; returns the output
template <bool STEP>
__device__ __forceinline__ float gl_value(const GlArgs& A, float x, float scale_or_up, float acc)
{
    if (!STEP) return -0.5f * scale_or_up * acc;
    const float sc = scale_or_up;
    const float xs = x * sc;
    return xs + A.half_alpha * (acc * sc);
}

// Rows (and chunks of split rows): a sub-warp of SL lanes per (item, segment
// of SL*VEC columns).  The segments run one after the other over the whole
// grid, so one segment's columns of G (n x SL*VEC floats; 84 MB for 656k
// vertices at 32 columns) stay in L2 while every row gathers from them.
// Within a segment the sub-warps take blocks of IB consecutive items in turn:
// the chunks of one long row spread over many sub-warps, and a block (rows in
// vertex order) rarely crosses a graph of a batch.  A graph too small for
// every sub-warp to get GL_ROWS_PER_SUB rows takes them one at a time: with
// blocks of 16, 1000 rows kept 63 of 4864 warps busy, each with 16 rows in
// turn (33.7 us a descent step at 5 columns, now 6.4).  Batches of graphs take
// blocks earlier, and a step over a batch always: a sub-warp's column maxima go
// to its graph's accumulators whenever the graph changes, and rows one at a time
// change it at every row (256 graphs of 3000 vertices, 32 columns: 627 us a step,
// 155 in blocks).  Gradient over 4096 graphs of 50 vertices, one by one against
// blocks: 39 / 45 us at 8 rows per sub-warp (32 columns), 72 / 58 at 16 (64),
// 193 / 138 at 32 (256).
#define GL_ITEM_BLOCK 16
#define GL_ROWS_PER_SUB 32
#define GL_ROWS_PER_SUB_BATCH 12
//
// What bounds it: the gathers.  Long-scoreboard stalls led at half the warps
// resident, so a lane keeps GL_INFLIGHT neighbour rows in flight (the last,
// partial group too: most rows are short), adds two columns per instruction
// (fma.rn.f32x2 by the edge's sign instead of a sign flip and an add per
// column), and leaves the discrete loss, which took five integer operations
// per element here, to k_gl_count: this kernel only writes the sign words of
// its output.  More rows in flight than that is slower (6 or 8 in registers,
// or 16 per warp through a cp.async ring in shared memory: 3.4-4.0 ms against
// 2.93 for the step below): 11.6 TB/s of gathered rows out of L2, a third of
// them from DRAM, is what the memory system gives.  Rows that are not 16-byte
// aligned (R not a multiple of 4) are taken in 32-column pieces, up to four
// per lane (STRIDED): 25 traced steps at 37 columns 53.9 -> 34.0 ms.  Traced
// step on the 2^20 R-MAT graph, 256 columns: 4.58 -> 2.98 ms (and 0.12 for
// k_gl_count); 64 columns without a trace: 1.47 -> 0.89 ms.
template <int VEC, int SL, bool STRIDED, bool STEP, int IB>
__global__ void __launch_bounds__(GL_THREADS, STRIDED && VEC > 1 ? 4 : GL_ROWS_MIN_BLOCKS) k_gl_rows(GlArgs A)
{
    extern __shared__ uint32_t smax[];  // R (STEP)
    const int R = A.R;
    if (STEP) {
        for (int i = threadIdx.x; i < R; i += GL_THREADS) smax[i] = 0;
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const int sl = lane & (SL - 1);
    const unsigned smask = SL == 32 ? 0xffffffffu : (((1u << SL) - 1u) << (lane & ~(SL - 1)));
    const int64_t subs_total = (int64_t)gridDim.x * (GL_THREADS / SL);
    const int64_t sub_id = (int64_t)blockIdx.x * (GL_THREADS / SL) + threadIdx.x / SL;
    constexpr int seg_w = SL * VEC;
    const int nseg = (R + seg_w - 1) / seg_w;
    // split-row chunks one at a time, then whole rows by blocks: work unit w
    // covers items [lo(w), hi(w))
    const int64_t nsplit = A.n_split_items;
    const int64_t nunits = nsplit + sb_cdiv(A.n_items - nsplit, IB);
    for (int seg = 0; seg < nseg; seg++) {
        // a lane's columns: VEC adjacent ones, or every 32nd from r0 on
        constexpr int CS = STRIDED ? 32 : 1;
        const int r0 = STRIDED ? seg * seg_w + sl : seg * seg_w + sl * VEC;
        const bool act = r0 < R;
        GlCols<VEC> cols;
        for (int64_t wu = sub_id; wu < nunits; wu += subs_total)
        for (int64_t it = wu < nsplit ? wu : nsplit + (wu - nsplit) * IB,
                     it_end = wu < nsplit ? wu + 1 : min(A.n_items, nsplit + (wu - nsplit + 1) * IB);
             it < it_end; it++) {
            const int4 q = __ldg((const int4*)(A.items + it));  // vertex, CSR range, split row or -1
            const int64_t v = q.x;
            const int64_t g = A.vgid ? A.vgid[v] : 0;
            if (STEP && g != cols.g) {
                if (act) cols.flush(A, r0, CS, smax);
                cols.reset(g);
            }
            float acc[VEC];
#pragma unroll
            for (int k = 0; k < VEC; k++) acc[k] = 0.f;
            // blocks of 32 neighbours (fixed order), SL column ids loaded at a time
            for (int j0 = q.y; j0 < q.z; j0 += 32) {
                const int cnt = min(32, q.z - j0);
                uint64_t b01 = 0, b23 = 0;
                float bs[STRIDED ? VEC : 1];
#pragma unroll
                for (int k = 0; k < (STRIDED ? VEC : 1); k++) bs[k] = 0.f;
                for (int jj = 0; jj < cnt; jj += SL) {
                    const int cc_n = min(SL, cnt - jj);
                    const uint32_t mycol = sl < cc_n ? (uint32_t)__ldg(A.col + j0 + jj + sl) : 0u;
                    for (int q0 = 0; q0 < cc_n; q0 += GL_INFLIGHT) {
                        uint32_t cc[GL_INFLIGHT];
#pragma unroll
                        for (int i = 0; i < GL_INFLIGHT; i++) cc[i] = __shfl_sync(smask, mycol, (q0 + i) & (SL - 1), SL);
                        if constexpr (!STRIDED) {
                            ulonglong2 x[GL_INFLIGHT];
#pragma unroll
                            for (int i = 0; i < GL_INFLIGHT; i++)
                                if (act && q0 + i < cc_n)
                                    x[i] = __ldg((const ulonglong2*)(A.gin + (int64_t)(cc[i] & SB_ID_MASK) * R + r0));
#pragma unroll
                            for (int i = 0; i < GL_INFLIGHT; i++)
                                if (act && q0 + i < cc_n) {
                                    const uint32_t sg = 0x3F800000u | (cc[i] & 0x80000000u);
                                    const uint64_t ss = ((uint64_t)sg << 32) | sg;
                                    add_signed2(b01, x[i].x, ss);
                                    add_signed2(b23, x[i].y, ss);
                                }
                        } else {
                            float x[GL_INFLIGHT][VEC];
#pragma unroll
                            for (int i = 0; i < GL_INFLIGHT; i++) {
                                const float* p = A.gin + (int64_t)(cc[i] & SB_ID_MASK) * R + r0;
#pragma unroll
                                for (int k = 0; k < VEC; k++)
                                    if (r0 + CS * k < R && q0 + i < cc_n) x[i][k] = __ldg(p + CS * k);
                            }
#pragma unroll
                            for (int i = 0; i < GL_INFLIGHT; i++)
#pragma unroll
                                for (int k = 0; k < VEC; k++)
                                    if (r0 + CS * k < R && q0 + i < cc_n)
                                        bs[STRIDED ? k : 0] += flip_sign(x[i][k], cc[i] & 0x80000000u);
                        }
                    }
                }
                if constexpr (!STRIDED) {
                    acc[0] += lo2(b01);
                    acc[1 % VEC] += hi2(b01);
                    acc[2 % VEC] += lo2(b23);
                    acc[3 % VEC] += hi2(b23);
                } else {
#pragma unroll
                    for (int k = 0; k < VEC; k++) acc[k] += bs[STRIDED ? k : 0];
                }
            }
            if (q.w >= 0) {
                const int64_t slot = A.hub_first[q.w] + (q.y - A.rowptr[v]) / SB_GL_CHUNK;
                if (act) {
                    if constexpr (!STRIDED)
                        *(float4*)(A.partial + slot * R + r0) = make_float4(acc[0], acc[1 % VEC], acc[2 % VEC], acc[3 % VEC]);
                    else
#pragma unroll
                        for (int k = 0; k < VEC; k++)
                            if (r0 + CS * k < R) A.partial[slot * R + r0 + CS * k] = acc[k];
                }
                continue;
            }
            float out[VEC];
            if (act) {
                const float* pin = A.gin + v * R + r0;
                const float* pup = (STEP ? A.scale : A.upstream) + g * R + r0;
                if (!STRIDED && A.vec_out) {
                    const float4 up = *(const float4*)pup;
                    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (STEP) x = __ldg((const float4*)pin);
                    const float xv[4] = {x.x, x.y, x.z, x.w}, uv[4] = {up.x, up.y, up.z, up.w};
#pragma unroll
                    for (int k = 0; k < VEC; k++) out[k] = gl_value<STEP>(A, xv[k], uv[k], acc[k]);
                    *(float4*)(A.gout_rows + v * R + r0) =
                        make_float4(out[0], out[1 % VEC], out[2 % VEC], out[3 % VEC]);
                } else {
#pragma unroll
                    for (int k = 0; k < VEC; k++) {
                        out[k] = 0.f;
                        if (r0 + CS * k >= R) continue;
                        out[k] = gl_value<STEP>(A, STEP ? __ldg(pin + CS * k) : 0.f, pup[CS * k], acc[k]);
                        A.gout_rows[v * R + r0 + CS * k] = out[k];
                    }
                }
                if (STEP) {
#pragma unroll
                    for (int k = 0; k < VEC; k++) cols.mx[k] = max(cols.mx[k], __float_as_uint(fabsf(out[k])));
                }
            }
            if (STEP && A.signs) {
                if constexpr (!STRIDED) {
                    uint32_t w = 0;  // sign word of this lane's 8-lane group
#pragma unroll
                    for (int k = 0; k < 4; k++)
                        w |= ((__ballot_sync(smask, act && is_neg(out[k % VEC])) >> (lane & ~7)) & 255u) << (8 * k);
                    if (act && (sl & 7) == 0) A.signs[v * A.sign_words + r0 / 32] = w;
                } else {
#pragma unroll
                    for (int k = 0; k < VEC; k++) {
                        const uint32_t w = sign_word(r0 + 32 * k < R && is_neg(out[k]), R % 4 == 0);
                        if (lane == 0 && r0 + 32 * k < R) A.signs[v * A.sign_words + r0 / 32 + k] = w;
                    }
                }
            }
        }
        if (STEP && act) cols.flush(A, r0, CS, smax);
    }
    if (STEP) {
        __syncthreads();
        if (!A.vgid)
            for (int i = threadIdx.x; i < R; i += GL_THREADS)
                if (smax[i]) atomicMax(A.colmax + i, smax[i]);
    }
}

// Split rows: add chunk partials in chunk order, then the same epilogue.  A
// warp takes 32 columns of one row; eight partials are loaded before they are
// added in order (the longest rows have hundreds).
template <bool STEP>
__global__ void __launch_bounds__(GL_THREADS) k_gl_combine(GlArgs A, const int32_t* __restrict__ hub_vertex,
                                                           const int32_t* __restrict__ hub_count, int64_t n_hubs)
{
    const int R = A.R, lane = threadIdx.x & 31;
    const int nb = (R + 31) / 32;
    const int64_t warps = (int64_t)gridDim.x * (GL_THREADS / 32);
    for (int64_t x = ((int64_t)blockIdx.x * GL_THREADS + threadIdx.x) >> 5; x < n_hubs * nb; x += warps) {
        const int64_t h = x / nb;
        const int blk = (int)(x - h * nb), r = 32 * blk + lane;
        const bool act = r < R;
        const float* part = A.partial + (int64_t)A.hub_first[h] * R + r;
        const int cnt = act ? hub_count[h] : 0;
        float acc = 0.f;
        int k = 0;
        for (; k + 8 <= cnt; k += 8) {
            float p[8];
#pragma unroll
            for (int i = 0; i < 8; i++) p[i] = part[(int64_t)(k + i) * R];
#pragma unroll
            for (int i = 0; i < 8; i++) acc += p[i];
        }
        for (; k < cnt; k++) acc += part[(int64_t)k * R];
        const int64_t v = hub_vertex[h];
        const int64_t g = A.vgid ? A.vgid[v] : 0;
        float out = 0.f;
        if (act) {
            const int64_t idx = v * R + r;
            out = gl_value<STEP>(A, STEP ? A.gin[idx] : 0.f, STEP ? A.scale[g * R + r] : A.upstream[g * R + r], acc);
            A.gout_rows[idx] = out;
            if (STEP) {
                const uint32_t b = __float_as_uint(fabsf(out));
                uint32_t* m = A.colmax + g * R + r;
                if (b > __ldcg(m)) atomicMax(m, b);
            }
        }
        if (STEP && A.signs) {
            const uint32_t w = sign_word(act && is_neg(out), R % 4 == 0);
            if (lane == 0) A.signs[v * A.sign_words + blk] = w;
        }
    }
}

// Sign words of a whole matrix: a warp takes 32 columns of one vertex at a time,
// eight such words loaded together (one by one: 44 us at n = 100,000 and 130
// columns, 24 so).  Clears `clear` for the counts that follow.
__global__ void __launch_bounds__(GL_THREADS) k_gl_signs(const float* __restrict__ g, int64_t n, int R,
                                                         uint32_t* __restrict__ signs, int sign_words,
                                                         int32_t* __restrict__ clear, int64_t nclear)
{
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (GL_THREADS / 32);
    const int64_t t0 = (int64_t)blockIdx.x * GL_THREADS + threadIdx.x;
    for (int64_t i = t0; i < nclear; i += 32 * warps) clear[i] = 0;
    for (int64_t x = (t0 >> 5) * 8; x < n * sign_words; x += 8 * warps) {
        int64_t v = x / sign_words;
        int blk = (int)(x - v * sign_words);
        float y[8];
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int r = 32 * blk + lane;
            y[i] = 0.f;
            if (v < n && r < R) y[i] = g[v * R + r];
            if (++blk == sign_words) {
                blk = 0;
                v++;
            }
        }
        uint32_t mine = 0;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const uint32_t w = sign_word(is_neg(y[i]), R % 4 == 0);
            if (lane == i) mine = w;
        }
        if (lane < 8 && x + lane < n * sign_words) signs[x + lane] = mine;
    }
}

// Frustrated edges per column of one graph from the sign words (vertical
// counters, as in the scorer): a group of G lanes takes an edge, lane = 64
// columns, a warp a contiguous range of the edges.  Latency bounds it: 490 us per
// pass (16.8 M edges, 256 columns) with a check before every load, 264 without,
// 115 with the next batch's edges loaded ahead and the counters flushed by
// transposes.
template <int G>
__global__ void __launch_bounds__(GL_THREADS) k_gl_count(const int2* __restrict__ edges, int64_t m,
                                                         const uint64_t* __restrict__ signs, int W, int R,
                                                         int32_t* __restrict__ F)
{
    __shared__ uint32_t scnt[64 * G];
    const int lane = threadIdx.x & 31, gl = lane & (G - 1), grp = lane / G;
    const int word = blockIdx.y * 32 + gl;
    const bool act = word < W;
    constexpr int NG = 32 / G;
    for (int i = threadIdx.x; i < 64 * G; i += GL_THREADS) scnt[i] = 0;
    __syncthreads();
    const int64_t warps = (int64_t)gridDim.x * (GL_THREADS / 32);
    const int64_t per = sb_cdiv(sb_cdiv(m, 8 * NG), warps) * (8 * NG);
    const int64_t wid = (int64_t)blockIdx.x * (GL_THREADS / 32) + (threadIdx.x >> 5);
    const int64_t e1 = min(m, (wid + 1) * per);
    ScoreAcc acc;
    acc.reset();
    int2 nx[8];
    auto load = [&](int64_t e) {
#pragma unroll
        for (int k = 0; k < 8; k++) {
            nx[k] = make_int2(0, 0);
            if (e + k * NG < e1) nx[k] = __ldg(edges + e + k * NG);
        }
    };
    if (act) load(wid * per + grp);
    if (act)
        for (int64_t e = wid * per + grp; e < e1; e += 8 * NG) {
            uint64_t x[8];
            int2 ed[8];
            // the next batch's edges are loaded while this one is counted; no
            // branches between the loads of a batch, so that all are in flight
#pragma unroll
            for (int k = 0; k < 8; k++) ed[k] = nx[k];
            load(e + 8 * NG);
#pragma unroll
            for (int k = 0; k < 8; k++)
                x[k] = signs[(int64_t)ed[k].x * W + word] ^ signs[(int64_t)((uint32_t)ed[k].y & SB_ID_MASK) * W + word] ^
                       (uint64_t)(int64_t)(ed[k].y >> 31);  // 0 past the end: an edge (0, 0)
            acc.add8(x);
            if (acc.nb == SC_FLUSH) acc.flush(scnt + 64 * gl);
        }
    acc.template flush_warp<G>(scnt);
    __syncthreads();
    for (int i = threadIdx.x; i < 64 * G; i += GL_THREADS) add_count(F, R, blockIdx.y * 64 + i / 32, i & 31, scnt[i]);
}

// The same for a batch: F[graph * R + column].  A warp takes a contiguous range of
// the edges (graph after graph) and 64 columns (blockIdx.y), a lane an edge.  256
// edges of one graph go into vertical counters; where graphs change, 32 edges at a
// time are transposed and each graph's share is counted under its lanes' mask, so
// that a graph costs its own edges and one flush.  With vertical counters alone
// every lane flushed 64 counters whenever it met another graph (20,000 graphs of
// 9 edges, 5 columns: 166 us a pass, 6 here).
__global__ void __launch_bounds__(GL_THREADS) k_gl_count_graphs(const int2* __restrict__ edges, int64_t m,
                                                                const int32_t* __restrict__ vgid,
                                                                const uint64_t* __restrict__ signs, int W, int R,
                                                                int32_t* __restrict__ F)
{
    const int lane = threadIdx.x & 31, word = blockIdx.y;
    const int64_t warps = (int64_t)gridDim.x * (GL_THREADS / 32);
    const int64_t per = sb_cdiv(m, 32 * warps) * 32;
    const int64_t wid = (int64_t)blockIdx.x * (GL_THREADS / 32) + (threadIdx.x >> 5);
    const int64_t e1 = min(m, (wid + 1) * per);
    ScoreAcc acc;
    acc.reset();
    int64_t gcur = -1;
    uint32_t lo = 0, hi = 0;  // of graph gcur, this lane's columns
    auto sum = [&]() {
        if (!acc.nb) return;
        uint32_t l, h;
        acc.template sum_warp<1>(&l, &h);
        lo += l;
        hi += h;
        acc.reset();
    };
    auto turn = [&](int64_t g) {  // to graph g
        if (g == gcur) return;
        if (gcur >= 0) {
            sum();
            add_count(F + gcur * R, R, 2 * word, lane, lo);
            add_count(F + gcur * R, R, 2 * word + 1, lane, hi);
        }
        gcur = g;
        lo = hi = 0;
    };
    for (int64_t e = wid * per; e < e1; e += 256) {
        int2 ed[8];
        int32_t gk[8];
        uint64_t x[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            ed[k] = make_int2(-1, 0);
            if (e + 32 * k + lane < e1) ed[k] = __ldg(edges + e + 32 * k + lane);
        }
#pragma unroll
        for (int k = 0; k < 8; k++) {
            gk[k] = -1;
            x[k] = 0;
            if (ed[k].x >= 0) {
                gk[k] = vgid[ed[k].x];
                x[k] = signs[(int64_t)ed[k].x * W + word] ^ signs[(int64_t)((uint32_t)ed[k].y & SB_ID_MASK) * W + word] ^
                       (uint64_t)(int64_t)(ed[k].y >> 31);
            }
        }
        const int32_t g0 = __shfl_sync(0xffffffffu, gk[0], 0);
        if (g0 == __shfl_sync(0xffffffffu, gk[7], 31)) {  // 256 edges of one graph
            turn(g0);
            acc.add8(x);
            if (acc.nb == SC_FLUSH) sum();
            continue;
        }
#pragma unroll
        for (int k = 0; k < 8; k++) {
            uint32_t rem = __ballot_sync(0xffffffffu, gk[k] >= 0);
            if (!rem) break;
            const uint32_t a = warp_transpose32((uint32_t)x[k], lane), b = warp_transpose32((uint32_t)(x[k] >> 32), lane);
            while (rem) {
                const int32_t g = __shfl_sync(0xffffffffu, gk[k], __ffs((int)rem) - 1);
                const uint32_t mask = __ballot_sync(0xffffffffu, gk[k] == g);
                turn(g);
                lo += (uint32_t)__popc(a & mask);
                hi += (uint32_t)__popc(b & mask);
                rem &= ~mask;
            }
        }
    }
    turn(-1);
}

// Alg. 2 rounding: bit per edge and column, from the sign words: a warp takes
// 4 words of 64 edges and 32 columns, lane = edge, and two 32 x 32 bit
// transposes per word give lane j the edges of the column at bit j.  For one
// graph it also counts them into F (nullable): a warp keeps its columns, since
// the launch's warps are a multiple of the column blocks.
__global__ void __launch_bounds__(GL_THREADS) k_gl_flips(const int2* __restrict__ edges, int64_t m,
                                                         const uint32_t* __restrict__ signs, int sign_words, int R,
                                                         uint64_t* __restrict__ flips, int32_t* __restrict__ F)
{
    const int lane = threadIdx.x & 31, nb = (R + 31) / 32;
    const int64_t nw = sb_cdiv(m, 64), nq = sb_cdiv(nw, 4);
    const int64_t rows = (int64_t)gridDim.x * (GL_THREADS / 32) / nb;
    const int64_t wid = ((int64_t)blockIdx.x * GL_THREADS + threadIdx.x) >> 5;
    const int blk = (int)(wid % nb);
    const int r = 32 * blk + sign_col(lane, R % 4 == 0);
    uint32_t count = 0;
    for (int64_t wq = wid / nb; wq < nq; wq += rows) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int64_t w = 4 * wq + i;
            if (w >= nw) break;
            uint32_t half[2];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int64_t e = 64 * w + 32 * h + lane;
                uint32_t f = 0;
                if (e < m) {
                    const int2 ed = __ldg(edges + e);
                    f = signs[(int64_t)ed.x * sign_words + blk] ^
                        signs[(int64_t)((uint32_t)ed.y & SB_ID_MASK) * sign_words + blk] ^ (uint32_t)(ed.y >> 31);
                }
                half[h] = warp_transpose32(f, lane);
                count += (uint32_t)__popc(half[h]);
            }
            if (r < R) flips[(int64_t)r * nw + w] = ((uint64_t)half[1] << 32) | half[0];
        }
    }
    if (F && r < R && count) atomicAdd(F + r, (int32_t)count);
}

// per-(graph, column) renorm decision after one step
__global__ void k_gl_step_final(int64_t GR, uint32_t* colmax, float* scale, int32_t* exps, int renorm_log2)
{
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < GR; r += (int64_t)gridDim.x * blockDim.x) {
        const float mx = __uint_as_float(colmax[r]);
        colmax[r] = 0;
        float sc = 1.0f;
        if (renorm_log2 > 0 && mx >= ldexpf(1.0f, renorm_log2)) {
            sc = ldexpf(1.0f, -renorm_log2);
            exps[r] += renorm_log2;
        }
        scale[r] = sc;
    }
}

__global__ void k_gl_fill(float* p, int64_t n, float v)
{
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) p[r] = v;
}

// Pending power-of-two scale of the last step, and the sign words (nullable)
// of what it changes (a scaled value can underflow to zero): a warp takes 32
// columns of four vertices at a time, and columns without a pending scale cost
// one read of the scale.
__global__ void __launch_bounds__(GL_THREADS) k_gl_apply_scale(float* g, int64_t n, int R, const float* scale,
                                                               const int32_t* vgid, uint32_t* signs, int sign_words)
{
    const int lane = threadIdx.x & 31, nb = (R + 31) / 32;
    const int64_t warps = (int64_t)gridDim.x * (GL_THREADS / 32), quads = sb_cdiv(n, 4);
    for (int64_t x = ((int64_t)blockIdx.x * GL_THREADS + threadIdx.x) >> 5; x < quads * nb; x += warps) {
        const int64_t q = x / nb;
        const int blk = (int)(x - q * nb), r = 32 * blk + lane;
        float sc[4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int64_t v = 4 * q + i;
            sc[i] = 1.0f;
            if (r < R && v < n) sc[i] = scale[(vgid ? (int64_t)vgid[v] : 0) * R + r];
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int64_t v = 4 * q + i;
            if (!__any_sync(0xffffffffu, sc[i] != 1.0f)) continue;
            float y = 0.f;
            if (r < R) {
                y = g[v * R + r] * sc[i];
                g[v * R + r] = y;
            }
            if (signs) {
                const uint32_t w = sign_word(r < R && is_neg(y), R % 4 == 0);
                if (lane == 0) signs[v * sign_words + blk] = w;
            }
        }
    }
}

// Edge-parallel forward: per column the compensated sum of e_uv G_u G_v, and
// the count of frustrated edges under theta = sign(G) (>= 0 -> +1).  A block
// takes a contiguous edge range and its sub-warps of SL lanes (VEC columns
// each) a contiguous part of it, so that the row of the edge's first endpoint
// (the edges are sorted by it) comes from L1; GL_FWD_INFLIGHT edges are loaded
// before they are added in order.  Sums per block, in sub-warp order, then over
// the blocks in a fixed order.  One column per thread and one edge at a time
// kept 64 of 256 threads busy at R = 64 and waited for every gather: 3.88 ms on
// the 2^20 R-MAT graph, now 0.94 (4.3 GB of rows gathered beside those from L1).
#define GL_FWD_INFLIGHT 4
template <int VEC, int SL>
__global__ void __launch_bounds__(GL_THREADS, 3) k_gl_fwd(const int2* __restrict__ edges, int64_t m,
                                                          const float* __restrict__ g, int R,
                                                          double* __restrict__ red, int32_t* __restrict__ Facc)
{
    constexpr int SUBS = GL_THREADS / SL, SEG = SL * VEC;
    __shared__ double ssum[SUBS][SEG];
    __shared__ int32_t sf[SUBS][SEG];
    const int lane = threadIdx.x & 31, sl = lane & (SL - 1), sub = threadIdx.x / SL;
    const unsigned smask = SL == 32 ? 0xffffffffu : (((1u << SL) - 1u) << (lane & ~(SL - 1)));
    const int64_t per = sb_cdiv(m, (int64_t)gridDim.x), spr = sb_cdiv(per, SUBS);
    const int64_t b0 = (int64_t)blockIdx.x * per, b1 = min(m, b0 + per);
    const int64_t e0 = min(b1, b0 + sub * spr), e1 = min(b1, e0 + spr);
    for (int r00 = 0; r00 < R; r00 += SEG) {
        const int r0 = r00 + sl * VEC;
        const bool act = r0 < R;
        float s[VEC], comp[VEC];
        int32_t f[VEC];
#pragma unroll
        for (int k = 0; k < VEC; k++) {
            s[k] = comp[k] = 0.f;
            f[k] = 0;
        }
        for (int64_t e = e0; e < e1; e += SL) {
            const int cnt = (int)min((int64_t)SL, e1 - e);
            const int2 my = sl < cnt ? __ldg(edges + e + sl) : make_int2(0, 0);
            for (int q0 = 0; q0 < cnt; q0 += GL_FWD_INFLIGHT) {
                float a[GL_FWD_INFLIGHT][VEC], b[GL_FWD_INFLIGHT][VEC];
                uint32_t nb[GL_FWD_INFLIGHT];
#pragma unroll
                for (int i = 0; i < GL_FWD_INFLIGHT; i++) {
                    const uint32_t u = (uint32_t)__shfl_sync(smask, my.x, (q0 + i) & (SL - 1), SL);
                    const uint32_t y = (uint32_t)__shfl_sync(smask, my.y, (q0 + i) & (SL - 1), SL);
                    nb[i] = y & 0x80000000u;
                    if (act && q0 + i < cnt) {
                        const float* pa = g + (int64_t)u * R + r0;
                        const float* pb = g + (int64_t)(y & SB_ID_MASK) * R + r0;
                        if constexpr (VEC == 4) {
                            const float4 xa = __ldg((const float4*)pa), xb = __ldg((const float4*)pb);
                            a[i][0] = xa.x, a[i][1 % VEC] = xa.y, a[i][2 % VEC] = xa.z, a[i][3 % VEC] = xa.w;
                            b[i][0] = xb.x, b[i][1 % VEC] = xb.y, b[i][2 % VEC] = xb.z, b[i][3 % VEC] = xb.w;
                        } else {
                            a[i][0] = __ldg(pa);
                            b[i][0] = __ldg(pb);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < GL_FWD_INFLIGHT; i++)
                    if (act && q0 + i < cnt) {
#pragma unroll
                        for (int k = 0; k < VEC; k++) {
                            const float p = flip_sign(__fmul_rn(a[i][k], b[i][k]), nb[i]);
                            // s + p and its exact rounding error (Knuth's two-sum)
                            const float t = __fadd_rn(s[k], p);
                            const float z = __fsub_rn(t, s[k]);
                            comp[k] = __fadd_rn(comp[k], __fadd_rn(__fsub_rn(s[k], __fsub_rn(t, z)), __fsub_rn(p, z)));
                            s[k] = t;
                            f[k] += (int32_t)(is_neg(a[i][k]) ^ is_neg(b[i][k]) ^ (nb[i] >> 31));
                        }
                    }
            }
        }
#pragma unroll
        for (int k = 0; k < VEC; k++) {
            ssum[sub][sl * VEC + k] = (double)s[k] + (double)comp[k];
            sf[sub][sl * VEC + k] = f[k];
        }
        __syncthreads();
        for (int c = threadIdx.x; c < SEG && r00 + c < R; c += GL_THREADS) {
            double t = 0.0;
            int32_t ft = 0;
            for (int i = 0; i < SUBS; i++) {
                t += ssum[i][c];
                ft += sf[i][c];
            }
            red[(int64_t)blockIdx.x * R + r00 + c] = t;
            if (ft) atomicAdd(Facc + r00 + c, ft);
        }
        __syncthreads();
    }
}

// one warp per column
__global__ void __launch_bounds__(GL_THREADS) k_gl_fwd_final(const double* __restrict__ red, int nblocks, int R,
                                                             int64_t m, float* loss, int32_t* Facc, int32_t* F_out)
{
    const int lane = threadIdx.x & 31;
    const int r = (int)(((int64_t)blockIdx.x * GL_THREADS + threadIdx.x) >> 5);
    if (r >= R) return;
    double s = 0.0;
    for (int b = lane; b < nblocks; b += 32) s += red[(int64_t)b * R + r];
    for (int d = 16; d; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if (lane == 0) {
        loss[r] = (float)(0.5 * (double)m - 0.5 * s);
        if (F_out) F_out[r] = Facc[r];
    }
}

// Relaxed and discrete loss of every graph of a batch: one block per graph
// sums its own edges in order (Kahan-Babuska), so no cross-block reduction.
__global__ void __launch_bounds__(GL_THREADS) k_gl_fwd_graph(const int2* __restrict__ edges,
                                                             const int32_t* __restrict__ eoff,
                                                             const float* __restrict__ g, int R,
                                                             float* __restrict__ loss, int32_t* __restrict__ F)
{
    const int64_t gg = blockIdx.x;
    const int64_t e0 = eoff[gg], e1 = eoff[gg + 1];
    for (int r = threadIdx.x; r < R; r += GL_THREADS) {
        float s = 0.f, comp = 0.f;
        int32_t f = 0;
        for (int64_t e = e0; e < e1; e++) {
            const int2 ed = edges[e];
            const uint32_t nb = (uint32_t)ed.y & 0x80000000u;
            const float a = g[(int64_t)ed.x * R + r];
            const float b = g[(int64_t)((uint32_t)ed.y & SB_ID_MASK) * R + r];
            const float p = flip_sign(a * b, nb);
            const float t = s + p;
            comp += fabsf(s) >= fabsf(p) ? (s - t) + p : (p - t) + s;
            s = t;
            f += (int32_t)(is_neg(a) ^ is_neg(b) ^ (nb >> 31));
        }
        loss[gg * R + r] = (float)(0.5 * (double)(e1 - e0) - 0.5 * ((double)s + (double)comp));
        if (F) F[gg * R + r] = f;
    }
}

// ----------------------------------------------------------------- host
// sign words per vertex (32-bit, even)
static int gl_sign_words(int R) { return 2 * (int)sb_cdiv(R, 64); }

static sb_status gl_scratch(sb_ctx* c, int R)
{
    SB_TRY(sb_ensure(c, (void**)&c->gl_partial, &c->gl_partial_cap,
                     sizeof(float) * (size_t)std::max<int64_t>(c->n_gl_partials, 1) * R));
    SB_TRY(sb_ensure(c, (void**)&c->gl_red, &c->gl_red_cap, sizeof(double) * (size_t)c->num_sms * 8 * R));
    return sb_ensure(c, (void**)&c->gl_misc, &c->gl_misc_cap, sizeof(int32_t) * (size_t)R);
}

static sb_status gl_signs_scratch(sb_ctx* c, int R, int copies)
{
    return sb_ensure(c, (void**)&c->gl_signs, &c->gl_signs_cap,
                     sizeof(uint32_t) * (size_t)c->n * gl_sign_words(R) * copies);
}

// (clear: nclear counters set to zero, nullable)
static sb_status gl_signs_launch(sb_ctx* c, const float* gamma, int R, uint32_t* signs, int32_t* clear, int64_t nclear)
{
    const int sw = gl_sign_words(R);
    const unsigned blocks =
        (unsigned)std::min<int64_t>(sb_cdiv(c->n * sw, 8 * (GL_THREADS / 32)), (int64_t)c->num_sms * 8);
    k_gl_signs<<<blocks, GL_THREADS, 0, c->stream>>>(gamma, c->n, R, signs, sw, clear, nclear);
    return sb_after_launch(c, "k_gl_signs");
}

static const void* gl_count_kernel(int W)
{
    return W > 16  ? (const void*)k_gl_count<32>
           : W > 8 ? (const void*)k_gl_count<16>
           : W > 4 ? (const void*)k_gl_count<8>
           : W > 2 ? (const void*)k_gl_count<4>
           : W > 1 ? (const void*)k_gl_count<2>
                   : (const void*)k_gl_count<1>;
}

// adds the frustrated edges of every (graph, column) to F
static sb_status gl_count_launch(sb_ctx* c, const uint32_t* signs, int R, int32_t* F)
{
    if (c->m == 0) return SB_OK;
    int W = gl_sign_words(R) / 2;
    const int2* edges = c->sc_edges;  // first endpoints repeat over a run of edges, second ones are often hubs
    int64_t m = c->m;
    if (c->batch_G > 0) {  // (the scorer's edges lie graph after graph, as the sorted ones)
        // a warp takes at least 64 edges
        const unsigned bx = (unsigned)std::max<int64_t>(
            1, std::min<int64_t>(sb_cdiv(m, 64 * (GL_THREADS / 32)), sb_cdiv((int64_t)c->num_sms * 8, std::min(W, 8))));
        k_gl_count_graphs<<<dim3(bx, (unsigned)W), GL_THREADS, 0, c->stream>>>(edges, m, c->vgid, (const uint64_t*)signs, W, R, F);
        return sb_after_launch(c, "k_gl_count_graphs");
    }
    // a warp takes at least 4 batches of 8 edges per group
    const int64_t batches = sb_cdiv(m * std::min(W, 32), 8 * 32 * 4 * (GL_THREADS / 32));
    const unsigned bx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(batches, (int64_t)c->num_sms * 4));
    void* args[] = {(void*)&edges, &m, (void*)&signs, &W, &R, &F};
    SB_CHECK_CUDA(c, cudaLaunchKernel(gl_count_kernel(W), dim3(bx, (unsigned)sb_cdiv(W, 32)), dim3(GL_THREADS), args, 0, c->stream));
    return sb_after_launch(c, "k_gl_count");
}

static GlArgs gl_args(sb_ctx* c, int R)
{
    GlArgs A;
    memset(&A, 0, sizeof(A));
    A.items = c->gl_items;
    A.n_items = c->n_gl_items;
    A.n_split_items = c->n_gl_partials;
    A.rowptr = c->rowptr;
    A.col = c->col;
    A.hub_first = c->gl_hub_first;
    A.partial = c->gl_partial;
    A.n = c->n;
    A.R = R;
    A.vgid = c->batch_G > 0 ? c->vgid : nullptr;
    return A;
}

template <bool STEP, int IB>
static const void* gl_rows_kernel(bool vec4, int64_t lanes, int R)
{
    if (vec4)
        return lanes == 32   ? (const void*)k_gl_rows<4, 32, false, STEP, IB>
               : lanes == 16 ? (const void*)k_gl_rows<4, 16, false, STEP, IB>
                             : (const void*)k_gl_rows<4, 8, false, STEP, IB>;
    return R > 64   ? (const void*)k_gl_rows<4, 32, true, STEP, IB>
           : R > 32 ? (const void*)k_gl_rows<2, 32, true, STEP, IB>
                    : (const void*)k_gl_rows<1, 32, true, STEP, IB>;
}

// Lanes per row segment: the knob, or the width whose segments take least in
// all.  A segment costs 1.03 / 1.24 / 1.62 ms with 8 / 16 / 32 lanes (descent
// step on the 2^20 R-MAT graph), so a wide one pays as soon as it saves one.
static int64_t gl_lanes(const sb_ctx* c, int R)
{
    if (c->tune[SB_TUNE_GL_LANES] > 0) return c->tune[SB_TUNE_GL_LANES];
    const int64_t t8 = 103 * sb_cdiv(R, 32), t16 = 124 * sb_cdiv(R, 64), t32 = 162 * sb_cdiv(R, 128);
    return t32 < t16 && t32 < t8 ? 32 : t16 < t8 ? 16 : 8;
}

template <bool STEP>
static sb_status gl_rows_launch(sb_ctx* c, GlArgs& A)
{
    const bool vec4 = (A.R % 4 == 0) && (((uintptr_t)A.gin & 15) == 0);
    const int64_t lanes = gl_lanes(c, A.R);
    A.vec_out = (((uintptr_t)A.gout_rows | (uintptr_t)A.upstream) & 15) == 0;
    const int subs = GL_THREADS / (vec4 && lanes != 32 ? (lanes == 16 ? 16 : 8) : 32);
    const int64_t rows = A.n_items - A.n_split_items;
    const int64_t fill = (int64_t)c->num_sms * GL_ROWS_MIN_BLOCKS * subs;
    const bool small = !(STEP && A.vgid) && rows < fill * (A.vgid ? GL_ROWS_PER_SUB_BATCH : GL_ROWS_PER_SUB);
    const void* fn = small ? gl_rows_kernel<STEP, 1>(vec4, lanes, A.R) : gl_rows_kernel<STEP, GL_ITEM_BLOCK>(vec4, lanes, A.R);
    size_t smem = STEP ? sizeof(uint32_t) * (size_t)A.R : 0;
    if (smem > 48 * 1024) SB_CHECK_CUDA(c, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    SB_CHECK_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, GL_THREADS, smem));
    // blocks without a work unit are not launched
    const int64_t units = A.n_split_items + sb_cdiv(rows, small ? 1 : GL_ITEM_BLOCK);
    unsigned blocks = (unsigned)std::max<int64_t>(
        1, std::min<int64_t>((int64_t)c->num_sms * std::max(per_sm, 1), sb_cdiv(units, subs)));
    void* args[] = {&A};
    SbProf prof(c, SB_PROF_GL_ROWS);
    SB_CHECK_CUDA(c, cudaLaunchKernel(fn, dim3(blocks), dim3(GL_THREADS), args, smem, c->stream));
    SB_TRY(sb_after_launch(c, "k_gl_rows"));
    if (c->n_gl_hubs > 0) {
        const void* fc = (const void*)k_gl_combine<STEP>;
        const int32_t* hv = c->gl_hub_vertex;
        const int32_t* hc = c->gl_hub_count;
        int64_t nh = c->n_gl_hubs;
        unsigned gb = (unsigned)std::min<int64_t>(sb_cdiv(nh * sb_cdiv(A.R, 32), GL_THREADS / 32), (int64_t)c->num_sms * 8);
        void* cargs[] = {&A, (void*)&hv, (void*)&hc, &nh};
        SB_CHECK_CUDA(c, cudaLaunchKernel(fc, dim3(gb), dim3(GL_THREADS), cargs, 0, c->stream));
        SB_TRY(sb_after_launch(c, "k_gl_combine"));
    }
    return SB_OK;
}

static sb_status gl_check(sb_ctx* c, int32_t R)
{
    if (!c) return SB_ERR_ARG;
    if (!c->has_graph) return sb_fail(c, SB_ERR_STATE, "no graph loaded");
    if (R < 1 || R > 65536) return sb_fail(c, SB_ERR_ARG, "R must be in [1, 65536]");
    SB_CHECK_CUDA(c, cudaSetDevice(c->device));
    return SB_OK;
}

// the two launches of the forward pass on at most max_blocks blocks (red:
// blocks x R, Facc: R)
static cudaError_t gl_fwd_launch(const int2* edges, int64_t m, const float* gamma, int R, double* red, int32_t* Facc,
                                 int max_blocks, float* loss_out, int32_t* F_out, cudaStream_t st)
{
    const bool vec4 = R % 4 == 0 && ((uintptr_t)gamma & 15) == 0;
    const int w = vec4 ? R / 4 : R;  // lanes the columns need
    const int SL = w > 16 ? 32 : w > 8 ? 16 : 8;
    // a sub-warp takes at least 16 edges
    int nblocks = (int)std::max<int64_t>(1, std::min<int64_t>(max_blocks, sb_cdiv(m, 16 * (GL_THREADS / SL))));
    cudaError_t e = cudaMemsetAsync(Facc, 0, sizeof(int32_t) * (size_t)R, st);
    if (e != cudaSuccess) return e;
    const void* fn = vec4 ? (SL == 32   ? (const void*)k_gl_fwd<4, 32>
                             : SL == 16 ? (const void*)k_gl_fwd<4, 16>
                                        : (const void*)k_gl_fwd<4, 8>)
                          : (SL == 32   ? (const void*)k_gl_fwd<1, 32>
                             : SL == 16 ? (const void*)k_gl_fwd<1, 16>
                                        : (const void*)k_gl_fwd<1, 8>);
    void* args[] = {(void*)&edges, &m, (void*)&gamma, &R, &red, &Facc};
    e = cudaLaunchKernel(fn, dim3((unsigned)nblocks), dim3(GL_THREADS), args, 0, st);
    if (e != cudaSuccess) return e;
    k_gl_fwd_final<<<(unsigned)sb_cdiv(R, GL_THREADS / 32), GL_THREADS, 0, st>>>(red, nblocks, R, m, loss_out, Facc, F_out);
    return cudaGetLastError();
}

extern "C" sb_status sb_graphL_fwd(sb_ctx* c, const float* gamma, int32_t R, float* loss_out, int32_t* F_out)
{
    SB_TRY(gl_check(c, R));
    if (!gamma || !loss_out) return sb_fail(c, SB_ERR_ARG, "null pointer");
    if (c->batch_G > 0) {  // one block per graph; loss_out / F_out are G x R
        SbProf prof(c, SB_PROF_GL_FWD);
        k_gl_fwd_graph<<<(unsigned)c->batch_G, GL_THREADS, 0, c->stream>>>(c->edges, c->b_eoff, gamma, R, loss_out,
                                                                          F_out);
        return sb_after_launch(c, "k_gl_fwd_graph");
    }
    SB_TRY(gl_scratch(c, R));
    SbProf prof(c, SB_PROF_GL_FWD);
    const cudaError_t e = gl_fwd_launch(c->sc_edges, c->m, gamma, R, c->gl_red, c->gl_misc, c->num_sms * 8, loss_out,
                                        F_out, c->stream);
    if (e != cudaSuccess) return sb_cuda_fail(c, e, "k_gl_fwd");
    c->prof_launch[SB_PROF_GL_FWD] += 2;
    return SB_OK;
}

extern "C" sb_status sb_graphL_bwd(sb_ctx* c, const float* gamma, int32_t R, const float* gout, float* grad_out)
{
    SB_TRY(gl_check(c, R));
    if (!gamma || !gout || !grad_out) return sb_fail(c, SB_ERR_ARG, "null pointer");
    SB_TRY(gl_scratch(c, R));
    GlArgs A = gl_args(c, R);
    A.gin = gamma;
    A.gout_rows = grad_out;
    A.upstream = gout;
    return gl_rows_launch<false>(c, A);
}

extern "C" sb_status sb_graphL_round(sb_ctx* c, const float* gamma, int32_t R, int32_t* F_out, uint64_t* flip_out)
{
    SB_TRY(gl_check(c, R));
    if (!gamma || !F_out) return sb_fail(c, SB_ERR_ARG, "null pointer");
    SB_TRY(gl_signs_scratch(c, R, 1));
    SbProf prof(c, SB_PROF_GL_FWD);
    // two launches, three for the flips of a batch: 2.5 us each is what counts on
    // a small graph
    SB_TRY(gl_signs_launch(c, gamma, R, c->gl_signs, F_out, (c->batch_G > 0 ? c->batch_G : 1) * (int64_t)R));
    const bool flips = flip_out && c->m > 0;
    if (!flips || c->batch_G > 0) SB_TRY(gl_count_launch(c, c->gl_signs, R, F_out));
    if (flips) {
        const int64_t nb = sb_cdiv(R, 32), units = sb_cdiv(sb_cdiv(c->m, 64), 4) * nb;
        const int64_t blocks = std::min<int64_t>(sb_cdiv(units, GL_THREADS / 32), (int64_t)c->num_sms * 8);
        k_gl_flips<<<(unsigned)(sb_cdiv(blocks, nb) * nb), GL_THREADS, 0, c->stream>>>(
            c->edges, c->m, c->gl_signs, gl_sign_words(R), R, flip_out, c->batch_G > 0 ? nullptr : F_out);
        return sb_after_launch(c, "k_gl_flips");
    }
    return SB_OK;
}

// Captures the descent loop into a CUDA graph (or reuses the captured one
// when the key matches) and launches it on c->stream.
static sb_status gl_descent_graph(sb_ctx* c, GlArgs& A, const uint64_t* key, const float* src, float* const* dst,
                                  int steps, unsigned rb, int64_t GR, int32_t* F_trace, uint32_t* sign_last,
                                  int32_t* exps_out, int renorm_log2)
{
    const bool reuse = c->gl_exec && memcmp(key, c->gl_exec_key, sizeof(c->gl_exec_key)) == 0;
    const size_t sign_len = (size_t)c->n * A.sign_words;
    if (!reuse) {
        if (c->gl_exec) cudaGraphExecDestroy(c->gl_exec);
        c->gl_exec = nullptr;
        cudaGraph_t graph = nullptr;
        SB_CHECK_CUDA(c, cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
        c->capturing = true;
        sb_status st = SB_OK;
        const float* cur = src;
        for (int s = 0; s < steps && st == SB_OK; s++) {
            A.gin = cur;
            A.gout_rows = dst[s & 1];
            // sign words of step s's input: buffer s & 1
            A.signs = F_trace && s + 1 < steps ? c->gl_signs + ((s + 1) & 1) * sign_len : nullptr;
            if (s == steps - 1) A.signs = sign_last;
            if (F_trace) st = gl_count_launch(c, c->gl_signs + (s & 1) * sign_len, A.R, F_trace + (int64_t)s * GR);
            if (st == SB_OK) st = gl_rows_launch<true>(c, A);
            if (st == SB_OK) {
                k_gl_step_final<<<rb, 256, 0, c->stream>>>(GR, c->gl_colmax, c->gl_scale, exps_out, renorm_log2);
                st = sb_after_launch(c, "k_gl_step_final");
            }
            cur = A.gout_rows;
        }
        c->capturing = false;
        cudaError_t ec = cudaStreamEndCapture(c->stream, &graph);
        if (st != SB_OK) {
            if (graph) cudaGraphDestroy(graph);
            return st;
        }
        if (ec != cudaSuccess) return sb_cuda_fail(c, ec, "cudaStreamEndCapture");
        ec = cudaGraphInstantiate(&c->gl_exec, graph, 0);
        cudaGraphDestroy(graph);
        if (ec != cudaSuccess) {
            c->gl_exec = nullptr;
            return sb_cuda_fail(c, ec, "cudaGraphInstantiate");
        }
        memcpy(c->gl_exec_key, key, sizeof(c->gl_exec_key));
    } else {
        // the kernels of a replay are counted like launched ones
        c->prof_launch[SB_PROF_GL_ROWS] += (int64_t)steps * (c->n_gl_hubs > 0 ? 2 : 1);
        c->prof_launch[SB_PROF_OTHER] += (int64_t)steps * (F_trace && c->m > 0 ? 2 : 1);
    }
    SbProf prof(c, SB_PROF_GL_ROWS);
    SB_CHECK_CUDA(c, cudaGraphLaunch(c->gl_exec, c->stream));
    return SB_OK;
}

extern "C" sb_status sb_graphL_descent(sb_ctx* c, const float* gamma0, float* gamma_out, int32_t R, float alpha,
                                       int32_t steps, int32_t renorm_log2, int32_t* exps_out, int32_t* F_trace,
                                       int32_t* F_final)
{
    SB_TRY(gl_check(c, R));
    if (!gamma0 || !gamma_out || !exps_out || steps < 0 || renorm_log2 < 0 || renorm_log2 > 100)
        return sb_fail(c, SB_ERR_ARG, "bad descent argument");
    SB_TRY(gl_scratch(c, R));
    const int64_t GR = (c->batch_G > 0 ? c->batch_G : 1) * (int64_t)R;  // per (graph, column)
    SB_TRY(sb_ensure(c, (void**)&c->gl_scale, &c->gl_scale_cap, sizeof(float) * (size_t)GR));
    SB_TRY(sb_ensure(c, (void**)&c->gl_colmax, &c->gl_colmax_cap, sizeof(uint32_t) * (size_t)GR));
    const size_t bytes = sizeof(float) * (size_t)c->n * R;
    if (steps > 1 || gamma0 == gamma_out) SB_TRY(sb_ensure(c, (void**)&c->gl_buf, &c->gl_buf_cap, bytes));
    // sign words of the current and the next step's input; of the result
    // without a trace
    const int sw = gl_sign_words(R);
    if (F_trace || F_final) {
        SB_TRY(gl_signs_scratch(c, R, F_trace ? 2 : 1));
        SB_CHECK_CUDA(c, cudaMemsetAsync(c->gl_signs, 0, sizeof(uint32_t) * (size_t)c->n * sw * (F_trace ? 2 : 1), c->stream));
    }
    if (F_trace && steps > 0) SB_CHECK_CUDA(c, cudaMemsetAsync(F_trace, 0, sizeof(int32_t) * (size_t)GR * steps, c->stream));
    if (F_final) SB_CHECK_CUDA(c, cudaMemsetAsync(F_final, 0, sizeof(int32_t) * (size_t)GR, c->stream));
    SB_CHECK_CUDA(c, cudaMemsetAsync(c->gl_colmax, 0, sizeof(uint32_t) * GR, c->stream));
    SB_CHECK_CUDA(c, cudaMemsetAsync(exps_out, 0, sizeof(int32_t) * GR, c->stream));
    unsigned rb = (unsigned)sb_cdiv(GR, 256);
    k_gl_fill<<<rb, 256, 0, c->stream>>>(c->gl_scale, GR, 1.0f);
    SB_TRY(sb_after_launch(c, "k_gl_fill"));
    // the buffers alternate so that the last step writes gamma_out
    float* const dst[2] = {steps & 1 ? gamma_out : c->gl_buf, steps & 1 ? c->gl_buf : gamma_out};
    const float* src = gamma0;
    if (steps == 0 && gamma0 != gamma_out)
        SB_CHECK_CUDA(c, cudaMemcpyAsync(gamma_out, gamma0, bytes, cudaMemcpyDeviceToDevice, c->stream));
    if (gamma0 == dst[0] && steps > 0) {
        SB_CHECK_CUDA(c, cudaMemcpyAsync(c->gl_buf, gamma0, bytes, cudaMemcpyDeviceToDevice, c->stream));
        src = c->gl_buf;
    }
    if (F_trace && steps > 0) SB_TRY(gl_signs_launch(c, src, R, c->gl_signs, nullptr, 0));
    uint32_t* const sign_last = !F_final ? nullptr : c->gl_signs + (F_trace ? (size_t)(steps & 1) * c->n * sw : 0);
    GlArgs A = gl_args(c, R);
    A.scale = c->gl_scale;
    A.half_alpha = 0.5f * alpha;
    A.colmax = c->gl_colmax;
    A.sign_words = sw;
    // The step loop has no host synchronisation: it is captured once into a
    // CUDA graph and replayed while the call's buffers and parameters repeat.
    uint32_t abits;
    memcpy(&abits, &alpha, sizeof(abits));
    const uint64_t key[18] = {(uint64_t)(uintptr_t)src, (uint64_t)(uintptr_t)gamma_out, (uint64_t)R, abits,
                              (uint64_t)steps, (uint64_t)renorm_log2, (uint64_t)(uintptr_t)exps_out,
                              (uint64_t)(uintptr_t)F_trace, (uint64_t)(uintptr_t)c->gl_buf,
                              (uint64_t)(uintptr_t)c->gl_scale, (uint64_t)(uintptr_t)c->gl_partial,
                              (uint64_t)(uintptr_t)c->gl_misc, (uint64_t)(uintptr_t)c->gl_colmax,
                              (uint64_t)(uintptr_t)c->gl_items, (uint64_t)c->n,
                              1 + (uint64_t)c->tune[SB_TUNE_GL_LANES],  // the captured kernels depend on it
                              (uint64_t)(uintptr_t)c->gl_signs, (uint64_t)(uintptr_t)sign_last};
    if (steps > 0) {
        // capture and replay on a private stream ordered after / before the
        // context stream (the legacy default stream cannot be captured)
        if (!c->cap_stream) {
            SB_CHECK_CUDA(c, cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking));
            SB_CHECK_CUDA(c, cudaEventCreateWithFlags(&c->cap_in, cudaEventDisableTiming));
            SB_CHECK_CUDA(c, cudaEventCreateWithFlags(&c->cap_out, cudaEventDisableTiming));
        }
        cudaStream_t main_stream = c->stream;
        SB_CHECK_CUDA(c, cudaEventRecord(c->cap_in, main_stream));
        SB_CHECK_CUDA(c, cudaStreamWaitEvent(c->cap_stream, c->cap_in, 0));
        c->stream = c->cap_stream;
        sb_status stg = gl_descent_graph(c, A, key, src, dst, steps, rb, GR, F_trace, sign_last, exps_out, renorm_log2);
        c->stream = main_stream;
        SB_CHECK_CUDA(c, cudaEventRecord(c->cap_out, c->cap_stream));
        SB_CHECK_CUDA(c, cudaStreamWaitEvent(main_stream, c->cap_out, 0));
        SB_TRY(stg);
    }
    // pending power-of-two scale of the last step
    if (steps > 0) {
        const unsigned gb = (unsigned)std::min<int64_t>(sb_cdiv(sb_cdiv(c->n, 4) * sb_cdiv(R, 32), GL_THREADS / 32),
                                                        (int64_t)c->num_sms * 8);
        k_gl_apply_scale<<<gb, GL_THREADS, 0, c->stream>>>(gamma_out, c->n, R, c->gl_scale,
                                                           c->batch_G > 0 ? c->vgid : nullptr, sign_last, sw);
        SB_TRY(sb_after_launch(c, "k_gl_apply_scale"));
    }
    if (F_final) {
        SbProf prof(c, SB_PROF_GL_FWD);
        if (steps == 0) SB_TRY(gl_signs_launch(c, gamma_out, R, sign_last, nullptr, 0));
        SB_TRY(gl_count_launch(c, sign_last, R, F_final));
    }
    return SB_OK;
}

// ------------------------------------------- allocation-free relaxed loss
// sb_graphL_fwd_static runs the same two kernels as sb_graphL_fwd, but its
// scratch (per-block partial sums and the discrete-loss accumulators) lives in
// the fixed array below instead of context memory, so the call allocates
// nothing.  Every GPU that loads this library holds the array until the
// process exits.  All calls on a device share it and it keeps the last call's
// contents: the accumulators are cleared at the start of each call, and calls
// that overlap on the GPU (other streams, other host threads) race on it.
#define GL_STATIC_BLOCKS 304
#define GL_STATIC_RMAX 1024
static __device__ __align__(256) unsigned char g_gl_static_scratch[sizeof(double) * GL_STATIC_BLOCKS * GL_STATIC_RMAX +
                                                                   sizeof(int32_t) * GL_STATIC_RMAX];

#include <mutex>
static std::mutex g_static_mu;
static void* g_static_ptr[256];  // device address of the array, per device

extern "C" sb_status sb_graphL_fwd_static(const int32_t* edges, int64_t m, const float* gamma, int32_t R,
                                          float* loss_out, int32_t* F_out, void* cuda_stream)
{
    if (R < 1 || R > GL_STATIC_RMAX || m < 0 || m >= (1ll << 31) || !gamma || !loss_out || (m > 0 && !edges))
        return SB_ERR_ARG;
    // an error left pending by the caller's own earlier work is not ours to
    // clear; refuse to run rather than report it as this call's failure
    if (cudaPeekAtLastError() != cudaSuccess) return SB_ERR_CUDA;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) {
        cudaGetLastError();
        return SB_ERR_CUDA;
    }
    void* base = nullptr;
    {
        // first call on this device: look up the array's device address with
        // the device current (the host-side symbol is not a device address)
        std::lock_guard<std::mutex> lock(g_static_mu);
        if (!g_static_ptr[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_gl_static_scratch) != cudaSuccess || !p) {
                cudaGetLastError();
                return SB_ERR_CUDA;
            }
            g_static_ptr[dev] = p;
        }
        base = g_static_ptr[dev];
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    double* red = (double*)base;
    int32_t* Facc = (int32_t*)(red + (size_t)GL_STATIC_BLOCKS * GL_STATIC_RMAX);
    if (gl_fwd_launch((const int2*)edges, m, gamma, R, red, Facc, GL_STATIC_BLOCKS, loss_out, F_out, st) != cudaSuccess) {
        cudaGetLastError();
        return SB_ERR_CUDA;
    }
    return SB_OK;
}
