// sb_count.cuh -- vertical counters: 64 one-bit streams, one 64-bit word at a
// time, counted with carry-save adders (ones, twos, fours) and ripple planes of
// eights, and flushed into 32-bit counts before the planes can overflow.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sb_internal.cuh"

#define SC_PLANES 12                     // ripple planes of the eights
#define SC_RIPPLE_EXIT 1                 // stop the ripple when no carry is left
#define SC_FLUSH ((1 << SC_PLANES) - 1)  // batches of 8 words between flushes

__device__ __forceinline__ void csa(uint64_t& h, uint64_t& l, uint64_t a, uint64_t b, uint64_t c)
{
    const uint64_t u = a ^ b;
    h = (a & b) | (u & c);
    l = u ^ c;
}

struct ScoreAcc {
    uint64_t ones, twos, fours, P[SC_PLANES];
    int nb;  // batches added since the last flush
    __device__ __forceinline__ void reset()
    {
        ones = twos = fours = 0;
#pragma unroll
        for (int b = 0; b < SC_PLANES; b++) P[b] = 0;
        nb = 0;
    }
    __device__ __forceinline__ void add8(const uint64_t* x)
    {
        uint64_t twosA, twosB, foursA, foursB, eights;
        csa(twosA, ones, ones, x[0], x[1]);
        csa(twosB, ones, ones, x[2], x[3]);
        csa(foursA, twos, twos, twosA, twosB);
        csa(twosA, ones, ones, x[4], x[5]);
        csa(twosB, ones, ones, x[6], x[7]);
        csa(foursB, twos, twos, twosA, twosB);
        csa(eights, fours, fours, foursA, foursB);
        uint64_t cy = eights;
#pragma unroll
        for (int b = 0; b < SC_PLANES; b++) {
            if (SC_RIPPLE_EXIT && !cy) break;  // carries die out after a few planes
            const uint64_t t = P[b] & cy;
            P[b] ^= cy;
            cy = t;
        }
        nb++;
    }
    __device__ __forceinline__ uint32_t count(int t) const
    {
        uint32_t hi = 0;
#pragma unroll
        for (int b = 0; b < SC_PLANES; b++) {
            if (!(nb >> b)) break;  // nb batches hold at most nb eights
            hi |= (uint32_t)((P[b] >> t) & 1ull) << b;
        }
        return 8u * hi + 4u * (uint32_t)((fours >> t) & 1ull) + 2u * (uint32_t)((twos >> t) & 1ull) +
               (uint32_t)((ones >> t) & 1ull);
    }
    // add8 for words of several graphs (graph gk[k] of word k, the words in `rem`
    // valid, equal graphs next to one another): runs of one graph, flushed to
    // dst0 + graph * KP when the graph changes
    __device__ __forceinline__ void add8_runs(const uint64_t* x, const int32_t* gk, uint32_t rem, int64_t& gcur,
                                              uint32_t* dst0, int64_t KP)
    {
        while (rem) {
            int32_t g = -1;
#pragma unroll
            for (int k = 7; k >= 0; k--)
                if ((rem >> k) & 1u) g = gk[k];  // graph of the first remaining word
            uint64_t xm[8];
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const bool tk = ((rem >> k) & 1u) && gk[k] == g;
                xm[k] = tk ? x[k] : 0ull;
                if (tk) rem &= ~(1u << k);
            }
            if (g != gcur) {
                if (gcur >= 0) flush(dst0 + gcur * KP);
                gcur = g;
            }
            add8(xm);
            if (nb == SC_FLUSH) flush(dst0 + gcur * KP);
        }
    }
    // adds the 64 counters into dst[0..63] (shared or global memory)
    __device__ __forceinline__ void flush(uint32_t* dst)
    {
        if (nb == 0) return;
        for (int t = 0; t < 64; t++) {
            const uint32_t val = count(t);
            if (val) atomicAdd(dst + t, val);
        }
        reset();
    }
    // the same for a whole warp whose lanes gl, gl + G, .. count word gl of
    // dst[64 * G] (lanes that count nothing hold zeros).  Up to 16 words: every
    // plane is transposed, so that lane j has all lanes' bits of stream j and a
    // population count per word sums the lanes that share it, instead of 64
    // bit extractions per lane and as many atomics on one address.  32 words:
    // nothing is shared, and the lanes start at different streams so that
    // their atomics fall in different banks.
    template <int G>
    __device__ __forceinline__ void flush_warp(uint32_t* dst)
    {
        const unsigned lane = threadIdx.x & 31u;
        if constexpr (G == 32) {
            for (int i = 0; i < 64; i++) {
                const int t = (i + (int)lane) & 63;
                const uint32_t val = count(t);
                if (val) atomicAdd(dst + 64 * lane + t, val);
            }
        } else {
            uint32_t lo[G], hi[G];
            sum_warp<G>(lo, hi);
#pragma unroll
            for (int w = 0; w < G; w++) {
                if (lo[w]) atomicAdd(dst + 64 * w + lane, lo[w]);
                if (hi[w]) atomicAdd(dst + 64 * w + 32 + lane, hi[w]);
            }
        }
    }
    // the warp's counts of streams `lane` and `lane + 32` of word w in lo[w], hi[w]
    template <int G>
    __device__ __forceinline__ void sum_warp(uint32_t* lo, uint32_t* hi) const
    {
        constexpr uint32_t M = G == 1 ? 0xFFFFFFFFu : G == 2 ? 0x55555555u : G == 4 ? 0x11111111u
                             : G == 8 ? 0x01010101u : 0x00010001u;  // lanes of word 0
        const unsigned lane = threadIdx.x & 31u;
#pragma unroll
        for (int w = 0; w < G; w++) lo[w] = hi[w] = 0;
        auto add = [&](uint64_t x, int shift) {
            if (!__any_sync(0xffffffffu, x != 0)) return;
            const uint32_t a = warp_transpose32((uint32_t)x, lane), b = warp_transpose32((uint32_t)(x >> 32), lane);
#pragma unroll
            for (int w = 0; w < G; w++) {
                lo[w] += (uint32_t)__popc(a & (M << w)) << shift;
                hi[w] += (uint32_t)__popc(b & (M << w)) << shift;
            }
        };
        add(ones, 0);
        add(twos, 1);
        add(fours, 2);
#pragma unroll
        for (int b = 0; b < SC_PLANES; b++) add(P[b], 3 + b);
    }
};
