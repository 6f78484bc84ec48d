// Device functions that run as kernels of their own and inside the kernel in front of a block step (layer_step.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace dash {

constexpr int kPlanRows = 128;           // query rows of a tile of the attention kernel

// Where an attention call's item list goes in its workspace and, fp32 tensors, the bf16 copies of Q, K and V: for a step that fills them
// in a kernel of its own ahead of attention_planned()
struct AttnPlanWs { int4* plan; int* n_items; unsigned int* ticket; int64_t max_entries; int sms; __nv_bfloat16 *q, *k, *v; };
int attention_plan_ws(int S, int64_t n, int Hq, int Hkv, int D, dash_dtype dt, void* ws, size_t ws_bytes, AttnPlanWs* out);

// Whether the items of a call are pairs of neighbouring query tiles (every second tile of a sequence from its last one down, each standing for itself
// and the tile below it) or single tiles.  A pair takes 2700 cycles per key block, a tile alone about 1700, and a call lasts at least as long as its
// longest item: tiles go alone while the SMs have no more than 5/4 of the longest tile's key blocks each (blocks: of one head).  us, alone / pairs,
// and blocks per SM over those of the longest tile: 8192 rows of 4 heads of 64 79 / 101 (0.88), 1024 rows of 28 / 4 heads of 128 17.1 / 20.5 (0.85), 1300 24.2 / 26.2
// (1.14), 6000 of 7 / 1 72.6 / 76.6 (1.14), 1500 of 28 / 4 27.3 / 27.0 (1.23), 12000 of 4 heads of 64 157 / 144 (1.28), 1700 of 28 / 4 33.6 / 30.3 (1.42), 2048 40.4 / 32.7 (1.6).
// Of a pair of two tiles all in all the lower one has one block, the upper two, and single tiles take turns as well until there are many:
// 40 sequences of 200 tokens, 8 / 2 heads of 128 23.4 / 26.4 (3.2), 16 heads of 64 30.5 / 31.9 (6.5), 32 / 8 51.2 / 49.9 (13), 64 of 256, 32 / 8 78.5 / 72.5 (21).
__host__ __device__ __forceinline__ bool attention_in_pairs(int64_t blocks, int64_t longest, int Hq, int sms) {
    return longest > 2 ? 4 * blocks * Hq > 5 * longest * sms : blocks * Hq > 10 * longest * sms;
}

// The items of a call (sequence, query tile) from its true lengths, ordered by falling number of key blocks; x of an entry is 1 where it stands for a
// pair.  Called by all THREADS threads of one CTA.
template <int THREADS>
__device__ __forceinline__ void attention_plan_items(const int32_t* __restrict__ cu, int S, int Hq, int sms, int4* __restrict__ plan, int* __restrict__ n_items,
                                                     unsigned int* __restrict__ ticket, int64_t max_entries) {
    constexpr int NW = THREADS / 32;
    __shared__ int s_warp[33];
    __shared__ uint32_t s_lengths[3][32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    auto tiles = [&](int s) { return (cu[s + 1] - cu[s] + kPlanRows - 1) / kPlanRows; };
    // tiles of the longest sequence, key blocks of all (in two parts of 24 bits and the rest, which sums of a warp's 32 words cannot overflow)
    uint32_t mx = 0;
    uint64_t sum = 0;
    for (int s = tid; s < S; s += THREADS) {
        const int nq = tiles(s);
        if (nq > 0) { mx = max(mx, (uint32_t)nq); sum += (uint64_t)nq * (nq + 1) / 2; }
    }
    auto over_lanes = [&](uint32_t& m, uint64_t& t) {
        m = __reduce_max_sync(0xffffffffu, m);
        t = __reduce_add_sync(0xffffffffu, (uint32_t)t & 0xffffffu) + ((uint64_t)__reduce_add_sync(0xffffffffu, (uint32_t)(t >> 24)) << 24);
    };
    over_lanes(mx, sum);
    if (lane == 0) { s_lengths[0][w] = mx; s_lengths[1][w] = (uint32_t)sum; s_lengths[2][w] = (uint32_t)(sum >> 32); }
    __syncthreads();
    mx = lane < NW ? s_lengths[0][lane] : 0;
    sum = lane < NW ? s_lengths[1][lane] | (uint64_t)s_lengths[2][lane] << 32 : 0;
    over_lanes(mx, sum);
    const int max_nq = (int)mx;
    const int pairs = attention_in_pairs((int64_t)sum, max_nq, Hq, sms) ? 1 : 0;
    int64_t offset = 0;
    auto is_top = [&](int nq, int qt) { return nq > qt && !((nq - 1 - qt) & pairs); };
    auto put = [&](int64_t k, int s, int qt) { if (k < max_entries) plan[k] = make_int4(pairs && qt > 0, qt, cu[s], cu[s + 1]); };
    // Up to NW levels (numbers of key blocks), that is short sequences: a warp to each, its lanes over the sequences.  More: a thread to each.  (200
    // sequences of 100 tokens are one level: with a thread to it a call with 4 heads of 64 took 32.0 us, 18.0 as it is.)
    const bool wide = max_nq <= NW;
    for (int top = max_nq - 1; top >= 0; top -= THREADS) {
        const int qt = top - (wide ? w : tid);              // the first takes the heaviest level of this chunk
        int cnt = 0;
        if (wide) {
            int c = 0;
            for (int s = lane; s < S; s += 32) c += qt >= 0 && is_top(tiles(s), qt);
            c = __reduce_add_sync(0xffffffffu, c);
            if (lane == 0) cnt = c;
        } else if (qt >= 0) {
            for (int s = 0; s < S; ++s) cnt += is_top(tiles(s), qt);
        }
        // exclusive scan over the block
        int inc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { int t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
        if (lane == 31) s_warp[w] = inc;
        __syncthreads();
        if (w == 0) {
            int x = lane < NW ? s_warp[lane] : 0, xi = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { int t = __shfl_up_sync(0xffffffffu, xi, o); if (lane >= o) xi += t; }
            s_warp[lane] = xi - x;
            if (lane == 31) s_warp[32] = xi;
        }
        __syncthreads();
        int64_t k = offset + s_warp[w] + (wide ? 0 : inc - cnt);
        const int chunk_total = s_warp[32];
        if (wide) {
            for (int s0 = 0; s0 < S && qt >= 0; s0 += 32) {
                const int s = s0 + lane;
                const bool mine = s < S && is_top(tiles(s), qt);
                const uint32_t all = __ballot_sync(0xffffffffu, mine);
                if (mine) put(k + __popc(all & ((1u << lane) - 1)), s, qt);
                k += __popc(all);
            }
        } else if (qt >= 0) {
            for (int s = 0; s < S; ++s)
                if (is_top(tiles(s), qt)) put(k++, s, qt);
        }
        offset += chunk_total;
        __syncthreads();
    }
    if (tid == 0) {
        if (offset > max_entries) offset = max_entries;     // cannot happen for cu_seqlens[S] <= n; keeps every read in bounds
        *n_items = (int)(offset * Hq);
        *ticket = 0u;
    }
}

struct RopeFreqs { double inv_freq[64]; };

// Per row (one warp): (cos, sin) of pos[t] * base^(-2i/D) for i < D/2, angles formed and reduced in fp64 (positions reach 1e5 rad
// at i = 0: fp32 would lose the angle), evaluated in fp32 on the reduced angle; and, when asked, the row factor of the RMSNorm, 1 / sqrt(mean(h^2) + eps), from one pass over the bf16 row.
// Rows first_warp, first_warp + n_warps, ..
__device__ __forceinline__ void row_prep_rows(const int32_t* __restrict__ pos, int64_t n, int half, const RopeFreqs& fr, float2* __restrict__ table,
                                              const char* __restrict__ H, int64_t ldh_b, int nvec, float inv_d, float eps, float* __restrict__ inv_rms,
                                              const int32_t* __restrict__ n_dev, int64_t first_warp, int64_t n_warps) {
    if (n_dev) { int64_t nd = *n_dev; if (nd < n) n = nd; }
    const int lane = threadIdx.x & 31;
    for (int64_t t = first_warp; t < n; t += n_warps) {
        float ss = 0.f;
        if (inv_rms) {
            const char* h = H + t * ldh_b;
            for (int base = 0; base < nvec; base += 128) {
                uint4 x[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) { const int v = base + k * 32 + lane; if (v < nvec) x[k] = ld_nc_v4(h + ((int64_t)v << 4)); }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int v = base + k * 32 + lane;
                    if (v < nvec) {
                        const float f[8] = {bf16lo(x[k].x), bf16hi(x[k].x), bf16lo(x[k].y), bf16hi(x[k].y), bf16lo(x[k].z), bf16hi(x[k].z), bf16lo(x[k].w), bf16hi(x[k].w)};
#pragma unroll
                        for (int e = 0; e < 8; ++e) ss += f[e] * f[e];
                    }
                }
            }
        }
        if (table) {
            const double ps = pos ? (double)pos[t] : (double)t;
            for (int i = lane; i < half; i += 32) {
                // angle formed and reduced to [-pi, pi] in fp64 (three operations), sine and cosine of the reduced angle in fp32
                const double ang = ps * fr.inv_freq[i];
                const double red = fma(-6.283185307179586476925286766559, rint(ang * 0.15915494309189533576888376337251), ang);
                float sn, cs;
                sincosf((float)red, &sn, &cs);
                table[t * half + i] = make_float2(cs, sn);
            }
        }
        if (inv_rms) {
            ss = warp_sum(ss);
            if (lane == 0) inv_rms[t] = rsqrtf(ss * inv_d + eps);
        }
    }
}

}  // namespace dash
