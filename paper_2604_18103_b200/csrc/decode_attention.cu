// Decode-step attention: one new token per sequence attends over that sequence's packed KV cache
// (the cache of the deeper layers holds only the tokens that stayed active; it simply has fewer rows).
// HBM-bound: every cached key/value row is read once.  The G = Hq / Hkv query heads that share one KV
// head form the (mostly empty) 128-row operand of the tcgen05 MMAs, so K and V tiles stream through
// shared memory once per KV head; the keys of a sequence are split over persistent CTAs (flash-decoding),
// whose partial (max, sum, O) results a merge kernel spread over all SMs combines.
//   plan          : items (sequence, KV head, key-block range).  Batches of up to 128 sequences: every CTA makes it for itself, an even share of the key blocks per CTA
//                   or, where that makes more items than CTAs, the length that takes the fewest rounds (self_plan_build); more sequences: a plan kernel, about four
//                   items per SM, handed out by ticket
//   decode kernel : per item  S = Q K_j^T -> masked online softmax (one warp: the rows that exist) -> O += P V_j
//   merge kernel  : O = sum_i 2^((m_i - m) c) O_i / sum_i 2^((m_i - m) c) l_i
#include <math.h>

#include "common.cuh"
#include "dash_testing.h"
#include "sm100_ptx.cuh"

namespace dash {

using namespace ptx;

constexpr int kDecBN = 128;                  // keys per block
constexpr int kDecThreads = 64;              // warp 0: softmax (rows 0..31 of the tile, G of them real), warp 1: TMA + MMA issue
constexpr int kDecRows = 8;                  // query heads per KV head the tile can hold (box of the Q load)
constexpr long long kDecWaitCycles = 4000000000LL;
constexpr uint32_t kDecTmemCols = 256;       // S | O

struct DecItem { int s, kvh, b0, b1; };

struct DecParams {
    const int32_t* cu;
    int S, Hq, Hkv, G;
    float scale_log2, scale;
    float* partial;             // [item][kDecRows][D]: unnormalised O rows
    float2* ml;                 // [Hq][max_items]: their (m, l); the splits of one head lie next to each other
    int max_items;
    const DecItem* plan;        // not where the CTAs plan for themselves (S <= kSelfPlanSeqs)
    const int* n_items;
    unsigned int* ticket;
    int target;                 // twice the number of CTAs (see self_plan_build)
    int* status;
};

// Batches of up to kSelfPlanSeqs sequences need no plan kernel, no ticket and no scratch clear: every CTA derives the chunk
// length and its items (item i -> CTA i mod grid; the items are equally long) from cu_seqlens itself, and so does the merge.
constexpr int kSelfPlanSeqs = 128;
__device__ __forceinline__ int dec_blocks(const int32_t* cu, int s) { return (cu[s + 1] - cu[s] + kDecBN - 1) / kDecBN; }
// The plan of a self-planning launch, built once per CTA in shared memory by its first warp, a lane per sequence (four at most).  With
// thread 0 going through the sequences one by one, up to nine times, the plan of 24 sequences took 3 us of the decode kernel and
// again of the merge kernel.
struct SelfPlan {
    int nb[kSelfPlanSeqs];            // key blocks of sequence s
    int first[kSelfPlanSeqs + 1];     // first item of sequence s (its Hkv heads follow each other, `per` items each); then the number of items
    int per[kSelfPlanSeqs];           // items per (sequence, KV head)
    int cu[kSelfPlanSeqs + 1];        // the boundaries it was made from
    int chunk, n_items;
};
// Called by all threads of the CTA (it synchronises).  `target` is twice the number of CTAs; the items at a chunk length of ceil(all blocks / target) and more are
// never more than target + sequences x heads, which the workspace has room for.  Chunk length (key blocks per item): an even share per CTA, if
// that makes no more items than CTAs (the last chunk of every sequence and head is an item of its own, so it can overshoot); else, of that, the next one, and three
// from two items per CTA on, the one with the fewest rounds x (chunk + 1.5): a CTA goes through an item in about 2 us a block and 3 us beside.  us a call in
// a graph, 28 / 4 heads of 128: this rule / one item per CTA where that kept 17 of 20 CTAs busy, else about two / the best of all lengths: one cache
// of 8192 rows 7.7 / 7.7 / 7.6, of 20 000 12.5 / 14.9 / 12.5, 4 of 7500 on the average 16.4 / 18.3 / 16.4, 8 of 2500 13.3 / 16.4 / 13.3, 16 of 750 11.6 / 14.1 / 11.6, 24 of
// 3125 31.3 / 31.3 / 31.3, 33 of 485 14.3 / 15.4 / 14.3, 40 of 750 19.3 / 18.6 / 18.4, 80 of 625 28.8 / 31.7 / 28.8, 96 of 1250 54.1 / 60.3 / 53.8.  (Little
// code on purpose: with every length up to the first that fits tried, in two loops, a call took 0.4 to 1.7 us longer.)
__device__ __forceinline__ void self_plan_build(SelfPlan& sp, const int32_t* cu, int S, int Hkv, int target) {
    if (threadIdx.x < 32) {
        constexpr int PL = kSelfPlanSeqs / 32;
        const int lane = threadIdx.x;
        unsigned int nb[PL], all = 0;
#pragma unroll
        for (int j = 0; j <= PL; ++j) { const int s = lane + 32 * j; if (s <= S) sp.cu[s] = __ldcg(cu + s); }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < PL; ++j) { const int s = lane + 32 * j; nb[j] = s < S ? (unsigned int)dec_blocks(sp.cu, s) : 0u; all += nb[j]; }
        all = __reduce_add_sync(0xffffffffu, all) * (unsigned int)Hkv;
        auto count = [&](unsigned int chunk) {
            unsigned int k = 0;
#pragma unroll
            for (int j = 0; j < PL; ++j)
                if (32 * j < S) k += (nb[j] + chunk - 1) / chunk;
            return (int)(__reduce_add_sync(0xffffffffu, k) * (unsigned int)Hkv);
        };
        const unsigned int ctas = (unsigned int)target / 2, even = max(1u, (all + ctas - 1) / ctas), half = max(1u, (all + (unsigned int)target - 1) / (unsigned int)target);
        unsigned int chunk = even;
        if ((unsigned int)count(even) > ctas) {
            unsigned int least = 0xffffffffu;
#pragma unroll 1
            for (unsigned int i = 0; i < 5; ++i) {
                const unsigned int c = i < 2 ? even + i : half + i - 2;
                const unsigned int cost = ((unsigned int)count(c) + ctas - 1) / ctas * (2 * c + 3);
                if (cost < least) { least = cost; chunk = c; }
            }
        }
        int k = 0;                    // items in front of the current group of 32 sequences
#pragma unroll
        for (int j = 0; j < PL; ++j) {
            if (32 * j >= S) break;
            const int s = lane + 32 * j, per = (int)((nb[j] + chunk - 1) / chunk), mine = per * Hkv;
            int inc = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += x; }
            if (s < S) { sp.nb[s] = (int)nb[j]; sp.per[s] = per; sp.first[s] = k + inc - mine; }
            k += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) { sp.chunk = (int)chunk; sp.n_items = k; sp.first[S] = k; }
    }
    __syncthreads();
}
// Whether the boundaries have become others since the plan was made from them (called by all threads of the CTA)
__device__ __forceinline__ bool self_plan_outdated(const SelfPlan& sp, const int32_t* cu, int S) {
    int changed = 0;
    for (int s = threadIdx.x; s <= S; s += blockDim.x) changed |= __ldcg(cu + s) != sp.cu[s];
    return __syncthreads_or(changed) != 0;
}
__device__ __forceinline__ DecItem self_plan_item(const SelfPlan& sp, int S, int item) {
    int lo = 0, hi = S;               // first[lo] <= item < first[hi]: the last such lo owns the item (sequences without keys own none)
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (sp.first[mid] <= item) lo = mid; else hi = mid;
    }
    const unsigned int per = (unsigned int)sp.per[lo], r = (unsigned int)(item - sp.first[lo]), h = r / per, i = r - h * per;
    DecItem it = {lo, (int)h, (int)i * sp.chunk, min(((int)i + 1) * sp.chunk, sp.nb[lo])};
    return it;
}

// One CTA: per sequence the number of key blocks, a common chunk length (blocks per item) so that about
// `target` items exist, then the items of every (sequence, KV head) written next to each other.
__global__ void __launch_bounds__(256)
decode_plan_kernel(const int32_t* __restrict__ cu, int S, int Hkv, int target, DecItem* __restrict__ plan, int2* __restrict__ seg,
                   int* __restrict__ n_items, unsigned int* __restrict__ ticket, int max_items, int* __restrict__ seq_first) {
    __shared__ unsigned long long s_total;
    __shared__ int s_chunk;
    if (threadIdx.x == 0) s_total = 0;
    __syncthreads();
    unsigned long long mine = 0;
    for (int s = threadIdx.x; s < S; s += blockDim.x) mine += (unsigned long long)((cu[s + 1] - cu[s] + kDecBN - 1) / kDecBN);
    atomicAdd(&s_total, mine);
    __syncthreads();
    if (threadIdx.x == 0) {
        const long long all = (long long)s_total * Hkv;
        const long long chunk = (all + target - 1) / target;
        s_chunk = (int)(chunk < 1 ? 1 : chunk);
        // first item of every sequence (its Hkv heads follow each other): one short serial pass over the sequences
        int k = 0;
        for (int s = 0; s < S; ++s) {
            seq_first[s] = k;
            const int nb = (cu[s + 1] - cu[s] + kDecBN - 1) / kDecBN;
            k += ((nb + s_chunk - 1) / s_chunk) * Hkv;
        }
        *n_items = k < max_items ? k : max_items;
        *ticket = 0u;
    }
    __syncthreads();
    const int chunk = s_chunk;
    for (int sh = threadIdx.x; sh < S * Hkv; sh += blockDim.x) {
        const int s = sh / Hkv, h = sh % Hkv;
        const int nb = (cu[s + 1] - cu[s] + kDecBN - 1) / kDecBN;
        const int per = (nb + chunk - 1) / chunk;
        const int first = seq_first[s] + h * per;
        int cnt = 0;
        for (int i = 0; i < per && first + i < max_items; ++i, ++cnt) {
            DecItem it = {s, h, i * chunk, min((i + 1) * chunk, nb)};
            plan[first + i] = it;
        }
        seg[sh] = make_int2(first, cnt);
    }
}

template <int D>
struct DecSmem {
    static constexpr int kTileBytes = kDecBN * D * 2;
    static constexpr int kQ = 0, kK = kTileBytes, kV = 2 * kTileBytes, kBars = 3 * kTileBytes;
    static constexpr int kTotal = kBars + 128;
    // What a launch asks for: so much that a third CTA does not fit onto an SM, whose TMEM holds two (kDecTmemCols each).  With heads of 64
    // (50 KB) four fit.  Launched while the merge of the call in front still sits on some of the SMs, the CTAs stacked up on the others,
    // where the third and fourth waited for columns with their share of the items, which nobody else takes: 8 heads of 64,
    // in a graph, 33 caches of 1200 rows 36.7 us, 64 of 1000 72, 128 of 1000 112, one of 131 072 83; with two per SM 23.4, 45, 77, 52.
    static constexpr int kLaunch = kTotal + 1024 > 80 * 1024 ? kTotal + 1024 : 80 * 1024;
};

// SELF: the CTAs plan for themselves (a template argument: with the plan's code beside it, the loop over planned items took 128 registers
// instead of 116 and ran 2 % longer over more than 128 caches with heads of 64, 1 % with heads of 128)
template <int D, bool SELF>
__global__ void __launch_bounds__(kDecThreads)
decode_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
              const __grid_constant__ CUtensorMap mapV, const DecParams p, int q_box_heads) {
    extern __shared__ uint8_t smem_raw[];
    using L = DecSmem<D>;
    constexpr int KCH = D / 64;
    constexpr int kChunkBytes = kDecBN * 128;
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sQ = smem_base + L::kQ, sK = smem_base + L::kK, sV = smem_base + L::kV;
    const uint32_t bars = smem_base + L::kBars;
    const uint32_t bar_q = bars, bar_k = bars + 8, bar_v = bars + 16, bar_s = bars + 24, bar_o = bars + 32, bar_p0 = bars + 40, bar_p1 = bars + 48;
    const uint32_t tmem_slot = bars + 64;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    volatile uint32_t* tmem_slot_gen = reinterpret_cast<volatile uint32_t*>(smem_gen + L::kBars + 64);
    volatile uint32_t* abort_gen = reinterpret_cast<volatile uint32_t*>(smem_gen + L::kBars + 68);
    volatile int* item_gen = reinterpret_cast<volatile int*>(smem_gen + L::kBars + 72);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // rows of the Q tile that no load ever writes must not hold NaN patterns: clear the tile once
    for (int i = tid * 16; i < L::kTileBytes; i += kDecThreads * 16) *reinterpret_cast<uint4*>(smem_gen + L::kQ + i) = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
    if (warp == 1) {
        if (lane == 0) {
            mbar_init(bar_q, 1); mbar_init(bar_k, 1); mbar_init(bar_v, 1);
            mbar_init(bar_s, 1); mbar_init(bar_o, 1); mbar_init(bar_p0, 32); mbar_init(bar_p1, 32);
            *abort_gen = 0;
            fence_barrier_init();
            fence_proxy_async_smem();
            prefetch_tensormap(&mapQ); prefetch_tensormap(&mapK); prefetch_tensormap(&mapV);
        }
        __syncwarp();
        tmem_alloc(tmem_slot, kDecTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    __shared__ SelfPlan sp;
    if (SELF) {
        // While the kernel in front drains (the previous call's merge, in a decoding step): the plan from the boundaries as they stand, and
        // this CTA's first key block asked into L2.  Nothing of either counts if the boundaries turn out to be others (a prefetch
        // reads nothing; its rows are those of the map or none).
        self_plan_build(sp, p.cu, p.S, p.Hkv, p.target);
        if (tid == 32 && (int)blockIdx.x < sp.n_items) {
            const DecItem it = self_plan_item(sp, p.S, (int)blockIdx.x);
            const int row = sp.cu[it.s] + it.b0 * kDecBN;
            for (int c = 0; c < KCH; ++c) { tma_prefetch_3d(&mapK, c * 64, it.kvh, row); tma_prefetch_3d(&mapV, c * 64, it.kvh, row); }
        }
    }
    pdl_wait();                              // set-up done; from here on the kernel in front has completed
    pdl_launch_dependents();                 // the merge kernel may get onto the SMs now: all in front of this kernel is complete for it too
    const uint32_t tmem = *tmem_slot_gen;
    const uint32_t tS = tmem, tP = tmem, tO = tmem + 128;
    constexpr uint32_t idesc_s = idesc_bf16_f32(128, kDecBN, false, false);
    constexpr uint32_t idesc_o = idesc_bf16_f32(128, D, false, true);
    // Q and the first key block of an item (one thread)
    auto load_first = [&](const DecItem& it, int seq_a) {
        mbar_arrive_expect_tx(bar_q, (uint32_t)(KCH * q_box_heads * 128));
        for (int c = 0; c < KCH; ++c) tma_load_3d(sQ + c * kChunkBytes, &mapQ, bar_q, c * 64, it.kvh * p.G, it.s);
        mbar_arrive_expect_tx(bar_k, L::kTileBytes);
        for (int c = 0; c < KCH; ++c) tma_load_3d(sK + c * kChunkBytes, &mapK, bar_k, c * 64, it.kvh, seq_a + it.b0 * kDecBN);
        mbar_arrive_expect_tx(bar_v, L::kTileBytes);
        for (int c = 0; c < KCH; ++c) tma_load_3d(sV + c * kChunkBytes, &mapV, bar_v, c * 64, it.kvh, seq_a + it.b0 * kDecBN);
    };
    uint32_t blk0 = 0, items_done = 0;       // barrier phases run on across the items of this CTA
    uint32_t again = 0;                      // loads of Q, K and V that were thrown away: their barriers are that many phases ahead
    bool loaded = false;                     // the first item's first loads are out
    if (SELF) {
        // The loads of the plan made ahead of the wait go out before its boundaries have been compared with those that stand now (0.7 us, and as
        // much again when the loads read the boundaries from memory once more: Q and the first K were in 2.4 us after the wait, now 1.2).  If they
        // differ, what was loaded (rows of the maps, or zeros where a coordinate lies outside) is waited for and loaded again by a new plan.
        loaded = (int)blockIdx.x < sp.n_items;
        if (tid == 32 && loaded) {
            const DecItem it = self_plan_item(sp, p.S, (int)blockIdx.x);
            load_first(it, sp.cu[it.s]);
        }
        if (self_plan_outdated(sp, p.cu, p.S)) {
            if (loaded) {
                if (tid == 32 && !(mbar_wait(bar_q, 0, kDecWaitCycles) && mbar_wait(bar_k, 0, kDecWaitCycles) && mbar_wait(bar_v, 0, kDecWaitCycles))) {
                    *abort_gen = 1;
                    atomicExch(p.status, DASH_ERR_TIMEOUT);
                }
                again = 1;
                loaded = false;
            }
            self_plan_build(sp, p.cu, p.S, p.Hkv, p.target);
        }
    }
    const int n_items = SELF ? sp.n_items : *p.n_items;

    for (;;) {
        int item;
        if (SELF) {
            item = (int)blockIdx.x + (int)items_done * (int)gridDim.x;
        } else {
            if (tid == 0) *item_gen = (int)atomicAdd(p.ticket, 1u);
            __syncthreads();
            item = *item_gen;
        }
        if (item >= n_items || *abort_gen) break;
        tc_fence_after();
        const DecItem it = SELF ? self_plan_item(sp, p.S, item) : p.plan[item];
        const int32_t* cu = SELF ? sp.cu : p.cu;
        const int seq_a = cu[it.s], len = cu[it.s + 1] - seq_a;
        const int nblk = it.b1 - it.b0;
        const int last_blk = (len + kDecBN - 1) / kDecBN - 1;       // the block of the sequence with a ragged end
        if (warp == 1) {
            if (lane == 0) {
                bool ok = true;
                if (!loaded) load_first(it, seq_a);
                auto issue_s = [&]() {
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) {
                        const uint32_t off = (kk >> 2) * kChunkBytes + (kk & 3) * 32;
                        mma_ss(tS, smem_desc_sw128(sQ + off, 16, 1024), smem_desc_sw128(sK + off, 16, 1024), idesc_s, kk > 0);
                    }
                    tc_commit(bar_s);
                };
                ok = mbar_wait(bar_q, (items_done + again) & 1, kDecWaitCycles) && mbar_wait(bar_k, (blk0 + again) & 1, kDecWaitCycles);
                if (ok) issue_s();
                for (int j = 0; j < nblk && ok; ++j) {
                    const uint32_t ph = (blk0 + j) & 1;
                    ok = mbar_wait(bar_s, ph, kDecWaitCycles);               // S_j done: the K buffer is free
                    if (!ok) break;
                    if (j + 1 < nblk) {
                        mbar_arrive_expect_tx(bar_k, L::kTileBytes);
                        for (int c = 0; c < KCH; ++c) tma_load_3d(sK + c * kChunkBytes, &mapK, bar_k, c * 64, it.kvh, seq_a + (it.b0 + j + 1) * kDecBN);
                    }
                    ok = mbar_wait(bar_p0, ph, kDecWaitCycles) && mbar_wait(bar_v, ph ^ again, kDecWaitCycles);
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < kDecBN / 32; ++kk)
                        mma_ts(tO, tP + kk * 8, smem_desc_sw128(sV + kk * 2048, kChunkBytes, 1024), idesc_o, (j > 0) || (kk > 0));
                    ok = mbar_wait(bar_p1, ph, kDecWaitCycles);
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll
                    for (int kk = kDecBN / 32; kk < kDecBN / 16; ++kk)
                        mma_ts(tO, tP + kk * 8, smem_desc_sw128(sV + kk * 2048, kChunkBytes, 1024), idesc_o, 1);
                    tc_commit(bar_o);
                    if (j + 1 < nblk) {
                        ok = mbar_wait(bar_k, (blk0 + j + 1 + again) & 1, kDecWaitCycles);
                        if (!ok) break;
                        issue_s();                                         // in issue order behind PV_j, which reads P_j from the same columns
                    }
                    ok = mbar_wait(bar_o, ph, kDecWaitCycles);              // PV_j done: the V buffer is free
                    if (!ok) break;
                    if (j + 1 < nblk) {
                        mbar_arrive_expect_tx(bar_v, L::kTileBytes);
                        for (int c = 0; c < KCH; ++c) tma_load_3d(sV + c * kChunkBytes, &mapV, bar_v, c * 64, it.kvh, seq_a + (it.b0 + j + 1) * kDecBN);
                    }
                }
                if (!ok) { *abort_gen = 1; atomicExch(p.status, DASH_ERR_TIMEOUT); }
            }
        } else {
            // ---- softmax warp.  Only rows 0..G-1 of the 128-row tile exist, so the scores are fetched in the 16-row shape
            // (tcgen05.ld.16x256b): thread t holds, of row t / 4, the keys 8u + 2 (t % 4) + {0, 1} of every group u of 8 keys
            // (and the same of row t / 4 + 8, which is not a real head and is ignored).  Four threads share a row: 32 exponentials
            // per thread and block instead of 128.  P goes back in the 16x128b shape, whose 32-bit column 4u + (t % 4) is exactly
            // the pair of keys the thread holds. ----
            const int sub = lane & 3, hrow = lane >> 2;         // position within the row's four threads, row (query head of the group)
            float m = -INFINITY, l = 0.f;                       // m: common to the row's threads, l: this thread's share
            bool ok = true;
            for (int j = 0; j < nblk; ++j) {
                const uint32_t ph = (blk0 + j) & 1;
                ok = mbar_wait(bar_s, ph, kDecWaitCycles);
                if (!ok || *abort_gen) { ok = false; break; }
                tc_fence_after();
                uint32_t raw[64];
                tmem_ld16x256_x8(tS, &raw[0]);
                tmem_ld16x256_x8(tS + 64, &raw[32]);
                tmem_wait_ld();
                float sc[32];                                   // sc[2u + e] = score of key 8u + 2 sub + e
#pragma unroll
                for (int u = 0; u < 16; ++u) { sc[2 * u] = __uint_as_float(raw[4 * u]); sc[2 * u + 1] = __uint_as_float(raw[4 * u + 1]); }
                const bool ragged = (it.b0 + j == last_blk);
                const int valid = len - (it.b0 + j) * kDecBN;               // keys of this block that exist (>= 1)
                if (ragged) {
#pragma unroll
                    for (int u = 0; u < 16; ++u) {
                        if (8 * u + 2 * sub >= valid) sc[2 * u] = -INFINITY;         // past the end of the sequence's cache
                        if (8 * u + 2 * sub + 1 >= valid) sc[2 * u + 1] = -INFINITY;
                    }
                }
                float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
                for (int c = 0; c < 32; c += 4) {
                    mx0 = fmax3(mx0, sc[c], sc[c + 1]);
                    mx1 = fmax3(mx1, sc[c + 2], sc[c + 3]);
                }
                float mx = fmaxf(mx0, mx1);
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                // the reference max only moves when the block max exceeds it by more than 2^8 (then O is rescaled)
                const bool grow = (mx - m) * p.scale_log2 > 8.0f;
                const float m_new = grow ? mx : m;
                const float msl = m_new * p.scale_log2;
                const float alpha = grow ? ex2((m - m_new) * p.scale_log2) : 1.0f;
                if (j > 0 && __any_sync(0xffffffffu, grow)) {
                    ok = mbar_wait(bar_o, (blk0 + j - 1) & 1, kDecWaitCycles);
                    if (!ok) break;
                    tc_fence_after();
                    const float a_row = __shfl_sync(0xffffffffu, alpha, (lane * 4) & 31);   // lane r < 8 rescales row r of O
#pragma unroll 1
                    for (int c = 0; c < D / 8; ++c) {
                        uint32_t o[8];
                        tmem_ld8(tO + c * 8, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 8; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * (lane < 8 ? a_row : 1.0f));
                        tmem_st8(tO + c * 8, o);
                    }
                    tmem_wait_st();
                }
                if (ragged) {
                    // cached rows past the end of the sequence may hold anything: zero them (0 * garbage must not make a NaN)
                    ok = mbar_wait(bar_v, ph ^ again, kDecWaitCycles);
                    if (!ok) break;
                    for (int r = lane; r < kDecBN; r += 32) {
                        if (r >= valid) {
#pragma unroll
                            for (int c = 0; c < KCH; ++c) {
                                uint4* rowp = reinterpret_cast<uint4*>(smem_gen + L::kV + c * kChunkBytes + r * 128);
#pragma unroll
                                for (int e = 0; e < 8; ++e) rowp[e] = make_uint4(0, 0, 0, 0);
                            }
                        }
                    }
                    fence_proxy_async_smem();
                }
                float2 sum2 = make_float2(0.f, 0.f);
                const float2 sl2 = make_float2(p.scale_log2, p.scale_log2), nm2 = make_float2(-msl, -msl);
                uint32_t pk[32];                                // pk[2u] = P of (row, keys 8u + 2 sub + {0,1}); pk[2u + 1] = row + 8: nothing
#pragma unroll
                for (int half = 0; half < 2; ++half) {
#pragma unroll
                    for (int u = half * 8; u < half * 8 + 8; ++u) {
                        const float2 x = __ffma2_rn(make_float2(sc[2 * u], sc[2 * u + 1]), sl2, nm2);
                        float2 pe;
                        pe.x = ex2(x.x); pe.y = ex2(x.y);
                        sum2 = __fadd2_rn(sum2, pe);
                        pk[2 * u] = pack_bf16(pe.x, pe.y);
                        pk[2 * u + 1] = 0u;
                    }
                    // the first 64 keys of P go out (and their PV steps start) while the rest is still being formed
                    tmem_st16x128_x8(tP + half * 32, &pk[half * 16]);
                    tmem_wait_st();
                    tc_fence_before();
                    mbar_arrive(half == 0 ? bar_p0 : bar_p1);
                }
                l = l * alpha + (sum2.x + sum2.y);
                m = m_new;
            }
            if (ok) ok = mbar_wait(bar_o, (blk0 + nblk - 1) & 1, kDecWaitCycles);
            // row sum: the four threads' shares; the row leaves as it is read, four threads to 32 contiguous bytes (a lane per row wrote 8 bytes
            // of seven rows at a time: 64 store instructions, now 32 of whole sectors)
            l += __shfl_xor_sync(0xffffffffu, l, 1);
            l += __shfl_xor_sync(0xffffffffu, l, 2);
            if (ok && !*abort_gen) {
                tc_fence_after();
                float* dst = p.partial + ((size_t)item * kDecRows + hrow) * D + 2 * sub;
                uint32_t o[D / 2];
#pragma unroll
                for (int c = 0; c < KCH; ++c) tmem_ld16x256_x8(tO + c * 64, &o[c * 32]);
                tmem_wait_ld();
                if (hrow < p.G) {
#pragma unroll
                    for (int u = 0; u < D / 8; ++u)
                        *reinterpret_cast<float2*>(dst + 8 * u) = make_float2(__uint_as_float(o[4 * u]), __uint_as_float(o[4 * u + 1]));
                    if (sub == 0) p.ml[(size_t)(it.kvh * p.G + hrow) * p.max_items + item] = make_float2(m, l);
                }
            } else if (!ok && lane == 0) {
                *abort_gen = 1;
                atomicExch(p.status, DASH_ERR_TIMEOUT);
            }
        }
        tc_fence_before();
        __syncthreads();                      // end of the item: O read out, every tile buffer free
        blk0 += (uint32_t)nblk;
        ++items_done;
        loaded = false;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kDecTmemCols);
    }
}

// The merge of the key splits, spread over the whole machine.  A unit is 32 output columns of one (sequence, query head); it goes to a
// group of K warps (K = 1, 2, 4 or 8: as many as there are warps per unit, so that few units with many splits and many units with
// few splits both fill the SMs).  Every warp of the group loads the splits' (m, l) pairs, lane = split (they lie next to each other:
// coalesced), and forms the common maximum, the splits' weights and the denominator; then it sums its share of the splits, lane =
// column, with the weights handed round by shuffles.  All loads of a unit go out before the first is waited for; the group meets in
// shared memory.
constexpr int kMergeThreads = 256;
struct MergeParams {
    const float* partial; const float2* ml; int max_items;
    const int2* seg;            // with a plan: first item and number of items of every (sequence, KV head); else the CTAs plan for themselves
    const int32_t* cu; int S, target, Hq, Hkv, G;
    float scale_log2, scale;
    __nv_bfloat16* out; int64_t ldo; float* lse;
};
template <int D, int K>
__device__ __forceinline__ void decode_merge_units(const MergeParams& p, const SelfPlan& sp, float (*s_acc)[32]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = kMergeThreads / 32, CH = D / 32;
    constexpr int B = 32, ML = B * K / 32;               // splits of one round: B per warp, their (m, l) in ML registers per lane
    const int n_units = p.S * p.Hq * CH;
    const int sub = warp % K;
    const size_t stride = (size_t)kDecRows * D;
    const int u = (int)blockIdx.x * (NW / K) + warp / K;      // (there are as many groups as units at least)
    if (u >= n_units) return;
    const int ch = u % CH, hd = (u / CH) % p.Hq, s = u / (CH * p.Hq);
    const int kvh = hd / p.G, row = hd % p.G;
    int first, cnt;
    if (!p.seg) { cnt = sp.per[s]; first = sp.first[s] + kvh * cnt; }
    else { const int2 sg = p.seg[s * p.Hkv + kvh]; first = sg.x; cnt = sg.y; }
    const float* base = p.partial + ((size_t)first * kDecRows + row) * D + ch * 32 + lane;
    const float2* mlb = p.ml + (size_t)hd * p.max_items + first;
    float dv[B];
    float2 ml[ML];
#pragma unroll
    for (int b = 0; b < B; ++b) { const int i = sub + b * K; dv[b] = (i < cnt) ? __ldcg(base + i * stride) : 0.f; }
#pragma unroll
    for (int j = 0; j < ML; ++j) { const int i = lane + 32 * j; ml[j] = (i < cnt) ? __ldcg(mlb + i) : make_float2(-INFINITY, 0.f); }
    float mx = -INFINITY;
#pragma unroll
    for (int j = 0; j < ML; ++j) mx = fmaxf(mx, ml[j].x);
    for (int i = lane + 32 * ML; i < cnt; i += 32) mx = fmaxf(mx, __ldcg(mlb + i).x);          // more than B * K splits: further rounds
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float ls = 0.f;
#pragma unroll
    for (int j = 0; j < ML; ++j) {
        ml[j].x = exp2f((ml[j].x - mx) * p.scale_log2);     // the split's weight (0 where there is no split)
        ls = fmaf(ml[j].x, ml[j].y, ls);
    }
    for (int i = lane + 32 * ML; i < cnt; i += 32) { const float2 v = __ldcg(mlb + i); ls = fmaf(exp2f((v.x - mx) * p.scale_log2), v.y, ls); }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, o);
    float acc = 0.f;
#pragma unroll
    for (int b = 0; b < B; ++b) acc = fmaf(__shfl_sync(0xffffffffu, ml[(b * K) / 32].x, (sub + b * K) & 31), dv[b], acc);
    for (int i = sub + B * K; i < cnt; i += K) acc = fmaf(exp2f((__ldcg(mlb + i).x - mx) * p.scale_log2), __ldcg(base + i * stride), acc);
    if (K > 1) {
        s_acc[warp][lane] = acc;
        asm volatile("bar.sync %0, %1;" ::"r"(1 + warp / K), "n"(K * 32) : "memory");
        if (sub == 0) {
            acc = 0.f;
#pragma unroll
            for (int j = 0; j < K; ++j) acc += s_acc[warp + j][lane];
        }
    }
    if (sub == 0) {
        const float v = cnt > 0 ? acc / ls : 0.f;
        p.out[(int64_t)s * p.ldo + (int64_t)hd * D + ch * 32 + lane] = __float2bfloat16(v);
        if (p.lse && ch == 0 && lane == 0) p.lse[(int64_t)s * p.Hq + hd] = cnt > 0 ? mx * p.scale + logf(ls) : -INFINITY;
    }
}

// The same where there are more units than warps, that is few splits to a sequence and head: a warp takes the whole head, a lane D / 32 neighbouring
// columns, so that each warp goes through its loads once instead of two or three times.
template <int D>
__device__ __forceinline__ void decode_merge_heads(const MergeParams& p, const SelfPlan& sp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = kMergeThreads / 32, W = D / 32, B = 8;           // B: splits whose loads are in flight at a time
    const size_t stride = (size_t)kDecRows * D;
    struct alignas(4 * W) Cols { float v[W]; };
    for (int u = (int)blockIdx.x * NW + warp; u < p.S * p.Hq; u += (int)gridDim.x * NW) {
        const int hd = u % p.Hq, s = u / p.Hq, kvh = hd / p.G, row = hd % p.G;
        int first, cnt;
        if (!p.seg) { cnt = sp.per[s]; first = sp.first[s] + kvh * cnt; }
        else { const int2 sg = p.seg[s * p.Hkv + kvh]; first = sg.x; cnt = sg.y; }
        const float* base = p.partial + ((size_t)first * kDecRows + row) * D + lane * W;
        const float2* mlb = p.ml + (size_t)hd * p.max_items + first;
        auto fetch = [&](int i) {
            Cols c;
            if (W == 4) { const float4 t = __ldcg(reinterpret_cast<const float4*>(base + i * stride)); c.v[0] = t.x; c.v[1] = t.y; c.v[W - 2] = t.z; c.v[W - 1] = t.w; }
            else { const float2 t = __ldcg(reinterpret_cast<const float2*>(base + i * stride)); c.v[0] = t.x; c.v[1] = t.y; }
            return c;
        };
        Cols dv[B];
#pragma unroll
        for (int b = 0; b < B; ++b)
            if (b < cnt) dv[b] = fetch(b);
        float2 ml = lane < cnt ? __ldcg(mlb + lane) : make_float2(-INFINITY, 0.f);
        float mx = ml.x;
        for (int i = lane + 32; i < cnt; i += 32) mx = fmaxf(mx, __ldcg(mlb + i).x);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        float ls = 0.f, acc[W];
#pragma unroll
        for (int e = 0; e < W; ++e) acc[e] = 0.f;
        for (int i0 = 0; i0 < cnt; i0 += 32) {                          // 32 splits' weights at a time, lane = split
            if (i0 > 0) ml = i0 + lane < cnt ? __ldcg(mlb + i0 + lane) : make_float2(-INFINITY, 0.f);
            const float wgt = exp2f((ml.x - mx) * p.scale_log2);        // 0 where there is no split
            ls = fmaf(wgt, ml.y, ls);
            for (int j0 = 0; j0 < min(32, cnt - i0); j0 += B) {
                if (i0 + j0 > 0) {
#pragma unroll
                    for (int b = 0; b < B; ++b)
                        if (i0 + j0 + b < cnt) dv[b] = fetch(i0 + j0 + b);
                }
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    const float w = __shfl_sync(0xffffffffu, wgt, j0 + b);
                    if (i0 + j0 + b < cnt) {
#pragma unroll
                        for (int e = 0; e < W; ++e) acc[e] = fmaf(w, dv[b].v[e], acc[e]);
                    }
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, o);
#pragma unroll
        for (int e = 0; e < W; ++e) acc[e] = cnt > 0 ? acc[e] / ls : 0.f;
        __nv_bfloat16* dst = p.out + (int64_t)s * p.ldo + (int64_t)hd * D + lane * W;
        if (W == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16(acc[0], acc[1]), pack_bf16(acc[W - 2], acc[W - 1]));
        else *reinterpret_cast<uint32_t*>(dst) = pack_bf16(acc[0], acc[1]);
        if (p.lse && lane == 0) p.lse[(int64_t)s * p.Hq + hd] = cnt > 0 ? mx * p.scale + logf(ls) : -INFINITY;
    }
}

template <int D>
__global__ void __launch_bounds__(kMergeThreads)
decode_merge_kernel(const MergeParams p) {
    __shared__ SelfPlan sp;
    __shared__ float s_acc[kMergeThreads / 32][32];
    pdl_launch_dependents();
    // started while the decode kernel runs, which had waited for all in front of it before it let this one start: the boundaries stand
    if (!p.seg) self_plan_build(sp, p.cu, p.S, p.Hkv, p.target);
    pdl_wait();                              // the decode kernel's partial results are complete from here on
    // warps per unit: as many as the machine has per unit, at most the CTA's eight
    const long long n_units = (long long)p.S * p.Hq * (D / 32), warps = (long long)gridDim.x * (kMergeThreads / 32);
    if (n_units * 16 <= warps) decode_merge_units<D, 8>(p, sp, s_acc);
    else if (n_units * 8 <= warps) decode_merge_units<D, 4>(p, sp, s_acc);
    else if (n_units * 4 <= warps) decode_merge_units<D, 2>(p, sp, s_acc);
    else if (n_units <= warps) decode_merge_units<D, 1>(p, sp, s_acc);
    else decode_merge_heads<D>(p, sp);
}

static int decode_max_items(int S, int Hkv) { return 4 * sm_count() + S * Hkv; }

size_t decode_ws_bytes(int64_t n, int S, int Hq, int Hkv, int D) {
    (void)n; (void)Hq;
    const size_t items = (size_t)decode_max_items(S, Hkv);
    return 256 + align_up(items * sizeof(DecItem), 256) + align_up((size_t)S * Hkv * sizeof(int2), 256) + align_up((size_t)S * sizeof(int), 256) +
           align_up(items * kDecRows * (size_t)D * sizeof(float), 256) + align_up(items * (size_t)Hq * sizeof(float2), 256);
}

// bf16 tensor [rows, heads, D]: box = 64 x box_heads x box_rows, 128-byte swizzle
static int make_map_heads_box(CUtensorMap* map, const void* base, int64_t rows, int heads, int D, int64_t ld, int box_heads, int box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return DASH_ERR_CUDA;
    cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)heads, (cuuint64_t)rows};
    cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)ld * 2};
    cuuint32_t box[3] = {64, (cuuint32_t)box_heads, (cuuint32_t)box_rows};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? DASH_OK : DASH_ERR_CUDA;
}

template <int D, bool SELF>
static int launch_decode(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, const DecParams& p, int box_heads, int grid,
                         cudaStream_t st) {
    const int smem = DecSmem<D>::kLaunch;
    static std::atomic<uint64_t> configured{0};
    if (!set_max_smem_once(decode_kernel<D, SELF>, smem, configured)) return DASH_ERR_CUDA;
    return launch_pdl(decode_kernel<D, SELF>, grid, kDecThreads, (size_t)smem, st, mq, mk, mv, p, box_heads) == cudaSuccess ? DASH_OK : DASH_ERR_CUDA;
}

}  // namespace dash

using namespace dash;

extern "C" int dash_decode_attention(const void* q, const void* Kc, const void* Vc, void* out, float* lse,
                                     int64_t ldq, int64_t ldk, int64_t ldv, int64_t ldo,
                                     const int32_t* cu_seqlens, int S, int64_t n, int Hq, int Hkv, int D, float scale,
                                     dash_dtype dt, void* ws, size_t ws_bytes, void* stream) {
    if (n < 0 || S < 1 || Hq < 1 || Hkv < 1 || !cu_seqlens) return DASH_ERR_INVALID_ARG;
    if (dt != DASH_F32 && dt != DASH_BF16) return DASH_ERR_INVALID_ARG;
    if (dt != DASH_BF16) return DASH_ERR_UNSUPPORTED;                 // the cache is read as stored: bf16 only
    if (D != 64 && D != 128) return DASH_ERR_UNSUPPORTED;
    if (Hq % Hkv) return DASH_ERR_INVALID_ARG;
    const int G = Hq / Hkv;
    if (G > kDecRows) return DASH_ERR_UNSUPPORTED;
    if (n > 0x7fffffffLL || S > 0x7fffffff / (Hq * 4)) return DASH_ERR_INVALID_ARG;      // the merge counts its units in an int
    if (!q || !out || (n > 0 && (!Kc || !Vc))) return DASH_ERR_INVALID_ARG;
    if (ldq < (int64_t)Hq * D || ldo < (int64_t)Hq * D || ldk < (int64_t)Hkv * D || ldv < (int64_t)Hkv * D) return DASH_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(out) || (n > 0 && (!aligned16(Kc) || !aligned16(Vc)))) return DASH_ERR_INVALID_ARG;
    if ((ldq * 2) % 16 || (ldk * 2) % 16 || (ldv * 2) % 16 || (ldo * 2) % 16) return DASH_ERR_INVALID_ARG;
    if (!(scale > 0.f)) return DASH_ERR_INVALID_ARG;
    if (!ws || ((uintptr_t)ws % 256) || ws_bytes < decode_ws_bytes(n, S, Hq, Hkv, D)) return DASH_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    const int max_items = decode_max_items(S, Hkv);
    char* w = (char*)ws;
    DecItem* plan = (DecItem*)(w + 256);
    int2* seg = (int2*)(w + 256 + align_up((size_t)max_items * sizeof(DecItem), 256));
    int* seq_first = (int*)((char*)seg + align_up((size_t)S * Hkv * sizeof(int2), 256));
    float* partial = (float*)((char*)seq_first + align_up((size_t)S * sizeof(int), 256));
    float2* ml = (float2*)((char*)partial + align_up((size_t)max_items * kDecRows * D * sizeof(float), 256));
    const bool self_plan = S <= kSelfPlanSeqs;
    const int target = 4 * sm_count();        // twice the CTAs: items that the plan kernel aims at, bound of the lengths that self_plan_build looks at
    if (!self_plan) {
        decode_plan_kernel<<<1, 256, 0, st>>>(cu_seqlens, S, Hkv, target, plan, seg, (int*)(w + 4), (unsigned int*)w, max_items, seq_first);
        DASH_CUDA_TRY(cudaGetLastError());
    }
    const float scale_log2 = scale * 1.4426950408889634f;
    if (n > 0) {
        CUtensorMap mq, mk, mv;
        int rc;
        const int box_heads = Hq < kDecRows ? Hq : kDecRows;
        if ((rc = make_map_heads_box(&mq, q, S, Hq, D, ldq, box_heads, 1)) != DASH_OK) return rc;
        if ((rc = make_map_heads_box(&mk, Kc, n, Hkv, D, ldk, 1, kDecBN)) != DASH_OK) return rc;
        if ((rc = make_map_heads_box(&mv, Vc, n, Hkv, D, ldv, 1, kDecBN)) != DASH_OK) return rc;
        DecParams p;
        p.cu = cu_seqlens; p.S = S; p.Hq = Hq; p.Hkv = Hkv; p.G = G;
        p.scale = scale; p.scale_log2 = scale_log2;
        p.partial = partial; p.ml = ml; p.max_items = max_items; p.plan = self_plan ? nullptr : plan; p.n_items = (const int*)(w + 4); p.ticket = (unsigned int*)w;
        p.target = target;
        p.status = status_word_ptr();
        if (!p.status) return DASH_ERR_CUDA;
        int grid = 2 * sm_count();
        if (grid > max_items) grid = max_items;
        if (self_plan) rc = D == 128 ? launch_decode<128, true>(mq, mk, mv, p, box_heads, grid, st) : launch_decode<64, true>(mq, mk, mv, p, box_heads, grid, st);
        else rc = D == 128 ? launch_decode<128, false>(mq, mk, mv, p, box_heads, grid, st) : launch_decode<64, false>(mq, mk, mv, p, box_heads, grid, st);
        if (rc != DASH_OK) return rc;
    }
    MergeParams mp;
    mp.partial = partial; mp.ml = ml; mp.max_items = max_items; mp.seg = self_plan ? nullptr : seg;
    mp.cu = cu_seqlens; mp.S = S; mp.target = target; mp.Hq = Hq; mp.Hkv = Hkv; mp.G = G;
    mp.scale_log2 = scale_log2; mp.scale = scale;
    mp.out = (__nv_bfloat16*)out; mp.ldo = ldo; mp.lse = lse;
    // one warp per unit at least, never more CTAs than SMs
    const long long units = (long long)S * Hq * (D / 32);
    long long mgrid = (units * 8 + kMergeThreads / 32 - 1) / (kMergeThreads / 32);
    if (mgrid > sm_count()) mgrid = sm_count();
    if (mgrid < 1) mgrid = 1;
    if (n == 0) {                             // no decode kernel in front that has waited for what writes the boundaries: in plain stream order
        if (D == 128) decode_merge_kernel<128><<<(int)mgrid, kMergeThreads, 0, st>>>(mp);
        else decode_merge_kernel<64><<<(int)mgrid, kMergeThreads, 0, st>>>(mp);
        DASH_CUDA_TRY(cudaGetLastError());
        return DASH_OK;
    }
    if (D == 128) DASH_CUDA_TRY(launch_pdl(decode_merge_kernel<128>, (int)mgrid, kMergeThreads, 0, st, mp));
    else DASH_CUDA_TRY(launch_pdl(decode_merge_kernel<64>, (int)mgrid, kMergeThreads, 0, st, mp));
    return DASH_OK;
}

extern "C" int dash_testing_decode_smem_bytes(int D) {
    return D == 128 ? DecSmem<128>::kLaunch + (int)sizeof(SelfPlan) : D == 64 ? DecSmem<64>::kLaunch + (int)sizeof(SelfPlan) : -1;
}
