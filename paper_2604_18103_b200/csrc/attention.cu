// Causal grouped-query attention over a packed (varlen) batch of active tokens,
// on tcgen05 tensor cores with TMEM accumulators, operands staged by TMA.
//
// Work item: two neighbouring tiles of 128 query rows, or one (a sequence's odd tile; every tile of a call with few: attention_in_pairs), of one head of
// one sequence.  A plan lists the items that exist (from cu_seqlens, on the device), heaviest first; persistent CTAs, one per SM, take them
// by ticket, so that no CTA is spent on query tiles that a shorter sequence does not have.
// Thread roles: warps 0-3 and 4-7 are the softmax of tile 0 and of tile 1 (thread <-> query row <-> TMEM lane), warp 8 takes the items and
// loads their tiles (with warp 11, where rows are fetched by index), a thread of warp 9 issues the scores, one of warp 10 the products.
// Items of one tile take tile 0 and tile 1 in turn, so that one item's start overlaps the end of the one before it.
//
// Per key block j (128 keys) and tile x, with K_j and V_j in shared memory for both tiles:
//   S = Q_x K_j^T  (SS MMA, fp32 in TMEM)  ->  softmax warps of x: scores into registers, buffer handed back, mask, maximum, exp2, row
//   sum, P_x (bf16) into TMEM, O_x rescaled if the reference moved  ->  O_x += P_x V_j  (TS MMA: A operand read from TMEM)
// TMEM holds O of both tiles, P of both tiles and ONE score buffer (128 + 128 + 64 + 64 + 128 columns).  The scores are in it only until
// a tile's threads have loaded them, so the tiles take turns with it, and the next block's scores of a tile are made while its
// exponentials of this block are still being formed: neither the score nor the product is on the softmax's chain.  Where S and P
// share columns (one tile per CTA, two CTAs per SM, each a chain score -> softmax -> product -> next score) a key block of a tile took
// 1714 to 1800 cycles of an SM, here 1350; K and V come through shared memory once for two tiles.
// Heads of 128, 28 / 4, one B200, that form and this one, us a call: 8192 tokens 411 / 351 alone, 450 / 390 in a loop at the power cap (1.65 GHz), 26 214 tokens 4400 / 3920
// (1256 TFLOP/s), 5 sequences of 1337 94 / 72, 200 of 100 157 / 90.  What bounds it: per pair of tiles and block 2700 cycles, of which a softmax warp
// waits 200 for its scores, loads 130, looks for the maximum 385, forms exponentials 1660 (2 x 1024 cycles of the MUFU are the floor of a
// sub-partition, 2048 cycles that of the tensor pipe).
// Causal tile skipping: a query tile only visits key blocks 0..its own index.
//
// The kernel is launched to start while the kernel in front of it in the stream drains (barriers, TMEM and descriptor prefetch are
// set up before griddepcontrol.wait).  A second instantiation (GATHER) takes the query rows -- and, optionally, the key / value
// rows -- of the packed set by index from full-length tensors (TMA gather4 loads) instead of from packed copies.
#include <math.h>

#include "common.cuh"
#include "prologue.cuh"
#include "sm100_ptx.cuh"

namespace dash {

using namespace ptx;

EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        fn = (EncodeTiledFn)p;
    }
    return fn;
}

int make_map_rows_heads(CUtensorMap* map, const void* base, int64_t rows, int heads, int D, int64_t ld, int box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return DASH_ERR_CUDA;
    cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)heads, (cuuint64_t)rows};
    cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)ld * 2};
    cuuint32_t box[3] = {64, 1, (cuuint32_t)box_rows};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? DASH_OK : DASH_ERR_CUDA;
}

// bf16 tensor [rows, cols] (cols = heads * D), box = 64 columns of one row: the map of the four-row gather loads
int make_map_rows_gather(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return DASH_ERR_CUDA;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {64, 1};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? DASH_OK : DASH_ERR_CUDA;
}

constexpr int kBM = 128;                 // query rows per tile
constexpr int kBN = 128;                 // keys per block
constexpr int kSoftWarps = 8;            // warps 0-3: rows of tile 0, warps 4-7: rows of tile 1
constexpr int kLoadWarp = 8, kScoreWarp = 9, kProductWarp = 10, kHelpWarp = 11;
constexpr int kAttnThreads = 384;         // three warpgroups: two of softmax, one of the rest
// Registers: 384 threads x 168 at launch; the third warpgroup gives back what the softmax takes.
constexpr int kSoftRegs = 208, kOtherRegs = 80;
static_assert(2 * kSoftRegs + kOtherRegs <= 3 * 168, "a split above the launch's registers would wait for good");
constexpr long long kWaitCycles = 4000000000LL;   // ~2 s: a wait that long is reported, not retried
constexpr uint32_t kTmemCols = 512;

struct AttnParams {
    int Hq, Hkv;
    float scale_log2;       // softmax scale * log2(e)
    float scale;
    void* O;
    int64_t ldo;            // elements
    __nv_bfloat16* O16;     // OUT_F32: a bf16 copy of O as well ([n, Hq, D]), or null
    float* lse;             // [Hq, n] or null
    int64_t n;
    int* status;
    const int4* plan;           // (1: a pair of tiles, highest query tile, first row, end row of the sequence) of every item group, heaviest first; Hq items (heads) per entry
    const int* n_items;         // device: entries * Hq
    int64_t max_entries;        // entries that the plan has room for
    unsigned int* ticket;       // device: items handed out beyond the first one of every CTA
    const int32_t* idx;         // GATHER: packed row i is row idx[i] of the full-length Q (and of K, V unless kv_packed)
    int kv_packed;              // GATHER: K and V are packed already ([n, Hkv, D], tiled loads); only Q is fetched by index
};

// ---- plan kernel of a call that is not part of a block step ----
constexpr int kPlanThreads = 256;
__global__ void __launch_bounds__(kPlanThreads)
attention_plan_kernel(const int32_t* __restrict__ cu, int S, int Hq, int sms, int4* __restrict__ plan, int* __restrict__ n_items,
                      unsigned int* __restrict__ ticket, int64_t max_entries) {
    pdl_launch_dependents();
    pdl_wait();
    attention_plan_items<kPlanThreads>(cu, S, Hq, sms, plan, n_items, ticket, max_entries);
}

constexpr int kKSlots = 3, kVSlots = 2, kRecords = 4;      // rings of K tiles, V tiles and item records
template <int D>
struct AttnSmem {
    static constexpr int kTileBytes = kBM * D * 2;
    static constexpr int kQ = 0, kK = 2 * kTileBytes, kV = kK + kKSlots * kTileBytes, kBars = kV + kVSlots * kTileBytes;
    static constexpr int kTotal = kBars + 512;
    // one CTA per SM, whose TMEM columns it takes all: with heads of 64 the tiles alone would let a second one in
    static constexpr int kLaunch = kTotal + 1024 > 120 * 1024 ? kTotal + 1024 : 120 * 1024;
};

// Barriers of a CTA (8 bytes each, in this order behind the tiles): two per query tile or one per slot of a ring
enum AttnBar {
    kBarQFull = 0, kBarQFree = kBarQFull + 2, kBarKFull = kBarQFree + 2, kBarKFree = kBarKFull + kKSlots, kBarVFull = kBarKFree + kKSlots,
    kBarVFree = kBarVFull + kVSlots, kBarSFull = kBarVFree + kVSlots, kBarSFree = kBarSFull + 2, kBarPFull = kBarSFree + 2, kBarOFull = kBarPFull + 2,
    kBarItemFull = kBarOFull + 2, kBarItemFree = kBarItemFull + kRecords, kBarDrain = kBarItemFree + kRecords, kBarCount = kBarDrain + 2
};
// behind them: TMEM address, the flag of a role that has given up, item records
constexpr int kTmemSlot = 8 * kBarCount, kAbortFlag = kTmemSlot + 4, kRecordAt = kTmemSlot + 16;
static_assert(kRecordAt % 16 == 0 && kRecordAt + kRecords * 16 <= 512, "what AttnSmem keeps behind the tiles");
// An item: its sequence's first and end row, its highest query tile (-1: no more items), its head and the tiles 0 and 1 of the CTA that it takes, first .. last
struct AttnItem {
    int seq_a, seq_b, top, h, first, last;
    __device__ int4 pack() const { return make_int4(seq_a, seq_b, top, h << 2 | first << 1 | last); }
    __device__ explicit AttnItem(const int4& r) : seq_a(r.x), seq_b(r.y), top(r.z), h(r.w >> 2), first(r.w >> 1 & 1), last(r.w & 1) {}
    __device__ AttnItem(int a, int b, int t, int head, int lo, int hi) : seq_a(a), seq_b(b), top(t), h(head), first(lo), last(hi) {}
};

// A wait of a single thread, bounded in time and given up as soon as another role of the CTA has given up.
__device__ __forceinline__ bool attn_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (*abort_flag || clock64() - t0 > kWaitCycles) return false;
    return true;
}
// The same for a whole warp, with one answer for all lanes (tcgen05 loads and stores behind it need them together).
__device__ __forceinline__ bool attn_wait_warp(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const long long t0 = clock64();
    for (;;) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        if (__any_sync(0xffffffffu, *abort_flag != 0 || clock64() - t0 > kWaitCycles)) return false;
    }
}

// v[e] of lane i (of four neighbouring lanes) <-> v[i] of lane e
__device__ __forceinline__ void quad_transpose(uint4 (&v)[4], int lane) {
    auto swap_halves = [](uint4& a, uint4& b, bool up, int d) {        // the lanes with `up` send a and keep b, the others the other way round
        uint4 s = up ? a : b, r;
        r.x = __shfl_xor_sync(0xffffffffu, s.x, d); r.y = __shfl_xor_sync(0xffffffffu, s.y, d);
        r.z = __shfl_xor_sync(0xffffffffu, s.z, d); r.w = __shfl_xor_sync(0xffffffffu, s.w, d);
        if (up) a = r; else b = r;
    };
    const bool b0 = lane & 1, b1 = lane & 2;
    swap_halves(v[0], v[1], b0, 1); swap_halves(v[2], v[3], b0, 1);
    swap_halves(v[0], v[2], b1, 2); swap_halves(v[1], v[3], b1, 2);
}

// GATHER: Q, K and V are full-length [rows, heads * D] tensors and the packed active set is given by p.idx; tiles are fetched four
// rows per instruction (TMA gather4, issued by all lanes of the loading warp: lane l brings rows 4l .. 4l+3 of the tile), so the active rows
// of Q, K, V are never copied into packed buffers.  Everything else -- and the packed O -- is the same.
//
// Hand-overs.  A tile buffer, the score buffer, a P and an item record each come back through a "free" barrier before they are filled again; O of
// a tile is handed on by the P of its next product.  Loads, scores and products go through items, key blocks and tiles in one order.  Every waiter
// sees the phases of a barrier one by one, so none can overtake it, with one exception: a softmax warp waits for a V tile only where it
// has rows of it to clear, in the last block b of a sequence's last tile, and has to know that the tile before in that slot, of block b - 2, has
// arrived.  If the item has more blocks the warp has seen the product of b - 1 done, so that of b - 2 was issued.  If not, the warp waits for b - 2 to
// be given free, and can tell that phase from the one of b - 4: the load of b - 2 has waited for it, ahead of the item's record.
// (tests/test_attention_handover.py runs these roles and barriers through a model of them.)
template <int D, bool OUT_F32, bool GATHER>
__global__ void __launch_bounds__(kAttnThreads, 1)
attention_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                 const __grid_constant__ CUtensorMap mapV, const AttnParams p) {
    extern __shared__ uint8_t smem_raw[];
    using L = AttnSmem<D>;
    constexpr int KCH = D / 64;              // 64-element (128-byte) chunks along D
    constexpr int kChunkBytes = kBM * 128;   // one chunk: 128 rows x 128 B
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sQ = smem_base + L::kQ, sK = smem_base + L::kK, sV = smem_base + L::kV;
    const uint32_t bars = smem_base + L::kBars;
    auto bar = [&](int kind, uint32_t i) { return bars + 8u * ((uint32_t)kind + i); };
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t tmem_slot = bars + kTmemSlot;
    volatile uint32_t* tmem_slot_gen = reinterpret_cast<volatile uint32_t*>(smem_gen + L::kBars + kTmemSlot);
    volatile uint32_t* abort_gen = reinterpret_cast<volatile uint32_t*>(smem_gen + L::kBars + kAbortFlag);
    int4* const records = reinterpret_cast<int4*>(smem_gen + L::kBars + kRecordAt);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == kProductWarp) {
        if (lane == 0) {
            for (uint32_t x = 0; x < 2; ++x) {
                mbar_init(bar(kBarQFull, x), 1); mbar_init(bar(kBarQFree, x), 1); mbar_init(bar(kBarSFull, x), 1); mbar_init(bar(kBarSFree, x), 4);
                mbar_init(bar(kBarPFull, x), 4); mbar_init(bar(kBarOFull, x), 1); mbar_init(bar(kBarDrain, x), 1);
            }
            for (uint32_t i = 0; i < (uint32_t)kRecords; ++i) { mbar_init(bar(kBarItemFull, i), 1); mbar_init(bar(kBarItemFree, i), kSoftWarps + 2 + GATHER); }
            for (uint32_t i = 0; i < (uint32_t)kKSlots; ++i) { mbar_init(bar(kBarKFull, i), 1); mbar_init(bar(kBarKFree, i), 1); }
            for (uint32_t i = 0; i < (uint32_t)kVSlots; ++i) { mbar_init(bar(kBarVFull, i), 1); mbar_init(bar(kBarVFree, i), 1); }
            *abort_gen = 0;
            fence_barrier_init();
            fence_proxy_async_smem();
            prefetch_tensormap(&mapQ); prefetch_tensormap(&mapK); prefetch_tensormap(&mapV);
        }
        __syncwarp();
        tmem_alloc(tmem_slot, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // The kernel behind may set itself up from here on, when every CTA of this grid is on its SM and holds its TMEM: on SMs without one, as the register
    // file is full beside it, and on the others while this kernel drains.
    pdl_launch_dependents();
    pdl_wait();                                            // set-up done; from here on the kernel in front (plan, projection) has completed
    const uint32_t tmem = *tmem_slot_gen;
    const uint32_t tS = tmem;                              // | S 128 | P of tile 0: 64 | P of tile 1: 64 | O of tile 0: 128 | O of tile 1: 128 |
    auto tP = [&](int x) { return tmem + 128 + 64 * x; };
    auto tO = [&](int x) { return tmem + 256 + 128 * x; };
    const int G = p.Hq / p.Hkv;
    auto give_up = [&]() { *abort_gen = 1; atomicExch(p.status, DASH_ERR_TIMEOUT); };

    if (warp >= kSoftWarps) {
    reg_dec<kOtherRegs>();
    if (warp == kLoadWarp || (GATHER && warp == kHelpWarp)) {
        // ---- loads, and the hand-out of items: all lanes go along.  A fetch by index is shared by two warps, the loading one and its helper, which
        // go through the same tiles (the helper by the item records): a warp issues a gather4 of 512 bytes per 90 cycles, two of them twice that, as
        // two CTAs per SM did.  K and V by index, 28 / 4 heads of 128, us a call, two CTAs per SM / one CTA, one warp /
        // two warps: 8192 tokens 1231 / 1164 / 604, 100 sequences of 100 143 / 193 / 109; heads of 64, 8192 tokens 654 / 674 / 394. ----
        const bool helper = GATHER && warp == kHelpWarp;
        uint32_t k_fills = 0, v_fills = 0, items = 0, turn = 0, q_any = 0, q_par = 0;      // q_any, q_par: bit x = tile x was ever loaded, parity of its count
        const int n_items = *p.n_items;
        auto wait = [&](uint32_t b, uint32_t parity) { return attn_wait_warp(b, parity, abort_gen); };
        int seq_a = 0, seq_b = 0;
        // Tile of 128 packed rows starting at row0 into a buffer that has been given free.  By index: a lane brings rows 4 lane .. 4 lane + 3 of a
        // 64-column chunk, of two chunks each warp one, of one chunk each every second lane.
        auto load_tile = [&](uint32_t sT, const CUtensorMap* map, uint32_t full, bool used, uint32_t free, uint32_t parity, int head, int row0, bool by_index) {
            int r[4];
            const bool mine = KCH == 2 || (lane & 1) == (int)helper;
            if (GATHER && by_index && mine) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int pr = row0 + 4 * lane + k;                  // rows past the sequence's end: its last row again (masked / zeroed later)
                    r[k] = p.idx[pr < seq_b ? pr : seq_b - 1];
                }
            }
            if (used && !wait(free, parity)) return false;        // (a buffer's first load has nothing to wait for, and a wait takes its 60 to 100 cycles)
            if (lane == 0 && !helper) mbar_arrive_expect_tx(full, L::kTileBytes);
            if (GATHER && by_index) {
                __syncwarp();
                const int c = KCH == 2 ? (int)helper : 0;
                if (mine) tma_gather4(sT + c * kChunkBytes + lane * 512, map, full, head * D + c * 64, r[0], r[1], r[2], r[3]);
            } else if (lane == 0) {
#pragma unroll
                for (int c = 0; c < KCH; ++c) tma_load_3d(sT + c * kChunkBytes, map, full, c * 64, head, row0);
            }
            return true;
        };
        const bool kv_by_index = GATHER && !p.kv_packed;
        auto load_q = [&](int x, int head, int tile) {
            if (!load_tile(sQ + x * L::kTileBytes, &mapQ, bar(kBarQFull, x), (q_any >> x) & 1, bar(kBarQFree, x), ((q_par >> x) & 1) ^ 1, head, seq_a + tile * kBM, GATHER)) return false;
            q_any |= 1u << x; q_par ^= 1u << x;
            return true;
        };
        auto load_k = [&](int kvh, int j) {
            if (helper && !kv_by_index) return true;
            const uint32_t slot = k_fills % kKSlots;
            if (!load_tile(sK + slot * L::kTileBytes, &mapK, bar(kBarKFull, slot), k_fills >= kKSlots, bar(kBarKFree, slot), ((k_fills / kKSlots) & 1) ^ 1, kvh, seq_a + j * kBN, kv_by_index)) return false;
            ++k_fills;
            return true;
        };
        auto load_v = [&](int kvh, int j) {
            if (helper && !kv_by_index) return true;
            const uint32_t slot = v_fills % kVSlots;
            if (!load_tile(sV + slot * L::kTileBytes, &mapV, bar(kBarVFull, slot), v_fills >= kVSlots, bar(kBarVFree, slot), ((v_fills / kVSlots) & 1) ^ 1, kvh, seq_a + j * kBN, kv_by_index)) return false;
            ++v_fills;
            return true;
        };
        // Next item: its number, and then its plan entry (the sequence's bounds ride along); two round trips to L2, with loads in between.  The first
        // item is the CTA's own number, tickets count on from there, and its entry is fetched beside the number of items: one round trip instead of three
        // ahead of the first load (one sequence of 64 tokens, 28 / 4 heads of 128, 10.1 -> 9.5 us a call, with two CTAs per SM 9.0; two of 500 14.0 -> 13.4, 16.6).
        int item = (int)blockIdx.x, asked = 0;
        const int64_t at = item / p.Hq;
        int4 e = p.plan[at < p.max_entries ? at : 0];
        auto ask = [&]() { if (lane == 0 && !helper) asked = (int)(gridDim.x + atomicAdd(p.ticket, 1u)); };
        auto take = [&]() {
            if (helper) return;
            item = __shfl_sync(0xffffffffu, asked, 0);
            e = item < n_items ? p.plan[item / p.Hq] : make_int4(0, -1, 0, 0);
        };
        if (item >= n_items) e = make_int4(0, -1, 0, 0);
        bool ok = true;
        for (;;) {
            const uint32_t slot = items % kRecords;
            if (!helper) {
                // An item of one tile takes tile 0 and tile 1 of the CTA in turn (0 behind a pair, whose tile 0 ends first): its start overlaps the
                // end of the one before it, as it did with two CTAs per SM.  us a call, two CTAs of one tile / one CTA, every item in tile 1 / in
                // turn: 200 sequences of 100 tokens, 28 / 4 heads of 128 157 / 163 / 116, 32 / 8 heads of 64 120 / 146 / 103; 64 of 300, 28 / 4 175 / 148 / 133.
                const bool pair = e.x != 0;
                ok = items < kRecords || wait(bar(kBarItemFree, slot), ((items / kRecords) & 1) ^ 1);
                if (ok && lane == 0) {
                    records[slot] = AttnItem(e.z, e.w, e.y, item % p.Hq, pair ? 0 : (int)turn, pair ? 1 : (int)turn).pack();
                    mbar_arrive(bar(kBarItemFull, slot));
                }
                turn = pair ? 0 : turn ^ 1;
                __syncwarp();
            } else {
                ok = wait(bar(kBarItemFull, slot), (items / kRecords) & 1);
            }
            if (!ok) break;
            const AttnItem it(records[slot]);
            if (helper) {
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarItemFree, slot));
            }
            seq_a = it.seq_a; seq_b = it.seq_b;
            const int h = it.h, qt = it.top, kvh = h / G, nb = qt + 1, last = it.last;
            const bool pair = it.first < last;
            ++items;
            if (qt < 0) break;
            // in the order of use; the next item is asked for while this one's last tiles are waited for
            if (nb <= 2) ask();
            if (pair) ok = load_q(0, h, qt - 1);
            ok = ok && load_k(kvh, 0) && load_q(last, h, qt);
            for (int t = 1; t <= nb && ok; ++t) {
                if (nb > 2 && t == nb - 2) ask();
                if (t < nb) ok = load_k(kvh, t);
                ok = ok && load_v(kvh, t - 1);
            }
            if (!ok) break;
            take();
        }
        if (!ok && lane == 0) give_up();
        __syncwarp();
        // Nothing is left in flight: every tile has arrived and, unless a wait ran out, been given free by the products that read it.
        for (uint32_t i = 0; i < (uint32_t)kKSlots; ++i)
            if (k_fills > i) {
                const uint32_t use = (k_fills - 1 - i) / kKSlots;
                mbar_wait(bar(kBarKFull, i), use & 1, kWaitCycles);
                if (ok) mbar_wait(bar(kBarKFree, i), use & 1, kWaitCycles);
            }
        for (uint32_t i = 0; i < (uint32_t)kVSlots; ++i)
            if (v_fills > i) {
                const uint32_t use = (v_fills - 1 - i) / kVSlots;
                mbar_wait(bar(kBarVFull, i), use & 1, kWaitCycles);
                if (ok) mbar_wait(bar(kBarVFree, i), use & 1, kWaitCycles);
            }
        for (uint32_t x = 0; x < 2; ++x)
            if (q_any >> x & 1) {
                mbar_wait(bar(kBarQFull, x), ((q_par >> x) & 1) ^ 1, kWaitCycles);
                if (ok) mbar_wait(bar(kBarQFree, x), ((q_par >> x) & 1) ^ 1, kWaitCycles);
            }
    } else if (warp == kScoreWarp) {
        // ---- S = Q K_j^T of both tiles in turn into the one score buffer.  A thread of its own: a wait holds its thread for 60 to 100 cycles, in
        // which the tensor pipe runs on what the other one has issued. ----
        if (lane == 0) {
            constexpr uint32_t idesc_s = idesc_bf16_f32(kBM, kBN, false, false);
            uint32_t k_used = 0, items = 0, s_made = 0, q_used = 0;   // s_made, q_used: bit x = parity of tile x's count
            int holder = -1;                                      // tile whose scores the buffer holds
            bool ok = true;
            auto wait = [&](uint32_t b, uint32_t parity) { return attn_wait(b, parity, abort_gen); };
            while (ok) {
                const uint32_t slot = items % kRecords;
                if (!(ok = wait(bar(kBarItemFull, slot), (items / kRecords) & 1))) break;
                const AttnItem it(records[slot]);
                const int top = it.top, first = it.first, last = it.last;
                mbar_arrive(bar(kBarItemFree, slot));
                ++items;
                if (top < 0) break;
                for (int j = 0; j <= top && ok; ++j) {
                    const uint32_t ks = k_used % kKSlots;
                    ok = wait(bar(kBarKFull, ks), (k_used / kKSlots) & 1);
                    for (int x = j < top ? first : last; x <= last && ok; ++x) {        // (a pair's tile 0 has a block less)
                        if (j == 0) ok = wait(bar(kBarQFull, x), (q_used >> x) & 1);
                        if (ok && holder >= 0) ok = wait(bar(kBarSFree, holder), ((s_made >> holder) & 1) ^ 1);
                        if (!ok) break;
                        tc_fence_after();
                        const uint64_t dq = smem_desc_sw128(sQ + x * L::kTileBytes, 16, 1024), dk = smem_desc_sw128(sK + ks * L::kTileBytes, 16, 1024);
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk) {
                            const uint32_t off = ((kk >> 2) * kChunkBytes + (kk & 3) * 32) >> 4;
                            mma_ss(tS, dq + off, dk + off, idesc_s, kk > 0);
                        }
                        tc_commit(bar(kBarSFull, x));
                        s_made ^= 1u << x;
                        holder = x;
                        if (j == top - (last - x)) { tc_commit(bar(kBarQFree, x)); q_used ^= 1u << x; }
                    }
                    if (ok) tc_commit(bar(kBarKFree, ks));
                    ++k_used;
                }
            }
            if (!ok) {
                give_up();
                tc_commit(bar(kBarDrain, 0));
                mbar_wait(bar(kBarDrain, 0), 0, kWaitCycles);
            }
        }
    } else if (warp == kProductWarp) {
        // ---- O += P_j V_j of both tiles in turn ----
        if (lane == 0) {
            constexpr uint32_t idesc_o = idesc_bf16_f32(kBM, D, false, true);
            uint32_t v_used = 0, items = 0, p_used = 0;               // p_used: bit x = parity of tile x's count
            bool ok = true;
            auto wait = [&](uint32_t b, uint32_t parity) { return attn_wait(b, parity, abort_gen); };
            while (ok) {
                const uint32_t slot = items % kRecords;
                if (!(ok = wait(bar(kBarItemFull, slot), (items / kRecords) & 1))) break;
                const AttnItem it(records[slot]);
                const int top = it.top, first = it.first, last = it.last;
                mbar_arrive(bar(kBarItemFree, slot));
                ++items;
                if (top < 0) break;
                for (int j = 0; j <= top && ok; ++j) {
                    const uint32_t vs = v_used % kVSlots;
                    ok = wait(bar(kBarVFull, vs), (v_used / kVSlots) & 1);
                    const uint64_t dv = smem_desc_sw128(sV + vs * L::kTileBytes, kChunkBytes, 1024);
                    for (int x = j < top ? first : last; x <= last && ok; ++x) {        // (a pair's tile 0 has a block less)
                        ok = wait(bar(kBarPFull, x), (p_used >> x) & 1);
                        if (!ok) break;
                        p_used ^= 1u << x;
                        tc_fence_after();
#pragma unroll
                        for (int kk = 0; kk < kBN / 16; ++kk)
                            mma_ts(tO(x), tP(x) + kk * 8, dv + (uint32_t)((kk * 2048) >> 4), idesc_o, (j > 0) || (kk > 0));
                        tc_commit(bar(kBarOFull, x));
                    }
                    if (ok) tc_commit(bar(kBarVFree, vs));
                    ++v_used;
                }
            }
            if (!ok) {
                give_up();
                tc_commit(bar(kBarDrain, 1));
                mbar_wait(bar(kBarDrain, 1), 0, kWaitCycles);
            }
        }
    }
    } else {
        reg_inc<kSoftRegs>();
        // ---- softmax: thread <-> query row of tile x ----
        const int x = warp >> 2, row = tid & 127;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        uint32_t blocks = 0, items = 0, v_blocks = 0;             // blocks of this tile / key blocks of all items so far
        bool ok = true;
        auto wait = [&](uint32_t b, uint32_t parity) { return attn_wait_warp(b, parity, abort_gen); };
        while (ok) {
            const uint32_t slot = items % kRecords;
            if (!(ok = wait(bar(kBarItemFull, slot), (items / kRecords) & 1))) break;
            const AttnItem it(records[slot]);
            const int seq_a = it.seq_a, seq_b = it.seq_b, top = it.top, h = it.h, first = it.first, last = it.last;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarItemFree, slot));
            ++items;
            if (top < 0) break;
            const uint32_t v_first = v_blocks;
            v_blocks += (uint32_t)top + 1;
            if (x < first || x > last) continue;                  // the other tile's item
            const int qt = top - (last - x);                      // this tile; its key blocks are 0 .. qt
            const int len = seq_b - seq_a, q0 = qt * kBM;
            const bool row_valid = (q0 + row) < len;
            float m = -INFINITY, l = 0.f;
            for (int j = 0; j <= qt; ++j, ++blocks) {
                ok = wait(bar(kBarSFull, x), blocks & 1);
                if (!ok) break;
                tc_fence_after();
                uint32_t sreg[128];
#pragma unroll
                for (int c = 0; c < 4; ++c) tmem_ld32(tS + lane_base + c * 32, &sreg[c * 32]);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarSFree, x));    // the score buffer may take the next product
                const bool diag = (j == qt);
                if (diag) {
#pragma unroll
                    for (int c = 0; c < 128; ++c)
                        if (c > row) sreg[c] = 0xff800000u;       // -inf: keys after the query (and past the sequence end)
                }
                // four independent chains of three-input max
                float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
                for (int c = 0; c < 128; c += 8) {
                    mx0 = fmax3(mx0, __uint_as_float(sreg[c]), __uint_as_float(sreg[c + 1]));
                    mx1 = fmax3(mx1, __uint_as_float(sreg[c + 2]), __uint_as_float(sreg[c + 3]));
                    mx2 = fmax3(mx2, __uint_as_float(sreg[c + 4]), __uint_as_float(sreg[c + 5]));
                    mx3 = fmax3(mx3, __uint_as_float(sreg[c + 6]), __uint_as_float(sreg[c + 7]));
                }
                const float mx = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3));
                // The reference m of a row (exponentials are taken of s - m) moves only when a block's maximum is more than 2^8 above it: P up to
                // 2^8 has the same relative precision in bf16 and is harmless in the fp32 sums.  (Not much later either: of a row that one key dominates
                // P is 1, without rounding, once the reference has moved.)
                bool o_waited = (j == 0);
                if (j == 0) {
                    m = mx;                                       // finite: key 0 is visible to every query row
                } else {
                    const bool grow = (mx - m) * p.scale_log2 > 8.0f;
                    if (__any_sync(0xffffffffu, grow)) {
                        const float m_new = grow ? mx : m;
                        const float alpha = grow ? ex2((m - m_new) * p.scale_log2) : 1.0f;
                        ok = wait(bar(kBarOFull, x), (blocks - 1) & 1);
                        if (!ok) break;
                        o_waited = true;
                        tc_fence_after();
#pragma unroll 1
                        for (int c = 0; c < D / 8; ++c) {
                            uint32_t o[8];
                            tmem_ld8(tO(x) + lane_base + c * 8, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 8; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                            tmem_st8(tO(x) + lane_base + c * 8, o);
                        }
                        l *= alpha;
                        m = m_new;
                    }
                }
                const float2 sl2 = make_float2(p.scale_log2, p.scale_log2);
                const float msl = m * p.scale_log2;
                const float2 nm2 = make_float2(-msl, -msl);
                // scale-subtract and row sums on packed fp32 pairs (two lanes per FMA-pipe instruction); P is packed in place.  A row's sum is added
                // up per 64 keys, in four chains of 16 (A, B: the first 64, C, D: the rest): a chain of 32 loses more of what lies below 2^-24 of a
                // row's largest weight.  One loop over all of them: as two loops of 64 heads of 64 took 3 % longer (8192 tokens, 32 / 8: 350 us,
                // 342 as it is, 339 with chains of 32), heads of 128 the same.
                float2 sumA, sumB, sumC, sumD;
#pragma unroll
                for (int c = 0; c < 128; c += 4) {
                    const float2 xa = __ffma2_rn(make_float2(__uint_as_float(sreg[c]), __uint_as_float(sreg[c + 1])), sl2, nm2);
                    const float2 xb = __ffma2_rn(make_float2(__uint_as_float(sreg[c + 2]), __uint_as_float(sreg[c + 3])), sl2, nm2);
                    float2 pa, pb;
                    pa.x = ex2(xa.x);
                    pa.y = ex2(xa.y);
                    pb.x = ex2(xb.x);
                    pb.y = ex2(xb.y);
                    float2 &s0 = c < 64 ? sumA : sumC, &s1 = c < 64 ? sumB : sumD;
                    s0 = (c & 63) ? __fadd2_rn(s0, pa) : pa;
                    s1 = (c & 63) ? __fadd2_rn(s1, pb) : pb;
                    sreg[c >> 1] = pack_bf16(pa.x, pa.y);
                    sreg[(c >> 1) + 1] = pack_bf16(pb.x, pb.y);
                }
                const float2 sum = __fadd2_rn(__fadd2_rn(make_float2(sumA.x, sumC.x), make_float2(sumA.y, sumC.y)),
                                              __fadd2_rn(make_float2(sumB.x, sumD.x), make_float2(sumB.y, sumD.y)));
                // (waited for and stored behind all exponentials: a wait and a store between their halves cut the loop in two for the compiler, and a
                // pair's block took 5 % longer)
                if (!o_waited) {                                  // PV_{j-1} has read the P that is overwritten now
                    ok = wait(bar(kBarOFull, x), (blocks - 1) & 1);
                    if (!ok) break;
                    tc_fence_after();
                }
                tmem_st32(tP(x) + lane_base, &sreg[0]);
                tmem_st32(tP(x) + lane_base + 32, &sreg[32]);
                l += sum.x;
                l += sum.y;
                if (diag && x == last && q0 + (warp & 3) * 32 + 31 >= len) {
                    // keys past the end of the sequence (only its last tile meets them): their V rows may hold anything (another sequence, or
                    // never-written memory); zero them so 0 * garbage cannot make a NaN
                    const uint32_t vb = v_first + j, vs = vb % kVSlots, use = vb / kVSlots;
                    ok = (j > 0 || use == 0 || wait(bar(kBarVFree, vs), (use - 1) & 1)) && wait(bar(kBarVFull, vs), use & 1);
                    if (!ok) break;
                    if (j * kBN + row >= len) {
                        // 16 bytes at a time, neighbouring rows in other banks: with the same piece of every row the stores of a warp fell on four
                        // banks (200 sequences of 100 tokens, 28 / 4 heads of 128, 116 -> 103 us).  A loop: unrolled it cost heads of 64 2 %.
                        uint8_t* rowp = smem_gen + L::kV + vs * L::kTileBytes + row * 128;
#pragma unroll 1
                        for (int e = 0; e < 8; ++e) {
#pragma unroll
                            for (int c = 0; c < KCH; ++c)
                                *reinterpret_cast<uint4*>(rowp + c * kChunkBytes + ((e ^ row) & 7) * 16) = make_uint4(0, 0, 0, 0);
                        }
                        fence_proxy_async_smem();
                    }
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarPFull, x));
            }
            if (ok) ok = wait(bar(kBarOFull, x), (blocks - 1) & 1);
            if (!ok) break;
            tc_fence_after();
            const float inv = 1.0f / l;
            const int64_t grow = (int64_t)seq_a + q0 + row;
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {
                uint32_t o[32];
                tmem_ld32(tO(x) + lane_base + c * 32, o);
                tmem_wait_ld();
                if (OUT_F32) {
                    // as below, 16 columns at a time: 8 x 64 contiguous bytes a store, 8 x 32 of the bf16 copy (a row per lane: the results of a tile
                    // of heads of 64 took 2.3 us, 1.3 so)
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        uint4 v[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const uint32_t* s = &o[half * 16 + 4 * e];
                            v[e].x = __float_as_uint(__uint_as_float(s[0]) * inv); v[e].y = __float_as_uint(__uint_as_float(s[1]) * inv);
                            v[e].z = __float_as_uint(__uint_as_float(s[2]) * inv); v[e].w = __float_as_uint(__uint_as_float(s[3]) * inv);
                        }
                        quad_transpose(v, lane);
                        const int col = h * D + c * 32 + half * 16 + (lane & 3) * 4;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int r = q0 + (warp & 3) * 32 + (lane & ~3) + e;
                            if (r >= len) continue;
                            const int64_t at = (int64_t)seq_a + r;
                            st_v4(reinterpret_cast<float*>(p.O) + at * p.ldo + col, v[e]);
                            if (p.O16)
                                *reinterpret_cast<uint2*>(p.O16 + at * p.Hq * D + col) =
                                    make_uint2(pack_bf16(__uint_as_float(v[e].x), __uint_as_float(v[e].y)), pack_bf16(__uint_as_float(v[e].z), __uint_as_float(v[e].w)));
                        }
                    }
                } else {
                    // 64 bytes of a row per lane; four lanes turn their 4 x 4 pieces of 16 bytes round, so that each stores one piece of each of
                    // their four rows: a store of the warp writes 8 x 64 contiguous bytes instead of 32 x 16 (32 lines a store held a tile's
                    // results for 4200 cycles).  Not unrolled over c: code that runs once an item waits for its instructions.
                    // 2728 tokens 61.2 -> 58.3 us, 5 of 1337 90.5 -> 87.2, 64 of 300 168 -> 160, 8192 412 -> 407.
                    uint4 v[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        v[e].x = pack_bf16(__uint_as_float(o[8 * e]) * inv, __uint_as_float(o[8 * e + 1]) * inv);
                        v[e].y = pack_bf16(__uint_as_float(o[8 * e + 2]) * inv, __uint_as_float(o[8 * e + 3]) * inv);
                        v[e].z = pack_bf16(__uint_as_float(o[8 * e + 4]) * inv, __uint_as_float(o[8 * e + 5]) * inv);
                        v[e].w = pack_bf16(__uint_as_float(o[8 * e + 6]) * inv, __uint_as_float(o[8 * e + 7]) * inv);
                    }
                    quad_transpose(v, lane);
                    __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(p.O) + (int64_t)h * D + c * 32 + (lane & 3) * 8;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int r = q0 + (warp & 3) * 32 + (lane & ~3) + e;
                        if (r < len) st_v4(dst + ((int64_t)seq_a + r) * p.ldo, v[e]);
                    }
                }
            }
            tc_fence_before();                                    // O has been read: ahead of the hand-over of the next item's first P
            if (row_valid && p.lse) p.lse[(int64_t)h * p.n + grow] = m * p.scale + logf(l);
        }
        if (!ok && lane == 0) give_up();
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == kProductWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

__global__ void f32_to_bf16_rows_kernel(const float* __restrict__ src, int64_t ld_src, __nv_bfloat16* __restrict__ dst, int64_t ld_dst,
                                        int64_t rows, int cols) {
    const int64_t total = rows * (cols / 4);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = i / (cols / 4);
        int c = (int)(i % (cols / 4)) * 4;
        float4 v = *reinterpret_cast<const float4*>(src + r * ld_src + c);
        uint2 o = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
        *reinterpret_cast<uint2*>(dst + r * ld_dst + c) = o;
    }
}

int launch_f32_to_bf16(const float* src, int64_t ld_src, void* dst, int64_t ld_dst, int64_t rows, int64_t cols, cudaStream_t st) {
    if (rows <= 0 || cols <= 0) return DASH_OK;
    int64_t grid = (rows * (cols / 4) + 255) / 256, cap = (int64_t)sm_count() * 8;
    if (grid > cap) grid = cap;
    f32_to_bf16_rows_kernel<<<(int)grid, 256, 0, st>>>(src, ld_src, (__nv_bfloat16*)dst, ld_dst, rows, (int)cols);
    return cudaGetLastError() == cudaSuccess ? DASH_OK : DASH_ERR_CUDA;
}

// workspace: [0,256) ticket + item count; then the plan (one int4 per existing (sequence, query tile));
// then, for fp32 tensors, their bf16 copies
static size_t plan_entries(int64_t n, int S) { return (size_t)(n / kBM) + (size_t)S + 1; }
static size_t plan_bytes(int64_t n, int S) { return align_up(plan_entries(n, S) * sizeof(int4), 256); }
size_t attention_ws_bytes(int64_t n, int S, int Hq, int Hkv, int D, dash_dtype dt) {
    size_t b = 256 + plan_bytes(n, S);
    if (dt != DASH_BF16) b += align_up((size_t)n * (Hq + 2 * Hkv) * D * 2, 256);
    return b;
}

template <int D, bool OUT_F32, bool GATHER>
static int launch_attention(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, const AttnParams& p, int grid, cudaStream_t st) {
    using L = AttnSmem<D>;
    const int smem = L::kLaunch;
    static std::atomic<uint64_t> configured{0};
    if (!set_max_smem_once(attention_kernel<D, OUT_F32, GATHER>, smem, configured)) return DASH_ERR_CUDA;
    return launch_pdl(attention_kernel<D, OUT_F32, GATHER>, grid, kAttnThreads, (size_t)smem, st, mq, mk, mv, p) == cudaSuccess ? DASH_OK : DASH_ERR_CUDA;
}

// The item list of a call (see attention_plan_items) into the head of its workspace
static int attention_plan(const int32_t* cu_seqlens, int S, int64_t n, int Hq, void* ws, size_t ws_bytes, cudaStream_t st) {
    if (!cu_seqlens || S < 1 || n < 0 || n > 0x7fffffffLL || Hq < 1) return DASH_ERR_INVALID_ARG;
    if (n == 0) return DASH_OK;
    if (!ws || ((uintptr_t)ws % 256) || ws_bytes < 256 + plan_bytes(n, S)) return DASH_ERR_WORKSPACE;
    if ((int64_t)plan_entries(n, S) * Hq > 0x7fffffffLL) return DASH_ERR_UNSUPPORTED;
    return launch_pdl(attention_plan_kernel, 1, kPlanThreads, 0, st, cu_seqlens, S, Hq, sm_count(), (int4*)((char*)ws + 256), (int*)((char*)ws + 4), (unsigned int*)ws,
                      (int64_t)plan_entries(n, S)) == cudaSuccess ? DASH_OK : DASH_ERR_CUDA;
}

static int attention_impl(const void* Q, const void* K, const void* V, void* O, float* lse,
                          int64_t ldq, int64_t ldk, int64_t ldv, int64_t ldo,
                          const int32_t* cu_seqlens, int S, int64_t n, int64_t max_seqlen,
                          int Hq, int Hkv, int D, float scale, int causal, dash_dtype dt,
                          void* ws, size_t ws_bytes, void* stream, bool planned, const int32_t* idx = nullptr, int64_t n_full = 0,
                          bool kv_packed = false, void* O16 = nullptr) {
    if (n < 0 || S < 1 || max_seqlen < 0 || Hq < 1 || Hkv < 1 || !cu_seqlens) return DASH_ERR_INVALID_ARG;
    if (dt != DASH_F32 && dt != DASH_BF16) return DASH_ERR_INVALID_ARG;
    if (D != 64 && D != 128) return DASH_ERR_UNSUPPORTED;
    if (Hq % Hkv) return DASH_ERR_INVALID_ARG;
    if (causal != 1) return DASH_ERR_UNSUPPORTED;
    if (n > 0x7fffffffLL || max_seqlen > n) return DASH_ERR_INVALID_ARG;
    if (n == 0 || max_seqlen == 0) return DASH_OK;
    if (!Q || !K || !V || !O) return DASH_ERR_INVALID_ARG;
    const int es = (dt == DASH_BF16) ? 2 : 4;
    if (ldq < (int64_t)Hq * D || ldo < (int64_t)Hq * D || ldk < (int64_t)Hkv * D || ldv < (int64_t)Hkv * D) return DASH_ERR_INVALID_ARG;
    if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(O)) return DASH_ERR_INVALID_ARG;
    if ((ldq * es) % 16 || (ldk * es) % 16 || (ldv * es) % 16 || (ldo * es) % 16) return DASH_ERR_INVALID_ARG;
    if (!(scale > 0.f)) return DASH_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;

    const void *q = Q, *k = K, *v = V;
    int64_t lq = ldq, lk = ldk, lv = ldv;
    if (!ws || ((uintptr_t)ws % 256) || ws_bytes < attention_ws_bytes(n, S, Hq, Hkv, D, dt)) return DASH_ERR_WORKSPACE;
    if (idx && (dt != DASH_BF16 || n_full < 1 || n_full > 0x7fffffffLL)) return dt != DASH_BF16 ? DASH_ERR_UNSUPPORTED : DASH_ERR_INVALID_ARG;
    if (dt == DASH_F32) {
        __nv_bfloat16* qb = (__nv_bfloat16*)((char*)ws + 256 + plan_bytes(n, S));
        __nv_bfloat16* kb = qb + (size_t)n * Hq * D;
        __nv_bfloat16* vb = kb + (size_t)n * Hkv * D;
        if (!planned) {                          // (a planned call finds its copies there: the step's rotary pass wrote them)
            const int cap = sm_count() * 8;
            auto cvt = [&](const void* src, int64_t ld, __nv_bfloat16* dst, int cols) {
                int64_t total = n * (cols / 4);
                int grid = (int)((total + 255) / 256);
                if (grid > cap) grid = cap;
                f32_to_bf16_rows_kernel<<<grid, 256, 0, st>>>((const float*)src, ld, dst, cols, n, cols);
            };
            cvt(Q, ldq, qb, Hq * D); cvt(K, ldk, kb, Hkv * D); cvt(V, ldv, vb, Hkv * D);
            DASH_CUDA_TRY(cudaGetLastError());
        }
        q = qb; k = kb; v = vb;
        lq = (int64_t)Hq * D; lk = lv = (int64_t)Hkv * D;
    }
    CUtensorMap mq, mk, mv;
    int rc;
    if (idx) {
        if ((rc = make_map_rows_gather(&mq, q, n_full, (int64_t)Hq * D, lq)) != DASH_OK) return rc;
        if (kv_packed) {
            if ((rc = make_map_rows_heads(&mk, k, n, Hkv, D, lk, kBN)) != DASH_OK) return rc;
            if ((rc = make_map_rows_heads(&mv, v, n, Hkv, D, lv, kBN)) != DASH_OK) return rc;
        } else {
            if ((rc = make_map_rows_gather(&mk, k, n_full, (int64_t)Hkv * D, lk)) != DASH_OK) return rc;
            if ((rc = make_map_rows_gather(&mv, v, n_full, (int64_t)Hkv * D, lv)) != DASH_OK) return rc;
        }
    } else {
        if ((rc = make_map_rows_heads(&mq, q, n, Hq, D, lq, kBM)) != DASH_OK) return rc;
        if ((rc = make_map_rows_heads(&mk, k, n, Hkv, D, lk, kBN)) != DASH_OK) return rc;
        if ((rc = make_map_rows_heads(&mv, v, n, Hkv, D, lv, kBN)) != DASH_OK) return rc;
    }

    AttnParams p;
    p.Hq = Hq; p.Hkv = Hkv;
    p.scale = scale;
    p.scale_log2 = scale * 1.4426950408889634f;
    p.O = O; p.ldo = ldo; p.O16 = (__nv_bfloat16*)O16; p.lse = lse; p.n = n; p.idx = idx; p.kv_packed = kv_packed ? 1 : 0;
    p.status = status_word_ptr();
    if (!p.status) return DASH_ERR_CUDA;
    p.ticket = (unsigned int*)ws;
    p.n_items = (const int*)((char*)ws + 4);
    p.plan = (const int4*)((char*)ws + 256);
    p.max_entries = (int64_t)plan_entries(n, S);
    if (!planned && (rc = attention_plan(cu_seqlens, S, n, Hq, ws, ws_bytes, st)) != DASH_OK) return rc;
    // persistent CTAs, one per SM, never more than there can be items
    int64_t grid64 = (max_seqlen + kBM - 1) / kBM * Hq * S;
    if (grid64 > sm_count()) grid64 = sm_count();
    const int grid = (int)grid64;
    if (idx) return D == 128 ? launch_attention<128, false, true>(mq, mk, mv, p, grid, st) : launch_attention<64, false, true>(mq, mk, mv, p, grid, st);
    if (D == 128) return dt == DASH_F32 ? launch_attention<128, true, false>(mq, mk, mv, p, grid, st) : launch_attention<128, false, false>(mq, mk, mv, p, grid, st);
    return dt == DASH_F32 ? launch_attention<64, true, false>(mq, mk, mv, p, grid, st) : launch_attention<64, false, false>(mq, mk, mv, p, grid, st);
}

int attention_plan_ws(int S, int64_t n, int Hq, int Hkv, int D, dash_dtype dt, void* ws, size_t ws_bytes, AttnPlanWs* out) {
    if (!ws || ((uintptr_t)ws % 256) || ws_bytes < attention_ws_bytes(n, S, Hq, Hkv, D, dt)) return DASH_ERR_WORKSPACE;
    if ((int64_t)plan_entries(n, S) * Hq > 0x7fffffffLL) return DASH_ERR_UNSUPPORTED;
    char* w = (char*)ws;
    out->ticket = (unsigned int*)w; out->n_items = (int*)(w + 4); out->plan = (int4*)(w + 256);
    out->max_entries = (int64_t)plan_entries(n, S);
    out->sms = sm_count();
    out->q = out->k = out->v = nullptr;
    if (dt == DASH_F32) {
        out->q = (__nv_bfloat16*)(w + 256 + plan_bytes(n, S));
        out->k = out->q + (size_t)n * Hq * D;
        out->v = out->k + (size_t)n * Hkv * D;
    }
    return DASH_OK;
}

// same as dash_varlen_attention for a workspace whose item list (and copies) a kernel in front on this stream has filled in; O16: fp32
// tensors, a bf16 copy of O as well
int attention_planned(const void* Q, const void* K, const void* V, void* O, float* lse, int64_t ldq, int64_t ldk, int64_t ldv, int64_t ldo,
                      const int32_t* cu_seqlens, int S, int64_t n, int64_t max_seqlen, int Hq, int Hkv, int D, float scale, dash_dtype dt,
                      void* ws, size_t ws_bytes, cudaStream_t st, void* O16) {
    return attention_impl(Q, K, V, O, lse, ldq, ldk, ldv, ldo, cu_seqlens, S, n, max_seqlen, Hq, Hkv, D, scale, 1, dt, ws, ws_bytes, (void*)st, true,
                          nullptr, 0, false, O16);
}

}  // namespace dash

extern "C" int dash_varlen_attention(const void* Q, const void* K, const void* V, void* O, float* lse,
                                     int64_t ldq, int64_t ldk, int64_t ldv, int64_t ldo,
                                     const int32_t* cu_seqlens, int S, int64_t n, int64_t max_seqlen,
                                     int Hq, int Hkv, int D, float scale, int causal, dash_dtype dt,
                                     void* ws, size_t ws_bytes, void* stream) {
    return dash::attention_impl(Q, K, V, O, lse, ldq, ldk, ldv, ldo, cu_seqlens, S, n, max_seqlen, Hq, Hkv, D, scale, causal, dt, ws, ws_bytes,
                                stream, false);
}

extern "C" int dash_varlen_attention_indexed(const void* Q, const void* K, const void* V, void* O, float* lse,
                                             int64_t ldq, int64_t ldk, int64_t ldv, int64_t ldo,
                                             const int32_t* idx, int64_t n_full, int kv_packed,
                                             const int32_t* cu_seqlens, int S, int64_t n, int64_t max_seqlen,
                                             int Hq, int Hkv, int D, float scale, int causal, dash_dtype dt,
                                             void* ws, size_t ws_bytes, void* stream) {
    if ((!idx && n > 0) || (kv_packed != 0 && kv_packed != 1)) return DASH_ERR_INVALID_ARG;
    if (n > n_full) return DASH_ERR_INVALID_ARG;
    return dash::attention_impl(Q, K, V, O, lse, ldq, ldk, ldv, ldo, cu_seqlens, S, n, max_seqlen, Hq, Hkv, D, scale, causal, dt, ws, ws_bytes,
                                stream, false, idx, n_full, kv_packed != 0);
}
