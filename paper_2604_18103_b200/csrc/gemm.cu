// Projections of the block as persistent tcgen05 GEMMs: C[n, N] = A[n, K] W[K, N], bf16 operands, fp32 accumulation in
// TMEM, with the element-wise work that follows each projection done on the accumulators before anything is written:
//   PLAIN  : C = A W (bf16 or fp32 out; any N, K that keep rows 16-byte aligned: tiles past the edge of W or along K are
//            zero-filled by the loads, columns past N are not stored)   (down projection of the FFN; every projection of the
//            path that runs the norm, the rotary embedding and the residual as passes of their own; fp32 tensors, whose
//            operands are rounded to bf16 copies first)
//   ROPE   : Q | K | V = Hn Wqkv with the rotary embedding applied to the Q and K heads    (Eq. 1, inside Attn)
//   RESID  : U = O Wo is never stored: H~ = H + U goes straight to x_full[tok[row]], and the per-row partial sums of
//            u^2, h^2 and (h+u)^2 of this tile's columns go to a small buffer (the score of Eq. 2 and the next norm's row factor are
//            finished from them)
//   SWIGLU : one tile holds 128 gate and the matching 128 up columns: act = silu(g) * u      (FFN of Alg. 1)
// One CTA per SM, in clusters of two: a pair computes a 256 x 256 tile (256 x 128 where there are few, see gemm_narrow) with tcgen05.mma.cta_group::2 -- CTA r holds
// rows 128 r .. of the A tile and half r of the W tile's columns, so every SM loads only half of the W operand.  K in steps of 64
// through a TMA ring of 6 (8) stages; warp 0 of each CTA issues its loads (their bytes are counted on the pair's even CTA), warp 1 of
// the even CTA issues the MMAs and releases stages / hands over accumulators in both CTAs with multicast commits, warps 2-9
// of each CTA read their 128 accumulator rows (two TMEM buffers, so a tile's epilogue overlaps the next tile's MMAs).
//
// Epilogue.  A TMEM row belongs to a lane, a row of the output to 8 lanes: every warp turns its 32 x 32 fp32 (or 32 x 64 bf16) piece
// through 4 KB of shared memory of its own, so that the rows of H, x_full, C and the rotary table are touched in pieces of 32 to
// 128 contiguous bytes, and what an epilogue reads is asked for a piece ahead.  With a lane per row in the loads and stores too (and
// four warps) an epilogue took 23-30 thousand cycles (ROPE), 18-22 (RESID), 15 (SWIGLU), 7 (PLAIN) against 31 thousand of a
// 3584-deep tile's MMAs: the QKV projection waited for it at every tile (41.9 thousand cycles per tile), and the last tile's showed
// in every launch.  The fused epilogues' pieces of a tile come in loops: a launch with a tile per CTA runs their code once, and would
// wait for the instructions (PLAIN, with little code per piece, is unrolled).
#include <math.h>

#include "common.cuh"
#include "dash_testing.h"
#include "gemm.cuh"
#include "prologue.cuh"
#include "sm100_ptx.cuh"

namespace dash {

using namespace ptx;

constexpr int kGM = 128, kGN = 256, kGNarrow = 128, kGK = 64;    // kGM: rows per CTA (256 per pair); columns of a pair's tile
constexpr int kGABytes = kGM * kGK * 2;      // per CTA and stage
// tiles BN columns wide: bytes of a stage per CTA, stages of the ring (192 KB either way)
template <int BN> struct Ring { static constexpr int kStage = kGABytes + kGK * (BN / 2) * 2, kStages = BN == kGN ? 6 : 8; };
constexpr int kGRingBytes = Ring<kGN>::kStage * Ring<kGN>::kStages;
static_assert(kGRingBytes == Ring<kGNarrow>::kStage * Ring<kGNarrow>::kStages, "one size of shared memory");
constexpr int kGEpiWarps = 8;                // two per TMEM lane quarter, each with one half of the tile's columns
constexpr int kGThreads = 64 + 32 * kGEpiWarps;
constexpr int kGEpiBytes = 4096;             // staging per epilogue warp: 32 rows of 128 bytes
constexpr int kGGroup = 16;                  // tiles per group of the tile order
constexpr int kGSplitMaxRounds = 4;          // tiles may be cut along K where whole tiles take up to so many rounds
constexpr int kGSplitMaxParts = 4;           // parts of a tile, on the average
constexpr int kGSplitMinShare = 6;           // K steps of a pair's share, at least
constexpr int kGSplitCost = 60;              // K steps that a cut costs (see gemm_groups)
constexpr long long kGWait = 4000000000LL;

constexpr uint32_t kPeerMask = 0xFEFFFFFFu;   // clears the CTA-rank bit of a shared::cluster address: the pair's even CTA

__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// tiled load into this CTA's shared memory whose bytes are counted on the barrier of the pair's even CTA
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst_smem, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst_smem), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar & kPeerMask), "r"(c0), "r"(c1) : "memory");
}
// arrives, once every tcgen05 operation issued so far has completed, on the barrier at this offset in both CTAs of the pair
__device__ __forceinline__ void commit_pair(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void arrive_on_leader(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar & kPeerMask) : "memory");
}
// The low word of a shared-memory descriptor holds the start address (>> 4) and the leading offset, the high word
// everything that does not change inside a tile: stepping through a tile is a 32-bit add.
__device__ __forceinline__ uint32_t smem_desc_lo(uint32_t saddr, uint32_t lbo_bytes) {
    return ((saddr & 0x3FFFFu) >> 4) | (((lbo_bytes >> 4) & 0x3FFFu) << 16);
}
__device__ __forceinline__ constexpr uint32_t smem_desc_hi_sw128(uint32_t sbo_bytes) {
    return ((sbo_bytes >> 4) & 0x3FFFu) | (1u << 14) | (2u << 29);
}
__device__ __forceinline__ void mma_ss_lh(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %6, 0;\n\tmov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %5, {%7, %7, %7, %7, %7, %7, %7, %7}, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate), "r"(0u) : "memory");
}

// tile t -> (m tile of 256 rows, n tile): the n tiles come in groups of kGGroup; within a group the m tiles run one after the other and
// each visits the group's n tiles, so that the CTAs of a wave share a few A row-blocks and a few W column-blocks in L2.  by_m: the same with
// rows and columns exchanged
__device__ __forceinline__ void tile_coords(int t, int m_tiles, int n_tiles, bool by_m, int& mt, int& nt) {
    const int grouped = by_m ? m_tiles : n_tiles, swept = by_m ? n_tiles : m_tiles, per_group = swept * kGGroup;
    const int g = t / per_group, r = t - g * per_group;
    const int gw = min(kGGroup, grouped - g * kGGroup);          // the last group may be narrower
    const int in = g * kGGroup + r % gw, along = r / gw;
    mt = by_m ? in : along;
    nt = by_m ? along : in;
}

template <int N> struct Width { static constexpr int value = N; };

// What a pair of CTAs works on.  Whole tiles: t = pair, pair + P, .. in the order of tile_coords.  Cut along K (groups > 0): the pairs form
// `groups` groups with one pair per row of tiles; the K steps of all column tiles are dealt out evenly to the groups, in order, so that
// a group's share begins and ends anywhere inside a tile, and its pairs go through the same part of W at the same time (W comes from
// HBM once: with the tiles' K steps simply dealt out to the pairs, a 136 MB weight matrix was read 3.6 times for three rows of tiles).
template <bool CUT>
struct Work {
    int t, tiles, P, m_tiles, n_tiles, ksteps, mt;
    long long u, u1;
    bool by_m;
    __device__ __forceinline__ Work(int pair, int P_, int m_tiles_, int n_tiles_, int ksteps_, int groups, int by_m_)
        : t(pair), tiles(m_tiles_ * n_tiles_), P(P_), m_tiles(m_tiles_), n_tiles(n_tiles_), ksteps(ksteps_), mt(0), u(0), u1(0), by_m(by_m_ != 0) {
        if constexpr (CUT) {
            const int grp = pair / m_tiles;
            const long long U = (long long)n_tiles * ksteps;
            mt = pair % m_tiles;
            if (grp < groups) { u = grp * U / groups; u1 = (grp + 1) * U / groups; }
        }
    }
    __device__ __forceinline__ bool next(int& m, int& n, int& k0, int& k1) {
        if constexpr (!CUT) {
            if (t >= tiles) return false;
            tile_coords(t, m_tiles, n_tiles, by_m, m, n);
            k0 = 0; k1 = ksteps; t += P;
            return true;
        }
        if (u >= u1) return false;
        n = (int)(u / ksteps); m = mt;
        k0 = (int)(u - (long long)n * ksteps);
        k1 = (int)min((long long)ksteps, k0 + (u1 - u));
        u += k1 - k0;
        return true;
    }
};

struct GemmArgs {
    int n, N, K;                 // rows (upper bound), columns of W that one tile row of the output spans, depth
    int n_tiles;                 // tiles along the output columns
    void* C; int64_t ldc;        // PLAIN / ROPE / SWIGLU output (elements)
    int w_early;                 // W may be read before the kernel in front is complete
    const int32_t* n_dev;        // device: true number of rows (<= n), or null
    int* status;
    int by_m;                    // order of the tiles (see tile_coords)
    int groups;                  // > 0: tiles are cut along K (see Work)
    float* part;                 // partial tiles of the pairs: two of 256 x 256 fp32 each
    unsigned int* arrived;       // per tile, CTA of the pair and epilogue warp: parts that are in `part`
    uint32_t spin_limit;         // polls for parts that others are writing before a pair gives up
    GemmEpilogue e;
};

// ---- epilogue pieces -----------------------------------------------------------
// A warp's staging block holds 32 rows of 128 bytes; 16-byte chunk c of row r sits at chunk c ^ (r & 7), so that a lane per row
// (writes) and eight lanes per row (reads) are both free of bank conflicts.
__device__ __forceinline__ uint32_t stage_addr(uint32_t stage, int row, int chunk) { return stage + row * 128 + ((chunk ^ (row & 7)) << 4); }
__device__ __forceinline__ void sts_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint4 lds_v4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint2 ld_v2(const void* p) {       // coherent: x_full may be H itself
    uint2 v;
    asm volatile("ld.global.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_v2(void* p, uint32_t a, uint32_t b) {
    asm volatile("st.global.v2.u32 [%0], {%1,%2};" ::"l"(p), "r"(a), "r"(b) : "memory");
}
// v[i] summed over the eight lanes that share lane >> 3; lane j of them is left with v[j & 7]'s total (in v[0])
__device__ __forceinline__ void reduce_rows8(float (&v)[8], int lane) {
#pragma unroll
    for (int w = 4; w >= 1; w >>= 1) {
        const bool up = (lane & w) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const float send = up ? v[i] : v[i + w], keep = up ? v[i + w] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
        }
    }
}

// F32 (PLAIN, ROPE): C is fp32.  CUT: tiles may be cut along K; kernels of their own, because the adding up of parts beside their epilogue's code cost those of
// whole tiles registers (gate | up projection 544 cycles per K step without, 550 with it; in one kernel / apart, in a loop, us: layer of 5000 rows 368 / 360, of 8192 834 / 826, three blocks of 701
// rows 875 / 869, of 8192 7815 / 7755)
template <int EPI, int BN, bool F32, bool CUT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGThreads, 1)
gemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapW, const GemmArgs g) {
    static_assert(BN == kGN || (BN == kGNarrow && EPI != GEMM_SWIGLU && !CUT), "tile widths");
    constexpr int kGStages = Ring<BN>::kStages, kGStageBytes = Ring<BN>::kStage;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t bars = base + kGStages * kGStageBytes + kGEpiWarps * kGEpiBytes;
    auto full = [&](int s) { return bars + 8 * s; };
    auto empty = [&](int s) { return bars + 8 * (kGStages + s); };
    auto acc_full = [&](int b) { return bars + 8 * (2 * kGStages + b); };
    auto acc_empty = [&](int b) { return bars + 8 * (2 * kGStages + 2 + b); };
    const uint32_t slot = bars + 8 * (2 * kGStages + 4);
    volatile uint32_t* slot_gen = reinterpret_cast<volatile uint32_t*>(smem_raw + (slot - smem_u32(smem_raw)));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // the kernel behind may set itself up while this one drains, as this one does while the kernel in front of it drains
    pdl_launch_dependents();
    const int rank = (int)cluster_rank();                  // 0: the pair's even CTA (issues the MMAs, owns the full / acc_empty barriers)
    if (warp == 1) {
        if (lane == 0) {
            for (int s = 0; s < kGStages; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
            for (int b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), 2 * kGEpiWarps); }
            fence_barrier_init();
            fence_proxy_async_smem();
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else if (warp == 0 && lane == 0) {
        prefetch_tensormap(&mapA); prefetch_tensormap(&mapW);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                    // the peer's barriers exist before anything is signalled across
    tc_fence_after();
    const uint32_t tmem = *slot_gen;
    const int m_tiles = (g.n + 2 * kGM - 1) / (2 * kGM), n_tiles = g.n_tiles, ksteps = (g.K + kGK - 1) / kGK;
    const int n_pairs = (int)gridDim.x / 2, pair = (int)blockIdx.x / 2;
    constexpr uint32_t idesc = idesc_bf16_f32(2 * kGM, BN, false, true);
    constexpr uint32_t hi = smem_desc_hi_sw128(1024);

    if (warp == 0) {
        // ---- loads of this CTA: its 128 x 64 half of the A tile (K-major), its half of the W tile as one or two chunks of 64 columns ----
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            Work<CUT> w(pair, n_pairs, m_tiles, n_tiles, ksteps, g.groups, g.by_m);
            int mt, nt, k0, k1;
            // w_early: the first stages' W tiles are asked for while the kernel in front, which makes A, still drains (see gemm.cuh for when)
            bool first = true;
            while (ok && w.next(mt, nt, k0, k1)) {
                const int m0 = mt * 2 * kGM + rank * kGM;
                auto load_w = [&](int s, int k) {
                    if (rank == 0) mbar_arrive_expect_tx(full(s), 2 * kGStageBytes);     // both CTAs' bytes land on this barrier
#pragma unroll
                    for (int c = 0; c < BN / 2 / 64; ++c) {
                        // SWIGLU: columns 0-127 of the tile (the even CTA's half) are gate features nt * 128 .., columns 128-255 the same features of "up"
                        const int col = (EPI == GEMM_SWIGLU) ? (rank * g.e.m + nt * 128 + c * 64) : (nt * BN + rank * (BN / 2) + c * 64);
                        tma_load_2d_pair(base + s * kGStageBytes + kGABytes + c * (kGK * 128), &mapW, full(s), col, k * kGK);
                    }
                };
                auto load_a = [&](int s, int k) { tma_load_2d_pair(base + s * kGStageBytes, &mapA, full(s), k * kGK, m0); };
                int k = k0;
                if (first) {
                    const int pre = min(kGStages, k1 - k0);
                    if (!g.w_early) pdl_wait();
                    for (int s = 0; s < pre; ++s) load_w(s, k0 + s);
                    if (g.w_early) pdl_wait();
                    for (int s = 0; s < pre; ++s) load_a(s, k0 + s);
                    k += pre; it += pre;
                    first = false;
                }
                for (; k < k1 && ok; ++k, ++it) {
                    const int s = it % kGStages;
                    if (it >= kGStages) ok = mbar_wait(empty(s), ((it / kGStages) - 1) & 1, kGWait);
                    if (!ok) break;
                    load_w(s, k);
                    load_a(s, k);
                }
            }
            if (!ok) atomicExch(g.status, DASH_ERR_TIMEOUT);
        }
    } else if (warp == 1) {
        // ---- MMAs (even CTA only): four 256 x BN x 16 steps per stage into the tile's TMEM buffer of both CTAs ----
        if (lane == 0 && rank == 0) {
            uint32_t it = 0, tl = 0;
            bool ok = true;
            Work<CUT> w(pair, n_pairs, m_tiles, n_tiles, ksteps, g.groups, g.by_m);
            int mt, nt, k0, k1;
            for (; ok && w.next(mt, nt, k0, k1); ++tl) {
                const int b = tl & 1;
                if (tl >= 2) ok = mbar_wait(acc_empty(b), ((tl >> 1) - 1) & 1, kGWait);
                if (!ok) break;
                tc_fence_after();
                const uint32_t tD = tmem + b * BN;
                for (int k = k0; k < k1 && ok; ++k, ++it) {
                    const int s = it % kGStages;
                    ok = mbar_wait(full(s), (it / kGStages) & 1, kGWait);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t sA = base + s * kGStageBytes, sB = sA + kGABytes;
                    const uint32_t a_lo = smem_desc_lo(sA, 16), b_lo = smem_desc_lo(sB, kGK * 128);
#pragma unroll
                    for (int kk = 0; kk < kGK / 16; ++kk)
                        mma_ss_lh(tD, a_lo + ((kk * 32) >> 4), hi, b_lo + ((kk * 2048) >> 4), hi, idesc, (k > k0) || (kk > 0));
                    commit_pair(empty(s));
                }
                commit_pair(acc_full(b));
            }
            if (!ok) atomicExch(g.status, DASH_ERR_TIMEOUT);
        }
    } else {
        // ---- epilogue: warp (q, half) holds rows 32 q .. of this CTA's 128 and half of the tile's columns (SWIGLU: gate and up columns of
        // features 64 half ..).  A tile of 256 columns: the four pieces of 128 columns; of 128: two of its four pieces ----
        const int q = warp & 3, half = (warp - 2) >> 2;           // q: the TMEM lane quarter this warp may read
        const int wcol = BN == kGN ? half * 128 : 0;              // the 128 columns of the tile that this warp's pieces are counted in
        constexpr int kPieces = BN == kGN ? 4 : 2;                // of 32 columns
        const int p0 = BN == kGN ? 0 : 2 * half;                  // the first of them
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        const uint32_t stage = base + kGStages * kGStageBytes + (warp - 2) * kGEpiBytes;
        pdl_wait();
        int n_true = g.n;
        if (g.n_dev) { const int nd = *g.n_dev; if (nd < n_true) n_true = nd; }
        const int r8 = lane >> 3, c8 = lane & 7;                  // eight lanes per row: row r8 + 4 i, chunk c8
        uint32_t tl = 0;
        bool ok = true;
        Work<CUT> w(pair, n_pairs, m_tiles, n_tiles, ksteps, g.groups, g.by_m);
        int mt, nt, k0, k1;
        for (; w.next(mt, nt, k0, k1); ++tl) {
            const int b = tl & 1;
            const int row0 = mt * 2 * kGM + rank * kGM + q * 32;  // first row of this warp's 32
            const uint32_t tD = tmem + b * BN + lane_base;
            const bool cut = CUT && k1 - k0 != ksteps;      // (what an epilogue reads ahead it then reads behind leave_part, for the registers)
            auto wait_acc = [&]() { ok = __all_sync(0xffffffffu, mbar_wait(acc_full(b), (tl >> 1) & 1, kGWait)); tc_fence_after(); };
            // every TMEM read of this warp for the tile has completed: the buffer goes back to the MMA thread
            auto release_acc = [&]() {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) arrive_on_leader(acc_empty(b));
            };
            // A tile that was cut along K.  Every pair says that it is done; all but the last to say so leave their partial sums in `part` (a lane's
            // row in 16-byte pieces, so that a warp's piece is 512 contiguous bytes) and say that too.  The last one waits for what the others are
            // writing at that moment -- they wait for nothing -- adds the parts up in the order of K, its own from TMEM, and goes on as with a whole
            // tile.  Warp by warp: the same warp of every pair holds the same rows and columns.  Bound by that one SM's loads from L2, a few at a time: from the last
            // product of the down projection to its last result 9 us at 701 rows, 8 at 1500, 13 at 233, four parts to a tile.  (14, 14 and 18 with 64-bit divisions in
            // the place of every part, 14 and 13 with its own part written and read back as well.)
            auto part_col = [&](int k) { return EPI == GEMM_SWIGLU ? (k >> 1) * 128 + half * 64 + (k & 1) * 32 : half * 128 + k * 32; };   // of piece k
            auto leave_part = [&]() -> bool {                     // true: the tile is left to another pair
                if constexpr (!CUT) return false;
                const long long U = (long long)n_tiles * ksteps, u0 = (long long)nt * ksteps;
                const int first_grp = (int)(((u0 + 1) * g.groups - 1) / U), n_parts = (int)(((u0 + ksteps) * g.groups - 1) / U) - first_grp + 1;
                unsigned int* cnt = g.arrived + (size_t)((nt * m_tiles + mt) * 2 + rank) * kGEpiWarps + (warp - 2);
                if (row0 >= g.n) return true;                     // no rows here: nothing to add up, nothing to store
                const int own = pair / m_tiles - first_grp;
                // Part p of the tile: of the two places of its pair the first (the share begins in this tile) or, p = 0 only, the second (it begins in a tile in
                // front).  (With that found by 64-bit divisions for every part the four kernels spilled 44 to 120 bytes: RESID now 24, ROPE 8, the others none.
                // us, a block of 523 rows with output and down projection cut 162.6, now 156.0, with Q | K | V and gate | up cut 149.7 / 143.0, three blocks of
                // 701 rows of the 7B shape 868 / 863.  Without the last 24 and 8, rows' indices asked for behind this and 16 columns at a time: 158.5, 143.1, 865.)
                const bool cont = first_grp * U / g.groups < u0;
                auto part_of = [&](int p, int col) {
                    return reinterpret_cast<float4*>(g.part) + (size_t)(2 * ((first_grp + p) * m_tiles + mt) + (p == 0 && cont ? 1 : 0)) * (2 * kGM * kGN / 4) + (size_t)(col >> 2) * (2 * kGM) +
                           rank * kGM + q * 32 + lane;
                };
                constexpr unsigned int kLeft = 1u << 16;          // low half of the counter: pairs that are done, high half: parts that are in `part`
                unsigned int in = 0;
                if (lane == 0) in = atomicAdd(cnt, 1u) & (kLeft - 1u);
                in = __shfl_sync(0xffffffffu, in, 0);
                if (in == (unsigned int)(n_parts - 1)) {
                    bool all = true;
                    if (lane == 0) {
                        const unsigned int want = (unsigned int)(n_parts - 1) * kLeft + (unsigned int)n_parts;
                        uint32_t spins = 0;
                        while (*reinterpret_cast<volatile unsigned int*>(cnt) != want && all) {
                            __nanosleep(32);
                            all = ++spins <= g.spin_limit;
                        }
                        // Zero for the next launch, but not where the wait ran out: a pair that is late would still add its part, and what is neither
                        // zero nor told by the status would look like a count.  Every step clears its counters ahead of its projections.
                        if (all) *cnt = 0u;
                        else atomicExch(g.status, DASH_ERR_TIMEOUT);
                    }
                    __syncwarp();
                    __threadfence();
                    if (__any_sync(0xffffffffu, !all)) return true;
                    // into this warp's accumulators, 32 columns at a time, the loads of up to two of the other parts in flight (where registers are left)
                    constexpr bool kTwo = EPI == GEMM_PLAIN || EPI == GEMM_SWIGLU;
#pragma unroll 1
                    for (int k = 0; k < 4; ++k) {
                        const int col = part_col(k);
                        uint32_t o[32];
#pragma unroll
                        for (int e = 0; e < 32; ++e) o[e] = 0u;
#pragma unroll 1
                        for (int p = 0; p < n_parts;) {
                            uint32_t v[kTwo ? 64 : 32];
                            const bool mine = p == own, two = kTwo && !mine && p + 1 < n_parts && p + 1 != own;
                            if (mine) {
                                tmem_ld32(tD + col, v);
                                tmem_wait_ld();
                            } else {
                                const float4 *s0 = part_of(p, col), *s1 = two ? part_of(p + 1, col) : s0;
#pragma unroll
                                for (int c = 0; c < (kTwo ? 16 : 8); ++c) {
                                    if (c < 8 || two) {
                                        const float4 x = __ldcg((c < 8 ? s0 : s1) + (c & 7) * (2 * kGM));
                                        v[4 * c] = __float_as_uint(x.x); v[4 * c + 1] = __float_as_uint(x.y); v[4 * c + 2] = __float_as_uint(x.z); v[4 * c + 3] = __float_as_uint(x.w);
                                    }
                                }
                            }
#pragma unroll
                            for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) + __uint_as_float(v[e]));
                            if constexpr (kTwo) {
                                if (two) {
#pragma unroll
                                    for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) + __uint_as_float(v[32 + e]));
                                }
                            }
                            p += two ? 2 : 1;
                        }
                        tmem_st32(tD + col, o);
                    }
                    tmem_wait_st();
                    return false;
                }
#pragma unroll 1
                for (int k = 0; k < 4; ++k) {
                    const int col = part_col(k);
                    uint32_t o[32];
                    tmem_ld32(tD + col, o);
                    tmem_wait_ld();
                    float4* dst = part_of(own, col);
#pragma unroll
                    for (int c = 0; c < 8; ++c) st_v4(dst + c * (2 * kGM), make_uint4(o[4 * c], o[4 * c + 1], o[4 * c + 2], o[4 * c + 3]));
                }
                __threadfence();
                __syncwarp();
                if (lane == 0) atomicAdd(cnt, kLeft);
                return true;
            };
            // o[0 .. N) and o[N .. 2N): N columns of this lane's row from columns col0 and col1 of the tile
            auto load_acc = [&](auto width, int col0, int col1, uint32_t* o) {
                constexpr int N = decltype(width)::value;
                if constexpr (N == 32) { tmem_ld32(tD + col0, o); tmem_ld32(tD + col1, o + 32); }
                else { tmem_ld16(tD + col0, o); tmem_ld16(tD + col1, o + 16); }
                tmem_wait_ld();
            };
            const Width<16> w16; const Width<32> w32;
            auto stage_f32 = [&](const uint32_t* o) {             // 32 columns of this lane's row
#pragma unroll
                for (int c = 0; c < 8; ++c) sts_v4(stage_addr(stage, lane, c), o[4 * c], o[4 * c + 1], o[4 * c + 2], o[4 * c + 3]);
                __syncwarp();
            };
            if (EPI == GEMM_PLAIN) {
                // columns at or past N (a last, partial tile) are not stored; N is a multiple of 8 (bf16) / 4 (fp32)
                const int col0 = nt * BN + wcol;
                wait_acc();
                if (!ok) break;
                if (cut && leave_part()) { release_acc(); continue; }
                if (F32) {
#pragma unroll
                    for (int i = 0; i < kPieces; ++i) {
                        const int k = p0 + i;
                        uint32_t o[32];
                        load_acc(w16, wcol + k * 32, wcol + k * 32 + 16, o);
                        if (i == kPieces - 1) release_acc();
                        stage_f32(o);
                        const int col = col0 + k * 32 + c8 * 4;
#pragma unroll
                        for (int i2 = 0; i2 < 8; ++i2) {
                            const int r = r8 + 4 * i2, row = row0 + r;
                            const uint4 v = lds_v4(stage_addr(stage, r, c8));
                            if (row < n_true && col < g.N) st_v4(reinterpret_cast<float*>(g.C) + (int64_t)row * g.ldc + col, v);
                        }
                        __syncwarp();
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < kPieces / 2; ++i) {
                        const int k = p0 / 2 + i;
                        uint32_t o[64];
                        load_acc(w32, wcol + k * 64, wcol + k * 64 + 32, o);
                        if (i == kPieces / 2 - 1) release_acc();
                        auto pk = [&](int e) { return pack_bf16(__uint_as_float(o[e]), __uint_as_float(o[e + 1])); };
#pragma unroll
                        for (int c = 0; c < 8; ++c) sts_v4(stage_addr(stage, lane, c), pk(8 * c), pk(8 * c + 2), pk(8 * c + 4), pk(8 * c + 6));
                        __syncwarp();
                        const int col = col0 + k * 64 + c8 * 8;
#pragma unroll
                        for (int i2 = 0; i2 < 8; ++i2) {
                            const int r = r8 + 4 * i2, row = row0 + r;
                            const uint4 v = lds_v4(stage_addr(stage, r, c8));
                            if (row < n_true && col < g.N) st_v4(reinterpret_cast<__nv_bfloat16*>(g.C) + (int64_t)row * g.ldc + col, v);
                        }
                        __syncwarp();
                    }
                }
            } else if (EPI == GEMM_ROPE) {
                // heads of D columns; inside a head of Q or K the pair (i, i + D/2) is rotated by the angle of (row, i).  A piece is 16
                // pairs of a head: four lanes per row, four pairs each; rows in the order 0, 4, 1, 5, 2, 6, 3, 7 so that the two rows of
                // a quarter warp lie in different halves of the banks.
                const int D = g.e.D, hd2 = D >> 1, c4 = lane & 3, rr = (lane >> 3) + 4 * ((lane >> 2) & 1);
                float rsc[4];
                int tab[4];                                       // (cos, sin) entry of this row: its own, or its position's
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int row = row0 + rr + 8 * i;
                    const bool live = row < n_true;
                    int64_t trow = live ? row : 0;
                    if (g.e.rope_pos) { trow = live ? g.e.rope_pos[row] : 0; if (trow >= g.e.rope_len) trow = g.e.rope_len - 1; if (trow < 0) trow = 0; }
                    tab[i] = (int)trow;
                    rsc[i] = (g.e.row_scale && live) ? g.e.row_scale[row] : 1.0f;
                }
                const int colw = nt * BN + wcol;                  // first column of this warp's 128
                auto head_of = [&](int k) { return D == 128 ? 0 : (k >> 1) * 64; };
                auto pair_of = [&](int k) { return D == 128 ? k * 16 : (k & 1) * 16; };
                const bool tab16 = (reinterpret_cast<uint64_t>(g.e.rope_table) & 15u) == 0;
                uint4 cs[8];
                auto fetch_cs = [&](int k) {
                    if (colw + head_of(k) < g.e.n_rot_cols) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float2* p = g.e.rope_table + (int64_t)tab[i] * hd2 + pair_of(k) + c4 * 4;
                            if (tab16) {
                                cs[2 * i] = __ldg(reinterpret_cast<const uint4*>(p));
                                cs[2 * i + 1] = __ldg(reinterpret_cast<const uint4*>(p) + 1);
                            } else {                              // a caller's table need only be 8-byte aligned
                                const uint2* p2 = reinterpret_cast<const uint2*>(p);
                                const uint2 a0 = __ldg(p2), a1 = __ldg(p2 + 1), a2 = __ldg(p2 + 2), a3 = __ldg(p2 + 3);
                                cs[2 * i] = make_uint4(a0.x, a0.y, a1.x, a1.y);
                                cs[2 * i + 1] = make_uint4(a2.x, a2.y, a3.x, a3.y);
                            }
                        }
                    }
                };
                if (!cut) fetch_cs(p0);
                wait_acc();
                if (!ok) break;
                if (cut) {
                    if (leave_part()) { release_acc(); continue; }
                    fetch_cs(p0);
                }
#pragma unroll 1
                for (int k = p0; k < p0 + kPieces; ++k) {
                    const int h0 = head_of(k), c = pair_of(k), colh = colw + h0;
                    uint32_t o[32];
                    load_acc(w16, wcol + h0 + c, wcol + h0 + hd2 + c, o);
                    if (k == p0 + kPieces - 1) release_acc();
                    stage_f32(o);
                    const bool rotate = colh < g.e.n_rot_cols, is_q = colh < g.e.q_cols;
                    // a head of K or V goes to the caller's cache as well; fp32: every head to the bf16 copies that the attention kernel reads
                    __nv_bfloat16* cache = nullptr;
                    int64_t ld_cache = g.e.ld_cache;
                    if (g.e.k_cache && !is_q)
                        cache = reinterpret_cast<__nv_bfloat16*>(rotate ? g.e.k_cache : g.e.v_cache) + (colh - (rotate ? g.e.q_cols : g.e.n_rot_cols));
                    if (F32 && is_q) { cache = reinterpret_cast<__nv_bfloat16*>(g.e.q_copy) + colh; ld_cache = g.e.q_cols; }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int r = rr + 8 * i, row = row0 + r;
                        const uint4 v1 = lds_v4(stage_addr(stage, r, c4)), v2 = lds_v4(stage_addr(stage, r, 4 + c4));
                        const float x1[4] = {__uint_as_float(v1.x) * rsc[i], __uint_as_float(v1.y) * rsc[i], __uint_as_float(v1.z) * rsc[i], __uint_as_float(v1.w) * rsc[i]};
                        const float x2[4] = {__uint_as_float(v2.x) * rsc[i], __uint_as_float(v2.y) * rsc[i], __uint_as_float(v2.z) * rsc[i], __uint_as_float(v2.w) * rsc[i]};
                        float y1[4], y2[4];
                        if (rotate) {
                            const uint32_t t[8] = {cs[2 * i].x, cs[2 * i].y, cs[2 * i].z, cs[2 * i].w, cs[2 * i + 1].x, cs[2 * i + 1].y, cs[2 * i + 1].z, cs[2 * i + 1].w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float cv = __uint_as_float(t[2 * e]), sv = __uint_as_float(t[2 * e + 1]);
                                y1[e] = x1[e] * cv - x2[e] * sv;
                                y2[e] = x2[e] * cv + x1[e] * sv;
                            }
                        } else {
#pragma unroll
                            for (int e = 0; e < 4; ++e) { y1[e] = x1[e]; y2[e] = x2[e]; }
                        }
                        if (row < n_true) {
                            const uint32_t a0 = pack_bf16(y1[0], y1[1]), a1 = pack_bf16(y1[2], y1[3]), b0 = pack_bf16(y2[0], y2[1]), b1 = pack_bf16(y2[2], y2[3]);
                            const int64_t at = (int64_t)row * g.ldc + colh + c + c4 * 4;
                            if (F32) {
                                float* dst = reinterpret_cast<float*>(g.C) + at;
                                st_v4(dst, make_uint4(__float_as_uint(y1[0]), __float_as_uint(y1[1]), __float_as_uint(y1[2]), __float_as_uint(y1[3])));
                                st_v4(dst + hd2, make_uint4(__float_as_uint(y2[0]), __float_as_uint(y2[1]), __float_as_uint(y2[2]), __float_as_uint(y2[3])));
                            } else {
                                __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(g.C) + at;
                                st_v2(dst, a0, a1);
                                st_v2(dst + hd2, b0, b1);
                            }
                            if (cache) {
                                __nv_bfloat16* kv = cache + (int64_t)row * ld_cache + c + c4 * 4;
                                st_v2(kv, a0, a1);
                                st_v2(kv + hd2, b0, b1);
                            }
                        }
                    }
                    if (k < p0 + kPieces - 1) fetch_cs(k + 1);
                    __syncwarp();
                }
            } else if (EPI == GEMM_RESID) {
                // H~ = H + U (U in fp32, one rounding) to x_full[tok[row]]; sums of u^2, h^2 and (h+u)^2 over 128 columns
                const int col0 = nt * BN + wcol + c8 * 4;
                const __nv_bfloat16* hsrc = reinterpret_cast<const __nv_bfloat16*>(g.e.H) + col0;
                __nv_bfloat16* xdst = reinterpret_cast<__nv_bfloat16*>(g.e.x_full) + col0;
                int tok[8];
                uint2 hv[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int row = row0 + r8 + 4 * i;
                    tok[i] = row < n_true ? (g.e.tok_index ? g.e.tok_index[row] : row) : 0;
                }
                auto fetch_h = [&](int k) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int row = row0 + r8 + 4 * i;
                        if (row < n_true) hv[i] = ld_v2(hsrc + (int64_t)row * g.e.ldh + k * 32);
                    }
                };
                if (!cut) fetch_h(p0);
                float su[8], sh[8], st2[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) su[i] = sh[i] = st2[i] = 0.f;
                wait_acc();
                if (BN == kGN && !ok) break;
                if (!ok) n_true = 0;                              // a narrow tile's two warps meet below, come what may: nothing is stored
                if (cut) {
                    if (leave_part()) { release_acc(); continue; }
                    fetch_h(p0);
                }
#pragma unroll 1
                for (int k = p0; k < p0 + kPieces; ++k) {
                    uint32_t o[32];
                    load_acc(w16, wcol + k * 32, wcol + k * 32 + 16, o);
                    if (k == p0 + kPieces - 1) release_acc();
                    stage_f32(o);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int r = r8 + 4 * i, row = row0 + r;
                        const uint4 v = lds_v4(stage_addr(stage, r, c8));
                        if (row < n_true) {
                            const float u[4] = {__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w)};
                            const float h[4] = {bf16lo(hv[i].x), bf16hi(hv[i].x), bf16lo(hv[i].y), bf16hi(hv[i].y)};
                            float y[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                su[i] += u[e] * u[e];
                                sh[i] += h[e] * h[e];
                                y[e] = h[e] + u[e];
                                st2[i] += y[e] * y[e];
                            }
                            st_v2(xdst + (int64_t)tok[i] * g.e.ldx + k * 32, pack_bf16(y[0], y[1]), pack_bf16(y[2], y[3]));
                        }
                    }
                    if (k < p0 + kPieces - 1) fetch_h(k + 1);
                    __syncwarp();
                }
                reduce_rows8(su, lane); reduce_rows8(sh, lane); reduce_rows8(st2, lane);
                const int row = row0 + r8 + 4 * c8;               // this lane holds the sums of row r8 + 4 c8
                if (BN == kGN) {
                    if (row < n_true) g.e.sums[(int64_t)row * (2 * n_tiles) + 2 * nt + half] = make_float4(su[0], sh[0], st2[0], 0.f);
                } else {
                    // of 64 columns: the quarter's two warps add theirs up, the second one's through its staging block
                    if (half == 1) sts_v4(stage + lane * 16, __float_as_uint(su[0]), __float_as_uint(sh[0]), __float_as_uint(st2[0]), 0u);
                    asm volatile("bar.sync %0, 64;" ::"r"(1 + q) : "memory");
                    if (half == 0) {
                        const uint4 o = lds_v4(stage + 4 * kGEpiBytes + lane * 16);
                        if (row < n_true)
                            g.e.sums[(int64_t)row * n_tiles + nt] = make_float4(su[0] + __uint_as_float(o.x), sh[0] + __uint_as_float(o.y), st2[0] + __uint_as_float(o.z), 0.f);
                    }
                    asm volatile("bar.sync %0, 64;" ::"r"(1 + q) : "memory");
                }
            } else {
                // SWIGLU: columns 0-127 gate, 128-255 up of the same 128 features
                const float rsc = (g.e.row_scale && row0 + lane < n_true) ? g.e.row_scale[row0 + lane] : 1.0f;
                wait_acc();
                if (!ok) break;
                if (cut && leave_part()) { release_acc(); continue; }
#pragma unroll 1
                for (int k = 0; k < 4; ++k) {
                    uint32_t gu[32];                              // 16 gate, 16 up columns of this lane's row
                    load_acc(w16, half * 64 + k * 16, 128 + half * 64 + k * 16, gu);
                    if (k == 3) release_acc();
                    float a[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const float z = __uint_as_float(gu[e]) * rsc;
                        a[e] = z / (1.0f + __expf(-z)) * (__uint_as_float(gu[16 + e]) * rsc);
                    }
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        sts_v4(stage_addr(stage, lane, k * 2 + c), pack_bf16(a[8 * c], a[8 * c + 1]), pack_bf16(a[8 * c + 2], a[8 * c + 3]),
                               pack_bf16(a[8 * c + 4], a[8 * c + 5]), pack_bf16(a[8 * c + 6], a[8 * c + 7]));
                }
                __syncwarp();
                __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(g.C) + nt * 128 + half * 64 + c8 * 8;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = r8 + 4 * i, row = row0 + r;
                    const uint4 v = lds_v4(stage_addr(stage, r, c8));
                    if (row < n_true) st_v4(dst + (int64_t)row * g.ldc, v);
                }
                __syncwarp();
            }
        }
        if (!ok && lane == 0) atomicExch(g.status, DASH_ERR_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                    // nobody leaves while the peer may still signal its barriers or read its tiles
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// (cos, sin) of every position 0 .. n - 1
__global__ void __launch_bounds__(256)
rope_table_kernel(int64_t n, int half, RopeFreqs fr, float2* __restrict__ table) {
    row_prep_rows(nullptr, n, half, fr, table, nullptr, 0, 0, 0.f, 0.f, nullptr, nullptr, (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5), (int64_t)gridDim.x * 8);
}

static int make_map_2d_bf16(CUtensorMap* map, const void* basep, uint64_t inner, uint64_t outer, uint64_t ld_elems, uint32_t box_inner,
                            uint32_t box_outer) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return DASH_ERR_CUDA;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {ld_elems * 2};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(basep), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? DASH_OK : DASH_ERR_CUDA;
}

// Scratch of tiles cut along K: a counter per tile, CTA and epilogue warp; two partial tiles per pair (gemm_split_part_bytes)
size_t gemm_split_count_bytes() { return align_up((size_t)(sm_count() / 2) * kGSplitMaxRounds * 2 * kGEpiWarps * sizeof(unsigned int), 256); }

// Into how many groups of pairs the K steps are dealt out (0: whole tiles).  Whole tiles take ceil(tiles / P) rounds of `ksteps` steps, the last
// of which may be nearly empty; cut, a pair takes n_tiles / groups tiles' worth of steps.  What the cut costs, partial tiles out and
// in again, is worth about kGSplitCost steps.  Steps of the 7B shape and of one with d = 2048, m = 6144, every projection cut / none, in us: savings of 24
// and 24 steps (233 rows, d = 2048) 71 / 53, of 42 and 42 (233 rows, 7B) 76 / 68, of 64 to 74 (down projections) about even: 701 rows of
// d = 2048 151 / 146, in a graph 143 / 160, 1024 and 2100 rows of 7B 384 / 385 and 793 / 781; 72 at 233 rows of d = 2048 114 / 122, 123 at
// 701 rows of 7B 304 / 320, 184 at 300 233 / 268, 197 at 2728 1009 / 1047.  (Two rounds of tiles of which the second is half empty, 1500 rows of 7B,
// gain 11 us of 149 by cuts that save 28 and 46 steps: the rule leaves those.  In a loop at the power cap, three blocks, a cost of
// 60 / 45 / 25: 600 rows 863 / 865 / 873 us, 1500 1567 / 1570 / 1590, 2000 2005 / 2015 / 2010.)
static int gemm_groups(int m_tiles, int n_tiles, int ksteps, int P, bool can) {
    const long long tiles = (long long)m_tiles * n_tiles;
    if (!can || m_tiles > P || tiles > (long long)kGSplitMaxRounds * P) return 0;
    int groups = P / m_tiles;
    const int most = (int)min((long long)n_tiles * kGSplitMaxParts, (long long)n_tiles * ksteps / kGSplitMinShare);
    if (groups > most) groups = most;
    if (groups < 1) return 0;
    const long long whole = (tiles + P - 1) / P * ksteps, cut = ((long long)n_tiles * ksteps + groups - 1) / groups;
    return cut + kGSplitCost < whole ? groups : 0;
}

size_t gemm_split_part_bytes(int64_t n, int64_t N, int64_t K) {
    if (n < 1 || N < 1 || K < 1 || n > 0x7fffffffLL || N > 0x7fffffffLL || K > 0x7fffffffLL) return 0;
    const int m_tiles = (int)((n + 2 * kGM - 1) / (2 * kGM));
    return (size_t)gemm_groups(m_tiles, (int)((N + kGN - 1) / kGN), (int)((K + kGK - 1) / kGK), sm_count() / 2, true) * m_tiles * 2 * (2 * kGM * kGN) * sizeof(float);
}
int gemm_tile_rows() { return 2 * kGM; }
int64_t gemm_split_max_rows() { return (int64_t)(sm_count() / 2) * 2 * kGM; }

template <int EPI, int BN, bool F32, bool CUT>
static int launch_tiles(const CUtensorMap& ma, const CUtensorMap& mw, const GemmArgs& g, int pairs, cudaStream_t st) {
    const int smem = kGRingBytes + kGEpiWarps * kGEpiBytes + 1024 + 256;
    static std::atomic<uint64_t> configured{0};
    if (!set_max_smem_once(gemm_kernel<EPI, BN, F32, CUT>, smem, configured)) return DASH_ERR_CUDA;
    return launch_pdl(gemm_kernel<EPI, BN, F32, CUT>, 2 * pairs, kGThreads, (size_t)smem, st, ma, mw, g) == cudaSuccess ? DASH_OK : DASH_ERR_CUDA;
}

// Tiles of 128 columns instead of 256 where every one of them still has a pair of SMs to itself.  What that saves is epilogue: an epilogue warp
// has half the columns (a 256 x 128 x 16 MMA takes the 134 cycles of a 256 x 256 x 16, so a tile's products take as long).  First
// tile in to the last result out, us, 256 / 128 columns: Q | K | V of the 7B shape at 233 rows 27 / 21, at 375 27 / 24, output projection at 233 28 / 23, at 375 28 / 24;
// fp32, 1024 rows of d = 256, Q | K | V 4.0 / 3.6, output projection 4.2 / 2.4.
static bool gemm_narrow(int m_tiles, int n_tiles, int P) { return 2LL * m_tiles * n_tiles <= P; }

// Groups of rows of tiles or of columns: the group's operand (16 tiles of 256 x 3584 are 29 MB, of 256 x 8192 67 MB) stays in L2 while the other one streams past
// it, once per group; of a K too deep for that (16 tiles of 256 x 18 944 are 155 MB) the pairs of a wave share what they go through side by side.  So of
// the two orders the one that reads less: (groups - 1) times the other operand more than both once.  The gate | up projection of
// 8192 rows, 32 x 148 tiles, reads 1.01 GB from HBM in groups of columns, 0.83 in groups of rows (its operands are 0.33 GB); the
// step runs at the power cap, where bytes are time: three blocks of 701, 6683, 8192 rows in a loop, columns / rows, us 883 / 877, 5772 / 5737,
// 7817 / 7768.  Groups of 8, 11 and 32: 8192 rows 7812, 7828, 7910.  Blocks of d = 8192, m = 28 672, columns / this rule: 2500 rows 3720 / 3530, 4096
// 5825 / 5750 (all four projections by rows, the down projection 28 672 deep), 5000 7370 / 7280 (gate | up), 8192 12 115 / 12 040 (Q | K | V, gate | up).
static bool gemm_by_m(int m_tiles, int n_tiles) {
    auto more = [](int grouped, int swept) { return (int64_t)((grouped + kGGroup - 1) / kGGroup - 1) * swept; };
    return more(m_tiles, n_tiles) < more(n_tiles, m_tiles);
}

template <int EPI, bool F32>
static int launch_gemm(const CUtensorMap& ma, const CUtensorMap& mw, GemmArgs g, cudaStream_t st) {
    const int m_tiles = (g.n + 2 * kGM - 1) / (2 * kGM);
    int pairs = sm_count() / 2;
    g.groups = gemm_groups(m_tiles, g.n_tiles, (g.K + kGK - 1) / kGK, pairs, g.part != nullptr);
    if (EPI != GEMM_SWIGLU && !g.groups && gemm_narrow(m_tiles, g.n_tiles, pairs)) {
        g.n_tiles = (g.N + kGNarrow - 1) / kGNarrow;
        return launch_tiles<EPI, EPI == GEMM_SWIGLU ? kGN : kGNarrow, F32, false>(ma, mw, g, m_tiles * g.n_tiles, st);
    }
    if constexpr (!F32) {                                     // (fp32 results come with no scratch for parts)
        if (g.groups) return launch_tiles<EPI, kGN, F32, true>(ma, mw, g, g.groups * m_tiles, st);
    }
    g.groups = 0;
    g.by_m = gemm_by_m(m_tiles, g.n_tiles);
    const int tiles = m_tiles * g.n_tiles;
    return launch_tiles<EPI, kGN, F32, false>(ma, mw, g, pairs > tiles ? tiles : pairs, st);
}

bool gemm_shape_ok(GemmEpilogueKind kind, int64_t n, int64_t N, int64_t K, int64_t lda, int64_t ldw, const GemmEpilogue& e) {
    if (n < 1 || n > 0x7fffffffLL || N < 1 || N > 0x7fffffffLL || K < 1 || K > 0x7fffffffLL || (lda % 8) || (ldw % 8)) return false;
    if (kind == GEMM_PLAIN) return (N % 4) == 0 && (K % 8) == 0;      // rows of A, W and C start on 16-byte boundaries
    // the fused epilogues work on whole 256-column tiles and whole K steps
    if (K < kGK || (K % kGK)) return false;
    if (kind == GEMM_SWIGLU) return e.m >= 128 && (e.m % 128) == 0 && N == 2 * (int64_t)e.m;
    if (N < kGN || (N % kGN)) return false;
    if (kind == GEMM_ROPE) return (e.D == 64 || e.D == 128) && (e.n_rot_cols % kGN) == 0 && e.n_rot_cols <= N;
    return true;
}

int gemm_bf16(GemmEpilogueKind kind, const void* A, int64_t lda, const void* W, int64_t ldw, void* C, int64_t ldc, int64_t n, int64_t N,
              int64_t K, const GemmEpilogue& e, const int32_t* n_dev, cudaStream_t st, bool out_f32, const GemmSplit* sc, bool w_early) {
    if (!gemm_shape_ok(kind, n, N, K, lda, ldw, e)) return DASH_ERR_UNSUPPORTED;
    if (!aligned16(A) || !aligned16(W)) return DASH_ERR_INVALID_ARG;
    if (out_f32 && kind != GEMM_PLAIN && kind != GEMM_ROPE) return DASH_ERR_UNSUPPORTED;
    if (out_f32 && kind == GEMM_ROPE && (!e.q_copy || !e.k_cache || !aligned16(C) || (ldc % 4))) return DASH_ERR_INVALID_ARG;
    if (kind == GEMM_PLAIN && (!aligned16(C) || (ldc * (out_f32 ? 4 : 2)) % 16 || (!out_f32 && (N % 8)))) return DASH_ERR_UNSUPPORTED;
    CUtensorMap ma, mw;
    int rc;
    if ((rc = make_map_2d_bf16(&ma, A, (uint64_t)K, (uint64_t)n, (uint64_t)lda, 64, kGM)) != DASH_OK) return rc;
    if ((rc = make_map_2d_bf16(&mw, W, (uint64_t)N, (uint64_t)K, (uint64_t)ldw, 64, kGK)) != DASH_OK) return rc;
    GemmArgs g;
    g.n = (int)n; g.N = (int)N; g.K = (int)K;
    g.n_tiles = kind == GEMM_SWIGLU ? e.m / 128 : (int)((N + kGN - 1) / kGN);
    g.C = C; g.ldc = ldc; g.n_dev = n_dev; g.e = e;
    g.w_early = w_early ? 1 : 0;
    g.part = sc ? sc->part : nullptr; g.arrived = sc ? sc->arrived : nullptr; g.groups = 0; g.by_m = 0;
    g.spin_limit = sc ? sc->spin_limit : kSpinLimit;
    g.status = status_word_ptr();
    if (!g.status) return DASH_ERR_CUDA;
    switch (kind) {
        case GEMM_PLAIN: return out_f32 ? launch_gemm<GEMM_PLAIN, true>(ma, mw, g, st) : launch_gemm<GEMM_PLAIN, false>(ma, mw, g, st);
        case GEMM_ROPE: return out_f32 ? launch_gemm<GEMM_ROPE, true>(ma, mw, g, st) : launch_gemm<GEMM_ROPE, false>(ma, mw, g, st);
        case GEMM_RESID: return launch_gemm<GEMM_RESID, false>(ma, mw, g, st);
        default: return launch_gemm<GEMM_SWIGLU, false>(ma, mw, g, st);
    }
}

int launch_rope_table(int64_t n, int D, double rope_base, float2* table, cudaStream_t st) {
    RopeFreqs fr;
    for (int i = 0; i < D / 2; ++i) fr.inv_freq[i] = pow(rope_base, -2.0 * i / D);
    int64_t blocks = (n + 7) / 8, cap = (int64_t)sm_count() * 8;
    if (blocks > cap) blocks = cap;
    rope_table_kernel<<<(int)blocks, 256, 0, st>>>(n, D / 2, fr, table);
    return cudaGetLastError() == cudaSuccess ? DASH_OK : DASH_ERR_CUDA;
}

}  // namespace dash

extern "C" int dash_testing_gemm_groups(int64_t n, int64_t N, int64_t K) {
    using namespace dash;
    if (n < 1 || N < 1 || K < 1) return 0;
    return gemm_groups((int)((n + 2 * kGM - 1) / (2 * kGM)), (int)((N + kGN - 1) / kGN), (int)((K + kGK - 1) / kGK), sm_count() / 2, true);
}

extern "C" int dash_testing_gemm_cut(const void* A, const void* W, void* C, int64_t n, int64_t N, int64_t K, int stall, uint32_t spin_limit, void* ws, size_t ws_bytes,
                                     void* stream) {
    using namespace dash;
    if (!A || !W || !C || n < 1 || N < 1 || K < 1 || spin_limit < 1 || spin_limit > kSpinLimit) return DASH_ERR_INVALID_ARG;
    const size_t count = gemm_split_count_bytes(), part = gemm_split_part_bytes(n, N, K);
    if (!part) return DASH_ERR_UNSUPPORTED;
    if (!ws || ((uintptr_t)ws % 256) || ws_bytes < count + part) return DASH_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    DASH_CUDA_TRY(cudaMemsetAsync(ws, 0, count, st));
    if (stall) DASH_CUDA_TRY(cudaMemsetAsync(ws, 1, 1, st));      // the first counter says 1: one pair too many will have said that it is done
    const GemmSplit sc = {(float*)((char*)ws + count), (unsigned int*)ws, spin_limit};
    return gemm_bf16(GEMM_PLAIN, A, K, W, N, C, N, n, N, K, GemmEpilogue(), nullptr, st, false, &sc);
}
