// Multi-query attention over many query positions at once (Section 3, the attention lines of the batched function:
// logits = einsum(bhnk,bmk->bhnm), weights = softmax(logits + mask), O = einsum(bhnm,bmv->bhnv)) under the mask of
// Section 2.3 for an autoregressive model.  This is the one part of the method whose arithmetic intensity is high:
// every K/V row is used by all h heads and by every later position, so it runs against the tensor-core roofline.
//
// Shape of the work on sm_100a.  A CTA takes TWO tiles of 128 query rows of one sequence, each 128 positions of a head or,
// where that fills the tiles better, fewer positions of several heads (PfShape; "head" below stands for tile; multi-query:
// the heads share K and V, so one staged K/V tile of 128 rows serves 256 query rows), and walks the cache rows up to their
// last position in stages of 128:
//     S_w   = Q_w K_j^T       tcgen05.mma, M = 128 query rows (TMEM lanes), N = 128 cache rows, fp32 in TMEM
//     P_w   = exp2(S_w log2e - m)   one thread per query row: the row's maximum and sum need no other thread
//     O_w  += P_w V_j         tcgen05.mma with A = P_w read from TMEM (bf16 pairs), B = V_j (MN-major)
// for w = 0, 1.  TMEM: ONE buffer of logits (128 columns) that the two heads use in turn, P_0 and P_1 (64 columns each, bf16
// pairs) and O_0, O_1 (128 each): all 512.  A head's logits are in registers a hundred cycles after they are there, the
// buffer then takes the other head's, and the weights wait in registers until the product before them has read the ones
// in tensor memory: so a head's logits are ready before it has finished the weights of the stage before, its product runs
// under its next softmax, and the two heads fall half a period apart by themselves.  (With P written over S, every stage of a
// head was a chain logits - softmax - product - logits; two heads' chains side by side left the tensor cores and the
// exponentials half idle.)  The reference maximum of a row moves only when the row's largest logit leads it by more than
// kPfMaxLead (then O_w's row is rescaled in TMEM by the row's own thread); P is bounded by 2^kPfMaxLead.
// Rows of a tile whose memory is shorter than 1024 rows feed P as bf16 hi + lo parts (two products, of half of the
// stage's rows each), like the decoding kernels, so that the rounding of few large weights stays inside the
// tolerance.
//
// Roles: warps 0-3 softmax of head 0, warps 4-7 softmax of head 1, warp 8 TMA producer, warp 9 issues the logits'
// products, warp 10 the weights' (two warps: with one, the gaps between waiting for a barrier and the first instruction
// added up to as much as the products).  The issuing warps stay together and elect a lane (elect_one): from code that
// only lane 0 runs, every tcgen05.mma took its descriptors from per-thread registers one by one, 82 cycles instead of 54.
//
// What bounds it: power.  A stage of both heads takes 2630 cycles (4400 before the logits had a buffer of their own and
// the issuers were taken apart; the tensor cores need 2048, the exponentials 2048), and at that rate the card holds its
// clock near 1.2 GHz.  32 x 32 heads x 4096 positions, in a loop: 5.0 ms -> 4.13 ms (1070 TFLOP/s).  Calls with few tiles, which
// are bound by the longest tile's chain of stages, go to mqa_prefill_tile_kernel below.
// Every wait is bounded; a wait that runs out flags PIPELINE_TIMEOUT and the CTA drains and leaves.
#pragma once
#include "decode_umma.cuh"

namespace mqa {

constexpr int kPfRows = 128;                                   // query positions per tile = cache rows per stage
constexpr int kPfTileBytes = kPfRows * kRowBytes;              // 32 KiB: 128 rows x 128 bf16, two 64-column boxes
constexpr int kPfHalfBytes = kPfTileBytes / 2;
constexpr int kPfKSlots = 2, kPfVSlots = 2;
constexpr int kPfThreads = 12 * 32;                            // (warp 11 only completes the third warpgroup)
constexpr int kPfProducerWarp = 8, kPfSWarp = 9, kPfPvWarp = 10;
constexpr int kPfRegsSoftmax = 216, kPfRegsOther = 72;
constexpr int kPfMaxSplit = 8;                                 // CTAs that share a tile's stages (mqa_prefill_tile_kernel)
constexpr float kPfMaxLead = 8.f;                              // log2 units a logit may exceed its row's reference by
// barriers: q_full, k_full/k_empty[2], v_full/v_empty[2], s_ready[2], p_ready[2], pv_done[2], s_free, q_empty
constexpr int kPfBarriers = 1 + 2 * kPfKSlots + 2 * kPfVSlots + 6 + 2;
constexpr int kPfOutBytes = 32 * 128;                          // a softmax warp's rows of O on their way out, 32 columns at a time
constexpr int kPfSmemBytes = (2 + kPfKSlots + kPfVSlots) * kPfTileBytes + 8 * kPfOutBytes + kPfBarriers * 8 + 16 + 1024 /* alignment slack */;
// tensor memory columns: the logits of one stage and head, the two heads' weights, the two accumulators
constexpr uint32_t kPfTmemP = 128, kPfTmemO = 256;
static_assert(kPfSmemBytes <= 227 * 1024, "exceeds the shared memory of one SM");

// two fp32 values in one 64-bit register: packed multiply-add and add (one instruction for two elements)
__device__ __forceinline__ unsigned long long f2_pack(float lo, float hi) {
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ void f2_unpack(unsigned long long v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// A tile is `positions` consecutive positions of `heads` consecutive heads, positions * heads <= 128 rows: row r is position
// r % positions of head r / positions (one box of Q as a [b h][n][128] tensor).  A sequence's tiles are numbered position
// block by position block, the heads' blocks within it, and a unit of work is two tiles in a row.  Units go out in groups of
// those that share a position block, the longest memories first, all sequences of a group after one another; CTA c takes
// units c, 2 grid - 1 - c, ... one after the other (a persistent kernel: barriers, tensor memory and the K/V rings are set
// up once, and the next unit's Q and first stages are fetched, and its first logits computed, while the softmax warps
// still write the unit before out).
struct PfShape {
    int b, h, n, m_max;
    int positions, heads;                 // of a tile
    int head_blocks, n_tiles, n_units;    // of a sequence
    int group;                            // units that go out together for one sequence
    int n_items;
};
struct PfItem {
    int seq, raw, L, n_kv;
    int tile0, n_act;                     // its first tile, how many it has (the last unit of a sequence may have one)
    int L0, n_kv0;                        // L and n_kv of the first tile alone (its positions may be earlier than the second's)
    bool hilo;
};
__device__ __forceinline__ int pf_position(const PfShape& sh, int tile) { return tile / sh.head_blocks * sh.positions; }   // the tile's first
__device__ __forceinline__ int pf_head(const PfShape& sh, int tile) { return tile % sh.head_blocks * sh.heads; }
// A tile goes no further than its own last position: a weight of zero does not silence a V row that is not finite, so what
// the unit's other tile sees beyond that must not enter its products.  The first tile of a unit may end earlier, by stages,
// and inside its last stage by rows: of that stage the whole steps of 16 rows below L0 are multiplied as they lie, and the step
// that L0 falls into from a copy whose rows from L0 on are zeros (pf_cut).  (The copy is made by the warp that issues those products: made
// by the softmax warps it cost every stage of every call 2 %, by way of their registers.)  What it costs: 5 x 9 heads x 333
// positions over up to 3000 rows 29.5 -> 30.0 us, 1 x 21 x 480 over 1242 21.2 -> 22.1 (a unit runs that code once, cold; the
// same with loops, votes, or a block of zeros for the steps left out: 21.9 to 22.5).  Inside a tile, a later position's row still reaches the earlier ones.
__device__ __forceinline__ PfItem pf_item(int item, const int32_t* start, const PfShape& sh) {
    PfItem it;
    it.seq = (item / sh.group) % sh.b;
    const int unit = sh.n_units - 1 - (item / (sh.group * sh.b) * sh.group + item % sh.group);
    it.n_act = unit < 0 ? 0 : min(2, sh.n_tiles - 2 * unit);     // (the last group may be partly filled)
    it.raw = start ? min(__ldcg(start + it.seq), sh.m_max) : 0;
    it.tile0 = 2 * unit;
    // rows of the memory the unit's last position sees (rows of a tile past the last position or head are computed on
    // whatever the Q tile holds there and never stored); a memory that would pass m_max is cut there
    it.L = min(it.raw + min(pf_position(sh, it.tile0 + it.n_act - 1) + sh.positions, sh.n), sh.m_max);
    const bool empty = it.n_act == 0 || it.raw < 0 || it.L <= 0; // nothing to look at: zeros (like a bad lens)
    it.n_kv = empty ? 0 : (it.L + kPfRows - 1) / kPfRows;        // stages
    it.L0 = min(it.raw + min(pf_position(sh, it.tile0) + sh.positions, sh.n), sh.m_max);
    it.n_kv0 = empty ? 0 : (it.L0 + kPfRows - 1) / kPfRows;
    // one rounding of the weights where the last position of the block of 128 that the unit's FIRST tile begins in sees
    // kSingleRoundingMinRows rows (its second tile goes with it)
    it.hilo = min(it.raw + min((pf_position(sh, it.tile0) & ~(kPfRows - 1)) + kPfRows, sh.n), sh.m_max) < kSingleRoundingMinRows;
    return it;
}
// Rows of the first tile's last stage that are its own, if the unit's other tile sees more of them; else 0.
__device__ __forceinline__ int pf_cut(const PfItem& it) { return it.L0 < it.L ? it.L0 & (kPfRows - 1) : 0; }
// The row of [b h n, 128] that row r of the unit's tile w is, or -1.
__device__ __forceinline__ int pf_row(const PfItem& it, const PfShape& sh, int w, int r) {
    const int hh = r / sh.positions, head = pf_head(sh, it.tile0 + w) + hh, pos = pf_position(sh, it.tile0 + w) + r - hh * sh.positions;
    return hh < sh.heads && head < sh.h && pos < sh.n && w < it.n_act ? (it.seq * sh.h + head) * sh.n + pos : -1;
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}

__global__ void __launch_bounds__(kPfThreads, 1)
mqa_prefill_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                   const __grid_constant__ CUtensorMap map_v, const int32_t* start, float* __restrict__ O,
                   int32_t* __restrict__ status, const PfShape sh) {
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);     // the 128-byte swizzle repeats every 1 KiB
    const uint32_t q_s = smem_addr(base);
    const uint32_t k_ring = q_s + 2 * kPfTileBytes, v_ring = k_ring + kPfKSlots * kPfTileBytes;
    const uint32_t out_s = v_ring + kPfVSlots * kPfTileBytes, bars = out_s + 8 * kPfOutBytes;
    const uint32_t q_empty = bars + 8 * (kPfBarriers - 1);       // the unit's Q tiles have been read for the last time
    const uint32_t s_free = bars + 8 * (kPfBarriers - 2);        // the logits have been read into registers
    const uint32_t q_full = bars, k_full = bars + 8, k_empty = k_full + 8 * kPfKSlots, v_full = k_empty + 8 * kPfKSlots,
                   v_empty = v_full + 8 * kPfVSlots, s_ready = v_empty + 8 * kPfVSlots, p_ready = s_ready + 16,
                   pv_done = p_ready + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + (2 + kPfKSlots + kPfVSlots) * kPfTileBytes + 8 * kPfOutBytes + kPfBarriers * 8);
    __shared__ int timed_out;

    if (threadIdx.x == 0) {
        prefetch_tensormap(&map_q); prefetch_tensormap(&map_k); prefetch_tensormap(&map_v);
        mbar_init(q_full, 1);
        mbar_init(q_empty, 1);
        mbar_init(s_free, 4);
        for (int i = 0; i < kPfKSlots; ++i) { mbar_init(k_full + 8 * i, 1); mbar_init(k_empty + 8 * i, 1); }
        for (int i = 0; i < kPfVSlots; ++i) { mbar_init(v_full + 8 * i, 1); mbar_init(v_empty + 8 * i, 1); }
        for (int w = 0; w < 2; ++w) { mbar_init(s_ready + 8 * w, 1); mbar_init(p_ready + 8 * w, 4); mbar_init(pv_done + 8 * w, 1); }
        timed_out = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kPfSWarp) {
        tmem_alloc(smem_addr(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    grid_dependency_wait();              // Q, K, V and start may come from the kernel before
    grid_launch_dependents();
    // the units of this CTA: c, 2G - 1 - c, 2G + c, 4G - 1 - c, ... (G CTAs; the units come longest first, so taking them
    // forwards and backwards in turn evens the CTAs' totals out)
    const int n_items = sh.n_items;
    auto pf_unit = [&](int round) -> int {
        const int G = (int)gridDim.x, c = (int)blockIdx.x;
        return round * G + ((round & 1) ? G - 1 - c : c);
    };
    if (start && threadIdx.x < 32) {
        // a start that is negative or leaves too little room is flagged once (its rows are zeros, or the memory is cut at m_max)
        bool bad = false;
        for (int i = blockIdx.x * 32 + threadIdx.x; i < sh.b; i += gridDim.x * 32) {
            const int first = __ldcg(start + i);
            bad = bad || first < 0 || first > sh.m_max - sh.n;
        }
        if (bad && status) atomicOr(status, kStatusLenClamped);
    }

    if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPfRegsOther));
    if (warp == kPfProducerWarp) {
        // =============================================================== TMA producer
        if (lane == 0) {
            bool ok = true;
            int g = 0, qi = 0;                                   // stages and units so far (they number the barriers' phases)
            int issued_k = 0, issued_v = 0, issued_q = 0;
            // (for tests: CTA 0 never starts one copy of the second stage of its first unit)
            const bool withhold = blockIdx.x == 0 && test_withhold();
            for (int round = 0, item; (item = pf_unit(round)) < n_items && ok; ++round) {
                const PfItem it = pf_item(item, start, sh);
                const int n_kv = it.n_kv;
                if (n_kv == 0) continue;
                if (qi > 0) ok = mbar_wait(q_empty, (qi - 1) & 1);            // the unit before has read its Q for the last time
                if (!ok) break;
                mbar_expect_tx(q_full, it.n_act * sh.positions * sh.heads * kRowBytes);
                for (int w = 0; w < it.n_act; ++w)
                    for (int half = 0; half < 2; ++half)
                        tma_load_3d(q_s + w * kPfTileBytes + half * kPfHalfBytes, &map_q, half * kBoxCols, pf_position(sh, it.tile0 + w),
                                    it.seq * sh.h + pf_head(sh, it.tile0 + w), q_full);
                issued_q = qi + 1;
                for (int j = 0; j < n_kv && ok; ++j) {
                    const int G = g + j;
                    const int y = it.seq * sh.m_max + j * kPfRows;
                    const int ks = G % kPfKSlots, vs = G % kPfVSlots;
                    if (G >= kPfKSlots) ok = mbar_wait(k_empty + 8 * ks, ((G / kPfKSlots) - 1) & 1);
                    if (!ok) break;
                    mbar_expect_tx(k_full + 8 * ks, kPfTileBytes);
                    tma_load_2d(k_ring + ks * kPfTileBytes, &map_k, 0, y, k_full + 8 * ks);
                    tma_load_2d(k_ring + ks * kPfTileBytes + kPfHalfBytes, &map_k, kBoxCols, y, k_full + 8 * ks);
                    issued_k = G + 1;
                    if (G >= kPfVSlots) ok = mbar_wait(v_empty + 8 * vs, ((G / kPfVSlots) - 1) & 1);
                    if (!ok) break;
                    mbar_expect_tx(v_full + 8 * vs, kPfTileBytes);
                    tma_load_2d(v_ring + vs * kPfTileBytes, &map_v, 0, y, v_full + 8 * vs);
                    if (!(withhold && G == 1)) tma_load_2d(v_ring + vs * kPfTileBytes + kPfHalfBytes, &map_v, kBoxCols, y, v_full + 8 * vs);
                    issued_v = G + 1;
                }
                g += n_kv;
                ++qi;
            }
            if (!ok) {
                // a wait ran out: the copies already started are given a bounded wait each before the CTA may leave
                atomicExch(&timed_out, 1);
                if (issued_q > 0) mbar_wait(q_full, (issued_q - 1) & 1);
                for (int G = max(0, issued_k - kPfKSlots); G < issued_k; ++G) mbar_wait(k_full + 8 * (G % kPfKSlots), (G / kPfKSlots) & 1);
                for (int G = max(0, issued_v - kPfVSlots); G < issued_v; ++G) mbar_wait(v_full + 8 * (G % kPfVSlots), (G / kPfVSlots) & 1);
            }
        }
    } else if (warp == kPfSWarp) {
        // =============================================================== issuer of the logits: S = Q_w K^T, the heads in turn,
        // each as soon as the ones before are in registers
        constexpr uint32_t kIdescS = umma_idesc(128, 128, false, false);
        bool ok = true;
        int g = 0, qi = 0, n_s = 0;                              // stages, units and logits so far
        for (int round = 0, item; (item = pf_unit(round)) < n_items && ok; ++round) {
            const PfItem it = pf_item(item, start, sh);
            const int n_kv = __shfl_sync(0xffffffffu, it.n_kv, 0), n_act = it.n_act;
            const int n_kv0 = __shfl_sync(0xffffffffu, it.n_kv0, 0);
            if (n_kv == 0) continue;
            ok = warp_wait(q_full, qi & 1);
            for (int j = 0; j < n_kv && ok; ++j, ++g) {
                const int slot = g % kPfKSlots;
                const uint32_t k_s = k_ring + slot * kPfTileBytes;
                ok = warp_wait(k_full + 8 * slot, (g / kPfKSlots) & 1);
                for (int w = 0; w < n_act && ok; ++w) {
                    if (w == 0 && j >= n_kv0) continue;
                    if (n_s > 0) ok = warp_wait(s_free, (n_s - 1) & 1);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint32_t qw = q_s + w * kPfTileBytes;
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks) {         // 8 k-steps of 16 columns; 4 per 64-column box
                            const uint32_t off = (ks >> 2) * kPfHalfBytes + (ks & 3) * 32;
                            umma_ss(tmem_base, umma_desc(qw + off, 16, 1024), umma_desc(k_s + off, 16, 1024), kIdescS, ks ? 1u : 0u);
                        }
                        tc_commit(s_ready + 8 * w);
                        if (w == n_act - 1) {
                            tc_commit(k_empty + 8 * slot);
                            if (j == n_kv - 1) tc_commit(q_empty);       // the unit's last logits are on their way
                        }
                    }
                    __syncwarp();
                    ++n_s;
                }
            }
            ++qi;
        }
        if (!ok && lane == 0) atomicExch(&timed_out, 1);
    } else if (warp == kPfPvWarp) {
        // =============================================================== issuer of O_w += P_w V: P from tensor memory (bf16 pairs: 8
        // columns per 16 rows of V), in two parts where the weights have a hi and a lo one
        constexpr uint32_t kIdescO = umma_idesc(128, 128, false, true);
        bool ok = true;
        int g = 0, n_p[2] = {0, 0};                              // stages and each head's weights so far
        for (int round = 0, item; (item = pf_unit(round)) < n_items && ok; ++round) {
            const PfItem it = pf_item(item, start, sh);
            const int n_kv = __shfl_sync(0xffffffffu, it.n_kv, 0), n_act = it.n_act, parts = __any_sync(0xffffffffu, it.hilo) ? 2 : 1;
            const int n_kv0 = __shfl_sync(0xffffffffu, it.n_kv0, 0);
            // (the stage that is cut.  A reduction over the warp leaves its result where the issue of a product can test it: 0.4 us
            // less for a unit than with a shuffle)
            const int cut = __reduce_max_sync(0xffffffffu, pf_cut(it)), cut_j = cut > 0 ? it.n_kv0 - 1 : -1;
            for (int j = 0; j < n_kv && ok; ++j, ++g) {
                const int slot = g % kPfVSlots;
                const uint32_t v_s = v_ring + slot * kPfTileBytes;
                ok = warp_wait(v_full + 8 * slot, (g / kPfVSlots) & 1);
                for (int w = 0; w < n_act && ok; ++w) {
                    if (w == 0 && j >= n_kv0) continue;
                    const bool whole = __all_sync(0xffffffffu, w > 0 || j != cut_j);
                    if (!whole && (cut & 15)) {
                        // the 16 rows that the first tile ends in, zeros from its end on, to the place where its softmax warps hand O out
                        // (with those of the unit before they are through once this stage's weights are there)
                        ok = warp_wait(p_ready, n_p[0] & 1);
                        uint4 v[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {            // 16-byte pieces, eight to a row of a 64-column half
                            const int at = (i >> 2) * kPfHalfBytes + ((cut & ~15) + (i & 3) * 4) * 128 + lane * 16;
                            asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v[i].x), "=r"(v[i].y), "=r"(v[i].z), "=r"(v[i].w) : "r"(v_s + at) : "memory");
                        }
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            if ((i & 3) * 4 + (lane >> 3) >= (cut & 15)) v[i] = make_uint4(0u, 0u, 0u, 0u);
                            asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(out_s + (i * 32 + lane) * 16), "r"(v[i].x), "r"(v[i].y), "r"(v[i].z), "r"(v[i].w) : "memory");
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                    }
                    for (int part = 0; part < parts && ok; ++part) {
                        ok = warp_wait(p_ready + 8 * w, n_p[w] & 1);
                        if (!ok) break;
                        ++n_p[w];
                        tc_fence_after();
                        if (whole) {
                            if (elect_one()) {
                                // one rounding: the stage's 128 rows; hi and lo: 64 of them, twice over
                                const uint32_t v_p = v_s + part * 4 * 2048;
#pragma unroll
                                for (int kk = 0; kk < 8; ++kk)
                                    umma_ts(tmem_base + kPfTmemO + w * 128, tmem_base + kPfTmemP + w * 64 + kk * 8,
                                            umma_desc(v_p + (parts == 2 ? kk & 3 : kk) * 2048, kPfHalfBytes, 1024), kIdescO, (j == 0 && part == 0 && kk == 0) ? 0u : 1u);
                                tc_commit(pv_done + 8 * w);
                                if (w == n_act - 1 && part == parts - 1) tc_commit(v_empty + 8 * slot);
                            }
                        } else if (elect_one()) {
                            // the first tile's last stage, up to its last row (the other tile has the stage too)
#pragma unroll
                            for (int kk = 0; kk < 8; ++kk) {
                                const int row = (parts == 2 ? part * 4 + (kk & 3) : kk) * 16;
                                if (row < cut)
                                    umma_ts(tmem_base + kPfTmemO, tmem_base + kPfTmemP + kk * 8,
                                            row + 16 > cut ? umma_desc(out_s, 2048, 1024) : umma_desc(v_s + row * 128, kPfHalfBytes, 1024),
                                            kIdescO, (j == 0 && part == 0 && kk == 0) ? 0u : 1u);
                            }
                            tc_commit(pv_done);
                        }
                        __syncwarp();
                    }
                }
            }
        }
        if (!ok && lane == 0) atomicExch(&timed_out, 1);
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPfRegsSoftmax));
        // =============================================================== softmax warps: one thread per query row
        const int w = warp >> 2, quarter = warp & 3, r = quarter * 32 + lane;
        const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const uint32_t p_t = lane_base + kPfTmemP + w * 64, o_t = lane_base + kPfTmemO + w * 128;
        const uint32_t out_w = out_s + warp * kPfOutBytes;
        bool ok = true;
        int g = 0, n_s = 0, n_p = 0;                             // stages of the CTA, logits and weights of this head so far
        for (int round = 0, item; (item = pf_unit(round)) < n_items; ++round) {
            const PfItem it = pf_item(item, start, sh);
            const int n_kv = it.n_kv;
            const int my_row = pf_row(it, sh, w, r);             // where this thread's row of O goes (-1: nowhere)
            if (w >= it.n_act) { g += n_kv; continue; }        // (the last unit of a sequence may have one tile)
            if (n_kv == 0) {
                if (my_row >= 0)
                    for (int i = 0; i < kHeadDim; i += 4) *reinterpret_cast<float4*>(O + (size_t)my_row * kHeadDim + i) = make_float4(0.f, 0.f, 0.f, 0.f);
                continue;
            }
            const int p0 = pf_position(sh, it.tile0 + w);
            const int lim_first = min(it.raw + p0 + 1, it.L);            // rows the tile's first position sees
            const int lim = min(it.raw + min(p0 + r % sh.positions, sh.n - 1) + 1, it.L);   // rows this thread's position sees: >= 1
            float m = -INFINITY, l = 0.f;                        // reference maximum (log2 units), sum of weights
            const int n_own = w == 0 ? it.n_kv0 : n_kv;                                  // stages of this tile
            const bool clears = w == (it.n_kv0 == it.n_kv ? 0 : 1);                      // the first tile to see the unit's last stage
            for (int j = 0; j < n_own; ++j) {
                const int k0 = j * kPfRows;
                if (ok) ok = mbar_wait(s_ready + 8 * w, n_s & 1);
                ++n_s;
                tc_fence_after();
                const bool diag = k0 + kPfRows > lim_first;           // some position of the tile cannot see all of this stage
                // ---- the row's 128 logits, read once and kept in registers.  The mask of Section 2.3 is applied
                // by index, as a select: what lies behind a masked logit is never used.
                uint32_t x[128];
                tmem_ld_cols<128>(lane_base, x);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(s_free);                   // the other head's logits may take their place
                if (diag) {
#pragma unroll
                    for (int i = 0; i < 128; ++i)
                        if (k0 + i >= lim) x[i] = 0xff800000u;        // -inf
                }
                float mx8[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) mx8[i] = fmaxf(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1]));
#pragma unroll
                for (int i = 8; i < 64; ++i) mx8[i & 7] = max3(mx8[i & 7], __uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1]));
                const float mx = max3(max3(mx8[0], mx8[1], mx8[2]), max3(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7])) * kLog2e;
                // (a row that is nobody's does not count: its query is whatever shared memory held, and the moment at which a warp
                // moves its references shows in the last bits of all of them)
                if (__any_sync(0xffffffffu, my_row >= 0 && mx > m + kPfMaxLead)) {
                    const float m_new = fmaxf(m, mx);
                    if (j > 0) {
                        // (a row whose logits have all been -inf, or which has seen nothing yet of a run of stages, has m = -inf)
                        const float f = m == m_new ? 1.f : fast_exp2(m - m_new);
                        l *= f;
                        if (ok) ok = mbar_wait(pv_done + 8 * w, (n_p - 1) & 1);           // O holds the stages before this one
                        tc_fence_after();
#pragma unroll 1
                        for (int c = 0; c < 16; ++c) {
                            uint32_t y[8];
                            tmem_ld8(o_t + c * 8, y);
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < 8; ++i) y[i] = __float_as_uint(__uint_as_float(y[i]) * f);
                            tmem_st8(o_t + c * 8, y);
                        }
                    }
                    m = m_new;
                }
                const float neg_m = m == -INFINITY ? 0.f : -m;      // (weights of zero)
                const unsigned long long neg_m2 = f2_pack(neg_m, neg_m), log2e2 = f2_pack(kLog2e, kLog2e);
                unsigned long long sum2[2] = {0ull, 0ull};
                if (clears && it.L < k0 + kPfRows) {
                    // the last stage runs past the memory: the tensor core would multiply the zero weights with
                    // whatever lies there (NaN * 0 = NaN), so those V rows are cleared first
                    const int vs = (g + j) % kPfVSlots;
                    if (ok) ok = mbar_wait(v_full + 8 * vs, ((g + j) / kPfVSlots) & 1);
                    const uint32_t v_s = v_ring + vs * kPfTileBytes;
                    const int first = it.L - k0;
                    for (int i = r; i < (kPfRows - first) * 16; i += 128) {
                        const int vrow = first + (i >> 4), ch = i & 15;
                        const uint32_t a = v_s + (ch >> 3) * kPfHalfBytes + vrow * 128 + ((ch & 7) << 4);
                        asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(a), "r"(0u) : "memory");
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                }
                // the weights stay in registers until the product before has read the ones in tensor memory
                auto give = [&](const uint32_t (&p0)[32], const uint32_t (&p1)[32]) {
                    if (n_p > 0 && ok) ok = mbar_wait(pv_done + 8 * w, (n_p - 1) & 1);
                    tc_fence_after();
                    tmem_st32(p_t, p0);
                    tmem_st32(p_t + 32, p1);
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(p_ready + 8 * w);
                    ++n_p;
                };
                if (it.hilo) {
                    // hi and lo parts of half of the stage's rows at a time: the first half's product runs under the other's exponentials
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        uint32_t hi[32], lo[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            float a0, a1;
                            f2_unpack(f2_fma(f2_pack(__uint_as_float(x[64 * half + 2 * i]), __uint_as_float(x[64 * half + 2 * i + 1])), log2e2, neg_m2), a0, a1);
                            const float pa = fast_exp2(a0), pb = fast_exp2(a1);
                            sum2[i & 1] = f2_add(sum2[i & 1], f2_pack(pa, pb));
                            hi[i] = pack_bf16(pa, pb);
                            lo[i] = pack_bf16(pa - bf16_lo(hi[i]), pb - bf16_hi(hi[i]));
                        }
                        give(hi, lo);
                    }
                } else {
                    uint32_t hi[2][32];
#pragma unroll
                    for (int i = 0; i < 64; ++i) {
                        float a0, a1;
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1])), log2e2, neg_m2), a0, a1);
                        const float pa = fast_exp2(a0), pb = fast_exp2(a1);
                        sum2[i & 1] = f2_add(sum2[i & 1], f2_pack(pa, pb));
                        hi[i >> 5][i & 31] = pack_bf16(pa, pb);
                    }
                    give(hi[0], hi[1]);
                }
                {
                    float s0, s1;
                    f2_unpack(f2_add(sum2[0], sum2[1]), s0, s1);
                    l += s0 + s1;
                }
            }
            // ---- the row of O, divided by the sum of its weights
            if (ok) ok = mbar_wait(pv_done + 8 * w, (n_p - 1) & 1);
            tc_fence_after();
            const float inv = 1.f / l;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t y[32];
                tmem_ld32(o_t + c * 32, y);
                tmem_wait_ld();
                // 32 columns of the warp's 32 rows through shared memory, so that they leave as 128-byte pieces (straight from
                // here a store instruction would touch 32 rows, 16 bytes of each)
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(out_w + lane * 128 + ((i ^ (lane & 7)) << 4)),
                                 "f"(__uint_as_float(y[4 * i]) * inv), "f"(__uint_as_float(y[4 * i + 1]) * inv),
                                 "f"(__uint_as_float(y[4 * i + 2]) * inv), "f"(__uint_as_float(y[4 * i + 3]) * inv) : "memory");
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int rr = i * 4 + (lane >> 3), row = __shfl_sync(0xffffffffu, my_row, rr);
                    float4 v;
                    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                                 : "r"(out_w + rr * 128 + (((lane & 7) ^ (rr & 7)) << 4)) : "memory");
                    if (row >= 0) *reinterpret_cast<float4*>(O + (size_t)row * kHeadDim + c * 32 + (lane & 7) * 4) = v;
                }
                __syncwarp();
            }
            tc_fence_before();                                   // (the next unit's first product overwrites O once its weights are in)
            g += n_kv;
        }
        if (!ok) atomicExch(&timed_out, 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kPfSWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0 && timed_out && status) atomicOr(status, kStatusPipelineTimeout);
}

// ---- Few tiles (a chunk of a prompt, short prompts, few sequences): ONE tile per CTA, so that twice as many SMs work, and the two
// softmax warpgroups take its stages in turn (warpgroup w: stages w, w + 2, ...), each with weights, an O accumulator, reference
// maxima and sums of its own, merged on the way out -- the order of work of the many-rows step (decode_wide.cuh), under the mask of
// Section 2.3.  A cluster of 2, 4 or 8 CTAs shares a tile's stages where there are SMs for it, each a run of them; their partial
// results go straight to the CTA that merges them (128 / CTAs rows each), from the merge of the warpgroups into its V ring.
// (Before it the two tiles of a unit stayed together and a cluster shared the unit: its rows of O went into shared memory and were
// read from there by remote loads, 24 KB/us, 7 us in all after the last product.)  A stage takes 0.72 us (1.05 with two roundings of
// the weights), half of what it takes for two tiles, and 8 us are around them.  us per call: 5 x 9 heads x 333 positions over up to 3000
// rows 28.5 -> 25.5; 8 x 8 x 256 over 900 22.1 -> 16.7; 4 x 23 x 115 over 1682 24.6 -> 18.1; 1 x 8 x 1000 17.3 -> 16.1.
constexpr int kPtKSlots = 3, kPtVSlots = 3;
// barriers: q_full, k_full/k_empty, v_full/v_empty per slot, s_ready[2], p_ready[2], pv_done[2], s_free, recv
constexpr int kPtBarriers = 1 + 2 * kPtKSlots + 2 * kPtVSlots + 6 + 2;
constexpr int kPtSmemBytes = (1 + kPtKSlots + kPtVSlots) * kPfTileBytes + kPtBarriers * 8 + 16 + 1024 /* alignment slack */;
static_assert(kPtSmemBytes + kPfRows * 12 + 16 /* static */ <= 227 * 1024, "exceeds the shared memory of one SM");

__global__ void __launch_bounds__(kPfThreads, 1)
mqa_prefill_tile_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                        const __grid_constant__ CUtensorMap map_v, const int32_t* start, float* __restrict__ O,
                        int32_t* __restrict__ status, const PfShape sh) {
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int ctas = (int)cluster_size(), rank = (int)cluster_cta_rank(), item = (int)blockIdx.x / ctas;
    const int per = kPfRows / ctas;                              // rows that each CTA of the cluster merges

    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);     // the 128-byte swizzle repeats every 1 KiB
    const uint32_t q_s = smem_addr(base);
    const uint32_t k_ring = q_s + kPfTileBytes, v_ring = k_ring + kPtKSlots * kPfTileBytes, bars = v_ring + kPtVSlots * kPfTileBytes;
    const uint32_t q_full = bars, k_full = bars + 8, k_empty = k_full + 8 * kPtKSlots, v_full = k_empty + 8 * kPtKSlots,
                   v_empty = v_full + 8 * kPtVSlots, s_ready = v_empty + 8 * kPtVSlots, p_ready = s_ready + 16, pv_done = p_ready + 16,
                   s_free = pv_done + 16, recv_bar = s_free + 8;
    const uint32_t recv_ml = v_ring + kPfRows * 512;             // (the rows that come lie where the first two V slots were)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + (1 + kPtKSlots + kPtVSlots) * kPfTileBytes + kPtBarriers * 8);
    __shared__ int timed_out, ex_row[kPfRows];                   // where each row of O goes (-1: nowhere)
    __shared__ float2 ex_ml[kPfRows];                            // (maximum, sum) of warpgroup 1's rows, then each row's two factors

    if (threadIdx.x == 0) {
        prefetch_tensormap(&map_q); prefetch_tensormap(&map_k); prefetch_tensormap(&map_v);
        mbar_init(q_full, 1);
        mbar_init(s_free, 4);
        for (int i = 0; i < kPtKSlots; ++i) { mbar_init(k_full + 8 * i, 1); mbar_init(k_empty + 8 * i, 1); }
        for (int i = 0; i < kPtVSlots; ++i) { mbar_init(v_full + 8 * i, 1); mbar_init(v_empty + 8 * i, 1); }
        for (int w = 0; w < 2; ++w) { mbar_init(s_ready + 8 * w, 1); mbar_init(p_ready + 8 * w, 4); mbar_init(pv_done + 8 * w, 1); }
        mbar_init(recv_bar, 1);
        timed_out = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(recv_bar, (uint32_t)((ctas - 1) * per * (kHeadDim * 4 + 8)));
    }
    if (warp == kPfSWarp) {
        tmem_alloc(smem_addr(tmem_slot), 512);
        tmem_relinquish();
    }
    // the tile: everything but where its sequence starts is known ahead of the wait
    const int seq = (item / sh.group) % sh.b, tile = sh.n_units - 1 - (item / (sh.group * sh.b) * sh.group + item % sh.group);
    const int p0 = pf_position(sh, tile), head0 = pf_head(sh, tile);
    // where the block of 128 that the pair's first tile begins in ends (see hilo below)
    const int block_end = min((pf_position(sh, tile & ~1) & ~(kPfRows - 1)) + kPfRows, sh.n);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    grid_dependency_wait();              // Q, K, V and start may come from the kernel before
    grid_launch_dependents();
    const int raw = start ? min(__ldcg(start + seq), sh.m_max) : 0;
    if (start && threadIdx.x < 32) {
        // a start that is negative or leaves too little room is flagged once (its rows are zeros, or the memory is cut at m_max)
        bool bad = false;
        for (int i = blockIdx.x * 32 + threadIdx.x; i < sh.b; i += gridDim.x * 32) {
            const int first = __ldcg(start + i);
            bad = bad || first < 0 || first > sh.m_max - sh.n;
        }
        if (bad && status) atomicOr(status, kStatusLenClamped);
    }
    const int L = min(raw + min(p0 + sh.positions, sh.n), sh.m_max);     // rows of the memory that the tile's last position sees
    const int n_all = raw < 0 || L <= 0 ? 0 : (L + kPfRows - 1) / kPfRows;
    const int first = rank * n_all / ctas, n_kv = __shfl_sync(0xffffffffu, (rank + 1) * n_all / ctas - first, 0);   // this CTA's stages
    // two roundings of the weights: by the first of the two tiles that the other kernel takes together, as pf_item does, so that a
    // position's precision does not depend on which kernel the batch sends it to
    const bool hilo = __any_sync(0xffffffffu, min(raw + block_end, sh.m_max) < kSingleRoundingMinRows);

    if (warp >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPfRegsOther));
        if (warp == kPfProducerWarp) {
            // =========================================================== TMA producer: a box per lane
            bool ok = true;
            int issued_k = 0, issued_v = 0;
            // (for tests: CTA 0 never starts one copy of its second stage, or of its only one)
            const bool withhold = blockIdx.x == 0 && test_withhold();
            if (n_kv > 0) {
                if (lane == 0) mbar_expect_tx(q_full, sh.positions * sh.heads * kRowBytes);
                if (lane < 2) tma_load_3d(q_s + lane * kPfHalfBytes, &map_q, lane * kBoxCols, p0, seq * sh.h + head0, q_full);
            }
            for (int j = 0; j < n_kv; ++j) {
                const int y = seq * sh.m_max + (first + j) * kPfRows, ks = j % kPtKSlots, vs = j % kPtVSlots;
                if (j >= kPtKSlots) ok = warp_wait(k_empty + 8 * ks, ((j / kPtKSlots) - 1) & 1);
                if (!ok) break;
                if (lane == 0) mbar_expect_tx(k_full + 8 * ks, kPfTileBytes);
                if (lane < 2) tma_load_2d(k_ring + ks * kPfTileBytes + lane * kPfHalfBytes, &map_k, lane * kBoxCols, y, k_full + 8 * ks);
                issued_k = j + 1;
                if (j >= kPtVSlots) ok = warp_wait(v_empty + 8 * vs, ((j / kPtVSlots) - 1) & 1);
                if (!ok) break;
                if (lane == 0) mbar_expect_tx(v_full + 8 * vs, kPfTileBytes);
                if (lane < 2 && !(withhold && lane == 1 && j == min(1, n_kv - 1)))
                    tma_load_2d(v_ring + vs * kPfTileBytes + lane * kPfHalfBytes, &map_v, lane * kBoxCols, y, v_full + 8 * vs);
                issued_v = j + 1;
            }
            if (!ok) {
                // a wait ran out: the copies already started are given a bounded wait each before the CTA may leave
                if (lane == 0) atomicExch(&timed_out, 1);
                mbar_wait(q_full, 0);
                for (int j = max(0, issued_k - kPtKSlots); j < issued_k; ++j) mbar_wait(k_full + 8 * (j % kPtKSlots), (j / kPtKSlots) & 1);
                for (int j = max(0, issued_v - kPtVSlots); j < issued_v; ++j) mbar_wait(v_full + 8 * (j % kPtVSlots), (j / kPtVSlots) & 1);
            }
        } else if (warp == kPfSWarp) {
            // =========================================================== issuer of the logits, each stage as soon as the one before is
            // in registers
            constexpr uint32_t kIdescS = umma_idesc(128, 128, false, false);
            bool ok = n_kv == 0 || warp_wait(q_full, 0);
            for (int j = 0; j < n_kv && ok; ++j) {
                const int slot = j % kPtKSlots;
                ok = warp_wait(k_full + 8 * slot, (j / kPtKSlots) & 1);
                if (ok && j > 0) ok = warp_wait(s_free, (j - 1) & 1);
                if (!ok) break;
                const uint32_t k_s = k_ring + slot * kPfTileBytes;
                tc_fence_after();
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {             // 8 k-steps of 16 columns; 4 per 64-column box
                        const uint32_t off = (ks >> 2) * kPfHalfBytes + (ks & 3) * 32;
                        umma_ss(tmem_base, umma_desc(q_s + off, 16, 1024), umma_desc(k_s + off, 16, 1024), kIdescS, ks ? 1u : 0u);
                    }
                    tc_commit(s_ready + 8 * (j & 1));
                    tc_commit(k_empty + 8 * slot);
                }
                __syncwarp();
            }
            if (!ok && lane == 0) atomicExch(&timed_out, 1);
        } else if (warp == kPfPvWarp) {
            // =========================================================== issuer of O_w += P_w V_j, in two parts where the weights have a hi
            // and a lo one
            constexpr uint32_t kIdescO = umma_idesc(128, 128, false, true);
            const int parts = hilo ? 2 : 1;
            bool ok = true;
            int n_p[2] = {0, 0};
            for (int j = 0; j < n_kv && ok; ++j) {
                const int slot = j % kPtVSlots, w = j & 1;
                const uint32_t v_s = v_ring + slot * kPfTileBytes;
                ok = warp_wait(v_full + 8 * slot, (j / kPtVSlots) & 1);
                for (int part = 0; part < parts && ok; ++part) {
                    ok = warp_wait(p_ready + 8 * w, n_p[w] & 1);
                    if (!ok) break;
                    ++n_p[w];
                    tc_fence_after();
                    if (elect_one()) {
                        const uint32_t v_p = v_s + part * 4 * 2048;
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            umma_ts(tmem_base + kPfTmemO + w * 128, tmem_base + kPfTmemP + w * 64 + kk * 8,
                                    umma_desc(v_p + (parts == 2 ? kk & 3 : kk) * 2048, kPfHalfBytes, 1024), kIdescO, (j < 2 && part == 0 && kk == 0) ? 0u : 1u);
                        tc_commit(pv_done + 8 * w);
                        if (part == parts - 1) tc_commit(v_empty + 8 * slot);
                    }
                    __syncwarp();
                }
            }
            if (!ok && lane == 0) atomicExch(&timed_out, 1);
        }
        if (ctas > 1) {                      // (as the softmax warps do)
            cluster_sync();
            cluster_arrive_relaxed();
            cluster_wait();
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPfRegsSoftmax));
        // =============================================================== softmax warpgroups: one thread per query row
        const int w = warp >> 2, quarter = warp & 3, r = quarter * 32 + lane;
        const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const uint32_t p_t = lane_base + kPfTmemP + w * 64, o_t = lane_base + kPfTmemO + w * 128;
        const int hh = r / sh.positions, pos = p0 + r - hh * sh.positions;
        const bool mine = hh < sh.heads && head0 + hh < sh.h && pos < sh.n;
        const int lim_first = min(raw + p0 + 1, L), lim = min(raw + min(pos, sh.n - 1) + 1, L);      // rows the tile's first position sees, and this thread's: >= 1
        if (w == 0) ex_row[r] = mine ? (seq * sh.h + head0 + hh) * sh.n + pos : -1;
        float m = -INFINITY, l = 0.f;                            // reference maximum (log2 units), sum of weights
        bool ok = true;
        int n_p = 0;
        for (int j = w; j < n_kv; j += 2) {
            const int k0 = (first + j) * kPfRows;
            if (ok) ok = mbar_wait(s_ready + 8 * w, (j >> 1) & 1);
            tc_fence_after();
            // ---- the row's 128 logits, read once and kept in registers; the mask by index, as a select
            uint32_t x[128];
            tmem_ld_cols<128>(lane_base, x);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(s_free);                  // the next stage's logits may take their place
            if (k0 + kPfRows > lim_first) {
#pragma unroll
                for (int i = 0; i < 128; ++i)
                    if (k0 + i >= lim) x[i] = 0xff800000u;       // -inf
            }
            float mx8[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) mx8[i] = fmaxf(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1]));
#pragma unroll
            for (int i = 8; i < 64; ++i) mx8[i & 7] = max3(mx8[i & 7], __uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1]));
            const float mx = max3(max3(mx8[0], mx8[1], mx8[2]), max3(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7])) * kLog2e;
            if (__any_sync(0xffffffffu, mine && mx > m + kPfMaxLead)) {      // (rows that are nobody's do not count)
                const float m_new = fmaxf(m, mx);
                if (n_p > 0) {
                    const float f = m == m_new ? 1.f : fast_exp2(m - m_new);
                    l *= f;
                    if (ok) ok = mbar_wait(pv_done + 8 * w, (n_p - 1) & 1);  // O holds the warpgroup's stages before this one
                    tc_fence_after();
#pragma unroll 1
                    for (int c = 0; c < 16; ++c) {
                        uint32_t y[8];
                        tmem_ld8(o_t + c * 8, y);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i) y[i] = __float_as_uint(__uint_as_float(y[i]) * f);
                        tmem_st8(o_t + c * 8, y);
                    }
                }
                m = m_new;
            }
            const float neg_m = m == -INFINITY ? 0.f : -m;       // (nothing seen yet, or logits of -inf: weights of zero)
            const unsigned long long neg_m2 = f2_pack(neg_m, neg_m), log2e2 = f2_pack(kLog2e, kLog2e);
            unsigned long long sum2[2] = {0ull, 0ull};
            if (L < k0 + kPfRows) {
                // the tile's last stage runs past its memory: those V rows are cleared, zero weights or not (NaN * 0 = NaN)
                const int vs = j % kPtVSlots;
                if (ok) ok = mbar_wait(v_full + 8 * vs, (j / kPtVSlots) & 1);
                for (int i = r; i < (k0 + kPfRows - L) * 16; i += 128) {
                    const int vrow = L - k0 + (i >> 4), ch = i & 15;
                    const uint32_t a = v_ring + vs * kPfTileBytes + (ch >> 3) * kPfHalfBytes + vrow * 128 + ((ch & 7) << 4);
                    asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(a), "r"(0u) : "memory");
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            // the weights stay in registers until the product before has read the ones in tensor memory
            auto give = [&](const uint32_t (&p_0)[32], const uint32_t (&p_1)[32]) {
                if (n_p > 0 && ok) ok = mbar_wait(pv_done + 8 * w, (n_p - 1) & 1);
                tc_fence_after();
                tmem_st32(p_t, p_0);
                tmem_st32(p_t + 32, p_1);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(p_ready + 8 * w);
                ++n_p;
            };
            if (hilo) {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint32_t hi[32], lo[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        float a0, a1;
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(x[64 * half + 2 * i]), __uint_as_float(x[64 * half + 2 * i + 1])), log2e2, neg_m2), a0, a1);
                        const float pa = fast_exp2(a0), pb = fast_exp2(a1);
                        sum2[i & 1] = f2_add(sum2[i & 1], f2_pack(pa, pb));
                        hi[i] = pack_bf16(pa, pb);
                        lo[i] = pack_bf16(pa - bf16_lo(hi[i]), pb - bf16_hi(hi[i]));
                    }
                    give(hi, lo);
                }
            } else {
                uint32_t hi[2][32];
#pragma unroll
                for (int i = 0; i < 64; ++i) {
                    float a0, a1;
                    f2_unpack(f2_fma(f2_pack(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1])), log2e2, neg_m2), a0, a1);
                    const float pa = fast_exp2(a0), pb = fast_exp2(a1);
                    sum2[i & 1] = f2_add(sum2[i & 1], f2_pack(pa, pb));
                    hi[i >> 5][i & 31] = pack_bf16(pa, pb);
                }
                give(hi[0], hi[1]);
            }
            {
                float s0, s1;
                f2_unpack(f2_add(sum2[0], sum2[1]), s0, s1);
                l += s0 + s1;
            }
        }
        if (n_p > 0 && ok) ok = mbar_wait(pv_done + 8 * w, (n_p - 1) & 1);
        // (Q and the K ring are used below: a last stage that is the other warpgroup's must have its logits.  That warpgroup's logits
        // before those were ready before this one's last ones were issued, so the wait cannot be a phase early)
        if (n_p > 0 && n_kv > 1 && ((n_kv - 1) & 1) != w && ok) ok = mbar_wait(s_ready + 8 * (w ^ 1), ((n_kv - 1) >> 1) & 1);
        tc_fence_after();
        if (!ok) atomicExch(&timed_out, 1);
        // ---- each warpgroup leaves its rows of O in shared memory (where Q and the K ring were, 16-byte pieces swizzled by row)
        if (w == 1) ex_ml[r] = make_float2(m, l);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");         // (it was the copy engine's and the tensor core's; so was the V ring)
        if (n_p > 0) {
            const uint32_t ex_o = q_s + (w * kPfRows + r) * 512;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t y[32];
                tmem_ld32(o_t + c * 32, y);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(ex_o + (((c * 8 + i) ^ (r & 31)) << 4)), "r"(y[4 * i]), "r"(y[4 * i + 1]),
                                 "r"(y[4 * i + 2]), "r"(y[4 * i + 3]) : "memory");
            }
        }
        named_barrier(1, 256);                                   // (all of this CTA's products are done)
        if (ctas > 1) cluster_sync();                            // every CTA's V ring may be written
        if (w == 0) {
            // what each warpgroup's sums count for (-1: nothing, and its row may never have been written.  A share of logits that are
            // all -inf, or of which the row sees nothing, has a sum of 0; the maximum does not tell, that of NaN logits is -inf too)
            const float2 other = ex_ml[r];
            const bool one = n_kv > 0 && l != 0.f, two = n_kv > 1 && other.y != 0.f;
            const float top = fmaxf(one ? m : -INFINITY, two ? other.x : -INFINITY);
            float f0 = !one ? -1.f : m == top ? 1.f : fast_exp2(m - top), f1 = !two ? -1.f : other.x == top ? 1.f : fast_exp2(other.x - top);
            const float sum = (one ? f0 * l : 0.f) + (two ? f1 * other.y : 0.f);
            if (ctas == 1) {
                const float scale = n_all > 0 ? 1.f / sum : 0.f;
                if (one) f0 *= scale;
                if (two) f1 *= scale;
                if (!one && !two && n_all > 0) f0 = sum * scale;             // (nothing but logits of -inf: 0 / 0)
            } else {
                const int to = r / per;
                const uint32_t at = recv_ml + (rank * per + r - to * per) * 8;
                if (to == rank) asm volatile("st.shared.v2.f32 [%0], {%1,%2};" ::"r"(at), "f"(top), "f"(sum) : "memory");
                else cluster_send_f2(cluster_map(at, to), make_float2(top, sum), cluster_map(recv_bar, to));
            }
            ex_ml[r] = make_float2(f0, f1);
        }
        named_barrier(2, 256);
        // ---- whole rows, merged by a warp each on the way out: 512 contiguous bytes
        const float4* rows = reinterpret_cast<const float4*>(base);
#pragma unroll 4
        for (int i = 0; i < kPfRows / 8; ++i) {
            const int row = warp + 8 * i, to_row = ex_row[row];
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (to_row >= 0) {
                const float2 f = ex_ml[row];
                if (f.x >= 0.f || f.x != f.x) {
                    const float4 a = n_kv > 0 ? rows[row * 32 + (lane ^ (row & 31))] : v;
                    v = make_float4(a.x * f.x, a.y * f.x, a.z * f.x, a.w * f.x);
                }
                if (f.y >= 0.f || f.y != f.y) {
                    const float4 a = rows[(kPfRows + row) * 32 + (lane ^ (row & 31))];
                    v.x = fmaf(a.x, f.y, v.x); v.y = fmaf(a.y, f.y, v.y); v.z = fmaf(a.z, f.y, v.z); v.w = fmaf(a.w, f.y, v.w);
                }
            }
            if (ctas == 1) {
                if (to_row >= 0) reinterpret_cast<float4*>(O + (size_t)to_row * kHeadDim)[lane] = v;
            } else {
                const int to = row / per;
                const uint32_t at = v_ring + (rank * per + row - to * per) * 512 + lane * 16;
                if (to == rank) asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(at), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
                else cluster_send_f4(cluster_map(at, to), v, cluster_map(recv_bar, to));
            }
        }
        if (ctas > 1) {
            cluster_arrive_relaxed();                            // (this CTA's rows are on their way)
            named_barrier(1, 256);                               // its own are in place
            const bool got = mbar_wait(recv_bar, 0);
            for (int i = warp; i < per; i += 8) {
                const int to_row = ex_row[rank * per + i];
                if (to_row < 0) continue;
                float2 ml[kPfMaxSplit];
                float4 part[kPfMaxSplit];
                float top = -INFINITY, den = 0.f;
                float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int c = 0; c < kPfMaxSplit; ++c) {
                    if (c >= ctas) break;
                    asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];" : "=f"(ml[c].x), "=f"(ml[c].y) : "r"(recv_ml + (c * per + i) * 8) : "memory");
                    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(part[c].x), "=f"(part[c].y), "=f"(part[c].z), "=f"(part[c].w)
                                 : "r"(v_ring + (c * per + i) * 512 + lane * 16) : "memory");
                    top = fmaxf(top, ml[c].x);
                }
#pragma unroll
                for (int c = 0; c < kPfMaxSplit; ++c) {
                    if (c >= ctas) break;
                    if (ml[c].y == 0.f) continue;                // (nothing of this share counts: see above)
                    const float f = ml[c].x == top ? 1.f : fast_exp2(ml[c].x - top);
                    den = fmaf(f, ml[c].y, den);
                    num.x = fmaf(f, part[c].x, num.x); num.y = fmaf(f, part[c].y, num.y);
                    num.z = fmaf(f, part[c].z, num.z); num.w = fmaf(f, part[c].w, num.w);
                }
                const float inv = n_all > 0 ? 1.f / den : 0.f;
                reinterpret_cast<float4*>(O + (size_t)to_row * kHeadDim)[lane] = make_float4(num.x * inv, num.y * inv, num.z * inv, num.w * inv);
            }
            cluster_wait();                                      // everybody's rows have been sent
            if (!got) {
                // a wait ran out: what is still on its way here gets another bounded one before this CTA's shared memory goes
                mbar_wait(recv_bar, 0);
                if (lane == 0) atomicExch(&timed_out, 1);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kPfSWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0 && timed_out && status) atomicOr(status, kStatusPipelineTimeout);
}

}  // namespace mqa
