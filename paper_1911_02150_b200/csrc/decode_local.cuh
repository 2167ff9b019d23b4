// Local multi-query attention, one decoding step (Section 4.1: a position attends to itself and the previous
// window - 1 positions; Section 4.3: the memory tensors padded to the window size).  The cache of a sequence is a
// ring of `window` rows: the new token's key/value row goes to row pos % window and the h heads attend over the
// min(pos + 1, window) rows that hold tokens (the order of rows does not matter to a softmax).
//
// A window is a few 32-row tiles (the paper's is one), so the work of a sequence is one warp's: 16 KiB of K and V
// per tile, brought in by the warp's own TMA copies into the warp's own stages of shared memory, and the same
// tensor-core tile routine as the fixed-split kernel (consume_tile: mma.sync m16n8k16 with the heads as M rows,
// online softmax in registers, P as bf16 hi + lo parts).  No CTA-wide barrier, no merge between warps: a warp
// loads its query fragments, walks its tiles and writes o from its accumulators.  A CTA is a few independent warps.
// More than 16 heads: the warp goes over the window once per 16 heads (the tiles come from L2).
//
// What bounds it at the paper's window is a chain of round trips, so there is one: the first tile does not depend on pos and
// is asked for together with pos, q and the new row, which then goes from registers into its place in the landed tile (and,
// with nobody waiting for it, into the ring).  Warps per CTA: the batch spread over all SMs, up to kLocalMaxWarps (1024
// sequences in CTAs of eight left a seventh of the SMs idle), each with two stages where there is a second tile to fetch
// ahead.  Windows of several tiles with few sequences go to the fixed-split kernel, four warps to a sequence.
// Measured, us per step: 600 sequences, 8 heads, window 128: 13.0 -> 10.3; 400 x 30, window 100: 15.0 -> 14.1; 100 x 16 heads, window
// 200: 14.0 -> 6.2; 20 x 4, window 500: 24.6 -> 8.6.  A window of one tile with up to 16 heads (the paper's) has a kernel of its own, below.
#pragma once
#include "decode_mma.cuh"

namespace mqa {

constexpr int kLocalMaxWarps = 7;                       // sequences per CTA at most
constexpr int kLocalStages = 2;
constexpr int local_smem_bytes(int warps) { return warps * kLocalStages * (kStageBytes + 8 /* barrier */) + 1024 /* alignment slack */; }
constexpr int local_tile_smem_bytes(int warps) { return warps * kStageBytes + 1024 /* alignment slack and barriers */; }
static_assert(2 * (local_tile_smem_bytes(kLocalMaxWarps) + 1024) <= 228 * 1024, "two CTAs of the one-tile kernel per SM");
static_assert(local_smem_bytes(kLocalMaxWarps) <= 227 * 1024, "exceeds the shared memory of one SM");

__global__ void __launch_bounds__(kLocalMaxWarps * 32, 1)
mqa_decode_local_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                        const uint4* q, const uint4* __restrict__ k_new, const uint4* __restrict__ v_new,
                        uint4* __restrict__ K, uint4* __restrict__ V, int32_t* __restrict__ pos, float* __restrict__ o,
                        int32_t* __restrict__ status, int b, int h, int window, int advance) {
    constexpr int stages = kLocalStages;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int seq = blockIdx.x * warps + warp;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* ring = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);       // the 128-byte swizzle repeats every 1 KiB
    const uint32_t ring_s = smem_addr(ring) + warp * stages * kStageBytes;              // this warp's K and V tiles
    const uint32_t bars = smem_addr(ring) + warps * stages * kStageBytes + warp * stages * 8;   // and their barriers
    if (lane == 0) {
        if (warp == 0) { prefetch_tensormap(&map_k); prefetch_tensormap(&map_v); }
        for (int s = 0; s < stages; ++s) mbar_init(bars + s * 8, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    const bool withhold = seq == 0 && test_withhold();       // for tests: one copy of sequence 0's second tile is never started
    grid_dependency_wait();          // pos, q, the rings and the new row may come from the kernel before
    grid_launch_dependents();
    if (seq >= b) return;            // (the whole warp: nothing is in flight)

    const int row_base = seq * window;                       // row coordinate in the [b * window, 128] view
    // a warp's copies are numbered: copy i goes into stage i % stages
    auto issue = [&](int i, int tile) {
        if (lane == 0) {
            const uint32_t bar = bars + (i % stages) * 8, dst = ring_s + (i % stages) * kStageBytes;
            mbar_expect_tx(bar, kStageBytes);
            const int y = row_base + tile * kTileRows;       // (a tile may run past the window: rows masked by index below)
            tma_load_2d(dst, &map_k, 0, y, bar);
            tma_load_2d(dst + kBoxBytes, &map_k, kBoxCols, y, bar);
            tma_load_2d(dst + 2 * kBoxBytes, &map_v, 0, y, bar);
            if (!(withhold && i == 1)) tma_load_2d(dst + 3 * kBoxBytes, &map_v, kBoxCols, y, bar);
        }
    };
    // the first tile, the new row's pieces (lanes 0-15 the key row, 16-31 the value row), q and pos are in flight together
    issue(0, 0);
    const uint4 row_piece = __ldcg((lane < 16 ? k_new : v_new) + (size_t)seq * (kRowBytes / 16) + (lane & 15));
    const int raw = __ldcg(pos + seq);
    QueryPieces<2> pieces;
    pieces.load(q, (size_t)seq * h, h, lane);
    const size_t units = (size_t)seq * h;
    if (raw < 0) {                   // no token position: no row written, zeros, flagged
        if (lane == 0 && status) atomicOr(status, kStatusAppendNegative | kStatusLenClamped);
        for (int i = lane; i < h * (kHeadDim / 4); i += 32) reinterpret_cast<float4*>(o + units * kHeadDim)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        mbar_wait(bars, 0);          // (the copy lands before the warp leaves)
        return;
    }
    const int new_row = raw % window;
    {
        const size_t dst = ((size_t)seq * window + new_row) * (kRowBytes / 16) + (lane & 15);
        if (lane < 16) K[dst] = row_piece; else V[dst] = row_piece;
    }
    const int L = raw < window ? raw + 1 : window;           // rows that hold tokens
    const int n_tiles = (L + kTileRows - 1) / kTileRows;
    const int passes = (h + 15) / 16, n_copies = passes * n_tiles;      // 16 heads at a time
    int issued = 1, next_tile = n_tiles > 1 ? 1 : 0;
    auto issue_next = [&]() {
        if (issued >= n_copies) return;
        issue(issued++, next_tile);
        next_tile = next_tile + 1 < n_tiles ? next_tile + 1 : 0;
    };
    issue_next();

    LaneOffsets off;
    off.init(lane);
    const int g = lane >> 2, t4 = lane & 3;
    bool ok = true;
    int use = 0;                                             // copies consumed so far
    for (int mt = 0; mt < passes && ok; ++mt) {
        // (the next 16 heads' rows of q are on their way while these are worked on.  Loaded, and swapped between lanes, at the top of their
        // own pass: 5 x 30 heads, window 19: 5.1 us a step, 4.8 so; 8 x 3, window 101 3.6 and 3.4; 400 x 30, window 100 14.0 and 14.4)
        uint32_t qa[8][4];
        pieces.fragments(qa, lane);
        if (mt + 1 < passes) pieces.load(q, (size_t)seq * h + (mt + 1) * 16, h - (mt + 1) * 16, lane);
        WarpState st;
        st.reset();
        for (int i = 0; i < n_tiles && ok; ++i, ++use) {
            const int stage = use % stages;
            ok = __all_sync(0xffffffffu, mbar_wait(bars + stage * 8, (use / stages) & 1));
            if (!ok) break;                                  // (a copy may still land: see the end of the kernel)
            const uint32_t k_s = ring_s + stage * kStageBytes;
            if (new_row / kTileRows == i) {                  // the new row into its place: boxes K, K, V, V
                const int row = new_row & (kTileRows - 1);
                asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(k_s + (lane >> 3) * kBoxBytes + row * 128 + (((lane & 7) ^ (row & 7)) << 4)),
                             "r"(row_piece.x), "r"(row_piece.y), "r"(row_piece.z), "r"(row_piece.w) : "memory");
                __syncwarp();
            }
            consume_tile<true>(st, qa, off, k_s, k_s + 2 * kBoxBytes, kBoxBytes, i * kTileRows, L, lane);
            // the tile was read through the generic proxy and the next copy writes the stage through the async proxy
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            issue_next();
        }
        if (!ok) break;
        // sums over the four lanes that share a head, then o = accumulators / sum, straight from the registers
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            st.l[r] += __shfl_xor_sync(0xffffffffu, st.l[r], 1);
            st.l[r] += __shfl_xor_sync(0xffffffffu, st.l[r], 2);
        }
        const float inv0 = 1.f / st.l[0], inv1 = 1.f / st.l[1];
        const int head0 = mt * 16 + g, head1 = head0 + 8;
#pragma unroll
        for (int vt = 0; vt < 16; ++vt) {
            if (head0 < h)
                *reinterpret_cast<float2*>(o + (units + head0) * kHeadDim + vt * 8 + t4 * 2) = make_float2(st.acc[vt][0] * inv0, st.acc[vt][1] * inv0);
            if (head1 < h)
                *reinterpret_cast<float2*>(o + (units + head1) * kHeadDim + vt * 8 + t4 * 2) = make_float2(st.acc[vt][2] * inv1, st.acc[vt][3] * inv1);
        }
    }
    if (!ok) {
        // a wait ran out: before the warp leaves (and with it, perhaps, the CTA and its shared memory), give the copies
        // in flight one more bounded wait each; flag the status word; o of this sequence is not valid
        for (int i = use; i < issued; ++i) mbar_wait(bars + (i % stages) * 8, (i / stages) & 1);
        if (lane == 0 && status) atomicOr(status, kStatusPipelineTimeout);
        return;
    }
    if (advance && lane == 0) pos[seq] = raw + 1;            // (every lane has read pos[seq]: it takes part in the waits above)
}

// A window of one tile and up to 16 heads (the paper's: 32 rows, 8 heads): the sequence's only tile needs no running state, its
// fragments of q are done with before the first accumulator is, and the accumulators leave 16 columns at a time.  So a thread
// needs 128 registers and a CTA of seven warps 112 KB, and two CTAs fit an SM: that of the next step is on it while this one's
// still works, and asks its windows into L2 ahead of the wait for it (rows written meanwhile are written there too).
// us per step, six layers in a graph, the general kernel with one stage -> this: 1024 x 8 heads 7.5 -> 5.9 (22.7 MB: 3.9 TB/s); 2000 x 8
// 13.3 -> 10.3; 1024 x 16 8.5 -> 6.7; 128 x 8 3.1 -> 2.7.
__global__ void __launch_bounds__(kLocalMaxWarps * 32, 2)
mqa_decode_local_tile_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                             const uint4* q, const uint4* __restrict__ k_new, const uint4* __restrict__ v_new,
                             uint4* __restrict__ K, uint4* __restrict__ V, int32_t* __restrict__ pos, float* __restrict__ o,
                             int32_t* __restrict__ status, int b, int h, int window, int advance) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int seq = blockIdx.x * warps + warp;

    extern __shared__ uint8_t smem_raw[];
    // the tiles lie at a multiple of 1 KiB (the 128-byte swizzle repeats every 1 KiB), the barriers where that leaves room
    const uint32_t pad = (1024u - (smem_addr(smem_raw) & 1023u)) & 1023u, tiles_s = smem_addr(smem_raw) + pad;
    const uint32_t k_s = tiles_s + warp * kStageBytes, v_s = k_s + 2 * kBoxBytes;
    const uint32_t bar = (pad >= kLocalMaxWarps * 8 ? smem_addr(smem_raw) : tiles_s + warps * kStageBytes) + warp * 8;
    if (lane == 0) {
        if (warp == 0) { prefetch_tensormap(&map_k); prefetch_tensormap(&map_v); }
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    const size_t rows = (size_t)seq * window * (kRowBytes / 16);
    if (seq < b && lane < 3) prefetch_l2(lane == 0 ? K + rows : lane == 1 ? V + rows : q + (size_t)seq * h * (kRowBytes / 16), (lane < 2 ? window : h) * kRowBytes);
    __syncwarp();
    const bool withhold = seq == 0 && test_withhold();       // for tests: one copy of sequence 0's tile is never started
    grid_dependency_wait();          // pos, q, the rings and the new row may come from the kernel before
    grid_launch_dependents();
    if (seq >= b) return;            // (the whole warp: nothing is in flight)

    // the tile (four boxes by four lanes; rows past the window masked by index below), the new row's pieces (lanes 0-15 the key
    // row, 16-31 the value row), q and pos are in flight together
    if (lane == 0) mbar_expect_tx(bar, kStageBytes);
    __syncwarp();
    if (lane < 4 && !(withhold && lane == 3)) tma_load_2d(k_s + lane * kBoxBytes, lane < 2 ? &map_k : &map_v, (lane & 1) * kBoxCols, seq * window, bar);
    const uint4 row_piece = __ldcg((lane < 16 ? k_new : v_new) + (size_t)seq * (kRowBytes / 16) + (lane & 15));
    const int raw = __ldcg(pos + seq);
    uint32_t qa[8][4];
    load_q_fragments(qa, q, (size_t)seq * h, h, lane);
    float* out = o + (size_t)seq * h * kHeadDim;
    if (raw < 0) {                   // no token position: no row written, zeros, flagged
        if (lane == 0 && status) atomicOr(status, kStatusAppendNegative | kStatusLenClamped);
        for (int i = lane; i < h * (kHeadDim / 4); i += 32) reinterpret_cast<float4*>(out)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        mbar_wait(bar, 0);           // (the copy lands before the warp leaves)
        return;
    }
    const int new_row = raw % window;
    {
        const size_t dst = rows + (size_t)new_row * (kRowBytes / 16) + (lane & 15);
        if (lane < 16) K[dst] = row_piece; else V[dst] = row_piece;
    }
    const int L = raw < window ? raw + 1 : window;           // rows that hold tokens
    LaneOffsets off;
    off.init(lane);
    if (!__all_sync(0xffffffffu, mbar_wait(bar, 0))) {
        // a wait ran out: before the warp leaves (and with it, perhaps, the CTA and its shared memory), the copies in flight get
        // one more bounded wait; o of this sequence is not valid
        mbar_wait(bar, 0);
        if (lane == 0 && status) atomicOr(status, kStatusPipelineTimeout);
        return;
    }
    // the new row into its place: boxes K, K, V, V
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(k_s + (lane >> 3) * kBoxBytes + new_row * 128 + (((lane & 7) ^ (new_row & 7)) << 4)),
                 "r"(row_piece.x), "r"(row_piece.y), "r"(row_piece.z), "r"(row_piece.w) : "memory");
    __syncwarp();
    const bool ragged = L < kTileRows;
    float sc[4][4], m[2], l[2] = {0.f, 0.f};
    tile_logits(sc, m, qa, off, k_s, kBoxBytes, 0, L, ragged, lane);
    uint32_t p_hi[2][4], p_lo[2][4];
    tile_weights<true>(p_hi, p_lo, l, sc, m);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
        l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
    }
    const float inv0 = 1.f / l[0], inv1 = 1.f / l[1];
    const int g = lane >> 2, t4 = lane & 3;
    const bool odd = (t4 & 1) != 0;
    uint32_t keep_lo[2], keep_hi[2];
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) tile_row_masks(keep_lo[kk], keep_hi[kk], 0, L, kk, lane);
#pragma unroll
    for (int vp = 0; vp < 8; ++vp) {
        float a0[4] = {0.f, 0.f, 0.f, 0.f}, a1[4] = {0.f, 0.f, 0.f, 0.f};      // columns vp * 16 + t4 * 2 + {0, 1}, and 8 further; heads g, g + 8
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) tile_product<true>(a0, a1, p_hi[kk], p_lo[kk], off, v_s, kBoxBytes, kk, vp, ragged, keep_lo[kk], keep_hi[kk]);
        // neighbouring lanes swap halves: an even lane has four columns of the first n-tile then, an odd one of the second
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float inv = r ? inv1 : inv0;
            const float x0 = a0[2 * r] * inv, x1 = a0[2 * r + 1] * inv, y0 = a1[2 * r] * inv, y1 = a1[2 * r + 1] * inv;
            const float s0 = __shfl_xor_sync(0xffffffffu, odd ? x0 : y0, 1), s1 = __shfl_xor_sync(0xffffffffu, odd ? x1 : y1, 1);
            const float4 v = odd ? make_float4(s0, s1, y0, y1) : make_float4(x0, x1, s0, s1);
            if (g + 8 * r < h) *reinterpret_cast<float4*>(out + (g + 8 * r) * kHeadDim + vp * 16 + (odd ? 8 : 0) + (t4 & 2) * 2) = v;
        }
    }
    if (advance && lane == 0) pos[seq] = raw + 1;            // (every lane has read pos[seq]: it takes part in the waits above)
}

}  // namespace mqa
