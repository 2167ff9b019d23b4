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
// Measured, us per step: 1024 sequences, 8 heads, window 32: 7.9 -> 7.3 (22.7 MB: 3.4 at the copy rate); 128 of them: 4.8 -> 3.1;
// 600 with window 128: 13.0 -> 10.8; 100 x 16 heads, window 200: 14.0 -> 6.2; 20 x 4, window 500: 24.6 -> 8.6.  Registers for two
// CTAs per SM (launch bounds) spilled: 7.9.
#pragma once
#include "decode_mma.cuh"

namespace mqa {

constexpr int kLocalMaxWarps = 7;                       // sequences per CTA at most
constexpr int local_smem_bytes(int warps, int stages) { return warps * stages * kStageBytes + 1024 /* alignment slack */ + warps * stages * 8 /* barriers */; }
static_assert(local_smem_bytes(kLocalMaxWarps, 2) <= 227 * 1024, "exceeds the shared memory of one SM");

__global__ void __launch_bounds__(kLocalMaxWarps * 32, 1)
mqa_decode_local_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                        const uint32_t* q, const uint4* __restrict__ k_new, const uint4* __restrict__ v_new,
                        uint4* __restrict__ K, uint4* __restrict__ V, int32_t* __restrict__ pos, float* __restrict__ o,
                        int32_t* __restrict__ status, int b, int h, int window, int advance, int stages) {
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
    uint32_t qa[8][4];
    load_q_fragments(qa, q, (size_t)seq, h, 0, lane);
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
    if (stages > 1) issue_next();

    LaneOffsets off;
    off.init(lane);
    const int g = lane >> 2, t4 = lane & 3;
    bool ok = true;
    int use = 0;                                             // copies consumed so far
    for (int mt = 0; mt < passes && ok; ++mt) {
        if (mt > 0) load_q_fragments(qa, q, (size_t)seq, h, mt, lane);
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

}  // namespace mqa
