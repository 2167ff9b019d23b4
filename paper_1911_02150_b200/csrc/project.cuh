// The projections either side of the multi-query step (Section 3, MultiquerySelfAttentionIncremental):
//
//     q     = einsum("bd,hdk->bhk", x, P_q)     k_new = einsum("bd,dk->bk", x, P_k)     v_new = einsum("bd,dv->bv", x, P_v)
//     y     = einsum("bhv,hdv->bd", o, P_o)
//
// as bf16 tensor-core products with fp32 accumulation (tcgen05, accumulators in TMEM).  A decoding
// step has few rows (b sequences) and large weights, so the weights are the M operand and the
// batch is N ("swap A and B"): a CTA streams a 128-wide slab of a weight matrix through shared
// memory with TMA, once, and multiplies it with the batch's activations:
//
//   project_in_kernel    slab s < h: P_q[s] = [d rows x 128]; s = h: P_k; s = h + 1: P_v  (each [d x 128], d contiguous
//                        rows of 256 bytes -- the layout of a 128-column cache, fetched the same way)
//                        Out^T[128 features x NB] = sum over d in chunks of 128:  W_chunk^T (MN-major A) * x_chunk^T (K-major B)
//                        the d rows of a slab are shared out over the CTAs of one thread-block cluster
//   project_out_kernel   CTA (d tile j, head group g): Y^T[128 x NB] = sum over the group's heads:
//                        P_o[head][128 d-rows of tile j x 128] (K-major A) * o[:, head, :]^T (K-major B, converted
//                        from fp32 to bf16 by the CTA); the head groups of a tile are one thread-block cluster
//
// The CTAs of a cluster leave their sums in shared memory, send each other the batch rows that fall to each, and add them up
// in rank order (no float atomics): SumShares.
//
// What bounds these kernels is latency: the weights are in flight before the kernel ahead has finished, and a CTA's work
// after that is a chain of round trips (x or o, the products, the other CTAs' sums), each made one round trip: all of a
// head's o loads are in flight at once, another CTA's sums come in one copy.  How the chain is cut up over batch columns
// and CTAs: projection_cut in api.cu, with what it measured.
//
// NB = batch columns of a tile (16, 32, 64 or 128; larger batches take several tiles).  Every wait is bounded (mbar_wait);
// TMEM is freed on every path.
#pragma once
#include <cuda_bf16.h>

#include "decode_umma.cuh"

namespace mqa {

constexpr int kProjWorkWarps = 8;              // convert o, read the sums out, add them up
constexpr int kProjTmaWarp = 8, kProjMmaWarp = 9;
constexpr int kProjThreads = 10 * 32;
constexpr int kProjChunkBytes = 128 * 256;     // 128 rows x 128 bf16 of a weight matrix: 32 KiB, two 64-column boxes
constexpr int kProjMaxCluster = 8;             // CTAs that share the depth of a product

template <int NB>
struct ProjCfg {
    static_assert(NB == 16 || NB == 32 || NB == 64 || NB == 128, "batch columns of a tile");
    static constexpr int kActBytes = NB * 256;                 // NB rows x 128 bf16, two 64-column boxes
    static constexpr int kStages = NB == 128 ? 2 : NB == 64 ? 3 : 4;
    static constexpr int kStageBytes = kProjChunkBytes + kActBytes;
    static constexpr int kSumBytes = NB * 512;                 // a CTA's sums, [NB batch rows][128] fp32: where the stages were
    static constexpr int kRecvBytes = (NB + kProjMaxCluster) * 512;     // the other CTAs' sums of this one's rows (whole rows, rounded up per CTA)
    static constexpr int smem_bytes(int stages) { return stages * kStageBytes + kRecvBytes + 256 /* barriers */ + 1024 /* alignment slack */; }
    static constexpr int kSmemBytes = smem_bytes(kStages);
    static_assert(kSumBytes <= kStageBytes, "the sums take the first stage's place");
    static constexpr int kTmemCols = NB < 32 ? 32 : NB;
    static_assert(kSmemBytes <= 227 * 1024, "exceeds the shared memory of one SM");
};

// The accumulator Out^T (TMEM lane = feature, column = batch row of the tile) into this CTA's shared memory as
// [NB batch rows][128 features] fp32, by the eight work warps: a warp may read the 32 lanes of its quarter, and the two
// warps of a quarter take half of the batch rows each.  valid = false: zeros.
template <int NB>
__device__ __forceinline__ void leave_sums(uint32_t tmem, uint32_t dst, int warp, int lane, bool valid) {
    constexpr int CH = NB < 64 ? NB / 2 : 32;                      // columns per load
    const int feature = (warp & 3) * 32 + lane, col0 = (warp >> 2) * (NB / 2);
#pragma unroll
    for (int c = 0; c < NB / 2; c += CH) {
        uint32_t part[CH];
        tmem_ld_cols<CH>(tmem + ((uint32_t)((warp & 3) * 32) << 16) + col0 + c, part);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < CH; ++i)
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(dst + (uint32_t)((col0 + c + i) * 128 + feature) * 4), "r"(valid ? part[i] : 0u) : "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // (bulk copies read them)
}

// ---- the sums of a cluster's CTAs, added up: CTA r of C takes the batch rows [r * per, (r + 1) * per) of the tile.  Every CTA
// sends each other one the rows that fall to it as ONE bulk copy from shared memory to shared memory (SM to SM, signalled on the
// receiver's mbarrier; a place of its own per sender) and adds up what it has and what it gets, in rank order.  Read by
// 16-byte remote loads instead, between two cluster barriers, the 64 KB that a CTA needs took 3.2 to 3.9 us at 128 batch
// columns; this 2.3 to 3.1 (SM to SM a CTA
// gets about 24 KB/us), and at 16 batch columns 1.0 in place of 1.6.
__device__ __forceinline__ void send_rows(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {      // dst and bar: cluster addresses
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
// Chunk (or head) c's stage of S, and how often that stage has been used before it.  (As many stages as chunks is the common case: no
// division by a number that the compiler does not know, 0.2 us of a layer step.)
__device__ __forceinline__ int stage_of(int c, int S) { return c < S ? c : c % S; }
__device__ __forceinline__ int turn_of(int c, int S) { return c < S ? 0 : c / S; }

struct SumShares {
    int rank, ctas, rows, per;            // rows: of the tile; per: of a CTA (the last ones may have fewer)
    __device__ __forceinline__ int count(int r) const { return max(0, min(per, rows - r * per)); }
    // by one thread, before the cluster barrier that tells the others that this CTA's barrier is in place
    __device__ __forceinline__ void expect(uint32_t bar) const { mbar_expect_tx(bar, (uint32_t)((ctas - 1) * count(rank)) * 512); }
    // by one warp, once this CTA's sums lie in its shared memory
    __device__ __forceinline__ void send(uint32_t sums, uint32_t recv, uint32_t bar, int lane) const {
        const int to = lane;              // (a cluster has at most kProjMaxCluster CTAs)
        if (to < ctas && to != rank && count(to) > 0)
            send_rows(cluster_map(recv + (uint32_t)(rank * per) * 512, to), sums + (uint32_t)(to * per) * 512, (uint32_t)count(to) * 512, cluster_map(bar, to));
    }
    // row i of this CTA's, features lane * 4 .. + 3
    __device__ __forceinline__ float4 add_up(uint32_t sums, uint32_t recv, int i, int lane) const {
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int g = 0; g < ctas; ++g) {
            const uint32_t at = (g == rank ? sums + (uint32_t)(rank * per + i) * 512 : recv + (uint32_t)(g * per + i) * 512) + lane * 16;
            float4 v;
            asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(at) : "memory");
            sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
        }
        return sum;
    }
};
template <int NB>
__global__ void __launch_bounds__(kProjThreads, 1)
project_in_kernel(const __grid_constant__ CUtensorMap map_pq, const __grid_constant__ CUtensorMap map_pk,
                  const __grid_constant__ CUtensorMap map_pv, const __grid_constant__ CUtensorMap map_x,
                  __nv_bfloat16* __restrict__ q, __nv_bfloat16* __restrict__ k_new, __nv_bfloat16* __restrict__ v_new,
                  int32_t* __restrict__ status, int b, int h, int d, const int S) {
    using Cfg = ProjCfg<NB>;                                      // (S stages, as many as a CTA has chunks, at most Cfg::kStages)
    const int slab = blockIdx.x, row0 = blockIdx.z * NB;          // weight slab; first batch row of this tile
    const int part = blockIdx.y, parts = gridDim.y;                // this CTA's part of the slab's d rows: one cluster per slab
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int chunk0 = part * (d / 128) / parts;                   // chunks of 128 rows [chunk0, chunk0 + n_chunks)
    const int n_chunks = (part + 1) * (d / 128) / parts - chunk0;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* stages = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    const uint32_t stages_s = smem_addr(stages);
    const uint32_t recv_s = stages_s + S * Cfg::kStageBytes;       // the other CTAs' sums of this one's batch rows
    const uint32_t full_s = recv_s + Cfg::kRecvBytes, empty_s = full_s + S * 8, done_s = empty_s + S * 8, recv_bar = done_s + 8;
    const int rows = min(NB, b - row0);
    const SumShares shares{part, parts, rows, (rows + parts - 1) / parts};
    __shared__ uint32_t tmem_slot;
    __shared__ int timed_out, issued;

    // The weights do not depend on the kernel before this one, x does: a stage's barrier takes two arrivals, one with
    // the weight chunk's bytes and one with the x chunk's, and the weight copies of the first stages start before the wait.
    const CUtensorMap* wmap = slab < h ? &map_pq : (slab == h ? &map_pk : &map_pv);
    const int wrow0 = slab < h ? slab * d : 0;
    auto issue_weights = [&](int c) {
        const uint32_t bar = full_s + stage_of(c, S) * 8, w_s = stages_s + stage_of(c, S) * Cfg::kStageBytes;
        mbar_expect_tx(bar, kProjChunkBytes);
        tma_load_2d(w_s, wmap, 0, wrow0 + (chunk0 + c) * 128, bar);
        tma_load_2d(w_s + kProjChunkBytes / 2, wmap, kBoxCols, wrow0 + (chunk0 + c) * 128, bar);
    };
    auto issue_x = [&](int c) {
        const uint32_t bar = full_s + stage_of(c, S) * 8, x_s = stages_s + stage_of(c, S) * Cfg::kStageBytes + kProjChunkBytes;
        mbar_expect_tx(bar, Cfg::kActBytes);
        tma_load_2d(x_s, &map_x, (chunk0 + c) * 128, row0, bar);              // rows past b read as zero
        tma_load_2d(x_s + Cfg::kActBytes / 2, &map_x, (chunk0 + c) * 128 + kBoxCols, row0, bar);
        issued = c + 1;
    };
    if (warp == kProjTmaWarp && lane == 0) {                                  // by the thread that issues the copies
        prefetch_tensormap(&map_pq); prefetch_tensormap(&map_pk); prefetch_tensormap(&map_pv); prefetch_tensormap(&map_x);
        timed_out = 0;
        issued = 0;
        for (int s = 0; s < S; ++s) { mbar_init(full_s + s * 8, 2); mbar_init(empty_s + s * 8, 1); }
        mbar_init(done_s, 1);
        mbar_init(recv_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (parts > 1) shares.expect(recv_bar);
        for (int c = 0; c < n_chunks && c < S; ++c) issue_weights(c);
    }
    if (warp == kProjMmaWarp) { tmem_alloc(smem_addr(&tmem_slot), Cfg::kTmemCols); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    // for tests: the first CTA keeps its sums to itself, so that the others of its cluster wait for them in vain
    const bool withhold = blockIdx.x == 0 && part == 0 && row0 == 0 && test_withhold();
    if (parts > 1) cluster_sync();   // every CTA's barrier is in place
    grid_dependency_wait();          // x may come from the kernel before this one
    grid_launch_dependents();

    if (warp == kProjTmaWarp) {
        if (lane == 0) {
            bool ok = true;
            for (int c = 0; c < n_chunks && ok; ++c) {
                if (c >= S) {
                    ok = mbar_wait(empty_s + stage_of(c, S) * 8, (turn_of(c, S) - 1) & 1);
                    if (!ok) break;
                    issue_weights(c);
                }
                issue_x(c);
            }
            if (!ok) atomicExch(&timed_out, 1);
        }
    } else if (warp == kProjMmaWarp) {
        if (lane == 0) {
            constexpr uint32_t kIdesc = umma_idesc(128, NB, true, false);
            bool ok = true;
            for (int c = 0; c < n_chunks; ++c) {
                const int st = stage_of(c, S);
                if (ok) ok = mbar_wait(full_s + st * 8, turn_of(c, S) & 1);
                tc_fence_after();
                if (ok) {
                    const uint32_t w_s = stages_s + st * Cfg::kStageBytes, x_s = w_s + kProjChunkBytes;
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {                         // 8 k-steps of 16 rows of the weight chunk
                        const uint64_t a = umma_desc(w_s + kk * 2048, kProjChunkBytes / 2, 1024);
                        const uint64_t bd = umma_desc(x_s + (kk >> 2) * (Cfg::kActBytes / 2) + (kk & 3) * 32, 16, 1024);
                        umma_ss(tmem, a, bd, kIdesc, (c > 0 || kk > 0) ? 1u : 0u);
                    }
                }
                tc_commit(empty_s + st * 8);
            }
            tc_commit(done_s);
            if (!ok) atomicExch(&timed_out, 1);
        }
    } else {
        // this CTA's sums into its shared memory: the stages are free once the last product has completed
        const bool ok = mbar_wait(done_s, 0);
        tc_fence_after();
        leave_sums<NB>(tmem, stages_s, warp, lane, ok);
        if (!ok) atomicExch(&timed_out, 1);
    }
    tc_fence_before();
    __syncthreads();
    if (timed_out && threadIdx.x == 0) {
        // before anything else: the last copy started into each stage has to land
        for (int s = 0; s < S && s < issued; ++s) mbar_wait(full_s + s * 8, ((issued - 1 - s) / S) & 1);
        if (status) atomicOr(status, kStatusPipelineTimeout);
    }
    __syncthreads();
    if (parts > 1) {
        if (warp == 0 && !withhold) shares.send(stages_s, recv_s, recv_bar, lane);
        if (!mbar_wait(recv_bar, 0)) { if (status && lane == 0) atomicOr(status, kStatusPipelineTimeout); mbar_wait(recv_bar, 0); }
        cluster_arrive_relaxed();    // what the others send has landed
    }
    {
        __nv_bfloat16* out = slab < h ? q + (size_t)slab * 128 : (slab == h ? k_new : v_new);
        const size_t stride = slab < h ? (size_t)h * 128 : 128;
        for (int i = warp; i < shares.count(part); i += kProjThreads / 32) {
            const float4 v = shares.add_up(stages_s, recv_s, i, lane);
            *reinterpret_cast<uint2*>(out + (size_t)(row0 + part * shares.per + i) * stride + lane * 4) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
        }
    }
    if (parts > 1) cluster_wait();   // nobody leaves while its sums are on their way
    if (warp == kProjMmaWarp) { tc_fence_after(); tmem_dealloc(tmem, Cfg::kTmemCols); }
}

// The head groups of one (d tile, batch tile) form one thread-block cluster (gridDim.y CTAs): each CTA accumulates Y^T over its
// heads in TMEM, and the cluster adds the sums up.  No partial sums pass through global memory and no float atomics are used.
template <int NB>
__global__ void __launch_bounds__(kProjThreads, 1)
project_out_kernel(const __grid_constant__ CUtensorMap map_po, const float* __restrict__ o, float* __restrict__ y,
                   int32_t* __restrict__ status, int b, int h, int d, int heads_per_cta, const int S) {
    using Cfg = ProjCfg<NB>;                                       // a stage: a head's weights and its o tile (S of them, as in project_in_kernel)
    const int tile = blockIdx.x, group = blockIdx.y, row0 = blockIdx.z * NB;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int head0 = group * heads_per_cta;
    const int n_heads = max(0, min(heads_per_cta, h - head0));

    extern __shared__ uint8_t smem_raw[];
    uint8_t* stages = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    const uint32_t stages_s = smem_addr(stages);
    const uint32_t recv_s = stages_s + S * Cfg::kStageBytes;       // the other CTAs' sums of this one's batch rows
    const uint32_t w_full = recv_s + Cfg::kRecvBytes, o_full = w_full + S * 8, empty_s = o_full + S * 8, done_s = empty_s + S * 8, recv_bar = done_s + 8;
    const int rows = min(NB, b - row0), n_groups = gridDim.y;
    const SumShares shares{group, n_groups, rows, (rows + n_groups - 1) / n_groups};
    __shared__ uint32_t tmem_slot;
    __shared__ int timed_out, issued;

    if (warp == kProjTmaWarp && lane == 0) {                                  // by the thread that issues the copies
        prefetch_tensormap(&map_po);
        timed_out = 0;
        issued = 0;
        for (int s = 0; s < S; ++s) { mbar_init(w_full + s * 8, 1); mbar_init(o_full + s * 8, kProjWorkWarps); mbar_init(empty_s + s * 8, 1); }
        mbar_init(done_s, 1);
        mbar_init(recv_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        shares.expect(recv_bar);
    }
    if (warp == kProjMmaWarp) { tmem_alloc(smem_addr(&tmem_slot), Cfg::kTmemCols); tmem_relinquish(); }
    auto issue_weights = [&](int i) {
        const int st = stage_of(i, S);
        const uint32_t bar = w_full + st * 8, w_s = stages_s + st * Cfg::kStageBytes;
        mbar_expect_tx(bar, kProjChunkBytes);
        const int yrow = (head0 + i) * d + tile * 128;
        tma_load_2d(w_s, &map_po, 0, yrow, bar);
        tma_load_2d(w_s + kProjChunkBytes / 2, &map_po, kBoxCols, yrow, bar);
        issued = i + 1;
    };
    // the weights do not depend on the kernel before this one: the first copies start at once
    if (warp == kProjTmaWarp && lane == 0)
        for (int i = 0; i < n_heads && i < S; ++i) issue_weights(i);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const bool withhold = tile == 0 && group == 0 && row0 == 0 && test_withhold();     // (as in project_in_kernel)
    cluster_sync();                  // every CTA's barrier is in place
    grid_dependency_wait();          // o comes from the kernel before this one
    grid_launch_dependents();

    if (warp == kProjTmaWarp) {
        if (lane == 0) {
            bool ok = true;
            for (int i = S; i < n_heads && ok; ++i) {
                ok = mbar_wait(empty_s + stage_of(i, S) * 8, (turn_of(i, S) - 1) & 1);
                if (ok) issue_weights(i);
            }
            if (!ok) atomicExch(&timed_out, 1);
        }
    } else if (warp == kProjMmaWarp) {
        if (lane == 0) {
            constexpr uint32_t kIdesc = umma_idesc(128, NB, false, false);
            bool ok = true;
            for (int i = 0; i < n_heads; ++i) {
                const int st = stage_of(i, S);
                if (ok) ok = mbar_wait(w_full + st * 8, turn_of(i, S) & 1);
                if (ok) ok = mbar_wait(o_full + st * 8, turn_of(i, S) & 1);
                tc_fence_after();
                if (ok) {
                    const uint32_t w_s = stages_s + st * Cfg::kStageBytes, o_s = w_s + kProjChunkBytes;
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {                         // 8 k-steps of 16 columns; 4 per 64-column box
                        const uint64_t a = umma_desc(w_s + (ks >> 2) * (kProjChunkBytes / 2) + (ks & 3) * 32, 16, 1024);
                        const uint64_t bd = umma_desc(o_s + (ks >> 2) * (Cfg::kActBytes / 2) + (ks & 3) * 32, 16, 1024);
                        umma_ss(tmem, a, bd, kIdesc, (i > 0 || ks > 0) ? 1u : 0u);
                    }
                }
                tc_commit(empty_s + st * 8);                                 // the stage may be filled again
            }
            tc_commit(done_s);
            if (!ok) atomicExch(&timed_out, 1);
        }
    } else {
        // ---- o[:, head, :] (fp32) -> bf16 tile [NB rows x 128 columns], K-major with the 128-byte swizzle:
        // row n, 16-byte chunk c of its 64-column half at n * 128 + ((c ^ (n & 7)) << 4).  A warp takes whole rows (512
        // contiguous bytes per load); all of a head's loads are in flight before the first is converted.
        bool ok = true;
        for (int i = 0; i < n_heads; ++i) {
            const int st = stage_of(i, S);
            float4 v[NB / kProjWorkWarps];
#pragma unroll
            for (int k = 0; k < NB / kProjWorkWarps; ++k) {
                const int n = warp + k * kProjWorkWarps;
                v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (row0 + n < b) v[k] = __ldcg(reinterpret_cast<const float4*>(o + ((size_t)(row0 + n) * h + head0 + i) * kHeadDim + lane * 4));
            }
            if (i >= S && ok) ok = mbar_wait(empty_s + st * 8, (turn_of(i, S) - 1) & 1);   // the product that read this tile is done
            const uint32_t o_s = stages_s + st * Cfg::kStageBytes + kProjChunkBytes + (lane >> 4) * (Cfg::kActBytes / 2) + (lane & 1) * 8;
#pragma unroll
            for (int k = 0; k < NB / kProjWorkWarps; ++k) {
                const int n = warp + k * kProjWorkWarps;
                const uint32_t at = o_s + n * 128 + ((((lane >> 1) & 7) ^ (n & 7)) << 4);
                asm volatile("st.shared.v2.b32 [%0], {%1,%2};" ::"r"(at), "r"(pack_bf16(v[k].x, v[k].y)), "r"(pack_bf16(v[k].z, v[k].w)) : "memory");
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // the tile is read by the tensor core
            __syncwarp();
            if (lane == 0) mbar_arrive(o_full + st * 8);
        }
        // ---- this CTA's Y^T into its shared memory: the stages are free once the last product has completed
        if (ok) ok = mbar_wait(done_s, 0);
        tc_fence_after();
        leave_sums<NB>(tmem, stages_s, warp, lane, ok && n_heads > 0);
        if (!ok) atomicExch(&timed_out, 1);
    }
    tc_fence_before();
    __syncthreads();
    if (timed_out && threadIdx.x == 0) {
        // before anything else: the last copy started into each stage has to land
        for (int s = 0; s < S && s < issued; ++s) mbar_wait(w_full + s * 8, ((issued - 1 - s) / S) & 1);
        if (status) atomicOr(status, kStatusPipelineTimeout);
    }
    __syncthreads();
    if (warp == 0 && !withhold) shares.send(stages_s, recv_s, recv_bar, lane);
    if (!mbar_wait(recv_bar, 0)) { if (status && lane == 0) atomicOr(status, kStatusPipelineTimeout); mbar_wait(recv_bar, 0); }
    cluster_arrive_relaxed();        // what the others send has landed
    for (int i = warp; i < shares.count(group); i += kProjThreads / 32)
        *reinterpret_cast<float4*>(y + (size_t)(row0 + group * shares.per + i) * d + (size_t)tile * 128 + lane * 4) = shares.add_up(stages_s, recv_s, i, lane);
    cluster_wait();                  // nobody leaves while its sums are on their way
    if (warp == kProjMmaWarp) { tc_fence_after(); tmem_dealloc(tmem, Cfg::kTmemCols); }
}

}  // namespace mqa
