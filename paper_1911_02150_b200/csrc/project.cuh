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
// The CTAs of a cluster leave their sums in shared memory and add them up through distributed shared memory, each the
// batch rows that fall to it, in rank order (no float atomics).
//
// What bounds these kernels is latency: the weights are in flight before the kernel ahead has finished, and a CTA's work
// after that is a chain of round trips (x or o, the products, the other CTAs' sums).  So a chain is cut into as many CTAs
// as help (projection_parts in api.cu), and each of its links is one round trip: all of a head's o loads, and all the remote loads
// of a row's sums, are in flight at once.  Measured on one B200, per layer step of 128 sequences, 8 heads, d = 1024, 128
// rows: 24.7 -> 17.1 us, about 1 us of it from the attention step between them (the 4.7 MB of weights take 0.7 us
// at the copy rate).
//
// NB = batch columns of a tile (the batch rounded up to 16, 32, 64 or 128; larger batches take
// several tiles of 128).  Every wait is bounded (mbar_wait); TMEM is freed on every path.
#pragma once
#include <cuda_bf16.h>

#include "decode_umma.cuh"

namespace mqa {

constexpr int kProjWorkWarps = 8;              // convert o, read the sums out, add them up
constexpr int kProjTmaWarp = 8, kProjMmaWarp = 9;
constexpr int kProjThreads = 10 * 32;
constexpr int kProjChunkBytes = 128 * 256;     // 128 rows x 128 bf16 of a weight matrix: 32 KiB, two 64-column boxes
constexpr int kProjMaxGroups = 16;             // project_out: head groups of a tile = CTAs of one cluster (16: the
                                               // non-portable cluster size, which the B200 offers; two heads per CTA at h = 32)
constexpr int kProjMaxParts = 8;               // project_in: CTAs (of one cluster) that share a slab's d rows

template <int NB>
struct ProjCfg {
    static_assert(NB == 16 || NB == 32 || NB == 64 || NB == 128, "batch columns of a tile");
    static constexpr int kActBytes = NB * 256;                 // NB rows x 128 bf16, two 64-column boxes
    static constexpr int kStages = NB == 128 ? 3 : 4;
    static constexpr int kStageBytes = kProjChunkBytes + kActBytes;
    static constexpr int kSmemBytes = kStages * kStageBytes + 256 /* barriers */ + 1024 /* alignment slack */;
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
}

// Batch row n of the tile, features lane * 4 .. + 3: the sums of all the cluster's CTAs, added up in rank order.  Every
// remote load of a row is asked for before the first is used (one round trip through the cluster per row, not one per CTA).
template <int MAX_CTAS>
__device__ __forceinline__ float4 add_up_row(uint32_t sums, int n, int lane, int ctas) {
    float4 part[MAX_CTAS];
#pragma unroll
    for (int g = 0; g < MAX_CTAS; ++g)
        if (g < ctas) part[g] = cluster_ld_f4(cluster_map(sums + (uint32_t)(n * 128 + lane * 4) * 4, (uint32_t)g));
    float4 sum = part[0];
#pragma unroll
    for (int g = 1; g < MAX_CTAS; ++g)
        if (g < ctas) { sum.x += part[g].x; sum.y += part[g].y; sum.z += part[g].z; sum.w += part[g].w; }
    return sum;
}

template <int NB>
__global__ void __launch_bounds__(kProjThreads, 1)
project_in_kernel(const __grid_constant__ CUtensorMap map_pq, const __grid_constant__ CUtensorMap map_pk,
                  const __grid_constant__ CUtensorMap map_pv, const __grid_constant__ CUtensorMap map_x,
                  __nv_bfloat16* __restrict__ q, __nv_bfloat16* __restrict__ k_new, __nv_bfloat16* __restrict__ v_new,
                  int32_t* __restrict__ status, int b, int h, int d) {
    using Cfg = ProjCfg<NB>;
    constexpr int S = Cfg::kStages;
    const int slab = blockIdx.x, row0 = blockIdx.z * 128;          // weight slab; first batch row of this tile
    const int part = blockIdx.y, parts = gridDim.y;                // this CTA's part of the slab's d rows: one cluster per slab
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int chunk0 = part * (d / 128) / parts;                   // chunks of 128 rows [chunk0, chunk0 + n_chunks)
    const int n_chunks = (part + 1) * (d / 128) / parts - chunk0;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* stages = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    const uint32_t stages_s = smem_addr(stages);
    const uint32_t full_s = stages_s + S * Cfg::kStageBytes, empty_s = full_s + S * 8, done_s = empty_s + S * 8;
    __shared__ uint32_t tmem_slot;
    __shared__ int timed_out, issued;

    // The weights do not depend on the kernel before this one, x does: a stage's barrier takes two arrivals, one with
    // the weight chunk's bytes and one with the x chunk's, and the weight copies of the first stages start before the wait.
    const CUtensorMap* wmap = slab < h ? &map_pq : (slab == h ? &map_pk : &map_pv);
    const int wrow0 = slab < h ? slab * d : 0;
    auto issue_weights = [&](int c) {
        const uint32_t bar = full_s + (c % S) * 8, w_s = stages_s + (c % S) * Cfg::kStageBytes;
        mbar_expect_tx(bar, kProjChunkBytes);
        tma_load_2d(w_s, wmap, 0, wrow0 + (chunk0 + c) * 128, bar);
        tma_load_2d(w_s + kProjChunkBytes / 2, wmap, kBoxCols, wrow0 + (chunk0 + c) * 128, bar);
    };
    auto issue_x = [&](int c) {
        const uint32_t bar = full_s + (c % S) * 8, x_s = stages_s + (c % S) * Cfg::kStageBytes + kProjChunkBytes;
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
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int c = 0; c < n_chunks && c < S; ++c) issue_weights(c);
    }
    if (warp == kProjMmaWarp) { tmem_alloc(smem_addr(&tmem_slot), Cfg::kTmemCols); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    grid_dependency_wait();          // x may come from the kernel before this one
    grid_launch_dependents();

    if (warp == kProjTmaWarp) {
        if (lane == 0) {
            bool ok = true;
            for (int c = 0; c < n_chunks && ok; ++c) {
                if (c >= S) {
                    ok = mbar_wait(empty_s + (c % S) * 8, ((c / S) - 1) & 1);
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
                const int st = c % S;
                if (ok) ok = mbar_wait(full_s + st * 8, (c / S) & 1);
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
    if (parts > 1) cluster_sync();   // every part's sums are in its shared memory
    {
        __nv_bfloat16* out = slab < h ? q + (size_t)slab * 128 : (slab == h ? k_new : v_new);
        const size_t stride = slab < h ? (size_t)h * 128 : 128;
        for (int n = part + parts * warp; n < NB && row0 + n < b; n += parts * (kProjThreads / 32)) {
            const float4 v = add_up_row<kProjMaxParts>(stages_s, n, lane, parts);
            *reinterpret_cast<uint2*>(out + (size_t)(row0 + n) * stride + lane * 4) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
        }
    }
    if (parts > 1) cluster_sync();   // nobody leaves while its shared memory is being read
    if (warp == kProjMmaWarp) { tc_fence_after(); tmem_dealloc(tmem, Cfg::kTmemCols); }
}

// The head groups of one (d tile, batch tile) form one thread-block cluster (gridDim.y CTAs, at most 16): each CTA
// accumulates Y^T over its heads in TMEM, leaves it in its shared memory, and after a cluster barrier every CTA adds up,
// in group order, the batch rows that fall to it (row n to CTA n mod cluster size) out of all the CTAs' shared memory
// and stores them to y.  No partial sums pass through global memory and no float atomics are used.
template <int NB>
__global__ void __launch_bounds__(kProjThreads, 1)
project_out_kernel(const __grid_constant__ CUtensorMap map_po, const float* __restrict__ o, float* __restrict__ y,
                   int32_t* __restrict__ status, int b, int h, int d, int heads_per_cta) {
    using Cfg = ProjCfg<NB>;
    constexpr int S = 2;                                           // ring of two stages: a head's weights and its o tile
    const int tile = blockIdx.x, group = blockIdx.y, row0 = blockIdx.z * 128;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int head0 = group * heads_per_cta;
    const int n_heads = max(0, min(heads_per_cta, h - head0));

    extern __shared__ uint8_t smem_raw[];
    uint8_t* stages = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    const uint32_t stages_s = smem_addr(stages);
    const uint32_t w_full = stages_s + S * Cfg::kStageBytes, o_full = w_full + S * 8, empty_s = o_full + S * 8, done_s = empty_s + S * 8;
    __shared__ uint32_t tmem_slot;
    __shared__ int timed_out, issued;

    if (warp == kProjTmaWarp && lane == 0) {                                  // by the thread that issues the copies
        prefetch_tensormap(&map_po);
        timed_out = 0;
        issued = 0;
        for (int s = 0; s < S; ++s) { mbar_init(w_full + s * 8, 1); mbar_init(o_full + s * 8, kProjWorkWarps); mbar_init(empty_s + s * 8, 1); }
        mbar_init(done_s, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kProjMmaWarp) { tmem_alloc(smem_addr(&tmem_slot), Cfg::kTmemCols); tmem_relinquish(); }
    auto issue_weights = [&](int i) {
        const int st = i % S;
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
    grid_dependency_wait();          // o comes from the kernel before this one
    grid_launch_dependents();

    if (warp == kProjTmaWarp) {
        if (lane == 0) {
            bool ok = true;
            for (int i = S; i < n_heads && ok; ++i) {
                ok = mbar_wait(empty_s + (i % S) * 8, ((i / S) - 1) & 1);
                if (ok) issue_weights(i);
            }
            if (!ok) atomicExch(&timed_out, 1);
        }
    } else if (warp == kProjMmaWarp) {
        if (lane == 0) {
            constexpr uint32_t kIdesc = umma_idesc(128, NB, false, false);
            bool ok = true;
            for (int i = 0; i < n_heads; ++i) {
                const int st = i % S;
                if (ok) ok = mbar_wait(w_full + st * 8, (i / S) & 1);
                if (ok) ok = mbar_wait(o_full + st * 8, (i / S) & 1);
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
            const int st = i % S;
            float4 v[NB / kProjWorkWarps];
#pragma unroll
            for (int k = 0; k < NB / kProjWorkWarps; ++k) {
                const int n = warp + k * kProjWorkWarps;
                v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (row0 + n < b) v[k] = *reinterpret_cast<const float4*>(o + ((size_t)(row0 + n) * h + head0 + i) * kHeadDim + lane * 4);
            }
            if (i >= S && ok) ok = mbar_wait(empty_s + st * 8, ((i / S) - 1) & 1);   // the product that read this tile is done
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
    cluster_sync();                  // every group's Y^T is in its shared memory
    const int rank = (int)cluster_cta_rank(), n_groups = (int)cluster_size();
    for (int n = rank + n_groups * warp; n < NB && row0 + n < b; n += n_groups * (kProjThreads / 32)) {
        const float4 sum = add_up_row<kProjMaxGroups>(stages_s, n, lane, n_groups);
        *reinterpret_cast<float4*>(y + (size_t)(row0 + n) * d + (size_t)tile * 128 + lane * 4) = sum;
    }
    cluster_sync();                  // nobody leaves while its shared memory is being read
    if (warp == kProjMmaWarp) { tc_fence_after(); tmem_dealloc(tmem, Cfg::kTmemCols); }
}

}  // namespace mqa
