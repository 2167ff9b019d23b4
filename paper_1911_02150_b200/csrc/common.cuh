// Shared device helpers for the decode-attention kernels (sm_100a).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mqa {

constexpr int kHeadDim = 128;                 // k == v == 128 (Section 4.1: d_k = d_v = 128)
constexpr int kRowBytes = kHeadDim * 2;       // one bf16 cache row
constexpr float kLog2e = 1.4426950408889634f;
// Where a running maximum of logits stands once it has seen rows, however low: (-inf) - (-inf) is NaN, and rows whose logits are -inf
// have to weigh nothing.  A piece that holds only such rows has this maximum and a sum of 0 (one that holds no rows has -inf and 0), so
// that nothing but such rows gives 0 / 0 and an empty prefix zeros.
constexpr float kLowestMax = -3.402823466e38f;

// status bits (mirrors include/mqa_decode.h)
constexpr int kStatusAppendFull = 1;
constexpr int kStatusAppendNegative = 2;
constexpr int kStatusLenClamped = 4;
constexpr int kStatusPipelineTimeout = 8;

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 16-byte global load that does not allocate in L1 (each cache byte is used once).
__device__ __forceinline__ uint4 ldg_stream(const void* p) {
    uint4 r;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
    return r;
}

// Programmatic dependent launch.  grid_dependency_wait(): block until the kernels this launch was
// made dependent on have finished and their writes are visible (a no-op for an ordinary launch).
// grid_launch_dependents(): allow the next kernel in the stream, if it was launched as a
// programmatic dependent, to start its prologue while this grid is still running.  Every kernel
// here waits first and lets its dependents start afterwards: with second-pass kernels that let
// theirs start before their own wait, a decoding loop of four kernels per step gave results that
// differed from run to run.
// So a kernel may be resident while the one ahead of it still writes what it will read, and none of that is read-only for
// its lifetime: memory that a kernel ahead may have written (lens, positions, q, new rows, o, pieces, the cache) is read after the
// wait with ordinary loads or __ldcg, never with a read-only one (__ldg; a plain load through a const __restrict__ pointer becomes
// one too, so those pointers have no __restrict__), which need not see the write.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;"); }

// Clamp a sequence length into [0, m_max]; flag the status word if it had to move.
__device__ __forceinline__ int clamp_len(int L, int m_max, int32_t* status) {
    if (L < 0 || L > m_max) {
        if (status) atomicOr(status, kStatusLenClamped);
        L = L < 0 ? 0 : m_max;
    }
    return L;
}

// Rows to attend over when the caller's lens[] still holds the count from before this step's append
// (bias = 1): a sequence that could take the new row (0 <= lens < m_max) has one more row than lens says.
__device__ __forceinline__ int biased_len(int raw, int m_max, int bias) {
    return (bias && raw >= 0 && raw < m_max) ? raw + 1 : raw;
}

// ---- thread-block cluster helpers (the pieces of a sequence, and the CTAs that share a projection, are summed through
// distributed shared memory)
__device__ __forceinline__ uint32_t cluster_cta_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t n;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
    return n;
}
// every thread of every CTA of the cluster, the same number of times on every path: what a CTA wrote to its shared
// memory before is visible to the others after
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();                    // the aligned forms want the whole warp at the same instruction
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
// (without the release: where the barrier only keeps CTAs from leaving, and what was written is known to have arrived)
__device__ __forceinline__ void cluster_arrive_relaxed() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() { cluster_arrive(); cluster_wait(); }
// The address, in the cluster's shared window, of this CTA's shared address `local` in the CTA of rank `rank`.
__device__ __forceinline__ uint32_t cluster_map(uint32_t local, uint32_t rank) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    return remote;
}
__device__ __forceinline__ float4 cluster_ld_f4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float2 cluster_ld_f2(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}
// 16 (or 8) bytes from registers to an address in the cluster's shared window, counted on an mbarrier of the CTA that gets them.
__device__ __forceinline__ void cluster_send_f4(uint32_t addr, float4 v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1,%2,%3,%4}, [%5];"
                 ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ void cluster_send_f2(uint32_t addr, float2 v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1,%2}, [%3];"
                 ::"r"(addr), "f"(v.x), "f"(v.y), "r"(bar) : "memory");
}

}  // namespace mqa
