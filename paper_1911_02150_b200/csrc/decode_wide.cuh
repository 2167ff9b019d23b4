// Multi-query decoding step for MANY query rows per sequence (33 and more: many heads, or beams x heads over one shared
// memory, Section 4.2; 128 rows per CTA, more as grid.y row tiles over the same cache rows) -- the same three lines of Section 3 (logits = einsum(bhk,bmk->bhm), softmax over the valid
// prefix, o = einsum(bhm,bmv->bhv)), with the query rows as the ROWS of the tensor-core tiles.
//
// The streaming kernel (decode_umma.cuh) puts the cache rows on the TMEM lanes and the heads on the columns, which is
// right for a few heads (N = 16 .. 32) but makes the softmax a cross-thread affair; from 64 query rows on that kernel
// is bound by its softmax warps, not by HBM.  Here a CTA holds all the sequence's query rows as ONE 128-row Q tile
// (rows past h are whatever shared memory held: computed, never stored) and walks a fixed split of the
// sequence's cache rows in stages of 128:
//     S   = Q K_j^T        tcgen05.mma, M = 128 query rows (TMEM lanes), N = 128 cache rows, fp32 in TMEM
//     P   = exp2(S log2e - m)   one thread per query row: the row's maximum and sum need no other thread
//     O  += P V_j          tcgen05.mma with A = P read from TMEM (bf16 pairs in columns of their own), B = V_j (MN-major)
// The two softmax warpgroups take the stages in turn (warpgroup w: stages w, w + 2, ...), each with weights, an
// O accumulator, reference maxima and sums of its own -- two partial softmaxes over interleaved rows of the cache,
// merged exactly at the end (the same recombination as between splits) -- so the logits of a stage are computed and
// its weights formed while the other warpgroup's stage is multiplied with V.  TMEM: one buffer of logits that the stages
// use in turn, P_0, P_1, O_0, O_1 (512 columns; why they lie like this, and why two warps issue the products: prefill.cuh).
// A CTA writes o itself when the sequence has one split, else a piece (maximum, sum, unnormalised rows) for the
// second-pass kernel (combine.cuh).  Valid prefix: rows >= lens are never fetched except in a split's last stage,
// where they are masked by index (select) and their V rows cleared in shared memory.
//
// Roles: warps 0-3 and 4-7 the two softmax warpgroups, warp 8 TMA producer, warps 9 and 10 issue the products (warp 11 only
// completes the third warpgroup, which hands most of its registers to the other two).  The compiler may give a thread 168
// registers, whatever the softmax warps have in the end, and keeps 2 to 8 values of theirs in local memory (EARLY 0, 1, 2: 32, 8, 20
// bytes of spills).  Every wait is bounded.
#pragma once
#include "prefill.cuh"

namespace mqa {

constexpr int kWideRows = 128;                                 // query rows of the tile = cache rows per stage
constexpr int kWideKSlots = 3, kWideVSlots = 3;
constexpr int kWideThreads = 12 * 32;
constexpr int kWideProducerWarp = 8, kWideSWarp = 9, kWidePvWarp = 10;
// barriers: q_full, k_full/k_empty, v_full/v_empty per slot, s_ready[2], p_ready[2], pv_done[2], s_free
constexpr int kWideBarriers = 1 + 2 * kWideKSlots + 2 * kWideVSlots + 7;
constexpr int kWideSmemBytes = (1 + kWideKSlots + kWideVSlots) * kPfTileBytes + kWideBarriers * 8 + 16 + 1024 /* alignment slack */;
static_assert(kWideSmemBytes + 1024 + 16 /* static */ <= 227 * 1024, "exceeds the shared memory of one SM");

// grid: x = sequence * n_splits + split, y = tile of 128 query rows.  part_ml [b * h][n_splits], part_acc [b * h][n_splits][128] (combine.cuh).
// EARLY: what is fetched before the wait for the kernel ahead -- 0 nothing; 1 (the caller's promise of a decoding loop) the
// first stage, if it lies wholly below the prefix's last rows by lens as it reads now, which is final or one short (or else right
// after the wait, if the prefix has its rows in any case); 2 (behind the library's own projection or host-input kernel: lens
// is final) the first stages whatever they hold.  In a loop of two launches per step a CTA is on its SM, set up and idle, while
// the second pass of the step before runs.  One stage and no more: q has to come next, and behind 28 MB of stages (three per
// CTA) it took 4.7 us (us per step with 0 / 1 / 2 / 3 stages ahead: 32 x 128 rows x 8192: 30.3 / 30.4 / 31.8 / 32.1; 64 x 100 x 2048: 20.6 /
// 19.8 / 21.0 / 21.8; 8 x 16 x 32768: 27.9 / 26.9 / 27.3 / 29.0; 8 x 16 x 4096: 11.5 / 9.6 / 9.9 / 9.6).
template <int EARLY>
__global__ void __launch_bounds__(kWideThreads, 1)
mqa_decode_wide_kernel(const uint4* __restrict__ q, const __grid_constant__ CUtensorMap map_k,
                       const __grid_constant__ CUtensorMap map_v, const int32_t* __restrict__ lens, float* __restrict__ o,
                       float2* __restrict__ part_ml, float* __restrict__ part_acc, int32_t* __restrict__ status, int h,
                       int m_max, int chunk_rows, int n_splits, int len_bias, const FusedArgs fa, int32_t* __restrict__ lens_advance,
                       int mode) {
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int seq = blockIdx.x / n_splits, split = blockIdx.x % n_splits;
    const int row0 = blockIdx.y * kWideRows;                   // this CTA's first query row of the sequence (more than 128: grid.y tiles)

    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);     // the 128-byte swizzle repeats every 1 KiB
    const uint32_t q_s = smem_addr(base);
    const uint32_t k_ring = q_s + kPfTileBytes, v_ring = k_ring + kWideKSlots * kPfTileBytes;
    const uint32_t bars = v_ring + kWideVSlots * kPfTileBytes;
    const uint32_t q_full = bars, k_full = bars + 8, k_empty = k_full + 8 * kWideKSlots, v_full = k_empty + 8 * kWideKSlots,
                   v_empty = v_full + 8 * kWideVSlots, s_ready = v_empty + 8 * kWideVSlots, p_ready = s_ready + 16,
                   pv_done = p_ready + 16, s_free = pv_done + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + (1 + kWideKSlots + kWideVSlots) * kPfTileBytes + kWideBarriers * 8);
    __shared__ int timed_out;
    __shared__ float2 ex_ml[kWideRows];                       // (maximum, sum) of warpgroup 1's rows, then each row's two factors

    if (threadIdx.x == 0) {
        prefetch_tensormap(&map_k); prefetch_tensormap(&map_v);
        mbar_init(q_full, 8);
        mbar_init(s_free, 4);
        for (int i = 0; i < kWideKSlots; ++i) { mbar_init(k_full + 8 * i, 1); mbar_init(k_empty + 8 * i, 1); }
        for (int i = 0; i < kWideVSlots; ++i) { mbar_init(v_full + 8 * i, 1); mbar_init(v_empty + 8 * i, 1); }
        for (int w = 0; w < 2; ++w) { mbar_init(s_ready + 8 * w, 1); mbar_init(p_ready + 8 * w, 4); mbar_init(pv_done + 8 * w, 1); }
        timed_out = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kWideSWarp) {
        tmem_alloc(smem_addr(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);

    const int r0 = split * chunk_rows;                         // this CTA's rows of the sequence's cache begin here
    const bool producer = warp == kWideProducerWarp && lane == 0;
    const uint64_t policy = l2_stream_policy(true);            // the cache is read once per step
    constexpr int kAhead = EARLY == 1 ? 1 : kWideKSlots < kWideVSlots ? kWideKSlots : kWideVSlots;
    auto issue_k = [&](int j) {
        const int ks = j % kWideKSlots, y = seq * m_max + r0 + j * kWideRows;
        mbar_expect_tx(k_full + 8 * ks, kPfTileBytes);
        tma_load_2d_hint(k_ring + ks * kPfTileBytes, &map_k, 0, y, k_full + 8 * ks, policy);
        tma_load_2d_hint(k_ring + ks * kPfTileBytes + kPfHalfBytes, &map_k, kBoxCols, y, k_full + 8 * ks, policy);
    };
    auto issue_v = [&](int j) {
        const int vs = j % kWideVSlots, y = seq * m_max + r0 + j * kWideRows;
        mbar_expect_tx(v_full + 8 * vs, kPfTileBytes);
        tma_load_2d_hint(v_ring + vs * kPfTileBytes, &map_v, 0, y, v_full + 8 * vs, policy);
        // (for tests: one copy of the first CTA's second stage is never started, so that a wait runs out)
        if (!((mode & kMmaWithhold) != 0 && blockIdx.x == 0 && blockIdx.y == 0 && j == 1))
            tma_load_2d_hint(v_ring + vs * kPfTileBytes + kPfHalfBytes, &map_v, kBoxCols, y, v_full + 8 * vs, policy);
    };
    int pre = 0, guess = 0;                                    // stages asked for so far (by the producer's thread)
    if (EARLY != 0 && producer) {
        guess = max(0, __ldcg(lens + seq));
        // (2: rows in the prefix once the new one is in; 1: the step ahead writes row guess - 1 or row guess)
        const int rows = min((EARLY == 2 ? min(guess + 1, m_max) : min(guess - 1, m_max)) - r0, chunk_rows);
        const int ready = max(0, min(EARLY == 2 ? (rows + kWideRows - 1) / kWideRows : rows / kWideRows, kAhead));
        for (; pre < ready; ++pre) { issue_k(pre); issue_v(pre); }
    }

    grid_dependency_wait();              // q, lens and the newest cache row may come from the kernel before
    grid_launch_dependents();
    if (EARLY == 1 && producer) {        // the rows that the prefix has in any case (for tests, MQA_STEP_TEST_WRONG_GUESS: a stage more)
        const int rows = min(min(guess + 1 + ((mode & kMmaWrongGuess) != 0 ? kWideRows : 0), m_max) - r0, chunk_rows);
        const int sure = max(pre, min((rows + kWideRows - 1) / kWideRows, kAhead));
        for (; pre < sure; ++pre) { issue_k(pre); issue_v(pre); }
    }
    // The append-and-attend step (fa.k_new given): the CTA whose rows hold row lens[seq] puts the new key/value row into its
    // place in the landed stage (the warps that issue the products do) and stores it in the cache (its producer warp, with
    // nobody waiting for it), every split attends over one row more, and lens moves on at the end -- here when the sequence
    // has one split (lens_advance given), else in the second-pass kernel.
    uint4 row_piece = make_uint4(0u, 0u, 0u, 0u);              // lanes 0-15: of the key row (S and producer warp), or the value row
    if (fa.k_new != nullptr && warp >= kWideProducerWarp)      // (the producer warp's lanes 16-31 the value row)
        row_piece = __ldcg((warp == kWidePvWarp || (warp == kWideProducerWarp && lane >= 16) ? fa.v_new : fa.k_new) + (size_t)seq * (kRowBytes / 16) + (lane & 15));
    const int raw = __ldcg(lens + seq);
    const bool appended = fa.k_new != nullptr && raw >= 0 && raw < m_max;
    if (fa.k_new != nullptr && !appended && split == 0 && blockIdx.y == 0 && threadIdx.x == 0 && status)
        atomicOr(status, raw < 0 ? kStatusAppendNegative : kStatusAppendFull);
    const int L = clamp_len(appended ? raw + 1 : biased_len(raw, m_max, len_bias), m_max, (split == 0 && blockIdx.y == 0 && threadIdx.x == 0) ? status : nullptr);
    const int r1 = min(r0 + chunk_rows, L);                    // and end here
    const int n_kv = __shfl_sync(0xffffffffu, r1 > r0 ? (r1 - r0 + kWideRows - 1) / kWideRows : 0, 0);      // stages
    const bool hilo = __any_sync(0xffffffffu, L < kSingleRoundingMinRows);
    const bool holds_new = appended && raw >= r0 && raw - r0 < chunk_rows;
    const int new_stage = holds_new ? (raw - r0) / kWideRows : -1;
    // the new row into a landed K or V stage, by a warp's lanes 0-15
    auto place_row = [&](uint32_t stage_s) {
        const int row = (raw - r0) % kWideRows;
        if (lane < 16)
            asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(stage_s + (lane >> 3) * kPfHalfBytes + row * 128 + (((lane & 7) ^ (row & 7)) << 4)),
                         "r"(row_piece.x), "r"(row_piece.y), "r"(row_piece.z), "r"(row_piece.w) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // read by the tensor core
        __syncwarp();
    };

    if (warp >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPfRegsOther));
        if (warp == kWideProducerWarp) {
            // =========================================================== TMA producer
            if (holds_new) {
                const size_t at = ((size_t)seq * m_max + raw) * (kRowBytes / 16) + (lane & 15);
                if (lane < 16) fa.K[at] = row_piece; else fa.V[at] = row_piece;
            }
            if (lane == 0 && (n_kv > 0 || pre > 0)) {
                bool ok = true;
                int issued_k = pre, issued_v = pre;
                for (int j = pre; j < n_kv && ok; ++j) {
                    if (j >= kWideKSlots) ok = mbar_wait(k_empty + 8 * (j % kWideKSlots), ((j / kWideKSlots) - 1) & 1);
                    if (!ok) break;
                    issue_k(j);
                    issued_k = j + 1;
                    if (j >= kWideVSlots) ok = mbar_wait(v_empty + 8 * (j % kWideVSlots), ((j / kWideVSlots) - 1) & 1);
                    if (!ok) break;
                    issue_v(j);
                    issued_v = j + 1;
                }
                for (int j = n_kv; j < pre; ++j) ok = mbar_wait(k_full + 8 * j, 0) && mbar_wait(v_full + 8 * j, 0) && ok;   // (a broken promise)
                if (!ok) {
                    // a wait ran out: the copies already started are given a bounded wait each before the CTA may leave
                    atomicExch(&timed_out, 1);
                    for (int j = max(0, issued_k - kWideKSlots); j < issued_k; ++j) mbar_wait(k_full + 8 * (j % kWideKSlots), (j / kWideKSlots) & 1);
                    for (int j = max(0, issued_v - kWideVSlots); j < issued_v; ++j) mbar_wait(v_full + 8 * (j % kWideVSlots), (j / kWideVSlots) & 1);
                }
            }
        } else if (warp == kWideSWarp) {
            // =========================================================== issuer of the logits: S = Q K_j^T, each stage as soon as
            // the one before is in registers
            constexpr uint32_t kIdescS = umma_idesc(128, 128, false, false);
            bool ok = n_kv == 0 || warp_wait(q_full, 0);
            for (int j = 0; j < n_kv && ok; ++j) {
                const int slot = j % kWideKSlots;
                ok = warp_wait(k_full + 8 * slot, (j / kWideKSlots) & 1);
                if (ok && j > 0) ok = warp_wait(s_free, (j - 1) & 1);
                if (!ok) break;
                const uint32_t k_s = k_ring + slot * kPfTileBytes;
                if (j == new_stage) place_row(k_s);
                tc_fence_after();
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {            // 8 k-steps of 16 columns; 4 per 64-column box
                        const uint32_t off = (ks >> 2) * kPfHalfBytes + (ks & 3) * 32;
                        umma_ss(tmem_base, umma_desc(q_s + off, 16, 1024), umma_desc(k_s + off, 16, 1024), kIdescS, ks ? 1u : 0u);
                    }
                    tc_commit(s_ready + 8 * (j & 1));
                    tc_commit(k_empty + 8 * slot);
                }
                __syncwarp();
            }
            if (!ok && lane == 0) atomicExch(&timed_out, 1);
        } else if (warp == kWidePvWarp) {
            // =========================================================== issuer of O_w += P_w V_j: P from tensor memory (bf16 pairs: 8
            // columns per 16 rows of V), both parts of it where there are two
            constexpr uint32_t kIdescO = umma_idesc(128, 128, false, true);
            bool ok = true;
            int n_p[2] = {0, 0};
            for (int j = 0; j < n_kv && ok; ++j) {
                const int slot = j % kWideVSlots, w = j & 1;
                const uint32_t v_s = v_ring + slot * kPfTileBytes;
                ok = warp_wait(v_full + 8 * slot, (j / kWideVSlots) & 1);
                if (ok && j == new_stage) place_row(v_s);
                for (int part = 0; part < (hilo ? 2 : 1) && ok; ++part) {
                    ok = warp_wait(p_ready + 8 * w, n_p[w] & 1);
                    if (!ok) break;
                    ++n_p[w];
                    tc_fence_after();
                    if (elect_one()) {
                        // one rounding: the stage's 128 rows; hi and lo: 64 of them, twice over
                        const uint32_t v_p = v_s + part * 4 * 2048;
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            umma_ts(tmem_base + kPfTmemO + w * 128, tmem_base + kPfTmemP + w * 64 + kk * 8,
                                    umma_desc(v_p + (hilo ? kk & 3 : kk) * 2048, kPfHalfBytes, 1024), kIdescO, (j < 2 && part == 0 && kk == 0) ? 0u : 1u);
                        tc_commit(pv_done + 8 * w);
                        if (part == (hilo ? 1 : 0)) tc_commit(v_empty + 8 * slot);
                    }
                    __syncwarp();
                }
            }
            if (!ok && lane == 0) atomicExch(&timed_out, 1);
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPfRegsSoftmax));
        // =============================================================== softmax warpgroups: one thread per query row
        const int w = warp >> 2, quarter = warp & 3, r = quarter * 32 + lane;
        const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const uint32_t p_t = lane_base + kPfTmemP + w * 64, o_t = lane_base + kPfTmemO + w * 128;
        // q, by the threads that have nothing else to do yet: 16 bytes a thread and turn, all its loads in flight, in the layout of
        // a K-major operand with the 128-byte swizzle.  (A tensor copy waited for the producer to read lens, and queued behind
        // the stages already asked for.)
        const int n_rows = min(h - row0, kWideRows);                  // query rows of this tile
        {
            uint4 v[8];
            const uint4* src = q + ((size_t)seq * h + row0) * (kRowBytes / 16);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (threadIdx.x + i * 256 < n_rows * 16) v[i] = __ldcg(src + threadIdx.x + i * 256);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int item = threadIdx.x + i * 256, row = item >> 4, ch = item & 15;
                if (item < n_rows * 16)
                    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(q_s + (ch >> 3) * kPfHalfBytes + row * 128 + (((ch & 7) ^ (row & 7)) << 4)),
                                 "r"(v[i].x), "r"(v[i].y), "r"(v[i].z), "r"(v[i].w) : "memory");
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(q_full);
        }
        // a warp none of whose rows is one of the sequence's only keeps the barriers' counts
        const bool idle = quarter * 32 >= n_rows, mine = r < n_rows;
        float m = -INFINITY, l = 0.f;                                 // reference maximum (log2 units), sum of weights
        bool ok = true;
        int n_p = 0;                                                  // products of this warpgroup's weights so far
        for (int j = w; j < n_kv; j += 2) {
            const int ph = j >> 1;
            const int valid = r1 - (r0 + j * kWideRows);              // rows of the stage inside this split's prefix (> 0)
            if (ok) ok = mbar_wait(s_ready + 8 * w, ph & 1);
            tc_fence_after();
            auto clear_v = [&]() {
                if (valid < kWideRows) {
                    // the stage runs past the prefix: the tensor core would multiply the zero weights with whatever lies
                    // there (NaN * 0 = NaN), so those V rows are cleared first
                    const int vs = j % kWideVSlots;
                    if (ok) ok = mbar_wait(v_full + 8 * vs, (j / kWideVSlots) & 1);
                    const uint32_t v_s = v_ring + vs * kPfTileBytes;
                    for (int i = r; i < (kWideRows - valid) * 16; i += 128) {
                        const int vrow = valid + (i >> 4), ch = i & 15;
                        const uint32_t a = v_s + (ch >> 3) * kPfHalfBytes + vrow * 128 + ((ch & 7) << 4);
                        asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(a), "r"(0u) : "memory");
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                }
            };
            uint32_t x[128];
            if (idle) {
                if (lane == 0) mbar_arrive(s_free);
                clear_v();
                for (int part = 0; part < (hilo ? 2 : 1); ++part, ++n_p) {
                    if (n_p > 0 && ok) ok = mbar_wait(pv_done + 8 * w, (n_p - 1) & 1);    // (the arrival below belongs to the next phase)
                    __syncwarp();
                    if (lane == 0) mbar_arrive(p_ready + 8 * w);
                }
            } else {
                // ---- the row's 128 logits, read once and kept in registers; rows past the prefix masked by index (a select)
                tmem_ld_cols<128>(lane_base, x);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(s_free);                       // the next stage's logits may take their place
                if (valid < kWideRows) {
#pragma unroll
                    for (int i = 0; i < 128; ++i)
                        if (i >= valid) x[i] = 0xff800000u;               // -inf
                }
                float mx8[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) mx8[i] = fmaxf(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1]));
#pragma unroll
                for (int i = 8; i < 64; ++i) mx8[i & 7] = max3(mx8[i & 7], __uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1]));
                const float mx = max3(max3(mx8[0], mx8[1], mx8[2]), max3(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7])) * kLog2e;
                if (__any_sync(0xffffffffu, mine && mx > m + kPfMaxLead)) {  // (rows past the sequence's last hold no query)
                    // ---- a row of this warp leads its reference by too much: every row of the warp moves its reference
                    // to its largest logit so far and rescales its sum and its row of O
                    const float m_new = fmaxf(m, mx);
                    if (ph > 0) {
                        const float f = m == m_new ? 1.f : fast_exp2(m - m_new);     // (m = -inf while all logits were)
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
                // ---- P = exp2(S log2e - m) as bf16 pairs (hi) and, for a short prefix, their remainders (lo)
                const float neg_m = m == -INFINITY ? 0.f : -m;            // (nothing but logits of -inf so far: weights of zero)
                const unsigned long long neg_m2 = f2_pack(neg_m, neg_m), log2e2 = f2_pack(kLog2e, kLog2e);
                unsigned long long sum2[2] = {0ull, 0ull};
                clear_v();
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
                if (hilo) {
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
        }
        if (n_p > 0 && ok) ok = mbar_wait(pv_done + 8 * w, (n_p - 1) & 1);
        // (Q and the K ring are used below: a last stage that is the other warpgroup's must have its logits.  That warpgroup's
        // logits before those were ready before this one's last ones were issued, so the wait cannot be a phase early)
        if (n_p > 0 && n_kv > 1 && ((n_kv - 1) & 1) != w && ok) ok = mbar_wait(s_ready + 8 * (w ^ 1), ((n_kv - 1) >> 1) & 1);
        tc_fence_after();
        // ---- the two warpgroups' partial results become one: each leaves (maximum, sum) and its rows of O in shared memory
        // (warpgroup 0 where Q and the first K slot were, 1 in the other two; 16-byte pieces swizzled by row), then all eight
        // warps merge whole rows on the way out, 512 contiguous bytes per instruction.
        if (!idle) {
            if (w == 1) ex_ml[r] = make_float2(m, l);
            if (n_p > 0) {
                const uint32_t ex_o = q_s + (w * kWideRows + r) * 512;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");           // (it was the copy engine's and the tensor core's)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t y[32];
                    tmem_ld32(o_t + c * 32, y);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; i += 4)
                        asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(ex_o + ((((c * 8 + (i >> 2)) ^ (r & 31)) << 4))),
                                     "r"(y[i]), "r"(y[i + 1]), "r"(y[i + 2]), "r"(y[i + 3]) : "memory");
                }
            }
        }
        named_barrier(1, 256);
        const bool two = n_kv > 1;                                                     // warpgroup 1 had a stage
        if (w == 0 && mine) {
            // (maximum, sum) of the row, and what each warpgroup's sums count for
            float2 ml = make_float2(-INFINITY, 0.f);                                   // (nothing of this split inside the prefix: an empty piece)
            if (n_kv > 0) {
                const float2 other = ex_ml[r];
                const float top = two ? fmaxf(m, other.x) : m;
                // (a share of logits that are all -inf has that maximum and a sum of 0)
                const float f0 = m == top ? 1.f : fast_exp2(m - top), f1 = !two ? 0.f : other.x == top ? 1.f : fast_exp2(other.x - top);
                ml = make_float2(fmaxf(top, kLowestMax), f0 * l + (two ? f1 * other.y : 0.f));
                const float scale = n_splits == 1 ? 1.f / ml.y : 1.f;
                ex_ml[r] = make_float2(f0 * scale, f1 * scale);
            }
            if (n_splits > 1) part_ml[((size_t)seq * h + row0 + r) * n_splits + split] = ml;
        }
        named_barrier(2, 256);
        if (n_kv > 0 || n_splits == 1) {
#pragma unroll 4
            for (int i = 0; i < kWideRows / 8; ++i) {
                const int row = warp + 8 * i;
                if (row >= n_rows) break;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (n_kv > 0) {
                    const float4* rows = reinterpret_cast<const float4*>(base);
                    const float2 f = ex_ml[row];
                    const float4 a = rows[row * 32 + (lane ^ (row & 31))];
                    v = make_float4(a.x * f.x, a.y * f.x, a.z * f.x, a.w * f.x);
                    if (two) {
                        const float4 c = rows[(kWideRows + row) * 32 + (lane ^ (row & 31))];
                        v.x = fmaf(c.x, f.y, v.x); v.y = fmaf(c.y, f.y, v.y); v.z = fmaf(c.z, f.y, v.z); v.w = fmaf(c.w, f.y, v.w);
                    }
                }
                const size_t unit = (size_t)seq * h + row0 + row;
                float* dst = n_splits == 1 ? o + unit * kHeadDim : part_acc + (unit * n_splits + split) * kHeadDim;
                reinterpret_cast<float4*>(dst)[lane] = v;
            }
        }
        if (!ok) atomicExch(&timed_out, 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kWideSWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0 && timed_out && status) atomicOr(status, kStatusPipelineTimeout);
    // (one split: lens is this CTA's to move on -- with several row tiles, the sequence's other CTAs read it too, so then the
    // host leaves it to a kernel of its own)
    if (lens_advance && appended && n_splits == 1 && threadIdx.x == 0) lens_advance[seq] = raw + 1;
}

}  // namespace mqa
