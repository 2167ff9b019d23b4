// C-ABI entry points of the decode-attention library (declared in include/mqa_decode.h):
// argument validation, the launch plan, and the kernel launches.  Host code here never
// synchronises, allocates or frees device memory.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>

#include "../../include/mqa_decode.h"
#include "append.cuh"
#include "combine.cuh"
#include "common.cuh"
#include "decode_mma.cuh"
#include "project.cuh"
#include "decode_simt.cuh"
#include "decode_umma.cuh"
#include "decode_local.cuh"
#include "prefill.cuh"
#include "decode_wide.cuh"

namespace mqa {
namespace {

constexpr int kMaxDevices = 64;
std::atomic<int> g_sm_count[kMaxDevices];

// Number of SMs of the current device (148 on a B200); 148 when no device can be queried,
// so that the host-only planning calls still answer on a machine without a GPU.
int sm_count() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 148; }
    if (dev < 0 || dev >= kMaxDevices) return 148;
    int n = g_sm_count[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
        cudaGetLastError();
        return 148;
    }
    g_sm_count[dev].store(n, std::memory_order_relaxed);
    return n;
}

enum class Kernel { kSimt, kMma1, kMma2, kUmma, kWide };
std::atomic<int> g_test_cluster_room{-1};      // mqa_set_test_cluster_room
constexpr int kMergeInKernelMaxPieces = 10;
constexpr int kFewHeads = 8;                  // FEW of the fixed-split kernel: the rows of one half of a fragment
// Fixed splits of up to kMmaMaxCluster per sequence are one thread-block cluster that merges the pieces itself: one launch in place
// of two.  Measured, us per step called directly (the second launch is 2 of the host's) / in a graph: 1 x 16 heads x 512 rows 6.9 / 5.1 ->
// 4.8 / 4.9; 4 x 16 x 1000 7.6 / 5.3 -> 5.2 / 5.1; 1 x 32 x 600 8.0 / 7.5 -> 6.9 / 6.7; 30 x 8 x 900 7.9 / 7.1 -> 6.8 / 6.5; sixteen pieces
// (clusters beyond the portable eight): 1 x 16 x 2048 8.0 / 5.3 -> 5.9 / 5.0.
// A cluster of S CTAs has to fit one GPC, and a launch whose clusters do not all fit at once takes a second round: at one CTA per SM (17
// to 32 heads) 10 clusters of 8 took 6.4 us where 16 took 12.2, at two per SM 24 took 5.7 and 48 12.7.  So many as eight (of more than four
// CTAs: seven) GPCs of 17 SMs hold, and no more than the device at hand says it can run at once, which on a part of a card may be
// none of that size: those sizes keep the second pass.
int mma_clusters_at_once(int S, int ctas_per_sm);
bool clusters_fit(int sequences, int S, int ctas_per_sm) {
    return S <= kMmaMaxCluster && sequences <= 17 * ctas_per_sm / S * (S <= 4 ? 8 : 7) && sequences <= mma_clusters_at_once(S, ctas_per_sm);
}
constexpr int kMaxClusterCtas = 4;            // a sequence's CTAs as one thread-block cluster.  Measured per step: clusters of 8
                                              // (16 sequences x 16384 rows) 43 us against 29 us without, clusters of 16
                                              // (8 x 32768) 43 against 30: too few of them fit the GPCs at once

struct Plan {
    int n_splits = 0;     // 0 = invalid.  Fixed-split kernels: splits per sequence.  Persistent kernel: the
                          // most CTAs that can hold pieces of one sequence.
    int chunk_rows = 0;   // rows of the memory axis per split (persistent kernel: per CTA for full caches)
    size_t units = 0;     // b * h
    int b = 0, h = 0;
    int grid = 0;         // persistent kernel: number of CTAs
    Kernel kernel = Kernel::kSimt;
    bool merge_in_kernel = false;   // tcgen05 plan: pieces merged by the CTA that delivers a sequence's last one (single launch)
    bool cluster = false;           // fixed-split plan: the splits of a sequence are a thread-block cluster that merges them (single launch)
    bool stream() const { return kernel == Kernel::kUmma; }
};

bool dims_ok(int b, int h, int m_max) { return b > 0 && h > 0 && m_max > 0; }

// Split plan for the CUDA-core kernel (one CTA per (unit, split)): enough CTAs to fill every
// SM several times over, but not chunks shorter than 256 rows, and a single split (no
// combine launch) when the cache is short.  Where that leaves SMs short of the CTAs that fit them at once, chunks down to 128
// rows, two rounds of a CTA's warps: us per append and step, 8 sequences x 1 head x 1000 rows 9.1 -> 6.3, 20 x 4 x 1000 13.7 -> 9.2,
// 64 x 1 x 1000 13.6 -> 8.6, 8 x 1 x 8000 14.8 -> 12.7 (beyond a wave of CTAs shorter chunks lose: 20 x 4 x 2000 18.2 in 560 CTAs,
// 19.9 in 1280).
Plan plan_simt(int b, int h, int m_max) {
    Plan p;
    p.units = (size_t)b * h;
    p.b = b; p.h = h;
    const long target_ctas = (long)sm_count() * 16;
    long want = (target_ctas + (long)p.units - 1) / (long)p.units;
    const long cap = m_max / 256 > 1 ? m_max / 256 : 1;
    if (want > cap) want = cap;
    if (want > 1024) want = 1024;                 // the second pass keeps one (max, sum) per split in shared memory
    if (want < 1) want = 1;
    int chunk = (int)((m_max + want - 1) / want);
    chunk = (chunk + 63) / 64 * 64;
    p.chunk_rows = chunk;
    p.n_splits = (m_max + chunk - 1) / chunk;
    const long at_once = (long)sm_count() * kSimtCtasPerSm;
    if (p.n_splits > 1 && (long)p.units * p.n_splits < at_once) {
        long more = at_once / (long)p.units;
        if (more > (m_max + 127) / 128) more = (m_max + 127) / 128;
        if (more > p.n_splits) {
            p.chunk_rows = ((int)((m_max + more - 1) / more) + 63) / 64 * 64;
            p.n_splits = (m_max + p.chunk_rows - 1) / p.chunk_rows;
        }
    }
    return p;
}

// Split plan for the tensor-core multi-query kernel (one CTA per (sequence, split), every CTA
// serving all h heads).  A small cost model in units of "cache rows streamed by one SM":
// CTAs run in waves over the resident slots, every CTA pays a fixed start-up/merge cost, and
// every split adds partial results that are written once and read once by the combine pass.
Plan plan_mma(int b, int h, int m_max) {
    Plan p;
    p.units = (size_t)b * h;
    p.b = b; p.h = h;
    p.kernel = h <= 16 ? Kernel::kMma1 : Kernel::kMma2;
    const int ctas_per_sm = h <= 16 ? MmaCfg<1>::kMinBlocks : MmaCfg<2>::kMinBlocks;
    const int sms = sm_count();
    const long slots = (long)sms * ctas_per_sm;
    const double overhead_rows = 128.0;                               // start-up + merge, per CTA
    const double partial_rows = (double)h * (kHeadDim + 2) * 4 * 2 / (2.0 * kRowBytes);   // per split
    const int max_splits = m_max / 128 > 1 ? (m_max / 128 < 256 ? m_max / 128 : 256) : 1;
    double best = 0;
    for (int s = 1; s <= max_splits; ++s) {
        int chunk = (m_max + s - 1) / s;
        chunk = (chunk + kTileRows - 1) / kTileRows * kTileRows;
        const int n = (m_max + chunk - 1) / chunk;
        if (n != s) continue;                                         // same plan as a smaller s
        const long ctas = (long)b * n;
        const long waves = (ctas + slots - 1) / slots;
        double cost = (double)waves * (chunk + overhead_rows) * ctas_per_sm;
        if (n > 1) cost += (double)ctas * partial_rows / sms;
        if (p.n_splits == 0 || cost < best) {
            best = cost;
            p.n_splits = n;
            p.chunk_rows = chunk;
        }
    }
    p.cluster = p.n_splits > 1 && clusters_fit(b, p.n_splits, ctas_per_sm);
    return p;
}

// Persistent tensor-core kernel: one CTA per SM, equal shares of the line of valid tiles.
Plan plan_stream(int b, int h, int m_max) {
    Plan p;
    p.units = (size_t)b * h;
    p.b = b; p.h = h;
    p.kernel = Kernel::kUmma;
    // One CTA per SM -- or a few fewer, when that makes the grid a multiple or a divisor of the batch: with
    // sequences of equal length every share then starts at a sequence's beginning, a sequence has the fewest
    // pieces (none when CTAs take whole sequences) and the CTAs that hold them finish together.  HBM is
    // saturated from about three quarters of the SMs on (measured: same pass time with 112..148 CTAs).
    // Among the multiples of the batch, first one that makes a sequence's CTAs a thread-block cluster.
    const int sms = sm_count();
    p.grid = sms;
    bool found = false;
    for (int g = sms; g >= (3 * sms + 3) / 4 && !found; --g)
        if (b % g == 0 || (g % b == 0 && g / b <= kMaxClusterCtas)) { p.grid = g; found = true; }
    for (int g = sms; g >= (3 * sms + 3) / 4 && !found; --g)
        if (g % b == 0) { p.grid = g; found = true; }
    const long long tiles = (long long)b * (((long long)m_max + kTileRows - 1) / kTileRows);
    p.chunk_rows = (int)((tiles + p.grid - 1) / p.grid) * kTileRows;
    int parts = (p.grid + b - 1) / b + 1;
    p.n_splits = parts < p.grid ? parts : p.grid;
    // a sequence cut into a few pieces is merged by one CTA inside the kernel; many pieces (few, long
    // sequences) are better spread over all SMs by the second-pass kernel
    // ... unless the batch divides the grid into clusters: then, with sequences
    // of equal length, a cluster merges its sequence through its shared memory however many pieces that is
    p.merge_in_kernel = p.kernel == Kernel::kUmma &&
                        (p.n_splits <= kMergeInKernelMaxPieces || (p.grid % b == 0 && p.grid / b >= 2 && p.grid / b <= kMaxClusterCtas));
    return p;
}

// Fixed splits for the kernel with the query rows as tile rows (decode_wide.cuh: 33 .. 128 query rows per sequence): one
// CTA per (sequence, split), about one CTA per SM, splits of whole 128-row stages and never shorter than two of them.
Plan plan_wide(int b, int h, int m_max) {
    Plan p;
    p.units = (size_t)b * h;
    p.b = b; p.h = h;
    p.kernel = Kernel::kWide;
    const int tiles = (h + kWideRows - 1) / kWideRows;           // row tiles of 128 query rows (grid.y)
    int want = sm_count() / (b * tiles);
    const int cap = m_max / (2 * kWideRows);
    if (want > cap) want = cap;
    if (want > 160) want = 160;                    // (the second pass merges up to 160 pieces in one go)
    if (want < 1) want = 1;
    const long long chunk = (((long long)m_max + want - 1) / want + kWideRows - 1) / kWideRows * kWideRows;
    p.chunk_rows = (int)chunk;
    p.n_splits = (int)((m_max + chunk - 1) / chunk);
    return p;
}

// The plan by rules on the sizes alone; make_plan below looks for a better one where there are up to 32 query rows.
Plan plan_by_size(bool multi_query, int b, int h, int m_max) {
    // a row space too large for the 32-bit TMA coordinates goes to the general CUDA-core kernel
    if (!(multi_query && (long long)b * m_max < 0x7fffffffLL)) return plan_simt(b, h, m_max);
    // More than 32 query rows per sequence: the kernel with the query rows as tile rows, 128 rows per CTA and more as row
    // tiles over the same cache rows.  (The streaming kernel used to take up to 64 rows on a tile of its own and more as
    // groups of 64: measured against that, per step, 32 x 64 rows x 8192: 30.5 vs 35.0 us; 128 x 64 x 2048: 26.2 vs 32.8;
    // 4 x 48 x 4096: 10.8 vs 20.7; 32 x 128 x 8192: 34.9 vs 68.8; 32 x 256 x 8192: 43.6 vs 122.7; 128 x 160 x 2048: 50.1 vs
    // 103.2 -- that tile and the groups are gone.)
    if (h > 32 && (h + kWideRows - 1) / kWideRows <= 65535 && (long long)b * h < 0x7fffffffLL) return plan_wide(b, h, m_max);
    // enough tiles to give every SM a real share: the persistent kernels; otherwise fixed splits
    const long long tiles = (long long)b * (((long long)m_max + kTileRows - 1) / kTileRows);
    const int sms = sm_count();
    if (b <= kStreamMaxSeqs && tiles >= 2LL * sms && m_max >= 1024 && sms <= 256) {
        const Plan p = plan_stream(b, h, m_max);
        // few, long sequences, each cut into more pieces than one CTA merges inside the kernel: the streaming kernel would
        // need its second pass as well, and the kernel with the query rows as tile rows (fixed splits, second pass) is
        // then the quicker of the two (measured per step: 1 x 32 heads x 32768 rows 16.2 vs 18.5 us, 4 x 32 x 4096 10.5 vs
        // 14.2, 8 x 32 x 32768 29.2 vs 30.6, 8 x 16 x 8192 16.1 vs 16.4)
        if (!p.merge_in_kernel) return plan_wide(b, h, m_max);
        return p;
    }
    return h <= 32 ? plan_mma(b, h, m_max) : plan_simt(b, h, m_max);
}

size_t plan_workspace_bytes(const Plan& p);

// ---- which of the multi-query kernels, and how many splits: a model of a step's time in us, for a launch of this kernel over caches
// that are a share `full` full.  Fitted to 9600 timings (1 to 512 sequences of 256 to 32768 rows, 8, 16 and 32 heads, full caches and
// ragged ones, splits from one to as many as there are tiles, steps in a graph); it is off by 9 to 12 % (rms).
// The two kernels that share out fixed splits take rounds (of the four row-warps, 128 rows, or of a stage) after a start, several
// CTAs per SM or waves of them, and no less than the bytes; then the merge.
struct SplitModel { double start, round, second, share, tail, floor, tbs, cluster, per_cluster, crowd, pass, pass_mb; };
constexpr SplitModel kMma1Model = {2.71, 1.78, 0.24, -0.16, 0.40, 2.64, 5.03, 0.96, 0.64, 1.11, 1.74, 0.56};
constexpr SplitModel kMma2Model = {3.85, 1.21, 0.63, 0.21, 0.18, 3.83, 4.46, 0.87, 0.08, 0.80, 1.74, 0.12};
struct WideModel { double start, stage, short_stage, pass, tail, floor, tbs; };
constexpr WideModel kWide1Model = {4.35, 0.70, 0.42, 2.07, 0.24, 4.39, 6.03}, kWide2Model = {4.87, 0.65, 0.37, 2.16, 0.31, 5.01, 6.03};
// The streaming kernel: what is around its stream, where the batch makes whole clusters or shares of whole sequences of full caches,
// where it does not, and for ragged ones.
struct StreamModel { double whole, cut, ragged, tbs; };
constexpr StreamModel kStream1Model = {7.43, 10.6, 11.7, 6.59}, kStream2Model = {8.72, 12.0, 14.1, 6.67};

double either(double a, double b) { return std::sqrt(std::sqrt(a * a * a * a + b * b * b * b)); }   // the larger, and some more where they are alike

double plan_us(const Plan& p, int m_max, double full, int sms) {
    const bool few = p.h <= 16;
    const double mb = (double)p.b * m_max * full * 2 * kRowBytes * 1e-6, per_sm = (double)p.b * p.n_splits / sms;
    double us;
    if (p.kernel == Kernel::kUmma) {
        const StreamModel& m = few ? kStream1Model : kStream2Model;
        const bool whole = p.b % p.grid == 0 || (p.grid % p.b == 0 && p.grid / p.b <= kMaxClusterCtas);
        us = (full < 1 ? m.ragged : whole ? m.whole : m.cut) + mb / m.tbs;
        // clusters that do not fit at once (3 x 48 sequences, 4 x 37): 18 us where 32 x 1024 rows take 9
        if (whole && p.grid > p.b && p.grid / p.b > 2 && p.grid > sms - 16) us *= 1.6;
        return us > 4.7 ? us : 4.7;
    }
    if (p.kernel == Kernel::kWide) {
        const WideModel& m = few ? kWide1Model : kWide2Model;
        const int stages = (p.chunk_rows + kWideRows - 1) / kWideRows;
        us = m.start + stages * (m.stage + (m_max < kSingleRoundingMinRows ? m.short_stage : 0));
        if (per_sm > 1) us *= per_sm + m.tail;
        us = either(us, m.floor + mb / m.tbs) + (p.n_splits > 1 ? m.pass : 0);
    } else {
        const SplitModel& m = few ? kMma1Model : kMma2Model;
        const int occ = few ? MmaCfg<1>::kMinBlocks : MmaCfg<2>::kMinBlocks, rounds = (p.chunk_rows + 4 * kTileRows - 1) / (4 * kTileRows);
        us = m.start + m.round * (rounds - 1) + (rounds > 1 ? m.second : 0);
        us *= 1 + m.share * ((per_sm > occ ? occ : per_sm > 1 ? per_sm : 1) - 1);
        if (per_sm > occ) us *= per_sm / occ + m.tail;
        us = either(us, m.floor + mb / m.tbs);
        if (p.n_splits > 1)
            us += p.cluster ? m.cluster + m.per_cluster * p.n_splits / 16 + (per_sm > 1 ? m.crowd * (per_sm - 1) : 0)
                            : m.pass + m.pass_mb * p.b * p.n_splits * p.h * (kHeadDim + 2) * 4e-6;
    }
    // called directly, a launch and the call take the host 4.7 us, two launches 6.6
    const double host = p.n_splits > 1 && !p.cluster ? 6.6 : 4.7;
    return us > host ? us : host;
}

// A plan is kept where it is expected to be faster, for full caches and for ragged ones (half of the rows on average; what lens holds is not
// known here), than the plan by size: by 13 % in all (18 % beyond 4096 rows, where fewer timings stand behind the model), and by 15 % more
// where it takes a second launch and the other does not.
// Measured against the plans by size over the sizes above: -13 % on average; us per step 16 x 16 heads x 1024 rows 11.3 -> 5.5,
// 32 x 8 x 1024 8.9 -> 7.0, 48 x 8 x 1500 20.9 -> 10.1, 8 x 8 x 2048 8.1 -> 5.2, 64 x 8 x up to 2048 rows 18.0 -> 13.0.
constexpr long long kMaxChunkRows = 0x7fffff00;          // (a chunk, and a stage more, in an int)
constexpr double kPlanGain = 0.87, kPlanGainLong = 0.82, kPlanSecondLaunch = 0.85;

Plan make_plan(bool multi_query, int b, int h, int m_max) {
    const Plan old = plan_by_size(multi_query, b, h, m_max);
    if (!multi_query || h > 32 || old.kernel == Kernel::kSimt || b > kStreamMaxSeqs) return old;
    const int sms = sm_count();
    // (a decoding loop asks for the same few plans at every step)
    struct Entry { int sms, room, b, h, m_max; Plan plan; };
    thread_local Entry kept[32] = {};
    Entry& e = kept[((unsigned)b * 7u + (unsigned)h * 31u + (unsigned)m_max) % 32u];
    const int room = g_test_cluster_room.load(std::memory_order_relaxed);
    if (e.sms == sms && e.room == room && e.b == b && e.h == h && e.m_max == m_max) return e.plan;
    const double us_full = plan_us(old, m_max, 1.0, sms), us_ragged = plan_us(old, m_max, 0.5, sms);
    auto one_launch = [](const Plan& p) { return p.stream() ? p.merge_in_kernel : p.n_splits == 1 || p.cluster; };
    auto launches = [&](const Plan& p) { return one_launch(p) ? 1.0 : 1.0 / (kPlanSecondLaunch * kPlanSecondLaunch); };
    Plan best = old;
    const double gain = m_max <= 4096 ? kPlanGain : kPlanGainLong;
    double best_cost = us_full * us_ragged * gain * gain * launches(old);
    auto consider = [&](const Plan& p) {
        const size_t need = plan_workspace_bytes(p);
        // (what the built-in scratch held it still holds, and what took no workspace takes none)
        if (need > plan_workspace_bytes(old) && (need > MQA_NOALLOC_SCRATCH_BYTES || plan_workspace_bytes(old) == 0)) return;
        const double full = plan_us(p, m_max, 1.0, sms), ragged = plan_us(p, m_max, 0.5, sms);
        if (full > us_full || ragged > us_ragged || full * ragged * launches(p) >= best_cost) return;
        best = p;
        best_cost = full * ragged * launches(p);
    };
    // more than 16 heads stay with the streaming kernel in whole clusters from 2048 rows on (32 x 32 x 2048: 12.7 us, 12.8 in four splits; 16 x
    // 32 x 4096 13.9, 12.1 so) and otherwise from 3584 on, where the model has it too slow (24 x 22 x 4080: 14.8 us, 16.5 in four splits; 22
    // x 30 x 3876 15.1 and 16.4; 20 x 32 x 3820 14.8 and 14.2)
    const bool whole = old.stream() && old.grid % b == 0 && old.grid / b <= kMaxClusterCtas;
    const bool search = !(old.stream() && h > 16 && m_max >= (whole ? 2048 : 3584));
    Plan p;
    p.units = (size_t)b * h;
    p.b = b; p.h = h;
    // fixed splits of 128 rows and multiples of them, one round of the four row-warps per 128, that fit the SMs in one wave (2 x 21 x
    // 9909 rows: 10.2 us by size, 12.9 in 156 splits for 148 SMs).  (By the number of splits: a walk over the multiples of 128 rows takes
    // as many rounds as a cache of any length has of them, and a chunk and a rounding up do not fit an int together for the longest.)
    p.kernel = h <= 16 ? Kernel::kMma1 : Kernel::kMma2;
    const int occ = h <= 16 ? MmaCfg<1>::kMinBlocks : MmaCfg<2>::kMinBlocks;
    auto splits_of = [&](long long rows) { return (m_max + rows - 1) / rows; };
    auto chunk_of = [&](int S, int step) { return ((m_max + (long long)S - 1) / S + step - 1) / step * step; };       // of S splits, whole steps
    auto most_splits = [&](int step, long long most) { return (int)std::max(1LL, std::min(most, splits_of(step))); };
    for (int S = most_splits(4 * kTileRows, std::min(128LL, (long long)occ * sms / b)); search && S >= 1; --S) {
        const long long chunk = chunk_of(S, kTileRows);
        if (splits_of(chunk_of(S, 4 * kTileRows)) != S || splits_of(chunk) != S || chunk > kMaxChunkRows) continue;
        p.n_splits = S;
        p.chunk_rows = (int)chunk;
        p.cluster = S > 1 && m_max <= kMmaMaxCluster * 256 && clusters_fit(b, S, occ);
        consider(p);
    }
    // and of whole stages on the kernel with the query rows as tile rows, one wave of CTAs
    p.kernel = Kernel::kWide;
    p.cluster = false;
    for (int S = most_splits(kWideRows, sms / b); search && (long long)S * b <= sms && S >= 1; --S) {
        const long long chunk = chunk_of(S, kWideRows);
        if (splits_of(chunk) != S || chunk > kMaxChunkRows) continue;
        p.n_splits = S;
        p.chunk_rows = (int)chunk;
        consider(p);
    }
    // Up to three rounds in one split are quicker than in two whose clusters crowd the SMs, which the model does not tell apart: us, full
    // caches, two splits / one: 76 x 8 x 257 6.4 / 5.9, 90 x 8 x 384 7.3 / 7.0, 136 x 8 x 300 7.4 / 6.2, 50 x 24 x 300 7.6 / 7.0, 64 x 24 x
    // 384 8.0 / 7.4; 74 x 8 x 300 6.0 / 6.2, 37 x 24 x 384 6.8 / 7.4, 110 x 8 x 512 8.4 / 8.2, 64 x 24 x 512 8.7 / 8.9.
    if (best.cluster && best.n_splits == 2 && m_max <= 3 * 4 * kTileRows && 2 * b > (h <= 16 ? sms : sms / 2)) {
        best.n_splits = 1;
        best.chunk_rows = (m_max + kTileRows - 1) / kTileRows * kTileRows;
        best.cluster = false;
    }
    e = Entry{sms, room, b, h, m_max, best};
    return best;
}

// Every workspace begins with the control block of the single-launch step (kStreamCtrlBytes: see decode_umma.cuh),
// whatever the plan: a workspace that serves several shapes then keeps one epoch for all of them, and the kernels of
// the other plans never write over it.  The plan's own scratch follows.
size_t plan_workspace_bytes(const Plan& p) {
    if (p.stream()) {
        const int slots = p.grid + p.b;
        return kStreamCtrlBytes + stream_span_bytes(p.b) + stream_ml_bytes(slots, p.h) + stream_acc_bytes(slots, p.h);
    }
    if (p.n_splits <= 1) return 0;
    return kStreamCtrlBytes + partial_ml_bytes(p.units, p.n_splits) + partial_acc_bytes(p.units, p.n_splits);
}

// Fixed-split plans: (max, sum) pairs, then the accumulators, after the control block.
float2* partials_ml(const void* workspace) {
    return workspace ? reinterpret_cast<float2*>(static_cast<char*>(const_cast<void*>(workspace)) + kStreamCtrlBytes) : nullptr;
}
float* partials_acc(const Plan& p, const void* workspace) {
    return workspace ? reinterpret_cast<float*>(static_cast<char*>(const_cast<void*>(workspace)) + kStreamCtrlBytes +
                                                partial_ml_bytes(p.units, p.n_splits))
                     : nullptr;
}

struct StreamWorkspace {
    int2* span;
    float2* ml;
    float* acc;
    unsigned long long* ctrl;     // control block of the single-launch step (tcgen05 kernel)
};
StreamWorkspace stream_workspace(const Plan& p, const void* workspace) {
    char* base = static_cast<char*>(const_cast<void*>(workspace));
    const int slots = p.grid + p.b;
    StreamWorkspace w;
    w.ctrl = reinterpret_cast<unsigned long long*>(base);
    base += kStreamCtrlBytes;
    w.span = reinterpret_cast<int2*>(base);
    w.ml = reinterpret_cast<float2*>(base + stream_span_bytes(p.b));
    w.acc = reinterpret_cast<float*>(base + stream_span_bytes(p.b) + stream_ml_bytes(slots, p.h));
    return w;
}

// Launch `kernel` so that it may begin while the kernel before it in the stream is still running
// (programmatic dependent launch).  Every kernel of this library waits (griddepcontrol.wait)
// before it touches memory an earlier kernel may write, so the only effect is that launch
// latency and set-up overlap the tail of the previous kernel.
template <typename... Params, typename... Args>
cudaError_t launch_dependent_clusters(unsigned cluster, void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem,
                                      cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cluster > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

template <typename... Params, typename... Args>
cudaError_t launch_dependent_2d(void (*kernel)(Params...), unsigned grid_x, unsigned grid_y, unsigned block, size_t smem,
                                cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid_x, grid_y);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

template <typename... Params, typename... Args>
cudaError_t launch_dependent(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem,
                             cudaStream_t stream, Args... args) {
    return launch_dependent_clusters(1u, kernel, grid, block, smem, stream, args...);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
bool aligned4(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }

int check_step_args(const void* q, const void* K, const void* V, const int32_t* lens, const float* o,
                    const int32_t* status, int b, int h, int m_max, int k, int v) {
    if (!q || !K || !V || !lens || !o) return MQA_ERR_INVALID_ARG;
    if (!dims_ok(b, h, m_max) || k <= 0 || v <= 0) return MQA_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(K) || !aligned16(V) || !aligned16(o) || !aligned4(lens) ||
        !aligned4(status))
        return MQA_ERR_INVALID_ARG;
    if (k != kHeadDim || v != kHeadDim) return MQA_ERR_UNSUPPORTED;
    return MQA_OK;
}

int check_workspace(const Plan& p, const void* workspace, size_t workspace_bytes) {
    const size_t need = plan_workspace_bytes(p);
    if (need == 0) return MQA_OK;
    if (!workspace || !aligned16(workspace)) return MQA_ERR_INVALID_ARG;
    if (workspace_bytes < need) return MQA_ERR_WORKSPACE_TOO_SMALL;
    return MQA_OK;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link against libcuda).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
std::atomic<EncodeTiledFn> g_encode{nullptr};

EncodeTiledFn encode_fn() {
    EncodeTiledFn f = g_encode.load(std::memory_order_acquire);
    if (f) return f;
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess || !sym) {
        cudaGetLastError();
        return nullptr;
    }
    f = reinterpret_cast<EncodeTiledFn>(sym);
    g_encode.store(f, std::memory_order_release);
    return f;
}

// A row-major bf16 tensor [planes][rows][cols] fetched in boxes of box_planes x box_rows rows x 64 columns (128-byte swizzle).
// A decoding loop asks for the same few maps at every step (the cache, the weights) and encoding one costs about a
// microsecond of host time, so every thread keeps the maps it encoded last, by (address, shape, box): a map describes
// nothing but those, so it stays valid whatever the memory holds.
bool encode_map(CUtensorMap* map, const void* base, long long planes, long long rows, long long cols, int box_planes, int box_rows) {
    struct Entry { const void* base; long long planes, rows, cols; int box_planes, box_rows; bool used; CUtensorMap map; };
    constexpr int kEntries = 64;
    thread_local Entry kept[kEntries] = {};
    size_t hash = reinterpret_cast<size_t>(base) >> 8;
    hash = (hash ^ (hash >> 7) ^ (size_t)rows * 31u ^ (size_t)cols * 131u ^ (size_t)box_rows * 7u) % kEntries;
    Entry& e = kept[hash];
    if (e.used && e.base == base && e.planes == planes && e.rows == rows && e.cols == cols && e.box_planes == box_planes &&
        e.box_rows == box_rows) {
        *map = e.map;
        return true;
    }
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
    const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)cols * (cuuint64_t)rows * 2};
    const cuuint32_t box[3] = {(cuuint32_t)kBoxCols, (cuuint32_t)box_rows, (cuuint32_t)box_planes};
    const cuuint32_t elem[3] = {1, 1, 1};
    if (enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, planes > 0 ? 3 : 2, const_cast<void*>(base), dims, strides, box, elem,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
    e.base = base; e.planes = planes; e.rows = rows; e.cols = cols; e.box_planes = box_planes; e.box_rows = box_rows; e.map = *map; e.used = true;
    return true;
}

// A matrix [rows][cols] in boxes of box_rows rows: a 2-D map.
bool encode_matrix_map(CUtensorMap* map, const void* base, long long rows, long long cols, int box_rows) {
    return encode_map(map, base, 0, rows, cols, 0, box_rows);
}

// The cache of one tensor (K or V) as a 2-D bf16 tensor [rows = b * m_max][128 columns], fetched in
// boxes of kTileRows rows x 64 columns (128 bytes, the span of the 128-byte swizzle).
bool encode_cache_map(CUtensorMap* map, const void* base, long long rows, int box_rows = kTileRows) {
    return encode_matrix_map(map, base, rows, kHeadDim, box_rows);
}

std::atomic<int> g_smem_opt_in[kMaxDevices][24];

// The shared memory of an instance of the fixed-split kernel, and clusters beyond the portable size, asked for once per device.
template <int M_TILES, int EARLY, bool CLUSTER, bool FEW = false>
bool mma_opt_in(int dev) {
    auto kernel = mqa_decode_split_mma_kernel<M_TILES, EARLY, CLUSTER, FEW>;
    constexpr int kSlot = (((M_TILES - 1) * 3 + EARLY) * 2 + (CLUSTER ? 1 : 0)) * 2 + (FEW ? 1 : 0);
    if (g_smem_opt_in[dev][kSlot].load(std::memory_order_acquire)) return true;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MmaCfg<M_TILES>::smem_bytes(CLUSTER)) != cudaSuccess ||
        (CLUSTER && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
        cudaGetLastError();
        return false;
    }
    g_smem_opt_in[dev][kSlot].store(1, std::memory_order_release);
    return true;
}

// How many clusters of S CTAs of the fixed-split kernel the current device runs at once (asked once per device and size; any
// number on a machine without one, where the plan assumes a whole B200).
template <int M_TILES>
int clusters_of(int S) {
    static std::atomic<int> known[kMaxDevices][kMmaMaxCluster + 1];      // the answer + 1
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 0x7fffffff; }
    if (dev < 0 || dev >= kMaxDevices) return 0;
    int n = known[dev][S].load(std::memory_order_relaxed);
    if (n > 0) return n - 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)S);
    cfg.blockDim = dim3(MmaCfg<M_TILES>::kThreads);
    cfg.dynamicSmemBytes = MmaCfg<M_TILES>::smem_bytes(true);
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)S; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (!mma_opt_in<M_TILES, 0, true>(dev) || cudaOccupancyMaxActiveClusters(&n, mqa_decode_split_mma_kernel<M_TILES, 0, true>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    known[dev][S].store(n + 1, std::memory_order_relaxed);
    return n;
}
int mma_clusters_at_once(int S, int ctas_per_sm) {
    const int room = g_test_cluster_room.load(std::memory_order_relaxed);
    if (room >= 0) return room;
    return ctas_per_sm == MmaCfg<1>::kMinBlocks ? clusters_of<1>(S) : clusters_of<2>(S);
}

template <int M_TILES, int EARLY, bool CLUSTER, bool FEW>
int launch_mma_instance(const Plan& p, const void* q, const void* K, const void* V, const int32_t* lens, float* o,
               float2* part_ml, float* part_acc, int32_t* status, int b, int h, int m_max, cudaStream_t stream, int len_bias,
               const void* k_new, const void* v_new, int32_t* lens_advance,
               int mode) {
    using Cfg = MmaCfg<M_TILES>;
    auto kernel = mqa_decode_split_mma_kernel<M_TILES, EARLY, CLUSTER, FEW>;
    constexpr int kSmem = Cfg::smem_bytes(CLUSTER);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return MQA_ERR_CUDA; }
    if (!mma_opt_in<M_TILES, EARLY, CLUSTER, FEW>(dev)) return MQA_ERR_CUDA;
    alignas(64) CUtensorMap map_k, map_v, map_k_big, map_v_big;
    if (!encode_cache_map(&map_k, K, (long long)b * m_max) || !encode_cache_map(&map_v, V, (long long)b * m_max)) return MQA_ERR_CUDA;
    // four tiles per copy: never with EARLY = 1 or from chunks of under three tiles (in_groups), which then do without these two maps (a
    // microsecond each on new buffers)
    if (EARLY == 1 || p.chunk_rows <= 2 * kTileRows) {
        map_k_big = map_k;
        map_v_big = map_v;
    } else if (!encode_cache_map(&map_k_big, K, (long long)b * m_max, 4 * kTileRows) ||
               !encode_cache_map(&map_v_big, V, (long long)b * m_max, 4 * kTileRows)) {
        return MQA_ERR_CUDA;
    }
    FusedArgs fa = {};
    if (k_new) {                                       // the append-and-attend step
        fa.k_new = static_cast<const uint4*>(k_new);
        fa.v_new = static_cast<const uint4*>(v_new);
        fa.K = static_cast<uint4*>(const_cast<void*>(K));
        fa.V = static_cast<uint4*>(const_cast<void*>(V));
    }
    launch_dependent_clusters(CLUSTER ? (unsigned)p.n_splits : 1u, kernel, (unsigned)((size_t)b * p.n_splits), Cfg::kThreads, kSmem, stream, map_k, map_v,
                     map_k_big, map_v_big, static_cast<const uint32_t*>(q), lens, o, part_ml, part_acc, status, h, m_max, p.chunk_rows,
                     p.n_splits, len_bias, fa, lens_advance, mode);
    return cudaGetLastError() == cudaSuccess ? MQA_OK : MQA_ERR_CUDA;
}

template <int M_TILES, int EARLY = 0, bool CLUSTER = false>
int launch_mma(const Plan& p, const void* q, const void* K, const void* V, const int32_t* lens, float* o,
               float2* part_ml, float* part_acc, int32_t* status, int b, int h, int m_max, cudaStream_t stream, int len_bias,
               const void* k_new = nullptr, const void* v_new = nullptr, int32_t* lens_advance = nullptr,
               int mode = 0) {
    auto launch = launch_mma_instance<M_TILES, EARLY, CLUSTER, false>;
    if constexpr (M_TILES == 1) {
        if (h <= kFewHeads) launch = launch_mma_instance<M_TILES, EARLY, CLUSTER, true>;
    }
    return launch(p, q, K, V, lens, o, part_ml, part_acc, status, b, h, m_max, stream, len_bias, k_new, v_new, lens_advance, mode);
}

// Sequences per SM up to which a window of several tiles gives each sequence a CTA of the fixed-split kernel (us per step, a warp per
// sequence against that: 100 x 16 heads, window 200: 14.0 / 6.2; 290 x 8, window 64: 6.5 / 4.8; beyond two per SM it takes waves).
constexpr int kLocalTeamSeqs = 2;
constexpr int kLocalMaxWindow = 4096;         // the longest window the local step takes (a warp per sequence: decode_local.cuh)
constexpr size_t kL2KeepBytes = 64u << 20;   // K and V together: half of the 126 MB L2
constexpr int kEarlyTestWithhold = 1 << 8;    // rides on `early`: MQA_STEP_TEST_WITHHOLD_COPY
std::atomic<int> g_umma_opt_in[kMaxDevices][13];

// The streaming kernel serves up to 32 query rows per sequence (HP = 16 or 32); more go to decode_wide.cuh.
template <int HP, bool FUSED, bool GUESS = false>
int launch_umma(const Plan& p, const void* q, const void* K, const void* V, const int32_t* lens, float* o,
                void* workspace, int32_t* status, int b, int h, int m_max, cudaStream_t stream, bool merge,
                const void* k_new = nullptr, const void* v_new = nullptr, int32_t* lens_advance = nullptr,
                int early = 0) {
    using Cfg = UmmaCfg<HP>;
    auto kernel = mqa_decode_stream_umma_kernel<HP, FUSED, GUESS>;
    static_assert(HP == 16 || HP == 32, "padded head count");
    constexpr int kSlot = (HP == 16 ? 0 : 1) * 3 + (GUESS ? 2 : FUSED ? 1 : 0);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return MQA_ERR_CUDA; }
    if (!g_umma_opt_in[dev][kSlot].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmemBytes) != cudaSuccess ||
            cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
            cudaGetLastError();
            return MQA_ERR_CUDA;
        }
        g_umma_opt_in[dev][kSlot].store(1, std::memory_order_release);
    }
    FusedArgs fa = {};
    if (FUSED) {
        fa.k_new = static_cast<const uint4*>(k_new);
        fa.v_new = static_cast<const uint4*>(v_new);
        fa.K = static_cast<uint4*>(const_cast<void*>(K));
        fa.V = static_cast<uint4*>(const_cast<void*>(V));
    }
    alignas(64) CUtensorMap map_k, map_v, map_k_sub, map_v_sub, map_q;
    const long long rows = (long long)b * m_max;
    if (!encode_cache_map(&map_k, K, rows, kUmmaStageRows) || !encode_cache_map(&map_v, V, rows, kUmmaStageRows) ||
        !encode_cache_map(&map_k_sub, K, rows) || !encode_cache_map(&map_v_sub, V, rows) ||
        !encode_cache_map(&map_q, q, (long long)b * h, HP))
        return MQA_ERR_CUDA;
    const StreamWorkspace w = stream_workspace(p, workspace);
    // a cache that cannot stay in L2 from one step to the next is streamed through it with the evict-first policy
    const int read_once = ((size_t)b * m_max * 2 * kRowBytes > kL2KeepBytes ? 1 : 0) | ((early & kEarlyTestWithhold) ? 2 : 0);
    early &= ~kEarlyTestWithhold;
    // The single-launch step of a batch that divides the grid runs as clusters of grid / b CTAs (2 to 4): with sequences of equal length a cluster then holds exactly one sequence's pieces and merges
    // them through its shared memory (the kernel decides from lens; otherwise the clusters change nothing).
    unsigned cluster = 1;
    if (merge && p.grid % p.b == 0 && p.grid / p.b >= 2 && p.grid / p.b <= kMaxClusterCtas) cluster = (unsigned)(p.grid / p.b);
    launch_dependent_clusters(cluster, kernel, (unsigned)p.grid, kUmmaThreads, Cfg::kSmemBytes, stream, map_k, map_v, map_k_sub,
                              map_v_sub, map_q, lens, o, w.span, w.ml, w.acc, status, p.b, p.h, m_max, share_magic(p.grid), fa,
                              merge ? w.ctrl : nullptr, lens_advance, early, read_once);
    return cudaGetLastError() == cudaSuccess ? MQA_OK : MQA_ERR_CUDA;
}

template <bool FUSED>
int launch_umma_for(const Plan& p, const void* q, const void* K, const void* V, const int32_t* lens, float* o,
                    void* workspace, int32_t* status, int b, int h, int m_max, cudaStream_t stream, bool merge,
                    const void* k_new = nullptr, const void* v_new = nullptr, int32_t* lens_advance = nullptr,
                    int early = 0) {
#define MQA_UMMA_ARGS p, q, K, V, lens, o, workspace, status, b, h, m_max, stream, merge, k_new, v_new, lens_advance, early
    if constexpr (FUSED) {
        if ((early & ~kEarlyTestWithhold) >= 2) {           // the kernels that carry the code for copies started on a guess
            if (p.h <= 16) return launch_umma<16, true, true>(MQA_UMMA_ARGS);
            return launch_umma<32, true, true>(MQA_UMMA_ARGS);
        }
    }
    if (p.h <= 16) return launch_umma<16, FUSED>(MQA_UMMA_ARGS);
    return launch_umma<32, FUSED>(MQA_UMMA_ARGS);
#undef MQA_UMMA_ARGS
}

int launch_status() { return cudaGetLastError() == cudaSuccess ? MQA_OK : MQA_ERR_CUDA; }

template <int EARLY = 0>
int launch_wide(const Plan& p, const void* q, const void* K, const void* V, const int32_t* lens, float* o, float2* part_ml,
                float* part_acc, int32_t* status, int b, int h, int m_max, cudaStream_t stream, int len_bias,
                const void* k_new = nullptr, const void* v_new = nullptr, int32_t* lens_advance = nullptr, int mode = 0) {
    FusedArgs fa = {};
    if (k_new) {
        fa.k_new = static_cast<const uint4*>(k_new);
        fa.v_new = static_cast<const uint4*>(v_new);
        fa.K = static_cast<uint4*>(const_cast<void*>(K));
        fa.V = static_cast<uint4*>(const_cast<void*>(V));
    }
    static std::atomic<int> opt_in[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return MQA_ERR_CUDA; }
    if (!opt_in[dev].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(mqa_decode_wide_kernel<EARLY>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWideSmemBytes) != cudaSuccess) {
            cudaGetLastError();
            return MQA_ERR_CUDA;
        }
        opt_in[dev].store(1, std::memory_order_release);
    }
    alignas(64) CUtensorMap map_k, map_v;
    if (!encode_cache_map(&map_k, K, (long long)b * m_max, kWideRows) ||
        !encode_cache_map(&map_v, V, (long long)b * m_max, kWideRows))
        return MQA_ERR_CUDA;
    launch_dependent_2d(mqa_decode_wide_kernel<EARLY>, (unsigned)((size_t)b * p.n_splits), (unsigned)((h + kWideRows - 1) / kWideRows),
                        (unsigned)kWideThreads, (size_t)kWideSmemBytes, stream, static_cast<const uint4*>(q),
                     map_k, map_v, lens, o, part_ml, part_acc, status, h, m_max, p.chunk_rows, p.n_splits, len_bias, fa, lens_advance,
                     mode);
    return launch_status();
}

int run_split(bool multi_query, const void* q, const void* K, const void* V, const int32_t* lens, float* o,
              void* workspace, size_t workspace_bytes, int32_t* status,
              int b, int h, int m_max, int k, int v, cudaStream_t stream, int len_bias = 0, bool merge_in_kernel = false) {
    int rc = check_step_args(q, K, V, lens, o, status, b, h, m_max, k, v);
    if (rc) return rc;
    const Plan p = make_plan(multi_query, b, h, m_max);
    if (p.units * (size_t)p.n_splits > 0x7fffffffull) return MQA_ERR_UNSUPPORTED;
    rc = check_workspace(p, workspace, workspace_bytes);
    if (rc) return rc;
    if (p.kernel == Kernel::kUmma)
        return launch_umma_for<false>(p, q, K, V, lens, o, workspace, status, b, h, m_max, stream, merge_in_kernel);
    float2* part_ml = partials_ml(workspace);
    float* part_acc = partials_acc(p, workspace);
    if (p.kernel == Kernel::kWide) return launch_wide(p, q, K, V, lens, o, part_ml, part_acc, status, b, h, m_max, stream, len_bias);
    if (p.kernel == Kernel::kMma1 || p.kernel == Kernel::kMma2) {
        auto launch = p.kernel == Kernel::kMma1 ? (merge_in_kernel ? launch_mma<1, 0, true> : launch_mma<1, 0>)
                                                : (merge_in_kernel ? launch_mma<2, 0, true> : launch_mma<2, 0>);
        return launch(p, q, K, V, lens, o, part_ml, part_acc, status, b, h, m_max, stream, len_bias, nullptr, nullptr, nullptr, 0);
    }
    const unsigned grid = (unsigned)(p.units * (size_t)p.n_splits);
    launch_dependent(decode_split_simt_kernel, grid, kSimtThreads, 0, stream, static_cast<const uint4*>(q),
                     static_cast<const uint4*>(K), static_cast<const uint4*>(V), lens, o, part_ml, part_acc, status, h,
                     multi_query ? h : 1, m_max, p.chunk_rows, p.n_splits, len_bias);
    return launch_status();
}

// Second pass of the persistent kernel: one CTA per (schedule sequence, query row) merges the sequence's pieces.
int launch_stream_combine(const Plan& p, const void* workspace, float* o, int32_t* lens_advance, int m_max, cudaStream_t stream) {
    const StreamWorkspace w = stream_workspace(p, workspace);
    const unsigned grid = (unsigned)((size_t)p.b * p.h);
    if (p.n_splits <= kCombineEager)
        launch_dependent(stream_combine_kernel<1>, grid, kHeadDim, 0, stream, w.span, w.ml, w.acc, o, p.b, p.h, lens_advance,
                         m_max, share_magic(p.grid));
    else if (p.n_splits <= 4 * kCombineEager)
        launch_dependent(stream_combine_kernel<4>, grid, 4 * kHeadDim, 0, stream, w.span, w.ml, w.acc, o, p.b, p.h,
                         lens_advance, m_max, share_magic(p.grid));
    else
        launch_dependent(stream_combine_kernel<kCombineManyGroups>, grid, 4 * kHeadDim, 0, stream, w.span, w.ml, w.acc, o,
                         p.b, p.h, lens_advance, m_max, share_magic(p.grid));
    return launch_status();
}

int run_combine(bool multi_query, const int32_t* lens, float* o, const void* workspace, size_t workspace_bytes,
                int b, int h, int m_max, int k, int v, cudaStream_t stream, int len_bias = 0,
                int32_t* lens_advance = nullptr, bool fused = false) {
    if (!lens || !o || !dims_ok(b, h, m_max) || !aligned16(o) || !aligned4(lens)) return MQA_ERR_INVALID_ARG;
    if (k != kHeadDim || v != kHeadDim) return MQA_ERR_UNSUPPORTED;
    const Plan p = make_plan(multi_query, b, h, m_max);
    if (p.units > 0x7fffffffull) return MQA_ERR_UNSUPPORTED;
    int rc = check_workspace(p, workspace, workspace_bytes);
    if (rc) return rc;
    if (p.stream()) {
        return launch_stream_combine(p, workspace, o, lens_advance, m_max, stream);
    }
    if (p.n_splits <= 1) return MQA_OK;
    const float2* part_ml = partials_ml(workspace);
    const float* part_acc = partials_acc(p, workspace);
    // fused (the append-and-attend step of a sequence cut into fixed splits): the pass wrote a piece for every split,
    // the second pass does not look at lens and moves it on when asked to
    const int32_t* lens_read = fused ? nullptr : lens;
    if (p.n_splits <= 32) {
        // a warp per (sequence, head); with few of them each warp is a CTA of its own, so that they spread over the SMs
        auto kernel = p.n_splits <= 8 ? combine_few_kernel<8> : p.n_splits <= 16 ? combine_few_kernel<16> : combine_few_kernel<32>;
        const size_t warps = p.units > (size_t)8 * sm_count() ? kCombineFewWarps : 1;
        launch_dependent(kernel, (unsigned)((p.units + warps - 1) / warps), (unsigned)(warps * 32), 0, stream, part_ml, part_acc, lens_read, o, h,
                         m_max, p.chunk_rows, p.n_splits, len_bias, fused ? lens_advance : static_cast<int32_t*>(nullptr), p.units);
    }
    else
        launch_dependent(combine_splits_kernel<4>, (unsigned)p.units, 4 * kHeadDim, 0, stream, part_ml, part_acc, lens_read, o, h,
                         m_max, p.chunk_rows, p.n_splits, len_bias, fused ? lens_advance : static_cast<int32_t*>(nullptr));
    return launch_status();
}

int run_step(bool multi_query, const void* q, const void* K, const void* V, const int32_t* lens, float* o,
             void* workspace, size_t workspace_bytes, int32_t* status,
             int b, int h, int m_max, int k, int v, cudaStream_t stream) {
    // a single launch where the kernel merges the pieces itself
    bool one_launch = false;
    if (dims_ok(b, h, m_max)) {
        const Plan p = make_plan(multi_query, b, h, m_max);
        one_launch = p.merge_in_kernel || p.cluster;
    }
    int rc = run_split(multi_query, q, K, V, lens, o, workspace, workspace_bytes, status, b, h, m_max, k, v, stream, 0,
                       one_launch);
    if (rc || one_launch) return rc;
    return run_combine(multi_query, lens, o, workspace, workspace_bytes, b, h, m_max, k, v, stream);
}

// lens[i] += 1 for the sequences that took a row (the multi-launch form of mqa_decode_append_step
// advances lens last, after the kernels that read the old value).
__global__ void lens_advance_kernel(int32_t* lens, int b, int m_max) {
    grid_dependency_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < b && lens[i] >= 0 && lens[i] < m_max) lens[i] += 1;
}

// ---- the whole layer step: projections, append + attention, output projection ---------------------
size_t align256(size_t n) { return (n + 255) & ~(size_t)255; }

struct LayerWorkspace {
    size_t q, k_new, v_new, o, step, total;             // byte offsets
};
LayerWorkspace layer_workspace(int b, int h, int d, int m_max) {
    LayerWorkspace w;
    size_t at = 0;
    w.q = at;      at += align256((size_t)b * h * kHeadDim * 2);
    w.k_new = at;  at += align256((size_t)b * kHeadDim * 2);
    w.v_new = at;  at += align256((size_t)b * kHeadDim * 2);
    w.o = at;      at += align256((size_t)b * h * kHeadDim * 4);
    w.step = at;   at += align256(plan_workspace_bytes(make_plan(true, b, h, m_max)));
    w.total = at;
    return w;
}

// How a projection is cut up: NB batch columns per tile (16, 32, 64 or 128) and the CTAs of a cluster that share the depth of the
// product (the chunks of d rows of an input slab; the heads of an output tile).  By a model of a CTA's chain, in microseconds: its
// activations (act_kb per batch column and chunk) at 60 KB/us, step_us per chunk (an output tile's chunk is a round trip for o), 0.4
// per chunk of weights beyond those fetched ahead of the wait, and what the cluster exchanges, which is slow (SM to SM about
// 24 KB/us per CTA).  A cut whose CTAs do not fit the SMs at once, or whose clusters do not fit the GPCs (of 8: about half of the
// SMs), is charged by its number of waves, total / most_ctas + 0.5; the input projection has about half of the SMs, where the attention kernel behind it
// does not yet set itself up.  Measured, us per layer step, one fixed cut (128 columns; 16 heads' groups) against this one:
// 128 x 8 heads x 1024 18.4 / 15.4; 200 x 16 x 1536 47.6 / 28.8; 256 x 8 x 2048 38.8 / 23.4; 8 x 32 x 2048 25.6 / 19.2; 1 x 16 x 2048 23.4 / 18.3.
// A CTA takes the shared memory of as many stages as it has chunks, so where the chunks of a CTA are few, two CTAs fit an SM and the
// weights are on their way while the kernel ahead still runs.  So a cut that leaves a CTA four chunks or more is halved once more where
// a second look, fitted to all cuts of 14 layer steps, finds that 5 % better (a chunk 0.38, activations at 25 KB/us, SM to SM 23.5, and
// two thirds of the SMs, times two where two fit); and clusters of 8 that do not all fit at once become clusters of 4.  us per layer step,
// without and with both: 128 x 8 x 1024 14.7 / 13.4; 256 x 32 x 2048 39.8 / 35.6; 8 x 32 x 2048 24.4 / 21.1; 1 x 16 x 2048 17.4 / 16.4; 7 x
// 11 x 1920 13.8 / 13.4.
struct ProjectionCut { int nb, ctas; };
int projection_stages(int nb, int chunks) {
    const int most = nb == 128 ? ProjCfg<128>::kStages : nb == 64 ? ProjCfg<64>::kStages : ProjCfg<32>::kStages;
    return chunks < most ? chunks : most;
}
bool two_projections_fit(int nb, int chunks) {
    const int s = projection_stages(nb, chunks);
    const int bytes = nb == 128 ? ProjCfg<128>::smem_bytes(s) : nb == 64 ? ProjCfg<64>::smem_bytes(s) : nb == 32 ? ProjCfg<32>::smem_bytes(s) : ProjCfg<16>::smem_bytes(s);
    return 2 * (bytes + 1024 + 16) <= 228 * 1024;
}
ProjectionCut projection_cut(int b, int columns, int depth, double act_kb, double step_us, int most_ctas) {
    ProjectionCut best = {128, 1};
    double best_us = -1;
    for (int nb = 16; nb <= 128 && (nb == 16 || nb < 2 * b); nb *= 2) {
        const int batch_tiles = (b + nb - 1) / nb, rows = b < nb ? b : nb;
        const int stages = nb == 128 ? ProjCfg<128>::kStages : nb == 64 ? ProjCfg<64>::kStages : ProjCfg<32>::kStages;
        for (int ctas = 1; ctas <= kProjMaxCluster && ctas <= depth; ctas *= 2) {
            const long long total = (long long)columns * batch_tiles * ctas;
            const int each = (depth + ctas - 1) / ctas;
            const double waves = total <= (ctas == 8 ? most_ctas * 5 / 9 : most_ctas) ? 1.0 : (double)total / most_ctas + 0.5;
            const double us = waves * (3.0 + each * step_us + rows * each * act_kb / 60 + (each > stages ? (each - stages) * 0.4 : 0) +
                                       (ctas > 1 ? 0.3 + rows * 0.5 * (ctas - 1) / ctas / 24 : 0));
            if (best_us < 0 || us < best_us) { best = {nb, ctas}; best_us = us; }
        }
    }
    const int batch_tiles = (b + best.nb - 1) / best.nb, rows = b < best.nb ? b : best.nb, each = (depth + best.ctas - 1) / best.ctas;
    if (best.ctas == 8 && columns * batch_tiles > (two_projections_fit(best.nb, each) ? 28 : 14)) return {best.nb, 4};
    auto second_look = [&](int ctas) {
        const int chunks = (depth + ctas - 1) / ctas;
        const bool two = two_projections_fit(best.nb, chunks);
        const double total = (double)columns * batch_tiles * ctas, slots = sm_count() * (two ? 2 : 1) * 0.66 * (ctas < 8 ? 1 : two ? 0.65 : 0.95);
        return (total <= slots ? 1.0 : total / slots) * (3.1 + chunks * 0.38 + rows * chunks * act_kb / 24.8 + rows * 0.5 * (ctas - 1) / ctas / 23.5);
    };
    // (not five chunks of a CTA into a cluster of three and two: 240 x 4 x 640 13.3 us a layer alone, 13.7 so; and not into more clusters of
    // eight than fit: 248 x 31 x 1152 35.3 in clusters of four, 39.9 so)
    const bool uneven = best.ctas == 1 && each == 5;
    const bool too_many = best.ctas * 2 == 8 && columns * batch_tiles > (two_projections_fit(best.nb, (depth + 7) / 8) ? 28 : 14);
    if (each >= 4 && !uneven && !too_many && best.ctas * 2 <= kProjMaxCluster && second_look(best.ctas * 2) < 0.95 * second_look(best.ctas)) best.ctas *= 2;
    return best;
}

ProjectionCut input_cut(int b, int h, int d) { return projection_cut(b, h + 2, d / 128, 0.25, 0.2, sm_count() * 5 / 9); }       // bf16 x
ProjectionCut output_cut(int b, int h, int d) { return projection_cut(b, d / 128, h, 0.5, 0.45, sm_count() * 8 / 9); }           // fp32 o

std::atomic<int> g_proj_opt_in[kMaxDevices][8];

template <int NB>
int launch_projections_in(const void* x, const void* P_q, const void* P_k, const void* P_v, void* q, void* k_new, void* v_new,
                          int32_t* status, int b, int h, int d, int parts, cudaStream_t stream) {
    using Cfg = ProjCfg<NB>;
    auto kernel = project_in_kernel<NB>;
    constexpr int kSlot = NB == 16 ? 0 : (NB == 32 ? 1 : (NB == 64 ? 2 : 3));
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return MQA_ERR_CUDA; }
    if (!g_proj_opt_in[dev][kSlot].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmemBytes) != cudaSuccess) {
            cudaGetLastError();
            return MQA_ERR_CUDA;
        }
        g_proj_opt_in[dev][kSlot].store(1, std::memory_order_release);
    }
    alignas(64) CUtensorMap map_pq, map_pk, map_pv, map_x;
    if (!encode_matrix_map(&map_pq, P_q, (long long)h * d, kHeadDim, 128) || !encode_matrix_map(&map_pk, P_k, d, kHeadDim, 128) ||
        !encode_matrix_map(&map_pv, P_v, d, kHeadDim, 128) || !encode_matrix_map(&map_x, x, b, d, NB))
        return MQA_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(h + 2), (unsigned)parts, (unsigned)((b + NB - 1) / NB));
    cfg.blockDim = dim3(kProjThreads);
    const int stages = projection_stages(NB, (d / 128 + parts - 1) / parts);
    cfg.dynamicSmemBytes = Cfg::smem_bytes(stages);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = (unsigned)parts;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = parts > 1 ? 2 : 1;
    cudaLaunchKernelEx(&cfg, kernel, map_pq, map_pk, map_pv, map_x, static_cast<__nv_bfloat16*>(q),
                       static_cast<__nv_bfloat16*>(k_new), static_cast<__nv_bfloat16*>(v_new), status, b, h, d, stages);
    return launch_status();
}

// The output projection: the head groups of a (d tile, batch tile) are the CTAs of one thread-block cluster (see
// project_out_kernel), each with ceil(h / ctas) heads.
template <int NB>
int launch_projection_out(const void* P_o, const float* o, float* y, int32_t* status, int b, int h, int d, int ctas, cudaStream_t stream) {
    using Cfg = ProjCfg<NB>;
    auto kernel = project_out_kernel<NB>;
    constexpr int kSlot = 4 + (NB == 16 ? 0 : (NB == 32 ? 1 : (NB == 64 ? 2 : 3)));
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return MQA_ERR_CUDA; }
    if (!g_proj_opt_in[dev][kSlot].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmemBytes) != cudaSuccess) {
            cudaGetLastError();
            return MQA_ERR_CUDA;
        }
        g_proj_opt_in[dev][kSlot].store(1, std::memory_order_release);
    }
    alignas(64) CUtensorMap map_po;
    if (!encode_matrix_map(&map_po, P_o, (long long)h * d, kHeadDim, 128)) return MQA_ERR_CUDA;
    const int heads_per_cta = (h + ctas - 1) / ctas;
    const int groups = (h + heads_per_cta - 1) / heads_per_cta;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(d / 128), (unsigned)groups, (unsigned)((b + NB - 1) / NB));
    cfg.blockDim = dim3(kProjThreads);
    const int stages = projection_stages(NB, heads_per_cta);
    cfg.dynamicSmemBytes = Cfg::smem_bytes(stages);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = (unsigned)groups;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaLaunchKernelEx(&cfg, kernel, map_po, o, y, status, b, h, d, heads_per_cta, stages);
    return launch_status();
}

}  // namespace
}  // namespace mqa

using namespace mqa;

extern "C" {
#ifdef MQA_DEBUG_TS
void mqa_debug_ts(unsigned long long* t) { cudaMemcpyFromSymbol(t, mqa::g_ts, sizeof(mqa::g_ts)); }
void mqa_debug_st(unsigned long long* t) { cudaMemcpyFromSymbol(t, mqa::g_st, sizeof(mqa::g_st)); }
#endif

int kv_cache_append(void* K, void* V, const void* k_new, const void* v_new, int32_t* lens, int advance,
                    int32_t* status, int b, int kv_heads, int m_max, int k, int v, mqa_stream_t stream) {
    if (!K || !V || !k_new || !v_new || !lens) return MQA_ERR_INVALID_ARG;
    if (b <= 0 || kv_heads <= 0 || m_max <= 0 || k <= 0 || v <= 0) return MQA_ERR_INVALID_ARG;
    if (!aligned16(K) || !aligned16(V) || !aligned16(k_new) || !aligned16(v_new) || !aligned4(lens) ||
        !aligned4(status))
        return MQA_ERR_INVALID_ARG;
    if (k != kHeadDim || v != kHeadDim) return MQA_ERR_UNSUPPORTED;
    launch_dependent(kv_cache_append_kernel, (unsigned)b, kAppendThreads, 0, static_cast<cudaStream_t>(stream),
                     static_cast<uint4*>(K), static_cast<uint4*>(V), static_cast<const uint4*>(k_new),
                     static_cast<const uint4*>(v_new), lens, advance, status, kv_heads, m_max);
    return launch_status();
}

int mqa_decode_step(const void* q, const void* K, const void* V, const int32_t* lens, float* o, void* workspace,
                    size_t workspace_bytes, int32_t* status, int b, int h, int m_max, int k, int v,
                    mqa_stream_t stream) {
    return run_step(true, q, K, V, lens, o, workspace, workspace_bytes, status, b, h, m_max, k, v,
                    static_cast<cudaStream_t>(stream));
}

int mha_decode_step(const void* q, const void* K, const void* V, const int32_t* lens, float* o, void* workspace,
                    size_t workspace_bytes, int32_t* status, int b, int h, int m_max, int k, int v,
                    mqa_stream_t stream) {
    return run_step(false, q, K, V, lens, o, workspace, workspace_bytes, status, b, h, m_max, k, v,
                    static_cast<cudaStream_t>(stream));
}

int mqa_decode_step_split(const void* q, const void* K, const void* V, const int32_t* lens, float* o,
                          void* workspace, size_t workspace_bytes, int32_t* status, int b, int h, int m_max,
                          int k, int v, mqa_stream_t stream) {
    return run_split(true, q, K, V, lens, o, workspace, workspace_bytes, status, b, h, m_max, k, v,
                     static_cast<cudaStream_t>(stream));
}

int mqa_decode_step_combine(const int32_t* lens, float* o, const void* workspace, size_t workspace_bytes, int b,
                            int h, int m_max, int k, int v, mqa_stream_t stream) {
    return run_combine(true, lens, o, workspace, workspace_bytes, b, h, m_max, k, v,
                       static_cast<cudaStream_t>(stream));
}

int mha_decode_step_split(const void* q, const void* K, const void* V, const int32_t* lens, float* o,
                          void* workspace, size_t workspace_bytes, int32_t* status, int b, int h, int m_max,
                          int k, int v, mqa_stream_t stream) {
    return run_split(false, q, K, V, lens, o, workspace, workspace_bytes, status, b, h, m_max, k, v,
                     static_cast<cudaStream_t>(stream));
}

int mha_decode_step_combine(const int32_t* lens, float* o, const void* workspace, size_t workspace_bytes, int b,
                            int h, int m_max, int k, int v, mqa_stream_t stream) {
    return run_combine(false, lens, o, workspace, workspace_bytes, b, h, m_max, k, v,
                       static_cast<cudaStream_t>(stream));
}

// early: what the persistent kernel may do before it waits for the kernel before it (see early in
// mqa_decode_stream_umma_kernel): kEarlyAfterProjection inside the layer step, kEarlyChained when the caller set
// MQA_STEP_CHAINED.  flags: MQA_STEP_ADVANCE | MQA_STEP_CHAINED.
constexpr int kEarlyNone = 0, kEarlyAfterProjection = 1, kEarlyChained = 2, kEarlyChainedWrongGuess = 3;
constexpr int kGuessMaxPieces = 6, kGuessMinShareRows = 8 * kUmmaStageRows;
// Every check of mqa_decode_append_step that needs no launch: flags, pointers, sizes, the plan, the workspace.
static int check_append_step(const void* q, const void* K, const void* V, const void* k_new, const void* v_new,
                             const int32_t* lens, int flags, const float* o, const void* workspace, size_t workspace_bytes,
                             const int32_t* status, int b, int h, int m_max, int k, int v, Plan* plan) {
    if (flags & ~(MQA_STEP_ADVANCE | MQA_STEP_CHAINED | MQA_STEP_TEST_WRONG_GUESS | MQA_STEP_TEST_WITHHOLD_COPY)) return MQA_ERR_INVALID_ARG;
    int rc = check_step_args(q, K, V, lens, o, status, b, h, m_max, k, v);
    if (rc) return rc;
    if (!k_new || !v_new || !aligned16(k_new) || !aligned16(v_new)) return MQA_ERR_INVALID_ARG;
    *plan = make_plan(true, b, h, m_max);
    if (plan->units * (size_t)plan->n_splits > 0x7fffffffull) return MQA_ERR_UNSUPPORTED;
    return check_workspace(*plan, workspace, workspace_bytes);
}

static int append_step_impl(const void* q, void* K, void* V, const void* k_new, const void* v_new, int32_t* lens,
                            int flags, float* o, void* workspace, size_t workspace_bytes, int32_t* status, int b,
                            int h, int m_max, int k, int v, mqa_stream_t stream_, bool after_projection,
                            const Plan* checked = nullptr) {
    // (checked: the caller has run check_append_step on these very arguments and passes the plan it gave)
    Plan p;
    int rc = MQA_OK;
    if (checked) p = *checked;
    else if ((rc = check_append_step(q, K, V, k_new, v_new, lens, flags, o, workspace, workspace_bytes, status, b, h, m_max, k, v, &p))) return rc;
    const int advance = flags & MQA_STEP_ADVANCE;
    int early = after_projection ? kEarlyAfterProjection
                : !(flags & MQA_STEP_CHAINED) ? kEarlyNone
                : (flags & MQA_STEP_TEST_WRONG_GUESS) ? kEarlyChainedWrongGuess : kEarlyChained;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const bool withhold = (flags & MQA_STEP_TEST_WITHHOLD_COPY) != 0;
    if (p.kernel == Kernel::kUmma) {
        // copies started on a guess pay where the step is one launch over long shares (measured: 0.4-0.7 us gained with
        // up to 6 pieces per sequence, 0.3-2.5 us lost with more pieces, short shares or a second-pass kernel)
        if (early == kEarlyChained && !(p.merge_in_kernel && p.n_splits <= kGuessMaxPieces && p.chunk_rows >= kGuessMinShareRows))
            early = kEarlyNone;
        if (withhold) early |= kEarlyTestWithhold;
        // one launch: append inside the pass, pieces merged by the last CTA to deliver one, lens advanced at the end
        if (p.merge_in_kernel)
            return launch_umma_for<true>(p, q, K, V, lens, o, workspace, status, b, h, m_max, stream, true, k_new, v_new,
                                         advance ? lens : nullptr, early);
        rc = launch_umma_for<true>(p, q, K, V, lens, o, workspace, status, b, h, m_max, stream, false, k_new, v_new, nullptr,
                                   early);
        if (rc) return rc;
        return run_combine(true, lens, o, workspace, workspace_bytes, b, h, m_max, k, v, stream, 0, advance ? lens : nullptr);
    }
    // what the fixed-split and the many-rows kernel fetch ahead of the wait (their EARLY), and the testing flags
    const int ahead = early >= kEarlyChained ? 1 : early == kEarlyAfterProjection ? 2 : 0;
    const int mode = (withhold ? kMmaWithhold : 0) | (early == kEarlyChainedWrongGuess ? kMmaWrongGuess : 0);
    // other plans: the same step as separate launches.  Without `advance` the append leaves lens alone and
    // the step is told that a sequence which took a row has one more row than lens says.
    if (p.kernel == Kernel::kWide) {
        // many query rows: the CTA whose rows hold the new one writes it; one split per sequence moves lens on itself,
        // otherwise the second pass does.  One or two launches.
        float2* part_ml = partials_ml(workspace);
        float* part_acc = partials_acc(p, workspace);
        // (one split and one tile of 128 rows: the CTA moves lens on itself)
        const bool alone = p.n_splits == 1 && h <= kWideRows;
        auto launch = ahead == 1 ? launch_wide<1> : ahead == 2 ? launch_wide<2> : launch_wide<0>;
        rc = launch(p, q, K, V, lens, o, part_ml, part_acc, status, b, h, m_max, stream, 0, k_new, v_new,
                    alone && advance ? lens : nullptr, mode);
        if (rc || alone) return rc;
        if (p.n_splits == 1) {                                   // several row tiles read lens: moved on by a kernel of its own
            if (advance) launch_dependent(lens_advance_kernel, (unsigned)((b + 255) / 256), 256u, 0, stream, lens, b, m_max);
            return launch_status();
        }
        return run_combine(true, lens, o, workspace, workspace_bytes, b, h, m_max, k, v, stream, 0, advance ? lens : nullptr, true);
    }
    if (p.kernel == Kernel::kMma1 || p.kernel == Kernel::kMma2) {
        // one CTA per sequence writes the row, attends and moves lens on, all in one launch; of several splits the CTA whose
        // rows hold the new one writes it and the second pass moves lens on.  What is fetched ahead of the wait: EARLY in
        // decode_mma.cuh.
        const bool alone = p.n_splits == 1 || p.cluster;
        float2* part_ml = alone ? nullptr : partials_ml(workspace);
        float* part_acc = alone ? nullptr : partials_acc(p, workspace);
        int32_t* move_lens = alone && advance ? lens : nullptr;
#define MQA_MMA_STEP(TILES, EARLY) \
    (p.cluster ? launch_mma<TILES, EARLY, true> : launch_mma<TILES, EARLY>)(p, q, K, V, lens, o, part_ml, part_acc, status, b, h, m_max, stream, 0, \
                                                                             k_new, v_new, move_lens, mode)
        if (p.kernel == Kernel::kMma1)
            rc = ahead == 1 ? MQA_MMA_STEP(1, 1) : ahead == 2 ? MQA_MMA_STEP(1, 2) : MQA_MMA_STEP(1, 0);
        else
            rc = ahead == 1 ? MQA_MMA_STEP(2, 1) : ahead == 2 ? MQA_MMA_STEP(2, 2) : MQA_MMA_STEP(2, 0);
#undef MQA_MMA_STEP
        if (rc || alone) return rc;
        return run_combine(true, lens, o, workspace, workspace_bytes, b, h, m_max, k, v, stream, 0, advance ? lens : nullptr, true);
    }
    rc = kv_cache_append(K, V, k_new, v_new, lens, 0, status, b, 1, m_max, k, v, stream_);
    if (rc) return rc;
    rc = run_split(true, q, K, V, lens, o, workspace, workspace_bytes, status, b, h, m_max, k, v, stream, 1);
    if (rc) return rc;
    rc = run_combine(true, lens, o, workspace, workspace_bytes, b, h, m_max, k, v, stream, 1);
    if (rc) return rc;
    if (advance) {
        launch_dependent(lens_advance_kernel, (unsigned)((b + 255) / 256), 256u, 0, stream, lens, b, m_max);
        return launch_status();
    }
    return MQA_OK;
}

int mqa_decode_append_step(const void* q, void* K, void* V, const void* k_new, const void* v_new, int32_t* lens,
                           int advance, float* o, void* workspace, size_t workspace_bytes, int32_t* status, int b,
                           int h, int m_max, int k, int v, mqa_stream_t stream) {
    return append_step_impl(q, K, V, k_new, v_new, lens, advance, o, workspace, workspace_bytes, status, b, h, m_max, k, v,
                            stream, false);
}

int mqa_decode_local_step(const void* q, void* K, void* V, const void* k_new, const void* v_new, int32_t* pos, int advance,
                          float* o, int32_t* status, int b, int h, int window, int k, int v, mqa_stream_t stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int rc = check_step_args(q, K, V, pos, o, status, b, h, window, k, v);
    if (rc) return rc;
    if (!k_new || !v_new || !aligned16(k_new) || !aligned16(v_new)) return MQA_ERR_INVALID_ARG;
    if ((long long)b * window >= 0x7fffffffLL) return MQA_ERR_UNSUPPORTED;
    if (window > kLocalMaxWindow) return MQA_ERR_UNSUPPORTED;   // a window that long is the ordinary step's business
    const int sms = sm_count();
    if (window > kTileRows && h <= 32 && b <= kLocalTeamSeqs * sms) {
        // few sequences, several tiles each: four warps to a sequence (and two head tiles side by side)
        Plan p;
        p.units = (size_t)b * h;
        p.b = b; p.h = h;
        p.n_splits = 1;
        p.chunk_rows = (window + kTileRows - 1) / kTileRows * kTileRows;
        auto launch = h <= 16 ? launch_mma<1, 0> : launch_mma<2, 0>;
        return launch(p, q, K, V, pos, o, nullptr, nullptr, status, b, h, window, stream, 0, k_new, v_new, advance ? pos : nullptr, kMmaRing);
    }
    // a warp per sequence: windows of a few tiles, any number of heads; and of one tile (the paper's) with up to 16
    static std::atomic<int> opted[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return MQA_ERR_CUDA; }
    if (!opted[dev].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(mqa_decode_local_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, local_smem_bytes(kLocalMaxWarps)) != cudaSuccess ||
            cudaFuncSetAttribute(mqa_decode_local_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, local_tile_smem_bytes(kLocalMaxWarps)) != cudaSuccess) {
            cudaGetLastError();
            return MQA_ERR_CUDA;
        }
        opted[dev].store(1, std::memory_order_release);
    }
    alignas(64) CUtensorMap map_k, map_v;
    if (!encode_cache_map(&map_k, K, (long long)b * window) || !encode_cache_map(&map_v, V, (long long)b * window)) return MQA_ERR_CUDA;
    const bool tile = window <= kTileRows && h <= 16;
    const int each = (b + sms - 1) / sms, warps = each < kLocalMaxWarps ? each : kLocalMaxWarps;
    launch_dependent(tile ? mqa_decode_local_tile_kernel : mqa_decode_local_kernel, (unsigned)((b + warps - 1) / warps), (unsigned)(warps * 32),
                     (size_t)(tile ? local_tile_smem_bytes(warps) : local_smem_bytes(warps)), stream, map_k, map_v, static_cast<const uint4*>(q),
                     static_cast<const uint4*>(k_new), static_cast<const uint4*>(v_new), static_cast<uint4*>(K), static_cast<uint4*>(V), pos, o, status,
                     b, h, window, advance ? 1 : 0);
    return launch_status();
}

size_t mqa_host_staging_bytes(int b, int h, int k, int v) {
    if (b <= 0 || h <= 0 || k != kHeadDim || v != kHeadDim) return 0;
    return align256((size_t)b * h * k * 2) + 2 * align256((size_t)b * kHeadDim * 2) + align256((size_t)b * h * v * 4);
}

// The device's address of pinned host memory that it can reach (16-byte aligned), or null.
static const void* host_device_pointer(const void* host) {
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, host) == cudaSuccess && attr.type == cudaMemoryTypeHost && attr.devicePointer &&
        aligned16(attr.devicePointer))
        return attr.devicePointer;
    cudaGetLastError();
    return nullptr;
}

int mqa_decode_append_step_host(const void* q_host, const void* k_new_host, const void* v_new_host, float* o_host,
                                void* K, void* V, int32_t* lens, int advance, void* staging, size_t staging_bytes,
                                void* workspace, size_t workspace_bytes, int32_t* status, int b, int h, int m_max, int k,
                                int v, mqa_stream_t stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!q_host || !k_new_host || !v_new_host || !o_host || !staging) return MQA_ERR_INVALID_ARG;
    if (!dims_ok(b, h, m_max) || k <= 0 || v <= 0 || !aligned16(staging)) return MQA_ERR_INVALID_ARG;
    if (k != kHeadDim || v != kHeadDim) return MQA_ERR_UNSUPPORTED;
    if (staging_bytes < mqa_host_staging_bytes(b, h, k, v)) return MQA_ERR_WORKSPACE_TOO_SMALL;
    const size_t q_bytes = (size_t)b * h * k * 2, row_bytes = (size_t)b * kHeadDim * 2, o_bytes = (size_t)b * h * v * 4;
    char* base = static_cast<char*>(staging);
    char* q_dev = base;
    char* k_dev = q_dev + align256(q_bytes);
    char* v_dev = k_dev + align256(row_bytes);
    float* o_dev = reinterpret_cast<float*>(v_dev + align256(row_bytes));
    // everything that can be refused is refused before the first copy is enqueued
    Plan plan;
    const int bad = check_append_step(q_dev, K, V, k_dev, v_dev, lens, advance, o_dev, workspace, workspace_bytes, status, b, h,
                                      m_max, k, v, &plan);
    if (bad) return bad;
    // the step's inputs.  Pinned memory that this device can address: a kernel fetches them, and the attention kernel
    // sets itself up and asks for its first stages while it does (what the layer step does behind its input projection).
    // Otherwise copy-engine transfers: one when the caller packed them back to back (256-byte aligned parts), else three.
    const char* qh = static_cast<const char*>(q_host);
    const void* q_map = host_device_pointer(q_host);
    const void* k_map = host_device_pointer(k_new_host);
    const void* v_map = host_device_pointer(v_new_host);
    const bool by_kernel = q_map && k_map && v_map && q_bytes / 16 <= 0xffffffffull;
    if (by_kernel) {
        const StageInPart pq = {static_cast<const uint4*>(q_map), reinterpret_cast<uint4*>(q_dev), (unsigned)(q_bytes / 16)};
        const StageInPart pk = {static_cast<const uint4*>(k_map), reinterpret_cast<uint4*>(k_dev), (unsigned)(row_bytes / 16)};
        const StageInPart pv = {static_cast<const uint4*>(v_map), reinterpret_cast<uint4*>(v_dev), (unsigned)(row_bytes / 16)};
        const size_t turns = (q_bytes / 16 + kStageInThreads - 1) / kStageInThreads;
        const unsigned grid = (unsigned)(turns < (size_t)(2 * sm_count()) ? (turns ? turns : 1) : 2 * sm_count());
        if (launch_dependent(stage_in_kernel, grid, (unsigned)kStageInThreads, 0, stream, pq, pk, pv) != cudaSuccess) {
            cudaGetLastError();
            return MQA_ERR_CUDA;
        }
    } else {
        const bool packed = static_cast<const char*>(k_new_host) == qh + align256(q_bytes) &&
                            static_cast<const char*>(v_new_host) == qh + align256(q_bytes) + align256(row_bytes);
        if (packed) {
            if (cudaMemcpyAsync(q_dev, qh, align256(q_bytes) + align256(row_bytes) + row_bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess) {
                cudaGetLastError();
                return MQA_ERR_CUDA;
            }
        } else {
            if (cudaMemcpyAsync(q_dev, q_host, q_bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
                cudaMemcpyAsync(k_dev, k_new_host, row_bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
                cudaMemcpyAsync(v_dev, v_new_host, row_bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess) {
                cudaGetLastError();
                return MQA_ERR_CUDA;
            }
        }
    }
    // the result: where o_host is pinned memory that this device can address, the kernels store o there themselves
    // (posted writes that overlap the end of the step); otherwise it goes through the staging buffer and a copy
    float* o_direct = static_cast<float*>(const_cast<void*>(host_device_pointer(o_host)));
    const int rc = append_step_impl(q_dev, K, V, k_dev, v_dev, lens, advance, o_direct ? o_direct : o_dev, workspace,
                                    workspace_bytes, status, b, h, m_max, k, v, stream_, by_kernel, &plan);
    if (rc || o_direct) return rc;
    if (cudaMemcpyAsync(o_host, o_dev, o_bytes, cudaMemcpyDeviceToHost, stream) != cudaSuccess) {
        cudaGetLastError();
        return MQA_ERR_CUDA;
    }
    return MQA_OK;
}

size_t mqa_layer_workspace_bytes(int b, int h, int d, int m_max, int k, int v) {
    if (!dims_ok(b, h, m_max) || d <= 0 || d % 128 != 0 || k != kHeadDim || v != kHeadDim) return 0;
    return layer_workspace(b, h, d, m_max).total;
}

int mqa_layer_cut(int b, int h, int d, int cut[4]) {
    if (!cut || !dims_ok(b, h, 1) || d <= 0 || d % 128 != 0) return MQA_ERR_INVALID_ARG;
    const ProjectionCut in = input_cut(b, h, d), out = output_cut(b, h, d);
    cut[0] = in.nb; cut[1] = in.ctas; cut[2] = out.nb; cut[3] = out.ctas;
    return MQA_OK;
}

int mqa_layer_decode_step(const void* x, const void* P_q, const void* P_k, const void* P_v, const void* P_o, void* K, void* V,
                          int32_t* lens, int advance, float* y, void* workspace, size_t workspace_bytes, int32_t* status,
                          int b, int h, int d, int m_max, int k, int v, mqa_stream_t stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!x || !P_q || !P_k || !P_v || !P_o || !K || !V || !lens || !y || !workspace) return MQA_ERR_INVALID_ARG;
    if (!dims_ok(b, h, m_max) || d <= 0 || k <= 0 || v <= 0) return MQA_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(P_q) || !aligned16(P_k) || !aligned16(P_v) || !aligned16(P_o) || !aligned16(K) ||
        !aligned16(V) || !aligned16(y) || !aligned16(workspace) || !aligned4(lens) || !aligned4(status))
        return MQA_ERR_INVALID_ARG;
    if (k != kHeadDim || v != kHeadDim || d % 128 != 0 || (long long)h * d >= 0x7fffffffLL) return MQA_ERR_UNSUPPORTED;
    const LayerWorkspace w = layer_workspace(b, h, d, m_max);
    if (workspace_bytes < w.total) return MQA_ERR_WORKSPACE_TOO_SMALL;
    char* base = static_cast<char*>(workspace);
    void* q = base + w.q;
    void* k_new = base + w.k_new;
    void* v_new = base + w.v_new;
    float* o = reinterpret_cast<float*>(base + w.o);
    const ProjectionCut in = input_cut(b, h, d), out = output_cut(b, h, d);
    int rc;
    switch (in.nb) {
        case 16: rc = launch_projections_in<16>(x, P_q, P_k, P_v, q, k_new, v_new, status, b, h, d, in.ctas, stream); break;
        case 32: rc = launch_projections_in<32>(x, P_q, P_k, P_v, q, k_new, v_new, status, b, h, d, in.ctas, stream); break;
        case 64: rc = launch_projections_in<64>(x, P_q, P_k, P_v, q, k_new, v_new, status, b, h, d, in.ctas, stream); break;
        default: rc = launch_projections_in<128>(x, P_q, P_k, P_v, q, k_new, v_new, status, b, h, d, in.ctas, stream); break;
    }
    if (rc) return rc;
    rc = append_step_impl(q, K, V, k_new, v_new, lens, advance ? MQA_STEP_ADVANCE : 0, o, base + w.step, w.total - w.step, status,
                          b, h, m_max, k, v, stream_, true);
    if (rc) return rc;
    switch (out.nb) {
        case 16: return launch_projection_out<16>(P_o, o, y, status, b, h, d, out.ctas, stream);
        case 32: return launch_projection_out<32>(P_o, o, y, status, b, h, d, out.ctas, stream);
        case 64: return launch_projection_out<64>(P_o, o, y, status, b, h, d, out.ctas, stream);
        default: return launch_projection_out<128>(P_o, o, y, status, b, h, d, out.ctas, stream);
    }
}

size_t mqa_workspace_bytes(int b, int h, int m_max, int k, int v) {
    if (!dims_ok(b, h, m_max) || k != kHeadDim || v != kHeadDim) return 0;
    const size_t a = plan_workspace_bytes(make_plan(true, b, h, m_max));
    const size_t c = plan_workspace_bytes(make_plan(false, b, h, m_max));
    return a > c ? a : c;
}

size_t mqa_workspace_bytes_up_to(int b, int h, int m_max, int k, int v) {
    size_t most = 0;
    // (a microsecond per batch size; caches of under 256 rows are never cut)
    for (int i = m_max < 256 ? b : 1; i <= b && i > 0; ++i) most = std::max(most, mqa_workspace_bytes(i, h, m_max, k, v));
    return most;
}

int mqa_append_step_launches(int b, int h, int m_max, int k, int v) {
    if (!dims_ok(b, h, m_max) || k != kHeadDim || v != kHeadDim) return 0;
    const Plan p = make_plan(true, b, h, m_max);
    if (p.merge_in_kernel) return 1;                   // append, pass, merge and lens advance in one kernel
    if ((p.kernel == Kernel::kMma1 || p.kernel == Kernel::kMma2) && (p.n_splits == 1 || p.cluster)) return 1;   // one CTA or cluster per sequence does it all
    if (p.stream()) return 2;                          // pass with the append inside, second pass
    if (p.kernel == Kernel::kMma1 || p.kernel == Kernel::kMma2) return 2;   // fixed splits: the same two
    if (p.kernel == Kernel::kWide) return p.n_splits == 1 && h <= kWideRows ? 1 : 2;
    return 2 + (p.n_splits > 1 ? 1 : 0) + 1;           // append, pass, (second pass), lens advance
}

int mqa_plan_splits(int multi_query, int b, int h, int m_max, int k, int v, int* chunk_rows) {
    if (!dims_ok(b, h, m_max) || k != kHeadDim || v != kHeadDim) return 0;
    const Plan p = make_plan(multi_query != 0, b, h, m_max);
    if (chunk_rows) *chunk_rows = p.chunk_rows;
    return p.n_splits;
}

// ---- the batched form (prefill) ---------------------------------------------------------------------------------
static int check_prefill_dims(int b, int h, int n, int m_max, int k, int v) {
    if (!dims_ok(b, h, m_max) || n <= 0 || k <= 0 || v <= 0) return MQA_ERR_INVALID_ARG;
    if (k != kHeadDim || v != kHeadDim || n > m_max) return MQA_ERR_UNSUPPORTED;
    const long long ctas = (long long)((n + kPfRows - 1) / kPfRows) * b * ((h + 1) / 2);
    if ((long long)b * m_max >= 0x7fffffffLL || (long long)b * h * n >= 0x7fffffffLL - kPfRows || ctas >= 0x7fffffffLL) return MQA_ERR_UNSUPPORTED;
    return MQA_OK;
}

// The tiles of a sequence: of all heads x positions with at most 128 rows the one with the fewest tiles (rows past the last
// position or head are work for nothing: with 128 positions of one head per tile, 16 positions of 32 heads would fill an eighth of
// their rows); among equals the most positions, whose tiles share their last stages.
static PfShape prefill_shape(int b, int h, int n, int m_max) {
    PfShape sh = {};
    sh.b = b; sh.h = h; sh.n = n; sh.m_max = m_max;
    for (int heads = 1; heads <= kPfRows && heads <= h; ++heads) {
        const int positions = kPfRows / heads < n ? kPfRows / heads : n;
        const int head_blocks = (h + heads - 1) / heads;
        const int tiles = (n + positions - 1) / positions * head_blocks;     // (at most 2 h n / 128 + h: checked with the sizes)
        if (heads == 1 || tiles < sh.n_tiles) {
            sh.positions = positions; sh.heads = heads; sh.head_blocks = head_blocks; sh.n_tiles = tiles;
        }
        if ((long long)sh.n_tiles * kPfRows < (long long)h * n + kPfRows) break;      // no shape has fewer
    }
    return sh;
}
// The units of work: two tiles each, or one (mqa_prefill_tile_kernel).
static void prefill_units(PfShape& sh, int tiles) {
    sh.n_units = (sh.n_tiles + tiles - 1) / tiles;
    sh.group = sh.head_blocks / tiles > 1 ? sh.head_blocks / tiles : 1;
    sh.n_items = (sh.n_units + sh.group - 1) / sh.group * sh.group * sh.b;
}

// Which kernel, by a model of the time in us: 0 for two tiles to a CTA (persistent, one CTA per SM), else the CTAs of a cluster that share
// one tile's stages.  Measured, us for two tiles / one tile by 1 / 2 / 4 / 8 CTAs: 120 tiles of up to 24 stages 37.8 / 25.6 / 35.7 (they do not
// fit at once); 64 of 32: 51.1 / 32.3 / 23.6 / 29.9; 10 of 12: 21.6 / 16.5 / 15.6 / 13.6 / 12.3; 1 of 16: 19.5 / 16.6 / 14.1 / 11.5 / 10.4; 240 of 3:
// 14.2 / 20.2; 256 of 16: 28.2 / 35.6; 15 of 15: 26.0 / 18.5 / 16.6 / 14.0 / 12.4.  (With two tiles to a unit throughout and clusters sharing
// units: 120 of 24 28.5, 128 of 8 22.0.)  An odd number of tiles leaves the longest alone in its unit, and quicker there than a pair (20 x 1 x
// 380 positions: 10.5 / 11.8 / 12.4); two CTAs' worth of units are not two rounds of the longest (5 x 16 x 471: 17.6 / 24.1).  Fitted to 330
// drawn calls of up to 30 Gflop by each way, off by 9 % (rms): 0.92 of what the calls took with clusters sharing units of two tiles; 2 % of
// them are more than 3 % slower than that, chunks of few rows (2 x 1 x 40 over 2096 10.1 -> 11.0).
static int prefill_tile_ctas(const PfShape& sh, int rows, int sms) {
    const int stages = (rows + kPfRows - 1) / kPfRows;
    const bool two_roundings = rows < kSingleRoundingMinRows;
    const long long tiles = (long long)sh.n_tiles * sh.b, units = (long long)((sh.n_tiles + 1) / 2) * sh.b;
    if (tiles > 2 * sms) return 0;
    // stages of the tile that the `before` longest ones come before
    auto stages_of = [&](long long before) {
        return std::max(1.0, stages - (double)(before / ((long long)sh.head_blocks * sh.b)) * sh.positions / kPfRows);
    };
    const double pair_us = two_roundings ? 1.95 : 1.34, tile_us = two_roundings ? 0.9 : 0.68;
    double best_us;
    if (units > sms)
        best_us = 7.3 + std::max((double)stages, stages_of(2 * (2 * sms - units)) + stages_of(2 * (units - 1)) + 3.4) * pair_us;
    else if (sh.n_tiles % 2 == 0)
        best_us = 7.3 + stages * pair_us;
    else
        best_us = std::max(6.0 + stages * (two_roundings ? 1.31 : 0.95),
                           sh.n_tiles > 1 ? 7.3 + (sh.head_blocks > 1 ? stages : std::max(1.0, stages - (double)sh.positions / kPfRows)) * pair_us : 0.0);
    best_us *= 0.92;                                             // (one tile has to be quicker by 8 %, a cluster by 3 % more: the calls that were slower for a tie)
    int best = 0;
    for (int ctas = 1, log2_ctas = 0; ctas <= kPfMaxSplit && ctas <= stages; ctas *= 2, ++log2_ctas) {
        const int slots = ctas == 8 ? sms * 2 / 21 : ctas == 4 ? sms * 9 / 40 : sms / ctas;      // clusters that fit at once
        if (slots < 1) break;
        double us = (ctas > 1 ? 3.1 : 0) - 0.32 * log2_ctas;
        for (long long first = 0; first < tiles; first += slots)
            us += (first ? 10.1 : 8.4) + std::ceil(stages_of(first) / ctas) * tile_us;
        if (ctas > 1) us *= 1.03;
        if (us < best_us) { best = ctas; best_us = us; }
    }
    return best;
}

const char* mqa_prefill_plan_kernel_name(int b, int h, int n, int m_max, int with_start, int k, int v, int* ctas) {
    if (ctas) *ctas = 0;
    if (check_prefill_dims(b, h, n, m_max, k, v) != MQA_OK) return "";
    const int share = prefill_tile_ctas(prefill_shape(b, h, n, m_max), with_start ? m_max : n, sm_count());
    if (ctas) *ctas = share > 0 ? share : 1;
    return share > 0 ? "mqa_prefill_tile_kernel" : "mqa_prefill_kernel";
}

size_t mqa_prefill_workspace_bytes(int b, int h, int n, int m_max, int k, int v) {
    return check_prefill_dims(b, h, n, m_max, k, v) == MQA_OK ? 16 : 0;     // (the kernel keeps everything on chip)
}

int mqa_prefill_attention(const void* Q, const void* K, const void* V, const int32_t* start, float* O, void* workspace,
                          size_t workspace_bytes, int32_t* status, int b, int h, int n, int m_max, int k, int v,
                          mqa_stream_t stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!Q || !K || !V || !O || !workspace) return MQA_ERR_INVALID_ARG;
    if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(O) || !aligned16(workspace) || !aligned4(start) ||
        !aligned4(status))
        return MQA_ERR_INVALID_ARG;
    const int rc = check_prefill_dims(b, h, n, m_max, k, v);
    if (rc) return rc;
    if (workspace_bytes < mqa_prefill_workspace_bytes(b, h, n, m_max, k, v)) return MQA_ERR_WORKSPACE_TOO_SMALL;
    static std::atomic<int> opt_in[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return MQA_ERR_CUDA; }
    if (!opt_in[dev].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(mqa_prefill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPfSmemBytes) != cudaSuccess ||
            cudaFuncSetAttribute(mqa_prefill_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPtSmemBytes) != cudaSuccess) {
            cudaGetLastError();
            return MQA_ERR_CUDA;
        }
        opt_in[dev].store(1, std::memory_order_release);
    }
    PfShape sh = prefill_shape(b, h, n, m_max);
    const int sms = sm_count(), ctas = prefill_tile_ctas(sh, start ? m_max : n, sms);
    prefill_units(sh, ctas > 0 ? 1 : 2);
    alignas(64) CUtensorMap map_q, map_k, map_v;
    if (!encode_map(&map_q, Q, (long long)b * h, n, kHeadDim, sh.heads, sh.positions) ||
        !encode_cache_map(&map_k, K, (long long)b * m_max, kPfRows) || !encode_cache_map(&map_v, V, (long long)b * m_max, kPfRows))
        return MQA_ERR_CUDA;
    if (ctas > 0)
        launch_dependent_clusters((unsigned)ctas, mqa_prefill_tile_kernel, (unsigned)(sh.n_items * ctas), (unsigned)kPfThreads,
                                  (size_t)kPtSmemBytes, stream, map_q, map_k, map_v, start, O, status, sh);
    else
        launch_dependent(mqa_prefill_kernel, (unsigned)(sh.n_items < sms ? sh.n_items : sms), (unsigned)kPfThreads,
                         (size_t)kPfSmemBytes, stream, map_q, map_k, map_v, start, O, status, sh);
    return launch_status();
}

int mqa_set_test_cluster_room(int most) {
    mqa::g_test_cluster_room.store(most < 0 ? -1 : most, std::memory_order_relaxed);
    return MQA_OK;
}

int mqa_set_test_withhold_copy(int on) {
    const int value = on ? 1 : 0;
    if (cudaMemcpyToSymbol(g_test_withhold, &value, sizeof value) != cudaSuccess) {
        cudaGetLastError();
        return MQA_ERR_CUDA;
    }
    return MQA_OK;
}

int mqa_set_wait_limit_cycles(long long cycles) {
    const long long value = cycles > 0 ? cycles : kWaitLimitCycles;
    if (cudaMemcpyToSymbol(g_wait_limit_cycles, &value, sizeof value) != cudaSuccess) {
        cudaGetLastError();
        return MQA_ERR_CUDA;
    }
    return MQA_OK;
}

const char* mqa_plan_kernel_name(int multi_query, int whole_step, int b, int h, int m_max, int k, int v) {
    if (!dims_ok(b, h, m_max) || k != kHeadDim || v != kHeadDim) return "";
    const Plan p = make_plan(multi_query != 0, b, h, m_max);
    switch (p.kernel) {
        case Kernel::kUmma: {
            const bool guess = whole_step && p.merge_in_kernel && p.n_splits <= kGuessMaxPieces && p.chunk_rows >= kGuessMinShareRows;
            if (h <= 16) return !whole_step ? "mqa_decode_stream_umma_kernel<16>" : guess ? "mqa_decode_stream_umma_kernel<16, fused, guess>" : "mqa_decode_stream_umma_kernel<16, fused>";
            return !whole_step ? "mqa_decode_stream_umma_kernel<32>" : guess ? "mqa_decode_stream_umma_kernel<32, fused, guess>" : "mqa_decode_stream_umma_kernel<32, fused>";
        }
        case Kernel::kMma1: return "mqa_decode_split_mma_kernel<1>";
        case Kernel::kMma2: return "mqa_decode_split_mma_kernel<2>";
        case Kernel::kWide: return "mqa_decode_wide_kernel";
        default: return "decode_split_simt_kernel";
    }
}

const char* mqa_status_string(int code) {
    switch (code) {
        case MQA_OK: return "ok";
        case MQA_ERR_INVALID_ARG: return "invalid argument (null or misaligned pointer, non-positive dimension)";
        case MQA_ERR_UNSUPPORTED: return "unsupported configuration (k and v must be 128)";
        case MQA_ERR_WORKSPACE_TOO_SMALL: return "workspace too small (see mqa_workspace_bytes)";
        case MQA_ERR_CUDA: return "CUDA launch error";
        case MQA_ERR_STATIC_SCRATCH_TOO_SMALL:
            return "these sizes need more scratch than the built-in array of mqa_decode_step_noalloc";
        default: return "unknown status code";
    }
}

}  // extern "C"
