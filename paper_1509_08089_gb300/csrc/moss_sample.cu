// moss_sample.cu -- the sampling loop of MOSS-4 (Algorithm 1), MOSS-4Min
// (Algorithm 2), T-5 (Algorithm 3) and Path-5 (Algorithm 4) on the device.
//
// One thread draws one sample at a time (grid-stride over sample ids), so
// every sample is an independent chain of dependent gathers:
//   random words -> vertex alias record (32 B, with the alias's vertex record;
//   vert[v] (16 B) only when the column keeps the draw) -> sigma
//   record(s) of N_v (32 B each, carrying the picked neighbour's list and
//   twin) -> uniform list picks (4 B) -> the unknown pairs, probed together
//   (hashed edge set, or lock-step binary searches) -> edge mask -> class
//   through a shared-memory table.
// Counts are aggregated per warp with __match_any_sync into shared-memory
// histograms, and each block adds its own to the launch's 22 sums.
//
// Word schedule (x_i = word i of the sample, output (4 s + method) 16 + i + 1
// of SplitMix64 seeded with seed, or Philox4x32-10 block i / 2; sample_words2
// in moss_internal.cuh):
//   MOSS-4 : x0,x1 vertex draw (column, threshold), x6 its level; x2,x3 sigma
//            draw of u; x4 w; x5 r.
//   T-5    : x0,x1 vertex draw, x7 its level; x2,x3 sigma of u; x4 w; x5 r;
//            x6 t.
//   MOSS-4Min: x0,x1 vertex draw (pi-check), x6 its level; x2,x3 sigma-check
//            draw of u; x4 w (uniform in N_{v,u}); x5 r (uniform in N_{u,v}).
//   Path-5 : x0,x1 vertex draw, x14 its level; x2 r; x3 t; attempts a = 0,1 use
//            x(4+4a)..x(7+4a) for two independent sigma draws (u, w), kept
//            when the positions differ (sigma_u sigma_w / (1 - sum sigma^2)
//            is exactly tau_u mu_w of Sec. 5.1.2); if both collide, x12 draws
//            u from tau^(v) and x13 draws w from mu^(v,u) with the interval of
//            u removed from ACC (Sec. 5.1.4).
// RandomVertex(N_v - X) (Sec. 4.1.3) takes the j-th admissible position,
// skipping the excluded positions of X in list order.
#include <algorithm>
#include <atomic>

#include "moss_sampler.cuh"

namespace moss {

namespace {

// Resident blocks per SM each sampler is compiled for: the loop is bound by
// memory latency, so more warps in flight help until register spills cost
// more than they hide (measured: 6 blocks of 256 threads for every main
// sampler; Path-5 reaches it only with its second attempt and fallback
// deferred).  Under Philox words they hold the generator's state beside their
// records and would spill at that register budget, so they are compiled for
// one block fewer; the grid of a launch follows each instance's occupancy.
template <int METHOD, int RNG>
constexpr int min_blocks() { return RNG == kRngPhilox ? 5 : 6; }
// The redraw launch: five blocks (48 registers) where that spills nothing, four
// with the filter's probes or the generator's state.
template <int PM, int RNG>
constexpr int redraw_blocks() { return PM == kPmFilter || RNG == kRngPhilox ? 4 : 5; }

template <int METHOD, bool RECORD, bool HASH, int PM, int RNG>
__global__ void __launch_bounds__(kThreads, min_blocks<METHOD, RNG>()) k_sample(DevGraph g, uint64_t first, uint64_t count, uint64_t seed,
                                                     uint64_t *sums, uint8_t *classes, uint32_t *verts) {
    __shared__ uint8_t lut[kLut];
    __shared__ uint8_t lutc[METHOD == 3 ? 4096 : 1];
    __shared__ uint32_t hist[kWarps][kSlots];
    let_next_begin();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint8_t *src = (METHOD == 0 || METHOD == 3) ? g_lut4 : g_lut5;
    const int lut_n = (METHOD == 0 || METHOD == 3) ? 64 : 1024;
    for (int i = threadIdx.x; i < lut_n; i += kThreads) lut[i] = src[i];
    if (METHOD == 3)
        for (int i = threadIdx.x; i < 4096; i += kThreads) lutc[i] = g_lutc[i];
    for (int i = threadIdx.x; i < kWarps * kSlots; i += kThreads) (&hist[0][0])[i] = 0;
    __syncthreads();
    const uint64_t stride = (uint64_t)gridDim.x * kThreads;
    // warp-uniform loop: every lane of a warp runs the same trip count
    const uint64_t warp_base = ((uint64_t)blockIdx.x * kThreads) + (uint64_t)warp * 32;
    for (uint64_t base = warp_base; base < count; base += stride) {
        const uint64_t i = base + lane;
        int cls = kSlots;  // no sample (tail)
        bool deferred = false;
        if (i < count) {
            const uint64_t s = first + i;
            Sample sm;
            if (METHOD == 0) sm = sample_moss4<RNG, HASH, PM>(g, lut, seed, s);
            else if (METHOD == 1) sm = sample_t5<RNG, HASH, PM>(g, lut, seed, s);
            else if (METHOD == 2) sm = sample_path5<RNG, HASH, 0, PM>(g, lut, seed, s);
            else sm = sample_min<RNG, HASH, PM>(g, lut, lutc, seed, s);
            deferred = METHOD == 2 && sm.cls == kDeferred;
            if (!deferred) {
                cls = METHOD == 3 ? min_slot(sm.cls, sm.v[4]) : sm.cls;
                if (RECORD) {
                    classes[i] = (uint8_t)sm.cls;
                    if (verts) {
#pragma unroll
                        for (int k = 0; k < 5; ++k) verts[5 * i + k] = sm.v[k];
                    }
                }
            }
        }
        if (METHOD == 2) {   // one bitmap word per 32 sample ids, written by the warp that drew them
            // (streaming store: the word is read once, by the next launch, and
            // should not push the tables out of L2 meanwhile)
            const uint32_t bits = __ballot_sync(0xffffffffu, deferred);
            if (lane == 0) __stcs(g.defer + (base >> 5), bits);
        }
        const uint32_t peers = __match_any_sync(0xffffffffu, cls);
        if (cls < kSlots && lane == __ffs(peers) - 1) atomicAdd(&hist[warp][cls], (uint32_t)__popc(peers));
    }
    __syncthreads();
    await_previous();
    add_sums<kWarps>(hist, sums);
}

// The Path-5 samples a launch deferred: their second attempt and, for those
// that collide again, the fallback.  A warp takes windows of `window` (up to
// 32) bitmap words, grid-stride; it appends each window's flagged ids to a
// list in shared memory (a warp scan of the words' popcounts places them) and
// draws from the list 32 at a time, one per lane, keeping fewer than 32 ids
// over to its next window; ids that collide again go to a second list, drawn
// in the same way.  So every round but the warp's last ones runs with all
// lanes busy however sparse the flags.  Bound by the rounds' chains of
// dependent gathers, with few warps' rounds in flight.  As two launches with
// 32-word windows (the fallback after every second attempt) it took 62 us of a
// 2M-edge mesh's estimate of 5e6 samples and 136 us of a 1M-edge graph's of
// 1e8; the estimates as a whole, two launches -> this one: 449 -> 433 us and
// 4.031 -> 4.013 ms.
constexpr uint32_t kDeferList = 1024 + 32;   // a window's ids plus the carry-over
constexpr uint32_t kAgainList = 64;          // fewer than 32 waiting plus a round's

template <bool RECORD, bool HASH, int PM, int RNG>
__global__ void __launch_bounds__(kThreads, redraw_blocks<PM, RNG>())
    k_sample_deferred(DevGraph g, uint64_t first, uint64_t count, uint32_t window, uint64_t seed, uint64_t *sums,
                      uint8_t *classes, uint32_t *verts) {
    __shared__ uint8_t lut[kLut];
    __shared__ uint32_t hist[kWarps][kSlots];
    __shared__ uint32_t list[kWarps][kDeferList], again[kWarps][kAgainList];   // ids relative to the chunk's first
    let_next_begin();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kLut; i += kThreads) lut[i] = g_lut5[i];
    for (int i = threadIdx.x; i < kWarps * kSlots; i += kThreads) (&hist[0][0])[i] = 0;
    __syncthreads();
    await_previous();
    const uint64_t words = (count + 31) / 32;
    const uint64_t stride = (uint64_t)gridDim.x * kWarps * window;
    uint32_t *lst = list[warp], *agn = again[warp];
    // counts (and records) the lanes' samples; kDeferred ones are left out
    auto put = [&](bool drawn, uint32_t i, const Sample &sm) {
        const int cls = drawn && sm.cls != kDeferred ? sm.cls : kSlots;
        if (RECORD && cls < kSlots) {
            classes[i] = (uint8_t)cls;
            if (verts) {
#pragma unroll
                for (int k = 0; k < 5; ++k) verts[5ull * i + k] = sm.v[k];
            }
        }
        const uint32_t peers = __match_any_sync(0xffffffffu, cls);
        if (cls < kSlots && lane == __ffs(peers) - 1) atomicAdd(&hist[warp][cls], (uint32_t)__popc(peers));
    };
    // the fallback of agn[from + lane] for lane < cnt (warp-uniform arguments)
    auto fallback = [&](uint32_t from, uint32_t cnt) {
        const bool mine = (uint32_t)lane < cnt;
        const uint32_t i = mine ? agn[from + lane] : 0u;   // < count: only drawn ids are flagged
        Sample sm;
        if (mine) sm = sample_path5<RNG, HASH, 2, PM>(g, lut, seed, first + i);
        put(mine, i, sm);
        __syncwarp();   // the places are free again
    };
    uint32_t m = 0;   // ids waiting in agn (warp-uniform, < 32 between rounds)
    // the second attempt of lst[from + lane] for lane < cnt
    auto attempt = [&](uint32_t from, uint32_t cnt) {
        const bool mine = (uint32_t)lane < cnt;
        const uint32_t i = mine ? lst[from + lane] : 0u;
        Sample sm;
        if (mine) sm = sample_path5<RNG, HASH, 1, PM>(g, lut, seed, first + i);
        put(mine, i, sm);
        const bool back = mine && sm.cls == kDeferred;
        const uint32_t bits = __ballot_sync(0xffffffffu, back);
        if (back) agn[m + __popc(bits & ((1u << lane) - 1u))] = i;
        __syncwarp();
        m += __popc(bits);
        if (m >= 32) fallback(m -= 32, 32);
    };
    uint32_t n = 0;   // ids waiting in lst (warp-uniform, < 32 between windows)
    for (uint64_t w0 = ((uint64_t)blockIdx.x * kWarps + warp) * window; w0 < words; w0 += stride) {
        const uint64_t w = w0 + lane;
        uint32_t bits = (uint32_t)lane < window && w < words ? __ldcs(g.defer + w) : 0u;
        const uint32_t c = __popc(bits);
        uint32_t incl = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += t;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        uint32_t at = n + incl - c;
        while (bits) {
            lst[at++] = (uint32_t)(w * 32 + __ffs(bits) - 1);
            bits &= bits - 1;
        }
        n += total;
        __syncwarp();
        uint32_t done = 0;
        for (; n - done >= 32; done += 32) attempt(done, 32);
        if (done) {   // move the remainder (< 32 ids) to the front
            const uint32_t rem = n - done;
            const uint32_t x = (uint32_t)lane < rem ? lst[done + lane] : 0u;
            __syncwarp();
            if ((uint32_t)lane < rem) lst[lane] = x;
            __syncwarp();
            n = rem;
        }
    }
    if (n) attempt(0, n);
    if (m) fallback(0, m);
    __syncthreads();
    add_sums<kWarps>(hist, sums);
}

// ---------------------------------------------------------------- batches --
// Many requests on many graphs in one persistent launch.  Warps take tiles
// (fixed-size runs of sample ids of one task) from a global counter -- one
// atomic per tile, none per sample -- and write each tile's class counts to
// the tile's own row, so a task's counts are the sum of its rows whatever
// warp ran which tile, and equal the counts of a solo launch of the task.
constexpr int kBatchBlocks = 4;   // resident blocks per SM (Path-5 bound)

// the count slot of sample s of a method: its class, or for MOSS-4Min its
// (class, c) slot
// (plain loads for every graph: a second, streaming body per method in the
// persistent batch kernel cost 12% on the 512-graph batch)
template <bool HASH, int RNG>
__device__ __forceinline__ int sample_any(const DevGraph &g, const uint8_t *lut4, const uint8_t *lut5,
                                          const uint8_t *lutc, uint32_t method, uint64_t seed, uint64_t s) {
    if (method == 0) return sample_moss4<RNG, HASH, kPmBatch>(g, lut4, seed, s).cls;
    if (method == 1) return sample_t5<RNG, HASH, kPmBatch>(g, lut5, seed, s).cls;
    if (method == 3) {
        const Sample sm = sample_min<RNG, HASH, kPmBatch>(g, lut4, lutc, seed, s);
        return min_slot(sm.cls, sm.v[4]);
    }
    return sample_path5<RNG, HASH, 3, kPmBatch>(g, lut5, seed, s).cls;
}

// Persistent sampler over a batch: warps take tiles of `tile_samples` ids of
// one task from a device counter.  THREADS per block is a tuning choice (the
// resident threads per SM stay the same: THREADS x blocks = 1,024).  RNGS:
// the generators the batch's graphs use (kBatchSplitMix, kBatchPhilox, or
// kBatchBoth: chosen per tile), so a single-generator batch carries one
// sampler body.  With tile_cycles non-null the first lane of a warp records
// each tile's duration in SM clock cycles (the autotuner's per-graph cost of
// a probe strategy).
template <int THREADS, int RNGS>
__global__ void __launch_bounds__(THREADS, kBatchBlocks * kThreads / THREADS)
    k_sample_batch(const DevGraph *graphs, const BatchTask *tasks, int ntasks, uint64_t ntiles, uint32_t tile_samples,
                   unsigned long long *next_tile, uint32_t *tile_counts, unsigned long long *tile_cycles) {
    constexpr int kW = THREADS / 32;
    __shared__ uint8_t lut4[64];
    __shared__ uint8_t lut5[kLut];
    __shared__ uint8_t lutc[4096];
    __shared__ uint32_t hist[kW][kSlots];
    __shared__ DevGraph gsh[kW];
    static_assert(sizeof(DevGraph) % 4 == 0 && sizeof(DevGraph) / 4 <= 64, "graph descriptor staging");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < 64; i += THREADS) lut4[i] = g_lut4[i];
    for (int i = threadIdx.x; i < kLut; i += THREADS) lut5[i] = g_lut5[i];
    for (int i = threadIdx.x; i < 4096; i += THREADS) lutc[i] = g_lutc[i];
    __syncthreads();
    for (;;) {
        const long long c0 = clock64();
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(next_tile, 1ull);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= ntiles) break;
        // the task of tile t: the last task whose first tile is <= t
        int lo = 0, len = ntasks;
        while (len > 0) {
            const int half = len >> 1;
            if (tasks[lo + half].tile0 <= t) { lo += half + 1; len -= half + 1; } else { len = half; }
        }
        const BatchTask tk = tasks[lo - 1];
        for (int wd = lane; wd < (int)(sizeof(DevGraph) / 4); wd += 32)
            reinterpret_cast<uint32_t *>(&gsh[warp])[wd] = reinterpret_cast<const uint32_t *>(graphs + tk.graph)[wd];
        if (lane < kSlots) hist[warp][lane] = 0;
        __syncwarp();
        const DevGraph &g = gsh[warp];
        const uint64_t f = tk.first + (t - tk.tile0) * tile_samples;
        const uint64_t left = tk.first + tk.count - f;
        const uint32_t cnt = (uint32_t)(left < tile_samples ? left : tile_samples);
        const bool hashed = g.hash != nullptr;
        // warp-uniform: a tile belongs to one graph
        const bool philox = RNGS == kBatchPhilox || (RNGS == kBatchBoth && g.rng == kRngPhilox);
        for (uint32_t base = 0; base < cnt; base += 32) {
            const uint32_t i = base + lane;
            int cls = kSlots;
            if (i < cnt) {
                if (philox)
                    cls = hashed ? sample_any<true, kRngPhilox>(g, lut4, lut5, lutc, tk.method, tk.seed, f + i)
                                 : sample_any<false, kRngPhilox>(g, lut4, lut5, lutc, tk.method, tk.seed, f + i);
                else
                    cls = hashed ? sample_any<true, kRngSplitMix>(g, lut4, lut5, lutc, tk.method, tk.seed, f + i)
                                 : sample_any<false, kRngSplitMix>(g, lut4, lut5, lutc, tk.method, tk.seed, f + i);
            }
            const uint32_t peers = __match_any_sync(0xffffffffu, cls);
            if (cls < kSlots && lane == __ffs(peers) - 1) atomicAdd(&hist[warp][cls], (uint32_t)__popc(peers));
        }
        __syncwarp();
        if (lane < kSlots) tile_counts[t * kSlots + lane] = hist[warp][lane];
        if (tile_cycles && lane == 0) tile_cycles[t] = (unsigned long long)(clock64() - c0);
        __syncwarp();
    }
}

// block per task, warp per class slot: sum the task's tile rows
__global__ void k_batch_reduce(const BatchTask *tasks, uint32_t tile_samples, const uint32_t *tile_counts,
                               uint64_t *task_counts) {
    const BatchTask tk = tasks[blockIdx.x];
    const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t nt = (tk.count + tile_samples - 1) / tile_samples;
    uint64_t s = 0;
    for (uint64_t j = lane; j < nt; j += 32) s += tile_counts[(tk.tile0 + j) * kSlots + c];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
    if (lane == 0) task_counts[(uint64_t)blockIdx.x * kSlots + c] = s;
}

__global__ void k_copy_counts(const uint64_t *sums, uint64_t *out) {
    await_previous();
    if (threadIdx.x < kSlots) out[threadIdx.x] = sums[threadIdx.x];
}

// T-5 and Path-5 (or, MIX, MOSS-4 and MOSS-4Min) samples 0.. in one launch:
// the first blocks_a blocks draw the first method's, counted at sums, the rest
// the second's, counted at sums + kSlots.  A small estimate is launches and latency, so
// its two sub-methods share the chip and Path-5 redraws in line (two more
// launches otherwise, each a few long dependent chains).
template <bool MIX, bool HASH, int PM, int RNG>
__global__ void __launch_bounds__(kThreads, 4)
    k_sample_pair(DevGraph g, uint32_t blocks_a, uint64_t count_a, uint64_t count_b, uint64_t seed,
                  uint64_t *sums) {
    __shared__ uint8_t lut[MIX ? 64 : kLut];
    __shared__ uint8_t lutc[MIX ? 4096 : 1];
    __shared__ uint32_t hist[kWarps][kSlots];
    let_next_begin();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < (MIX ? 64 : kLut); i += kThreads) lut[i] = MIX ? g_lut4[i] : g_lut5[i];
    if (MIX)
        for (int i = threadIdx.x; i < 4096; i += kThreads) lutc[i] = g_lutc[i];
    for (int i = threadIdx.x; i < kWarps * kSlots; i += kThreads) (&hist[0][0])[i] = 0;
    __syncthreads();
    const bool second = blockIdx.x >= blocks_a;   // block-uniform
    const uint32_t block = second ? blockIdx.x - blocks_a : blockIdx.x;
    const uint64_t count = second ? count_b : count_a;
    const uint64_t stride = (uint64_t)(second ? gridDim.x - blocks_a : blocks_a) * kThreads;
    for (uint64_t base = ((uint64_t)block * kWarps + warp) * 32; base < count; base += stride) {
        const uint64_t i = base + lane;
        int cls = kSlots;
        if (i < count) {
            if (!second) {
                cls = MIX ? sample_moss4<RNG, HASH, PM>(g, lut, seed, i).cls : sample_t5<RNG, HASH, PM>(g, lut, seed, i).cls;
            } else if (MIX) {
                const Sample sm = sample_min<RNG, HASH, PM>(g, lut, lutc, seed, i);
                cls = min_slot(sm.cls, sm.v[4]);
            } else {
                cls = sample_path5<RNG, HASH, 3, PM>(g, lut, seed, i).cls;
            }
        }
        const uint32_t peers = __match_any_sync(0xffffffffu, cls);
        if (cls < kSlots && lane == __ffs(peers) - 1) atomicAdd(&hist[warp][cls], (uint32_t)__popc(peers));
    }
    __syncthreads();
    add_sums<kWarps>(hist, second ? sums + kSlots : sums);
}

// the probe variant of a launch: 0 list search, 1 hashed set, 2 filter in
// front of it, 3 hashed set with two-level vertex tables (kPmStream)
int probe_variant(int method, const DevGraph &g) {
    if (!g.hash) return 0;
    if (g.filter) return 2;
    return g.nheavy[method] != 0 && g.nheavy[method] <= kStreamHeavy ? 3 : 1;
}

template <int M, bool R, int RNG>
cudaError_t launch_one_rng(const DevGraph &g, uint64_t first, uint64_t count, uint64_t seed, uint64_t *sums, int blocks,
                           uint8_t *classes, uint32_t *verts, cudaStream_t s, bool early) {
    auto *k = &k_sample<M, R, false, kPmPlain, RNG>;
    switch (probe_variant(M, g)) {
        case 2: k = &k_sample<M, R, true, kPmFilter, RNG>; break;
        case 3: k = &k_sample<M, R, true, kPmStream, RNG>; break;
        case 1: k = &k_sample<M, R, true, kPmPlain, RNG>; break;
        default: break;
    }
    return launch_early(early, k, blocks, kThreads, s, g, first, count, seed, sums, classes, verts);
}

template <int M, bool R>
cudaError_t launch_one(const DevGraph &g, uint64_t first, uint64_t count, uint64_t seed, uint64_t *sums, int blocks,
                       uint8_t *classes, uint32_t *verts, cudaStream_t s, bool early) {
    if (g.rng == kRngPhilox)
        return launch_one_rng<M, R, kRngPhilox>(g, first, count, seed, sums, blocks, classes, verts, s, early);
    return launch_one_rng<M, R, kRngSplitMix>(g, first, count, seed, sums, blocks, classes, verts, s, early);
}

}  // namespace

void upload_luts(const uint8_t *lut4, const uint8_t *lut5, const uint8_t *lutc) {
    upload_luts_here(lut4, lut5, lutc);
    upload_luts_group(lut4, lut5, lutc);
}

// resident blocks per SM of each sampler variant (probe 0 search, 1 hash, 2
// filter, 3 hash with two-level tables; + 4 under Philox words) on each
// device, 0 until queried
constexpr int kProbeVariants = 4;
constexpr int kVariants = 2 * kProbeVariants;
std::atomic<int> g_sample_per_sm[64][kMethods][kVariants];

template <int M, int RNG>
cudaError_t occupancy_probe(int *per) {
    cudaError_t e =
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per[0], k_sample<M, false, false, kPmPlain, RNG>, kThreads, 0);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per[1], k_sample<M, false, true, kPmPlain, RNG>, kThreads, 0);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per[2], k_sample<M, false, true, kPmFilter, RNG>, kThreads, 0);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per[3], k_sample<M, false, true, kPmStream, RNG>, kThreads, 0);
    return e;
}

template <int M>
cudaError_t occupancy_all(int (&per)[kVariants]) {
    cudaError_t e = occupancy_probe<M, kRngSplitMix>(per);
    if (e == cudaSuccess) e = occupancy_probe<M, kRngPhilox>(per + kProbeVariants);
    return e;
}

// resident blocks per SM of a variant (at least 1)
int sample_per_sm(int method, int device, int variant) {
    const bool cached = device >= 0 && device < 64 && method >= 0 && method < kMethods;
    if (cached) {
        const int c = g_sample_per_sm[device][method][variant].load(std::memory_order_relaxed);
        if (c > 0) return c;
    }
    int per[kVariants] = {1, 1, 1, 1, 1, 1, 1, 1};
    cudaError_t e;
    if (method == 0) e = occupancy_all<0>(per);
    else if (method == 1) e = occupancy_all<1>(per);
    else if (method == 2) e = occupancy_all<2>(per);
    else e = occupancy_all<3>(per);
    for (int v = 0; v < kVariants; ++v) {
        if (e != cudaSuccess || per[v] < 1) per[v] = 1;
        if (cached && e == cudaSuccess) g_sample_per_sm[device][method][v].store(per[v], std::memory_order_relaxed);
    }
    return per[variant];
}

// Blocks of a sampling launch: as many as fit, but for MOSS-4 behind the filter
// at most the 6 an SM that every sampler is compiled for.  Its registers would
// let 8 in, and their reads push one another's lines out of the L2 where no
// small heavy level holds most of the draws: 1.7e7 samples, ms, 8 -> 6 an SM:
// mesh of 2.3M edges 0.99 -> 0.93, 8M edges, 2M vertices 0.79 -> 0.76, 34M edges
// 1.44 -> 1.42.  With a heavy level of at most kStreamHeavy columns 8 stay (3.5M
// edges, degree order, 0.56 -> 0.60 with 6; 7M 0.59 -> 0.61).
int sample_launch_blocks(int method, int device, const DevGraph &g) {
    const int variant = probe_variant(method, g);
    int per = sample_per_sm(method, device, variant + (g.rng == kRngPhilox ? kProbeVariants : 0));
    const bool few_heavy = g.nheavy[method] != 0 && g.nheavy[method] <= kStreamHeavy;
    if (method == 0 && variant == 2 && !few_heavy) per = std::min(per, min_blocks<0, kRngSplitMix>());
    return device_sms(device) * per;
}

namespace {

cudaError_t launch_sample(int method, const DevGraph &g, uint64_t first, uint64_t count, uint64_t seed,
                          uint64_t *sums, int blocks, uint8_t *classes, uint32_t *verts, cudaStream_t s, bool early) {
    const bool rec = classes != nullptr;
    switch (method * 2 + (rec ? 1 : 0)) {
        case 0: return launch_one<0, false>(g, first, count, seed, sums, blocks, classes, verts, s, early);
        case 1: return launch_one<0, true>(g, first, count, seed, sums, blocks, classes, verts, s, early);
        case 2: return launch_one<1, false>(g, first, count, seed, sums, blocks, classes, verts, s, early);
        case 3: return launch_one<1, true>(g, first, count, seed, sums, blocks, classes, verts, s, early);
        case 4: return launch_one<2, false>(g, first, count, seed, sums, blocks, classes, verts, s, early);
        case 5: return launch_one<2, true>(g, first, count, seed, sums, blocks, classes, verts, s, early);
        case 6: return launch_one<3, false>(g, first, count, seed, sums, blocks, classes, verts, s, early);
        case 7: return launch_one<3, true>(g, first, count, seed, sums, blocks, classes, verts, s, early);
        default: return cudaErrorInvalidValue;
    }
}

template <bool HASH, int PM, int RNG>
cudaError_t launch_deferred(const DevGraph &g, uint64_t first, uint64_t count, uint64_t seed, uint64_t *sums,
                            uint8_t *classes, uint32_t *verts, cudaStream_t s) {
    // windows of 32 words, or smaller ones that give every resident warp one:
    // a warp draws its window's ids one round of 32 after the other
    const uint64_t warps = (uint64_t)current_sms() * redraw_blocks<PM, RNG>() * kWarps, words = (count + 31) / 32;
    const uint32_t window = (uint32_t)std::min<uint64_t>(32, (words + warps - 1) / warps);
    const uint64_t windows = (words + window - 1) / window;
    const int blocks = (int)std::min<uint64_t>(warps / kWarps, (windows + kWarps - 1) / kWarps);
    auto *k = classes ? &k_sample_deferred<true, HASH, PM, RNG> : &k_sample_deferred<false, HASH, PM, RNG>;
    return launch_early(true, k, blocks, kThreads, s, g, first, count, window, seed, sums, classes, verts);
}

template <int RNG>
cudaError_t launch_deferred_rng(const DevGraph &g, uint64_t first, uint64_t count, uint64_t seed, uint64_t *sums,
                                uint8_t *classes, uint32_t *verts, cudaStream_t s) {
    switch (probe_variant(2, g)) {
        case 2: return launch_deferred<true, kPmFilter, RNG>(g, first, count, seed, sums, classes, verts, s);
        case 3: return launch_deferred<true, kPmStream, RNG>(g, first, count, seed, sums, classes, verts, s);
        case 1: return launch_deferred<true, kPmPlain, RNG>(g, first, count, seed, sums, classes, verts, s);
        default: return launch_deferred<false, kPmPlain, RNG>(g, first, count, seed, sums, classes, verts, s);
    }
}

}  // namespace

cudaError_t launch_redraws(const DevGraph &g, uint64_t first, uint64_t count, uint64_t seed, uint64_t *sums,
                           uint8_t *classes, uint32_t *verts, cudaStream_t s) {
    if (g.rng == kRngPhilox) return launch_deferred_rng<kRngPhilox>(g, first, count, seed, sums, classes, verts, s);
    return launch_deferred_rng<kRngSplitMix>(g, first, count, seed, sums, classes, verts, s);
}

cudaError_t launch_copy_counts(const uint64_t *sums, uint64_t *out, bool early, cudaStream_t s) {
    return launch_early(early, k_copy_counts, 1, 32, s, sums, out);
}

cudaError_t launch_counts(int method, const DevGraph &g, uint64_t first, uint64_t count, uint64_t seed, uint64_t *sums,
                          uint8_t *classes, uint32_t *verts, cudaStream_t s, bool early) {
    int dev = 0;
    cudaGetDevice(&dev);
    const uint64_t chunk = method == 2 ? kDeferChunk : count;
    for (uint64_t c0 = 0; c0 < count; c0 += chunk) {
        const uint64_t len = std::min(chunk, count - c0);
        const int blocks = (int)std::min<uint64_t>(sample_launch_blocks(method, dev, g), (len + kThreads - 1) / kThreads);
        uint8_t *cl = classes ? classes + c0 : nullptr;
        uint32_t *vt = verts ? verts + 5 * c0 : nullptr;
        cudaError_t e = launch_sample(method, g, first + c0, len, seed, sums, blocks, cl, vt, s, early && c0 == 0);
        if (e == cudaSuccess && method == 2) e = launch_redraws(g, first + c0, len, seed, sums, cl, vt, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// ----------------------------------------------------------- small estimates --
namespace {

constexpr int kPairBlocks = 4;   // resident blocks per SM (Path-5 with its redraws in line)

template <bool MIX, int RNG>
cudaError_t launch_pair_rng(const DevGraph &g, int blocks, int blocks_a, uint64_t count_a, uint64_t count_b,
                            uint64_t seed, uint64_t *sums, cudaStream_t s) {
    if (!g.hash) k_sample_pair<MIX, false, kPmPlain, RNG><<<blocks, kThreads, 0, s>>>(g, blocks_a, count_a, count_b, seed, sums);
    else if (g.filter) k_sample_pair<MIX, true, kPmFilter, RNG><<<blocks, kThreads, 0, s>>>(g, blocks_a, count_a, count_b, seed, sums);
    else k_sample_pair<MIX, true, kPmPlain, RNG><<<blocks, kThreads, 0, s>>>(g, blocks_a, count_a, count_b, seed, sums);
    return cudaGetLastError();
}

}  // namespace

// At four resident blocks per SM against the single launches' six, and without
// their overlap, the pair stops paying once the chip is full for long.  Whole
// estimates, us, launches of their own -> one launch (20k-edge graph / 2M-edge
// mesh / 1M-edge power-law graph): k = 5, budget 1e5 55 -> 41 / 59 -> 44 / 52 ->
// 40, 1e6 87 -> 82 / 122 -> 119 / 92 -> 86, 2e6 117 -> 120 / 173 -> 188 / 126 ->
// 129; the mix, which has no redraws to save, 1e5 42 -> 40 / 45 -> 42 / 43 -> 40,
// 5e5 51 -> 51 / 68 -> 78 / 54 -> 57.
bool pair_fits(bool mix, uint64_t count_a, uint64_t count_b) {
    const uint64_t most = mix ? 1ull << 16 : 1ull << 19;
    return count_a <= most && count_b <= most;
}

cudaError_t launch_pair(bool mix, const DevGraph &g, uint64_t count_a, uint64_t count_b, uint64_t seed, uint64_t *sums,
                        cudaStream_t s) {
    if (count_a + count_b == 0) return cudaSuccess;
    // a block per 256 ids, or the resident blocks split in proportion
    const uint64_t most = (uint64_t)current_sms() * kPairBlocks;
    uint64_t na = (count_a + kThreads - 1) / kThreads, nb = (count_b + kThreads - 1) / kThreads;
    if (na + nb > most) {
        const uint64_t share = std::max<uint64_t>(most * na / (na + nb), na ? 1 : 0);
        nb = std::min(nb, std::max<uint64_t>(most - share, nb ? 1 : 0));
        na = share;
    }
    const int blocks = (int)(na + nb);
    if (g.rng == kRngPhilox)
        return mix ? launch_pair_rng<true, kRngPhilox>(g, blocks, (int)na, count_a, count_b, seed, sums, s)
                   : launch_pair_rng<false, kRngPhilox>(g, blocks, (int)na, count_a, count_b, seed, sums, s);
    return mix ? launch_pair_rng<true, kRngSplitMix>(g, blocks, (int)na, count_a, count_b, seed, sums, s)
               : launch_pair_rng<false, kRngSplitMix>(g, blocks, (int)na, count_a, count_b, seed, sums, s);
}

template <int T>
int max_per_sm_rngs(int rngs) {
    int per = 0;
    cudaError_t e;
    if (rngs == kBatchSplitMix) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sample_batch<T, kBatchSplitMix>, T, 0);
    else if (rngs == kBatchPhilox) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sample_batch<T, kBatchPhilox>, T, 0);
    else e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sample_batch<T, kBatchBoth>, T, 0);
    return e == cudaSuccess && per > 0 ? per : 1;
}

int batch_max_per_sm(int threads, int rngs) {
    if (threads == 128) return max_per_sm_rngs<128>(rngs);
    if (threads == 512) return max_per_sm_rngs<512>(rngs);
    return max_per_sm_rngs<256>(rngs);
}

int batch_blocks(int device, int threads, int per_sm, int rngs) {
    const int max = batch_max_per_sm(threads, rngs);
    const int per = per_sm <= 0 || per_sm > max ? max : per_sm;
    return device_sms(device) * per;
}

template <int T, int R>
void launch_batch_kernel(const DevGraph *graphs, const BatchTask *tasks, int ntasks, uint64_t ntiles,
                         uint32_t tile_samples, unsigned long long *next_tile, uint32_t *tile_counts, int blocks,
                         unsigned long long *tile_cycles, cudaStream_t s) {
    k_sample_batch<T, R><<<blocks, T, 0, s>>>(graphs, tasks, ntasks, ntiles, tile_samples, next_tile, tile_counts,
                                              tile_cycles);
}

template <int T>
void launch_batch_rngs(int rngs, const DevGraph *graphs, const BatchTask *tasks, int ntasks, uint64_t ntiles,
                       uint32_t tile_samples, unsigned long long *next_tile, uint32_t *tile_counts, int blocks,
                       unsigned long long *tile_cycles, cudaStream_t s) {
    if (rngs == kBatchSplitMix)
        launch_batch_kernel<T, kBatchSplitMix>(graphs, tasks, ntasks, ntiles, tile_samples, next_tile, tile_counts,
                                               blocks, tile_cycles, s);
    else if (rngs == kBatchPhilox)
        launch_batch_kernel<T, kBatchPhilox>(graphs, tasks, ntasks, ntiles, tile_samples, next_tile, tile_counts,
                                             blocks, tile_cycles, s);
    else
        launch_batch_kernel<T, kBatchBoth>(graphs, tasks, ntasks, ntiles, tile_samples, next_tile, tile_counts,
                                           blocks, tile_cycles, s);
}

cudaError_t launch_sample_batch(const DevGraph *graphs, const BatchTask *tasks, int ntasks, uint64_t ntiles,
                                uint32_t tile_samples, unsigned long long *next_tile, uint32_t *tile_counts,
                                int threads, int blocks, unsigned long long *tile_cycles, int rngs, cudaStream_t s) {
    if (ntasks <= 0 || ntiles == 0) return cudaSuccess;
    if (threads == 128)
        launch_batch_rngs<128>(rngs, graphs, tasks, ntasks, ntiles, tile_samples, next_tile, tile_counts, blocks,
                               tile_cycles, s);
    else if (threads == 512)
        launch_batch_rngs<512>(rngs, graphs, tasks, ntasks, ntiles, tile_samples, next_tile, tile_counts, blocks,
                               tile_cycles, s);
    else
        launch_batch_rngs<256>(rngs, graphs, tasks, ntasks, ntiles, tile_samples, next_tile, tile_counts, blocks,
                               tile_cycles, s);
    return cudaGetLastError();
}

cudaError_t launch_batch_reduce(const BatchTask *tasks, int ntasks, uint32_t tile_samples,
                                const uint32_t *tile_counts, uint64_t *task_counts, cudaStream_t s) {
    if (ntasks <= 0) return cudaSuccess;
    k_batch_reduce<<<ntasks, 32 * kSlots, 0, s>>>(tasks, tile_samples, tile_counts, task_counts);
    return cudaGetLastError();
}

}  // namespace moss
