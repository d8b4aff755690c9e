// moss_group.cu -- large sampling calls behind the edge filter, with the
// sample ids grouped by the vertex they draw first.
//
// A sample reads its first vertex v's own list (a slot record or two, one or
// two list entries) and then lists and edge tables all over the graph.  On a
// graph whose tables exceed the L2 every one of these reads is likely a DRAM
// line of its own.  Counts do not depend on the order samples are drawn in,
// so a large call first draws v for every id of a chunk, sorts the ids by a
// hash of v into kGroups groups (a counting sort: histogram with the draw,
// scan, placement through shared memory) and then draws the samples in that
// order: at any time the resident threads work on about a dozen groups, whose
// lists together are a few MB and stay in the L2.
//
// Bound: the sampling pass by DRAM lines and L1-to-L2 requests as before, at
// fewer of the former.  34M-edge graph, chunks of 2^26 ids, ncu: DRAM reads per
// sample and the pass's DRAM rate (a copy runs at 6.8 TB/s, random lines at 5.2),
// MOSS-4 / T-5 / Path-5: degree order 202 / 184 / 294 B, 5.7 / 4.0 / 5.7 TB/s
// (ungrouped 304 / 349 / 480 B); input ids 204 / 193 / 344 B, 4.6 / 3.6 / 4.8.
// The draw is bound by its ~130 instructions per id (0.29-0.31 ms per 2^26 ids),
// the placement by its 12 B per id and the shared-memory atomics (0.29 ms).
// Calls of 2e8 ids, ms, ungrouped -> grouped, same run:
//              34M edges, degree order   34M edges, input ids
//   MOSS-4          9.9 -> 8.7               15.2 -> 10.4
//   T-5            11.9 -> 10.9              19.3 -> 12.2
//   Path-5         15.9 -> 12.0              22.8 -> 16.1
//   MOSS-4Min      13.4 -> 10.9              17.5 -> 13.4
// Reads in the grouped pass must not skip L1 allocation: with
// ld.global.nc.L1::no_allocate the L2 gave the lines up early (T-5's DRAM reads
// per sample more than doubled).  Groups: 512 or 2,048 measured 2-4% slower than
// 1,024; chunks of 2^25 ids 4% slower than 2^26.
#include <algorithm>

#include "moss_sampler.cuh"

namespace moss {

namespace {

constexpr int kGroupBits = 10;
constexpr uint32_t kGroups = 1u << kGroupBits;
constexpr uint64_t kGroupChunk = kDeferChunk;   // ids per pass (the Path-5 deferral bitmap holds one chunk)
constexpr int kGroupThreads = 512;
constexpr int kGroupItems = 16;
constexpr uint32_t kGroupTile = kGroupThreads * kGroupItems;   // ids a block places at a time
constexpr int kGroupPerSm = 2;
// consecutive entries a block draws: the grid covers 152 x 6 x 1,024 ids (14
// groups of a full chunk) at a time; 256 and 8,192 measured slower (Path-5,
// degree order: 14.6 and 17.4 ms against 13.9)
constexpr uint32_t kDrawTile = 1024;
constexpr int kDrawIlp = 4;   // independent vertex draws in flight per thread

static_assert(kGroupChunk <= (1ull << 32) - kGroupTile, "chunk-relative ids are 32-bit");
static_assert(kGroups % kGroupThreads == 0, "a whole number of groups per thread");

// the group of a vertex: a multiplicative hash, so that neither the degree
// order (heavy vertices first) nor a pattern in the ids fills few groups
__device__ __forceinline__ uint32_t group_of(uint32_t v) { return (v * 0x9E3779B1u) >> (32 - kGroupBits); }

// Inclusive prefix of x over a block of WARPS warps; wsum: WARPS words.
template <int WARPS>
__device__ __forceinline__ uint32_t block_incl_scan(uint32_t x, uint32_t *wsum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += t;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    for (int w = 0; w < warp; ++w) x += wsum[w];
    return x;
}

// v of every id of the chunk (vout[i] of id first + i), and the group sizes
// added to sizes[kGroups] (zeroed beforehand)
template <int METHOD, int RNG>
__global__ void __launch_bounds__(kGroupThreads, kGroupPerSm)
    k_group_draw(DevGraph g, uint64_t first, uint32_t count, uint64_t seed, uint32_t *vout, uint32_t *sizes) {
    __shared__ uint32_t hist[kGroups];
    for (uint32_t i = threadIdx.x; i < kGroups; i += kGroupThreads) hist[i] = 0;
    __syncthreads();
    const uint32_t nh = g.nheavy[METHOD];
    const uint64_t tl = g.tlight[METHOD];
    const uint64_t stride = (uint64_t)gridDim.x * kGroupThreads * kDrawIlp;
    for (uint64_t base = (uint64_t)blockIdx.x * kGroupThreads * kDrawIlp; base < count; base += stride) {
        uint64_t xt[kDrawIlp];
        uint4 rec[kDrawIlp];   // {T lo, T hi, alias, self} of the column
#pragma unroll
        for (int k = 0; k < kDrawIlp; ++k) {
            const uint64_t i = base + k * kGroupThreads + threadIdx.x;
            const uint64_t s = first + i;
            const Words2 x01 = sample_words2<RNG>(seed, METHOD, s, 0);
            bool light = true;
            if (nh != 0) light = sample_word<RNG>(seed, METHOD, s, level_word(METHOD)) < tl;
            const uint32_t c = (light ? nh : 0u) + word_index32(x01.x[0], light ? g.n - nh : nh);
            xt[k] = x01.x[1];
            rec[k] = make_uint4(0, 0, 0, 0);
            if (i < count) rec[k] = ld4(g.seed[METHOD] + 2 * (uint64_t)c);
        }
#pragma unroll
        for (int k = 0; k < kDrawIlp; ++k) {
            const uint64_t i = base + k * kGroupThreads + threadIdx.x;
            if (i >= count) continue;
            const uint64_t T = ((uint64_t)rec[k].y << 32) | rec[k].x;
            const uint32_t v = xt[k] < T ? rec[k].w : rec[k].z;
            __stcs(vout + i, v);
            atomicAdd(&hist[group_of(v)], 1u);
        }
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < kGroups; i += kGroupThreads)
        if (hist[i]) atomicAdd(&sizes[i], hist[i]);
}

// group sizes to group starts, in place (one block)
__global__ void __launch_bounds__(kGroups) k_group_scan(uint32_t *sizes) {
    __shared__ uint32_t wsum[kGroups / 32];
    const uint32_t x = sizes[threadIdx.x];
    sizes[threadIdx.x] = block_incl_scan<kGroups / 32>(x, wsum) - x;
}

// entries {v, chunk-relative id} in group order: a block ranks a tile of ids
// within their groups, takes each group's next places from cursor[] and
// writes the tile from shared memory in runs of one group (8 entries, 64 B,
// on average)
__global__ void __launch_bounds__(kGroupThreads, kGroupPerSm)
    k_group_place(uint32_t count, const uint32_t *vin, uint32_t *cursor, uint2 *out) {
    extern __shared__ uint2 stage[];         // kGroupTile entries in group order
    __shared__ uint32_t start[kGroups];      // a group's size, then its first place in stage
    __shared__ uint32_t shift[kGroups];      // its place in out less its place in stage
    __shared__ uint32_t wsum[kGroupThreads / 32];
    constexpr uint32_t kPer = kGroups / kGroupThreads;
    for (uint64_t base = (uint64_t)blockIdx.x * kGroupTile; base < count; base += (uint64_t)gridDim.x * kGroupTile) {
        const uint32_t here = count - base < kGroupTile ? (uint32_t)(count - base) : kGroupTile;
        for (uint32_t i = threadIdx.x; i < kGroups; i += kGroupThreads) start[i] = 0;
        __syncthreads();
        uint32_t v[kGroupItems], rank[kGroupItems];
#pragma unroll
        for (int k = 0; k < kGroupItems; ++k) {
            const uint32_t i = k * kGroupThreads + threadIdx.x;
            v[k] = i < here ? __ldcs(vin + base + i) : 0u;
        }
#pragma unroll
        for (int k = 0; k < kGroupItems; ++k) {
            const uint32_t i = k * kGroupThreads + threadIdx.x;
            rank[k] = i < here ? atomicAdd(&start[group_of(v[k])], 1u) : 0u;
        }
        __syncthreads();
        uint32_t size[kPer], sum = 0;
#pragma unroll
        for (uint32_t k = 0; k < kPer; ++k) sum += size[k] = start[threadIdx.x * kPer + k];
        uint32_t at = block_incl_scan<kGroupThreads / 32>(sum, wsum) - sum;
#pragma unroll
        for (uint32_t k = 0; k < kPer; ++k) {
            const uint32_t i = threadIdx.x * kPer + k;
            start[i] = at;
            if (size[k]) shift[i] = atomicAdd(&cursor[i], size[k]) - at;
            at += size[k];
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kGroupItems; ++k) {
            const uint32_t i = k * kGroupThreads + threadIdx.x;
            if (i < here) stage[start[group_of(v[k])] + rank[k]] = make_uint2(v[k], (uint32_t)base + i);
        }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < here; i += kGroupThreads) {
            const uint2 e = stage[i];
            __stcs(out + (shift[group_of(e.x)] + i), e);
        }
        __syncthreads();
    }
}

// resident blocks per SM, as the ungrouped samplers'
template <int RNG>
constexpr int group_blocks() { return RNG == kRngPhilox ? 5 : 6; }

// The samples of the entries in order, a thread each; Path-5 samples whose
// first pair of sigma draws collides are flagged in the (zeroed) deferral
// bitmap for the redraws.
template <int METHOD, int RNG>
__global__ void __launch_bounds__(kThreads, group_blocks<RNG>())
    k_sample_group(DevGraph g, uint64_t first, uint32_t count, uint64_t seed, const uint2 *entries,
                   uint64_t *sums) {
    constexpr int PM = kPmGroup;
    __shared__ uint8_t lut[kLut];
    __shared__ uint8_t lutc[METHOD == 3 ? 4096 : 1];
    __shared__ uint32_t hist[kWarps][kSlots];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint8_t *src = (METHOD == 0 || METHOD == 3) ? g_lut4 : g_lut5;
    const int lut_n = (METHOD == 0 || METHOD == 3) ? 64 : 1024;
    for (int i = threadIdx.x; i < lut_n; i += kThreads) lut[i] = src[i];
    if (METHOD == 3)
        for (int i = threadIdx.x; i < 4096; i += kThreads) lutc[i] = g_lutc[i];
    for (int i = threadIdx.x; i < kWarps * kSlots; i += kThreads) (&hist[0][0])[i] = 0;
    __syncthreads();
    const uint4 *vrec = METHOD == 3 ? g.mvert : g.vert;
    for (uint64_t t = (uint64_t)blockIdx.x * kDrawTile; t < count; t += (uint64_t)gridDim.x * kDrawTile) {
        for (uint32_t j = 0; j < kDrawTile; j += kThreads) {
            const uint64_t i = t + j + threadIdx.x;
            int cls = kSlots;   // no sample (tail) or deferred
            if (i < count) {
                const uint2 e = __ldcs(entries + i);
                const uint64_t s = first + e.y;
                const VertexPick pv = {e.x, ld4(vrec + e.x)};
                Sample sm;
                if (METHOD == 0) sm = rest_moss4<RNG, true, PM>(g, lut, seed, s, pv);
                else if (METHOD == 1) sm = rest_t5<RNG, true, PM>(g, lut, seed, s, pv);
                else if (METHOD == 2) sm = rest_path5<RNG, true, 0, PM>(g, lut, seed, s, pv);
                else sm = rest_min<RNG, true, PM>(g, lut, lutc, seed, s, pv);
                if (METHOD == 2 && sm.cls == kDeferred) atomicOr(g.defer + (e.y >> 5), 1u << (e.y & 31));
                else cls = METHOD == 3 ? min_slot(sm.cls, sm.v[4]) : sm.cls;
            }
            const uint32_t peers = __match_any_sync(0xffffffffu, cls);
            if (cls < kSlots && lane == __ffs(peers) - 1) atomicAdd(&hist[warp][cls], (uint32_t)__popc(peers));
        }
    }
    __syncthreads();
    add_sums<kWarps>(hist, sums);
}

uint64_t align256(uint64_t x) { return (x + 255) & ~255ull; }

// scratch of a call: the group cursors, the chunk's v and its entries
struct Scratch {
    uint32_t *cursor, *v;
    uint2 *entries;
};
uint64_t scratch_bytes(uint64_t chunk) { return align256(kGroups * 4) + align256(chunk * 4) + chunk * 8; }
Scratch carve(void *mem, uint64_t chunk) {
    uint8_t *p = static_cast<uint8_t *>(mem);
    Scratch w;
    w.cursor = reinterpret_cast<uint32_t *>(p);
    w.v = reinterpret_cast<uint32_t *>(p + align256(kGroups * 4));
    w.entries = reinterpret_cast<uint2 *>(p + align256(kGroups * 4) + align256(chunk * 4));
    return w;
}

template <int M, int RNG>
cudaError_t run_chunk(const DevGraph &g, uint64_t first, uint32_t len, uint64_t seed, const Scratch &w,
                      uint64_t *sums, int sms, int blocks, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(w.cursor, 0, kGroups * 4, s);
    if (e != cudaSuccess) return e;
    constexpr int smem = kGroupTile * sizeof(uint2);
    e = cudaFuncSetAttribute(k_group_place, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_group_draw<M, RNG><<<sms * kGroupPerSm, kGroupThreads, 0, s>>>(g, first, len, seed, w.v, w.cursor);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_group_scan<<<1, kGroups, 0, s>>>(w.cursor);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_group_place<<<sms * kGroupPerSm, kGroupThreads, smem, s>>>(len, w.v, w.cursor, w.entries);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (M == 2 && (e = cudaMemsetAsync(g.defer, 0, ((uint64_t)len + 31) / 32 * 4, s)) != cudaSuccess) return e;
    k_sample_group<M, RNG><<<blocks, kThreads, 0, s>>>(g, first, len, seed, w.entries, sums);
    return cudaGetLastError();
}

template <int RNG>
cudaError_t run_method(int method, const DevGraph &g, uint64_t first, uint32_t len, uint64_t seed, const Scratch &w,
                       uint64_t *sums, int sms, int blocks, cudaStream_t s) {
    switch (method) {
        case 0: return run_chunk<0, RNG>(g, first, len, seed, w, sums, sms, blocks, s);
        case 1: return run_chunk<1, RNG>(g, first, len, seed, w, sums, sms, blocks, s);
        case 2: return run_chunk<2, RNG>(g, first, len, seed, w, sums, sms, blocks, s);
        case 3: return run_chunk<3, RNG>(g, first, len, seed, w, sums, sms, blocks, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

void upload_luts_group(const uint8_t *lut4, const uint8_t *lut5, const uint8_t *lutc) {
    upload_luts_here(lut4, lut5, lutc);
}

// Which calls are grouped: those behind the filter (the tables exceed the
// L2; on the 1M-edge graph, whose tables fit it, grouping cost 6-18%) with
// enough ids to pay for the draw and placement passes and their scattered
// scratch.  What it gains grows with the tables; it gains least where few heavy
// vertices hold most draws (the table's heavy level has kStreamHeavy columns at
// most), as their lists stay in the L2 anyway, and in degree order, where those
// lists lie together besides.  Grouped / ungrouped time of MOSS-4, T-5, Path-5,
// MOSS-4Min (power-law graphs unless a mesh; entries):
//   input ids, few heavy    2^22 ids                 2^23                     2^26
//     4.4M               1.28 1.13 1.05 1.05      1.19 1.13 1.01 0.99      1.13 1.08 0.96 0.93
//     6.9M               1.17 1.03 0.96 1.01      1.06 1.01 0.89 0.96      0.97 0.99 0.83 0.94
//     9.0M               1.13 1.04 0.95 0.99      0.99 1.01 0.89 0.94      0.89 0.98 0.85 0.91
//     14M                0.97 0.95 0.83 0.93      0.84 0.90 0.78 0.88      0.74 0.88 0.72 0.84
//   input ids, others
//     4.7M (mesh)        0.98 0.92 0.90 0.97      0.87 0.85 0.84 0.89      0.85 0.82 0.82 0.85
//     16M                1.04 0.89 0.95 1.02      0.95 0.87 0.91 0.96      0.89 0.85 0.89 0.95
//     24M                0.94 0.95 0.82 0.92      0.84 0.92 0.76 0.84      0.76 0.89 0.71 0.81
//     67M                0.82 0.75 0.83 0.89      0.76 0.72 0.79 0.84      0.72 0.70 0.75 0.82
//   degree order            2^23                     2^24                     2^26
//     4.4M, few heavy    1.23 1.00 0.88 1.03      1.21 0.98 0.84 0.97      1.18 0.97 0.82 0.94
//     14M, few heavy     1.09 0.99 0.98 0.87      1.08 0.98 0.97 0.86      1.06 0.96 0.97 0.86
//     4.7M (mesh)        0.88 0.88 0.84 0.91      0.86 0.88 0.82 0.89      0.86 0.89 0.82 0.90
//     16M                1.08 0.97 1.04 0.98      1.04 0.96 1.04 0.97      1.01 0.94 1.04 0.98
//     24M                1.09 0.99 1.01 1.00      1.05 0.97 0.99 0.96      1.03 0.96 0.97 0.95
//     47M                1.02 0.99 0.90 0.94      0.98 0.98 0.86 0.92      0.95 0.97 0.84 0.91
//     67M                0.93 0.95 0.85 0.90      0.89 0.93 0.77 0.87      0.86 0.91 0.73 0.85
static bool groups(int method, const DevGraph &g, bool degree_order, uint64_t nnz, uint64_t count) {
    if (!g.hash || !g.filter) return false;
    const bool few_heavy = g.nheavy[method] != 0 && g.nheavy[method] <= kStreamHeavy;
    const bool many_heavy = g.nheavy[method] > kStreamHeavy;
    if (degree_order) {
        if (few_heavy && method != 2) return false;
        if (many_heavy && nnz < (method == 0 ? 1ull << 25 : method == 2 ? 1ull << 24 : 0)) return false;
        return count >= 1ull << 24;
    }
    if (few_heavy && method <= 1 && nnz < 1ull << 23) return false;
    const bool late = method == 0 ? nnz < 1ull << 24 : (few_heavy || method == 3) && nnz < 3ull << 22;
    return count >= (late ? 1ull << 23 : 1ull << 22);
}

uint64_t group_bytes(int method, const DevGraph &g, bool degree_order, uint64_t nnz, uint64_t count) {
    return groups(method, g, degree_order, nnz, count) ? scratch_bytes(std::min(count, kGroupChunk)) : 0;
}

cudaError_t launch_counts_grouped(int method, const DevGraph &g, uint64_t first, uint64_t count, uint64_t seed,
                                  uint64_t *sums, void *scratch, cudaStream_t s) {
    const bool philox = g.rng == kRngPhilox;
    const int sms = current_sms(), blocks = sms * (philox ? group_blocks<kRngPhilox>() : group_blocks<kRngSplitMix>());
    const uint64_t chunk = std::min(count, kGroupChunk);
    const Scratch w = carve(scratch, chunk);
    cudaError_t e = cudaSuccess;
    for (uint64_t c0 = 0; e == cudaSuccess && c0 < count; c0 += chunk) {
        const uint32_t len = (uint32_t)std::min(chunk, count - c0);
        e = philox ? run_method<kRngPhilox>(method, g, first + c0, len, seed, w, sums, sms, blocks, s)
                   : run_method<kRngSplitMix>(method, g, first + c0, len, seed, w, sums, sms, blocks, s);
        if (e == cudaSuccess && method == 2) e = launch_redraws(g, first + c0, len, seed, sums, nullptr, nullptr, s);
    }
    return e;
}

}  // namespace moss
