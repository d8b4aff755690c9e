// moss_min.cu -- the MOSS-4Min tables (Sec. 4.2) on the device.
//
// The total order of Sec. 3.2 puts x above y when d_x > d_y, or d_x = d_y and
// x > y; the 64-bit key (d_x << 32) | x orders vertices exactly that way.
// N_{u,v} = {x in N_u : x above v}, d_{u,v} = |N_{u,v}|.  Every list N_v is
// stored sorted by that key, highest first (rlist), so N_{v,u} is its first
// d_{v,u} entries and d_{v,u} is the position of u in it:
//   * lists of at most 128 entries: a group of lanes or a warp per list, each
//     entry's rank is the count of keys above its own;
//   * lists of at most kTile entries: a block per list, merge sort in shared
//     memory, each key's list position moving with it;
//   * longer lists: a block per list sorts tiles of kTile keys in shared
//     memory, then merges runs pairwise in global memory.
// A merge places each key by one binary search in the partner run (keys are
// distinct).
// Then per slot (v -> u): u, d_u, off_u, d_{v,u} and d_{u,v} (the rank of the
// twin slot); per list: Gamma-check_v = sum_u d_{v,u} d_{u,v} and the alias
// table of sigma-check^(v) (eq. 3) -- the parallel closed form of the sweep
// used for sigma^(v) in moss_tables.cu, here in 128-bit arithmetic since
// q_j = w_j d_v can exceed 2^64; the exact total Gamma-check; and the vertex
// alias table of pi-check through the seed-table kernels.
#include <algorithm>
#include <atomic>

#include "moss_alias.cuh"
#include "moss_internal.cuh"

namespace moss {

namespace {

constexpr int kWarp = 32;
constexpr uint32_t kTile = 4096;      // keys sorted per shared-memory pass
constexpr int kSortThreads = 1024;
constexpr int kListThreads = 256;
constexpr uint32_t kWarpKeys = 4;     // k_rank_warp: lists up to 128 entries
constexpr uint32_t kLongList = 256;   // longer lists: k_min_alias_long, a block per list

__device__ __forceinline__ uint64_t order_key(uint32_t x, uint32_t dx) { return ((uint64_t)dx << 32) | x; }

// lists of at most kWarpKeys * 32 entries: an entry's rank is the number of
// keys above its own, counted against every key of the list broadcast by
// shuffles.  Short lists by groups of lanes, an entry per lane; longer ones a
// warp each, lane l holding entries l, l + 32, ...
template <int TILE>
__global__ void __launch_bounds__(kListThreads) k_rank_warp(uint32_t n, const uint4 *__restrict__ vert,
                                                           const uint32_t *__restrict__ col, uint2 *rlist,
                                                           uint32_t *rank) {
    const int lane = threadIdx.x & 31;
    auto small = [&](auto G, uint32_t, uint4 vr, uint32_t i, bool valid) {
        constexpr int g = decltype(G)::value;
        uint32_t x = 0, dx = 0, r = 0;
        if (valid) {
            x = col[vr.x + i];
            dx = vert[x].y;
        }
        const uint64_t key = order_key(x, dx);   // 0, below every real key, where there is no entry
#pragma unroll 8
        for (int j = 0; j < g; ++j) r += __shfl_sync(0xffffffffu, key, j, g) > key;
        if (valid) {
            rlist[vr.x + r] = make_uint2(x, dx);
            rank[vr.x + i] = r;
        }
    };
    auto large = [&](uint32_t, uint4 vr) {
        const uint32_t o = vr.x, d = vr.y;
        if (d > kWarpKeys * (uint32_t)kWarp) return;   // k_rank_block, k_rank_long
        const int rounds = (int)((d + kWarp - 1) / kWarp);
        uint32_t x[kWarpKeys], dx[kWarpKeys], r[kWarpKeys];
        uint64_t key[kWarpKeys];
#pragma unroll
        for (int k = 0; k < kWarpKeys; ++k) {
            const uint32_t i = k * kWarp + lane;
            x[k] = dx[k] = r[k] = 0;
            key[k] = 0;                               // below every real key (d_x >= 1)
            if (i < d) {
                x[k] = col[o + i];
                dx[k] = vert[x[k]].y;
                key[k] = order_key(x[k], dx[k]);
            }
        }
#pragma unroll
        for (int kk = 0; kk < kWarpKeys; ++kk) {
            if (kk >= rounds) break;                  // warp-uniform
            const int m = min((int)d - kk * kWarp, kWarp);
            for (int j = 0; j < m; ++j) {
                const uint64_t other = __shfl_sync(0xffffffffu, key[kk], j);
#pragma unroll
                for (int k = 0; k < kWarpKeys; ++k)
                    if (k < rounds) r[k] += other > key[k];   // warp-uniform
            }
        }
#pragma unroll
        for (int k = 0; k < kWarpKeys; ++k) {
            const uint32_t i = k * kWarp + lane;
            if (i < d) {
                rlist[o + r[k]] = make_uint2(x[k], dx[k]);
                rank[o + i] = r[k];
            }
        }
    };
    for_lists<TILE>(whole_grid(), n, vert, small, [](uint32_t, uint4) {}, large);
}

// Keys of col[o + base, o + base + len) sorted highest first, each with its
// position in the list from base: runs of 32 ranked by counting within a warp,
// then merged pairwise between the two halves of shared memory, every key
// placed by one binary search -- 35 dependent steps for 1,000 keys, where
// counting against the whole list took 1,000 and a bitonic sort 55 stages with
// a barrier each (lists of 129..1,024 entries of the 7.9M-edge graph 370 -> 108
// us, of the 1M-edge graph 116 -> 33).  k and id hold 2 MOST entries; returns the offset of the
// sorted half.  The block calls it together.
template <int THREADS, uint32_t MOST>
__device__ uint32_t sort_keys(const uint4 *vert, const uint32_t *col, uint32_t o, uint32_t base, uint32_t len,
                              uint64_t *k, uint16_t *id) {
    const int lane = threadIdx.x & 31;
    for (uint32_t i0 = threadIdx.x & ~31u; i0 < len; i0 += THREADS) {   // warp-uniform
        const uint32_t i = i0 + lane;
        uint64_t key = 0;   // below every real key (d_x >= 1)
        if (i < len) {
            const uint32_t x = col[o + base + i];
            key = order_key(x, vert[x].y);
        }
        uint32_t r = 0;
#pragma unroll 8
        for (int j = 0; j < kWarp; ++j) r += __shfl_sync(0xffffffffu, key, j) > key;
        if (i < len) {
            k[i0 + r] = key;
            id[i0 + r] = (uint16_t)i;
        }
    }
    __syncthreads();
    uint32_t src = 0, dst = MOST;
    for (uint32_t lg = 5; (1u << lg) < len; ++lg) {
        const uint32_t L = 1u << lg;
        for (uint32_t i = threadIdx.x; i < len; i += THREADS) {
            const uint64_t key = k[src + i];
            const uint32_t run = i >> lg, ps = (run ^ 1u) << lg;
            uint32_t lo = ps, n = ps < len ? min(L, len - ps) : 0;   // partner keys above key
            while (n > 0) {
                const uint32_t half = n >> 1;
                if (k[src + lo + half] > key) {
                    lo += half + 1;
                    n -= half + 1;
                } else {
                    n = half;
                }
            }
            const uint32_t at = dst + ((run & ~1u) << lg) + (i & (L - 1u)) + (lo - ps);
            k[at] = key;
            id[at] = id[src + i];
        }
        __syncthreads();
        const uint32_t t = src;
        src = dst;
        dst = t;
    }
    return src;
}

// lists of kWarpKeys * 32 + 1 .. kBlockList entries, a block each
constexpr uint32_t kBlockList = 1024;
constexpr int kBlockThreads = 256;

__global__ void __launch_bounds__(kBlockThreads) k_rank_block(uint32_t n, const uint4 *__restrict__ vert,
                                                             const uint32_t *__restrict__ col, uint2 *rlist,
                                                             uint32_t *rank) {
    __shared__ uint64_t k[2 * kBlockList];
    __shared__ uint16_t id[2 * kBlockList];
    for_each_vertex<kBlockThreads, kWarp>(
        whole_grid(), n, vert, [](uint4 vr) { return vr.y > kWarpKeys * (uint32_t)kWarp && vr.y <= kBlockList; },
        [&](uint32_t v) {
            const uint4 vr = vert[v];
            const uint32_t o = vr.x, d = vr.y;
            const uint32_t at = sort_keys<kBlockThreads, kBlockList>(vert, col, o, 0, d, k, id);
            for (uint32_t q = threadIdx.x; q < d; q += kBlockThreads) {
                const uint64_t key = k[at + q];
                rlist[o + q] = make_uint2((uint32_t)key, (uint32_t)(key >> 32));
                rank[o + id[at + q]] = q;
            }
            __syncthreads();   // k and id are refilled for the next list
        });
}

// lists longer than kBlockList: up to kTile entries sorted in shared memory;
// longer ones by tiles into a[], then runs of length L merged pairwise between
// a[] and b[] until one run is left
constexpr size_t kSortBytes = (size_t)2 * kTile * (sizeof(uint64_t) + sizeof(uint16_t));
__global__ void __launch_bounds__(kSortThreads) k_rank_long(uint32_t n, const uint4 *__restrict__ vert,
                                                           const uint32_t *__restrict__ col, uint64_t *a,
                                                           uint64_t *b, uint32_t *ia, uint32_t *ib, uint2 *rlist,
                                                           uint32_t *rank) {
    extern __shared__ uint64_t k[];   // 2 kTile keys, then their positions
    uint16_t *id = reinterpret_cast<uint16_t *>(k + 2 * kTile);
    for_each_vertex<kSortThreads>(whole_grid(), n, vert, [](uint4 vr) { return vr.y > kBlockList; }, [&](uint32_t v) {
        const uint4 vr = vert[v];
        const uint32_t o = vr.x, d = vr.y;
        if (d <= kTile) {
            const uint32_t at = sort_keys<kSortThreads, kTile>(vert, col, o, 0, d, k, id);
            for (uint32_t q = threadIdx.x; q < d; q += kSortThreads) {
                const uint64_t key = k[at + q];
                rlist[o + q] = make_uint2((uint32_t)key, (uint32_t)(key >> 32));
                rank[o + id[at + q]] = q;
            }
            __syncthreads();   // k and id are refilled for the next list
            return;
        }
        for (uint32_t base = 0; base < d; base += kTile) {
            const uint32_t len = min(kTile, d - base);
            const uint32_t at = sort_keys<kSortThreads, kTile>(vert, col, o, base, len, k, id);
            for (uint32_t i = threadIdx.x; i < len; i += blockDim.x) {
                a[(uint64_t)o + base + i] = k[at + i];
                ia[(uint64_t)o + base + i] = base + id[at + i];
            }
            __syncthreads();
        }
        uint64_t *src = a, *dst = b;
        uint32_t *isrc = ia, *idst = ib;
        for (uint64_t L = kTile; L < d; L <<= 1) {
            for (uint32_t i = threadIdx.x; i < d; i += blockDim.x) {
                const uint64_t run = i / L, start = run * L;
                const uint64_t ps = (run ^ 1) * L;               // the partner run
                const uint64_t ms = (run & ~1ull) * L;           // where the pair's merge starts
                const uint64_t key = src[(uint64_t)o + i];
                // partner keys above key (the partner run is sorted highest first)
                uint64_t lo = ps, len = ps < d ? min(ps + L, (uint64_t)d) - ps : 0;
                while (len > 0) {
                    const uint64_t half = len >> 1;
                    if (src[(uint64_t)o + lo + half] > key) {
                        lo += half + 1;
                        len -= half + 1;
                    } else {
                        len = half;
                    }
                }
                const uint64_t above = ps < d ? lo - ps : 0;
                dst[(uint64_t)o + ms + (i - start) + above] = key;
                idst[(uint64_t)o + ms + (i - start) + above] = isrc[(uint64_t)o + i];
            }
            __syncthreads();
            uint64_t *t = src;
            src = dst;
            dst = t;
            uint32_t *it = isrc;
            isrc = idst;
            idst = it;
        }
        for (uint32_t q = threadIdx.x; q < d; q += blockDim.x) {
            const uint64_t key = src[(uint64_t)o + q];
            rlist[o + q] = make_uint2((uint32_t)key, (uint32_t)(key >> 32));
            rank[o + isrc[(uint64_t)o + q]] = q;
        }
        __syncthreads();
    });
}

// per slot p (v -> u) of a list above kShortList entries: {0, 0, 0, u} and
// {off_u, d_u, d_{v,u}, d_{u,v}} (k_min_alias forms the short lists' itself)
__global__ void k_min_slots(uint64_t nnz, const uint4 *__restrict__ vert, const uint32_t *__restrict__ col,
                            const uint32_t *__restrict__ owner, const uint32_t *__restrict__ twin,
                            const uint32_t *__restrict__ rank, uint4 *mslot) {
    for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < nnz; p += (uint64_t)gridDim.x * blockDim.x) {
        if (vert[owner[p]].y <= kShortList) continue;
        const uint32_t u = col[p];
        const uint4 ur = vert[u];
        mslot[2 * p] = make_uint4(0u, 0u, 0u, u);
        mslot[2 * p + 1] = make_uint4(ur.x, ur.y, rank[p], rank[(uint64_t)ur.x + twin[p]]);
    }
}

// (a read-only load: the alias passes write only the first half of each record)
__device__ __forceinline__ uint64_t min_weight(const uint4 *mslot, uint64_t p) {
    const uint4 r = __ldg(mslot + 2 * p + 1);
    return (uint64_t)r.z * r.w;   // d_{v,u} d_{u,v}
}

// threshold and alias position into the first half of a slot record
__device__ __forceinline__ void set_min_alias(uint32_t *m32, uint64_t p, uint64_t thr, uint32_t alias) {
    *reinterpret_cast<uint2 *>(m32 + 8 * p) = make_uint2((uint32_t)thr, (uint32_t)(thr >> 32));
    m32[8 * p + 2] = alias;
}

// a list each: Gamma-check_v, mvert, and the alias table of sigma-check^(v)
// over capacity W = Gamma-check_v.  Lights (q_j = w_j d < W) carry the deficit
// W - q_j, heavies the excess q_j - W, both in list order; with A_i the
// exclusive prefix of the light deficits and P_k the inclusive prefix of the
// heavy excesses: light i keeps q_i and aliases heavy min{k : P_k >= A_i};
// heavy k keeps W + P_k - A_{i'} (i' = min{i : A_i > P_k}) and aliases heavy
// k+1, or keeps W when P_k is the total.  The split (idx, pre) of the list
// being built lives in the warp's share of shared memory.
// alias table of sigma-check^(v) for the list at o of d <= kLongList entries
// with total W > 0, one warp; pre and idx hold kLongList entries
__device__ void warp_min_alias(const uint4 *mslot, uint32_t *m32, uint32_t o, uint32_t d, uint64_t W, uint64_t *pre,
                               uint32_t *idx) {
    typedef uint64_t T;
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    // pass 1: lights to the front, heavies to the back, with their prefixes
    uint32_t nl = 0, nh = 0;
    T Arun = 0, Prun = 0;
    for (uint32_t base = 0; base < d; base += kWarp) {
        const uint32_t j = base + lane;
        const bool valid = j < d;
        const T q = valid ? (T)min_weight(mslot, (uint64_t)o + j) * (T)d : (T)0;
        const bool light = valid && q < W;
        const uint32_t lmask = __ballot_sync(0xffffffffu, light);
        const uint32_t hmask = __ballot_sync(0xffffffffu, valid && !light);
        const T D = light ? (T)W - q : (T)0;
        const T E = valid && !light ? q - (T)W : (T)0;
        const T Dincl = warp_incl_scan64(D, lane);
        const T Eincl = warp_incl_scan64(E, lane);
        if (light) {
            const uint32_t r = nl + __popc(lmask & below);
            idx[r] = j;
            pre[r] = Arun + Dincl - D;          // exclusive A_i
        } else if (valid) {
            const uint32_t r = nh + __popc(hmask & below);
            idx[d - 1 - r] = j;
            pre[d - 1 - r] = Prun + Eincl;      // inclusive P_k
        }
        nl += __popc(lmask);
        nh += __popc(hmask);
        Arun += __shfl_sync(0xffffffffu, Dincl, 31);
        Prun += __shfl_sync(0xffffffffu, Eincl, 31);
    }
    __syncwarp();
    const T Ptot = Prun;   // == Arun
    const uint64_t ob = o;
    // pass 2: each lane merges a contiguous run of lights, then of heavies
    {
        const uint32_t cl = (nl + kWarp - 1) / kWarp;
        const uint32_t i0 = lane * cl, i1 = min(nl, i0 + cl);
        if (i0 < i1) {
            const T A0 = pre[i0];
            uint32_t k = 0, len = nh;   // first heavy with P_k >= A
            while (len > 0) {
                const uint32_t half = len >> 1;
                if (pre[d - 1 - (k + half)] < A0) {
                    k += half + 1;
                    len -= half + 1;
                } else {
                    len = half;
                }
            }
            for (uint32_t i = i0; i < i1; ++i) {
                const T A = pre[i];
                while (pre[d - 1 - k] < A) ++k;
                const uint32_t j = idx[i];
                const uint64_t thr = min_weight(mslot, ob + j) * (uint64_t)d;   // q_j < W < 2^64
                set_min_alias(m32, ob + j, thr, idx[d - 1 - k]);
            }
        }
    }
    {
        const uint32_t ch = (nh + kWarp - 1) / kWarp;
        const uint32_t k0 = lane * ch, k1 = min(nh, k0 + ch);
        if (k0 < k1) {
            const T P0 = pre[d - 1 - k0];
            uint32_t i = 0, len = nl;   // first light with A_i > P_k
            while (len > 0) {
                const uint32_t half = len >> 1;
                if (pre[i + half] <= P0) {
                    i += half + 1;
                    len -= half + 1;
                } else {
                    len = half;
                }
            }
            for (uint32_t k = k0; k < k1; ++k) {
                const T Pk = pre[d - 1 - k];
                while (i < nl && pre[i] <= Pk) ++i;
                const uint32_t j = idx[d - 1 - k];
                uint64_t thr;
                uint32_t alias;
                if (Pk < Ptot) {
                    const T Ai = i < nl ? pre[i] : Ptot;
                    thr = (uint64_t)((T)W + Pk - Ai);
                    alias = idx[d - 1 - (k + 1)];
                } else {
                    thr = W;
                    alias = j;
                }
                set_min_alias(m32, ob + j, thr, alias);
            }
        }
    }
}

// A pick record (moss_internal.cuh) from a slot's record (a0 its threshold
// and u, a1 its fields) and its alias position's u and fields; narrow lists
// (Gamma-check_v < 2^32) whose fields fit 16 bits are marked usable.
__device__ __forceinline__ void store_pick(uint4 *mpick, uint64_t p, bool narrow, uint4 a0, uint4 a1, uint32_t bu,
                                           uint4 b1) {
    constexpr uint32_t kNarrow = 0xffffu;   // fields below this fit a half word
    const bool fits = narrow && a1.y < kNarrow && a1.z < kNarrow && a1.w < kNarrow && b1.y < kNarrow &&
                      b1.z < kNarrow && b1.w < kNarrow;
    mpick[2 * p] = make_uint4(a0.x, a0.w, a1.x, a1.z | a1.w << 16);
    mpick[2 * p + 1] = make_uint4(bu, b1.x, b1.z | b1.w << 16, fits ? (a1.y | b1.y << 16) : kSlotHub);
}

// Short lists (kShortList) by groups of lanes, in one pass from the ranks to
// the finished slot and pick records: d_{v,u} and d_{u,v}, Gamma-check_v, the
// alias, and the alias's fields from its lane.  Longer ones a warp each, from
// the slot records k_min_slots left; their pick records are k_min_pick's.
template <int TILE>
__global__ void __launch_bounds__(kListThreads) k_min_alias(uint32_t n, const uint4 *__restrict__ vert,
                                                           const uint32_t *__restrict__ col,
                                                           const uint32_t *__restrict__ twin,
                                                           const uint32_t *__restrict__ rank, uint4 *mslot,
                                                           uint4 *mpick, uint4 *mvert, u128 *gmin, u128 *partials) {
    __shared__ uint64_t s_pre[kListThreads / kWarp][kLongList];
    __shared__ uint32_t s_idx[kListThreads / kWarp][kLongList];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    uint32_t *m32 = reinterpret_cast<uint32_t *>(mslot);
    u128 total = 0;   // of the lists whose record this lane left
    auto leave = [&](uint32_t v, uint4 vr, uint64_t W) {
        mvert[v] = make_uint4(vr.x, vr.y, (uint32_t)W, (uint32_t)(W >> 32));
        gmin[v] = W;
        total += W;
    };
    auto small = [&](auto G, uint32_t v, uint4 vr, uint32_t j, bool valid) {
        constexpr int g = decltype(G)::value;
        const uint64_t p = (uint64_t)vr.x + j;
        uint32_t u = 0;
        uint4 f = make_uint4(0u, 0u, 0u, 0u);   // {off_u, d_u, d_{v,u}, d_{u,v}}
        if (valid) {
            u = col[p];
            const uint4 ur = vert[u];
            f = make_uint4(ur.x, ur.y, rank[p], rank[(uint64_t)ur.x + twin[p]]);
        }
        const uint64_t w = (uint64_t)f.z * f.w;
        const uint64_t W = __shfl_sync(0xffffffffu, group_scan<g>(w, j), g - 1, g);
        uint64_t thr;
        uint32_t alias;
        group_alias<g>(valid, w * vr.y, W, j, thr, alias);   // w d < 2^32 2^5 2^5
        if (W == 0) {   // never drawn: keep every column
            thr = 0;
            alias = j;
        }
        const uint32_t a = alias & (g - 1);
        uint4 b;
        b.x = __shfl_sync(0xffffffffu, f.x, a, g);
        b.y = __shfl_sync(0xffffffffu, f.y, a, g);
        b.z = __shfl_sync(0xffffffffu, f.z, a, g);
        b.w = __shfl_sync(0xffffffffu, f.w, a, g);
        const uint32_t bu = __shfl_sync(0xffffffffu, u, a, g);
        if (valid) {
            const uint4 head = make_uint4((uint32_t)thr, (uint32_t)(thr >> 32), alias, u);
            mslot[2 * p] = head;
            mslot[2 * p + 1] = f;
            store_pick(mpick, p, W >> 32 == 0, head, f, bu, b);
            if (j == 0) leave(v, vr, W);
        }
    };
    auto large = [&](uint32_t v, uint4 vr) {
        const uint32_t o = vr.x, d = vr.y;
        uint64_t W = 0;
        for (uint32_t j = lane; j < d; j += kWarp) W += min_weight(mslot, (uint64_t)o + j);
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) W += __shfl_down_sync(0xffffffffu, W, s);
        W = __shfl_sync(0xffffffffu, W, 0);
        if (lane == 0) leave(v, vr, W);
        if (d > kLongList && W != 0) return;   // k_min_alias_long
        if (W == 0) {
            for (uint32_t j = lane; j < d; j += kWarp) set_min_alias(m32, (uint64_t)o + j, 0, j);
            return;
        }
        // W = sum d_{v,u} d_{u,v} < d d 2^32, so q = w d <= W d < 2^56
        warp_min_alias(mslot, m32, o, d, W, s_pre[warp], s_idx[warp]);
        __syncwarp();
    };
    for_lists<TILE>(whole_grid(), n, vert, small, [&](uint32_t v, uint4 vr) { leave(v, vr, 0); }, large);
    total = warp_sum128(total);
    // block share of Gamma-check
    __shared__ u128 sh[kListThreads / kWarp];
    if (lane == 0) sh[warp] = total;
    __syncthreads();
    if (threadIdx.x == 0) {
        u128 s = 0;
        for (int w = 0; w < wpb; ++w) s += sh[w];
        partials[blockIdx.x] = s;
    }
}

// the alias tables of lists longer than kLongList, a block per list, 256
// threads up to kHubList entries and 1,024 above (moss_alias.cuh); each block
// forms Gamma-check_v itself (the same integer sum k_min_alias writes into
// mvert), so the kernels may run side by side.  The split of a list that fits
// the smem_bytes of dynamic shared memory is kept there, of a longer one in
// its range of the global scratch (idx, pre).  The arithmetic is 64-bit where
// d Gamma-check_v fits (always below 2^16 entries: d_{v,u} < d, d_{u,v} < d_u
// and S_v < 2^32), else 128-bit.
constexpr uint32_t kMidBytes = kHubList * (sizeof(uint64_t) + sizeof(uint32_t));
constexpr uint32_t kHubBytes = kHubSmemList * (sizeof(uint64_t) + sizeof(uint32_t));

template <typename T, int NT>
__device__ __forceinline__ void long_min_alias(const uint4 *mslot, uint32_t *m32, uint32_t o, uint32_t d, uint64_t W,
                                               u128 *smem, uint32_t smem_bytes, uint32_t *idx, u128 *pre) {
    const bool fits = d <= smem_bytes / (sizeof(T) + sizeof(uint32_t));
    T *s_pre = reinterpret_cast<T *>(smem);
    block_alias<T, NT>(
        d, (T)W, [&](uint32_t j) { return (T)min_weight(mslot, (uint64_t)o + j); },
        fits ? reinterpret_cast<uint32_t *>(s_pre + d) : idx + o, fits ? s_pre : reinterpret_cast<T *>(pre + o),
        [&](uint32_t j, T thr, uint32_t alias) { set_min_alias(m32, (uint64_t)o + j, (uint64_t)thr, alias); });
}

template <int NT, int CH, uint32_t LO, uint32_t HI>
__global__ void __launch_bounds__(NT) k_min_alias_long(uint32_t n, const uint4 *__restrict__ vert, uint4 *mslot,
                                                      uint32_t *idx, u128 *pre, uint32_t smem_bytes) {
    extern __shared__ u128 s_split[];   // the prefixes, then the positions
    __shared__ uint64_t s_w[NT / kWarp];
    uint32_t *m32 = reinterpret_cast<uint32_t *>(mslot);
    for_each_vertex<NT, CH>(
        whole_grid(), n, vert, [](uint4 vr) { return vr.y > LO && vr.y <= HI; },
        [&](uint32_t v) {
            const uint4 vr = vert[v];
            const uint32_t o = vr.x, d = vr.y;
            uint64_t W = 0;
            for (uint32_t j = threadIdx.x; j < d; j += NT) W += min_weight(mslot, (uint64_t)o + j);
#pragma unroll
            for (int sft = 16; sft > 0; sft >>= 1) W += __shfl_down_sync(0xffffffffu, W, sft);
            if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = W;
            __syncthreads();
            W = 0;
            for (int w = 0; w < NT / kWarp; ++w) W += s_w[w];
            __syncthreads();   // s_w is refilled for the next list
            if (W == 0) return;   // block-uniform: k_min_alias keeps every column
            if (W <= ~0ull / d) long_min_alias<uint64_t, NT>(mslot, m32, o, d, W, s_split, smem_bytes, idx, pre);
            else long_min_alias<u128, NT>(mslot, m32, o, d, W, s_split, smem_bytes, idx, pre);
        });
}
const auto k_min_alias_mid = k_min_alias_long<kListThreads, kWarp, kLongList, kHubList>;
const auto k_min_alias_hub = k_min_alias_long<kHubThreads, kHubThreads, kHubList, 0xffffffffu>;

__global__ void k_min_total(const u128 *partials, int blocks, DevTotals *tot) {
    const int lane = threadIdx.x;   // one warp
    u128 s = 0;
    for (int b = lane; b < blocks; b += kWarp) s += partials[b];
    s = warp_sum128(s);
    if (lane == 0) tot->gamma[3] = s;
}

unsigned grid_for(uint64_t items, int per_block, int cap_per_sm) {
    const int sms = current_sms();
    uint64_t b = (items + per_block - 1) / per_block;
    const uint64_t cap = (uint64_t)sms * cap_per_sm;
    if (b > cap) b = cap;
    return (unsigned)(b ? b : 1);
}

// blocks of k_min_alias (and rows of its partial totals)
unsigned alias_grid(uint32_t n) {
    unsigned b = 0;
    with_tile(n, [&](auto T) { b = tile_blocks(n, decltype(T)::value, kListThreads, current_sms(), 8); });
    return b;
}

struct MinScratch {
    uint32_t *rank;   // nnz
    uint64_t *a, *b;  // nnz each (long-list merges), then reused as u128 prefixes
    uint32_t *ia, *ib;  // nnz each: list positions of the keys in a, b, then the alias split order
    u128 *partials;
    void *seed;       // vertex alias scratch
    uint64_t bytes;
};

// per slot p of a list above kShortList entries: its pick record from p's
// mslot record and its alias position's
__global__ void k_min_pick(uint64_t nnz, const uint32_t *__restrict__ owner, const uint4 *__restrict__ mvert,
                           const uint4 *__restrict__ mslot, uint4 *mpick) {
    for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < nnz; p += (uint64_t)gridDim.x * blockDim.x) {
        const uint4 mv = mvert[owner[p]];
        if (mv.y <= kShortList) continue;
        const uint4 a0 = mslot[2 * p], a1 = mslot[2 * p + 1];
        const uint64_t ap = (uint64_t)mv.x + a0.z;
        store_pick(mpick, p, mv.w == 0, a0, a1, mslot[2 * ap].w, mslot[2 * ap + 1]);
    }
}

MinScratch carve(void *base, uint32_t n, uint64_t nnz) {
    MinScratch m{};
    uint8_t *p = static_cast<uint8_t *>(base);
    uint64_t off = 0;
    auto take = [&](uint64_t bytes) {
        off = (off + 255) & ~255ULL;
        uint8_t *r = p ? p + off : nullptr;
        off += bytes ? bytes : 1;
        return r;
    };
    const unsigned alias_blocks = alias_grid(n);
    m.rank = reinterpret_cast<uint32_t *>(take(nnz * 4));
    m.a = reinterpret_cast<uint64_t *>(take(nnz * 16));
    m.b = m.a ? m.a + nnz : nullptr;
    m.ia = reinterpret_cast<uint32_t *>(take(nnz * 8));
    m.ib = m.ia ? m.ia + nnz : nullptr;
    m.partials = reinterpret_cast<u128 *>(take((uint64_t)alias_blocks * 16));
    m.seed = take(seed_scratch_bytes(n));
    m.bytes = off;
    return m;
}

}  // namespace

uint64_t min_scratch_bytes(uint32_t n, uint64_t nnz) { return carve(nullptr, n, nnz).bytes; }

cudaError_t launch_min_tables(uint32_t n, uint64_t nnz, uint32_t d_max, const uint4 *vert, const uint32_t *col,
                              const uint32_t *owner, const uint32_t *twin, uint4 *mvert, uint4 *mslot, uint4 *mpick,
                              uint2 *rlist, u128 *gmin, uint4 *seed_min, DevTotals *tot, void *scratch,
                              uint32_t *flags, int split, cudaStream_t s, const AuxStreams *aux) {
    // With helper streams h0, h1 (aux->a[3], a[4]): the three sort tiers side
    // by side (disjoint lists), then the slot records on s; the short-list
    // alias tables, the total and the vertex table on s, beside the long-list
    // alias tables and (once the short ones are done) the pick records on h0.
    const MinScratch m = carve(scratch, n, nnz);
    cudaStream_t h0 = aux ? aux->a[3] : s, h1 = aux ? aux->a[4] : s;
    cudaError_t e = cudaSuccess, eh = cudaSuccess;
    static std::atomic<bool> attr_set[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !attr_set[dev].load(std::memory_order_relaxed)) {
        e = cudaFuncSetAttribute(k_min_alias_hub, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHubBytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_rank_long, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSortBytes);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev].store(true, std::memory_order_relaxed);
    }
    auto fork = [&](int k) {   // h0 (and h1) wait for what is queued on s
        if (!aux) return;
        if (e == cudaSuccess) e = cudaEventRecord(aux->sub_fork, s);
        for (int i = 0; i < k && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(aux->a[3 + i], aux->sub_fork, 0);
    };
    auto join = [&](int k) {   // s waits for h0 (and h1); done even after an error
        if (!aux) return;
        for (int i = 0; i < k; ++i) {
            cudaError_t ei = cudaEventRecord(aux->sub_done[i], aux->a[3 + i]);
            if (ei == cudaSuccess) ei = cudaStreamWaitEvent(s, aux->sub_done[i], 0);
            if (e == cudaSuccess) e = ei;
        }
    };
    if (nnz) {
        fork(2);
        if (e == cudaSuccess) {
            const unsigned chunks = (unsigned)(((uint64_t)n + kWarp - 1) / kWarp);
            if (d_max > kWarpKeys * kWarp) k_rank_block<<<chunks, kBlockThreads, 0, h0>>>(n, vert, col, rlist, m.rank);
            eh = cudaGetLastError();
            if (d_max > kBlockList)
                k_rank_long<<<grid_for((uint64_t)n, kSortThreads, 2), kSortThreads, kSortBytes, h1>>>(
                    n, vert, col, m.a, m.b, m.ia, m.ib, rlist, m.rank);
            if (eh == cudaSuccess) eh = cudaGetLastError();
            with_tile(n, [&](auto T) {
                constexpr int tile = decltype(T)::value;
                k_rank_warp<tile><<<tile_blocks(n, tile, kListThreads, current_sms(), 8), kListThreads, 0, s>>>(
                    n, vert, col, rlist, m.rank);
            });
            e = cudaGetLastError();
        }
        join(2);
        if (e == cudaSuccess) e = eh;
        if (e != cudaSuccess) return e;
        k_min_slots<<<grid_for(nnz, 256, 16), 256, 0, s>>>(nnz, vert, col, owner, twin, m.rank, mslot);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const unsigned ab = alias_grid(n);
    fork(1);
    if (e != cudaSuccess) return e;
    // the merges' scratch is dead now: the long-list kernel keeps its split
    // order in ia[] and its prefixes in a[], b[] (k_min_alias still reads the ranks)
    const unsigned chunks = (unsigned)(((uint64_t)n + kWarp - 1) / kWarp);
    u128 *pre = reinterpret_cast<u128 *>(m.a);
    if (d_max > kHubList) {
        const uint32_t bytes = std::min<uint64_t>(kHubBytes, (uint64_t)d_max * (sizeof(uint64_t) + sizeof(uint32_t)));
        k_min_alias_hub<<<hub_blocks(n), kHubThreads, bytes, h0>>>(n, vert, mslot, m.ia, pre, bytes);
    }
    if (d_max > kLongList)
        k_min_alias_mid<<<chunks, kListThreads, kMidBytes, h0>>>(n, vert, mslot, m.ia, pre, kMidBytes);
    eh = cudaGetLastError();
    with_tile(n, [&](auto T) {
        k_min_alias<decltype(T)::value><<<ab, kListThreads, 0, s>>>(n, vert, col, twin, m.rank, mslot, mpick, mvert,
                                                                    gmin, m.partials);
    });
    e = cudaGetLastError();
    if (aux && e == cudaSuccess) {   // the pick records need both alias passes and mvert
        e = cudaEventRecord(aux->sub_mid, s);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(h0, aux->sub_mid, 0);
    }
    if (e == cudaSuccess && eh == cudaSuccess && nnz) {
        k_min_pick<<<grid_for(nnz, 256, 16), 256, 0, h0>>>(nnz, owner, mvert, mslot, mpick);
        eh = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        k_min_total<<<1, kWarp, 0, s>>>(m.partials, (int)ab, tot);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        const int which[1] = {3};
        u128 *w[1] = {gmin};
        uint4 *sd[1] = {seed_min};
        const uint4 *vr[1] = {mvert};
        e = launch_seed_alias(n, tot, 1, which, w, sd, vr, m.seed, flags, split, s);
    }
    join(1);
    return e != cudaSuccess ? e : eh;
}

}  // namespace moss
