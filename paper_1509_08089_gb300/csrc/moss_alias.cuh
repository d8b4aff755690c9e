// moss_alias.cuh -- block-cooperative alias table of one long neighbour list.
//
// The closed form of moss_tables.cu (header comment there): q_j = w_j d,
// capacity W = sum w; lights (q_j < W) carry the deficit W - q_j, heavies the
// excess q_j - W, both in list order; with A_i the exclusive prefix of the
// light deficits and P_k the inclusive prefix of the heavy excesses, light i
// keeps q_i and aliases the first heavy k with P_k >= A_i; heavy k keeps
// W + P_k - A_{i'} (i' the first light with A_{i'} > P_k) and aliases heavy
// k+1, or keeps W when P_k is the total.  The warp-per-list kernels leave a
// hub's list to one warp, whose sequential merge then bounds the whole
// launch; here a block of NT threads shares one list: block scans split it,
// and each thread merges a run of about d / NT entries.
#pragma once

#include <type_traits>

#include "moss_internal.cuh"

namespace moss {

template <typename T>
__device__ __forceinline__ T shfl_up_any(T v, int d);
template <>
__device__ __forceinline__ uint32_t shfl_up_any<uint32_t>(uint32_t v, int d) {
    return __shfl_up_sync(0xffffffffu, v, d);
}
template <>
__device__ __forceinline__ uint64_t shfl_up_any<uint64_t>(uint64_t v, int d) {
    return __shfl_up_sync(0xffffffffu, v, d);
}
template <>
__device__ __forceinline__ u128 shfl_up_any<u128>(u128 v, int d) {
    return shfl_up_u128(v, d);
}

// inclusive scan over the block (blockDim.x == NT); total receives the block
// sum.  smem holds NT / 32 entries; every thread of the block must call it.
template <typename T, int NT>
__device__ __forceinline__ T block_incl_scan(T v, T &total, T *smem) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const T t = shfl_up_any<T>(v, d);
        if (lane >= d) v += t;
    }
    if (lane == 31) smem[warp] = v;
    __syncthreads();
    T off = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        const T s = smem[w];
        if (w < warp) off += s;
        tot += s;
    }
    __syncthreads();
    total = tot;
    return off + v;
}

// Inclusive scans over the block of three values at once (one pair of
// barriers): c, D and E become their inclusive prefixes, tc, tD and tE the
// block sums.  Every thread of the block must call it.
template <typename T, int NT>
__device__ __forceinline__ void block_scan3(uint64_t &c, T &D, T &E, uint64_t &tc, T &tD, T &tE) {
    __shared__ uint64_t s_c[NT / 32];
    __shared__ T s_D[NT / 32], s_E[NT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        const uint64_t c1 = shfl_up_any<uint64_t>(c, k);
        const T D1 = shfl_up_any<T>(D, k), E1 = shfl_up_any<T>(E, k);
        if (lane >= k) {
            c += c1;
            D += D1;
            E += E1;
        }
    }
    if (lane == 31) {
        s_c[warp] = c;
        s_D[warp] = D;
        s_E[warp] = E;
    }
    __syncthreads();
    uint64_t oc = 0, ac = 0;
    T oD = 0, aD = 0, oE = 0, aE = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        const uint64_t x = s_c[w];
        const T y = s_D[w], z = s_E[w];
        if (w < warp) {
            oc += x;
            oD += y;
            oE += z;
        }
        ac += x;
        aD += y;
        aE += z;
    }
    __syncthreads();
    c += oc;
    D += oD;
    E += oE;
    tc = ac;
    tD = aD;
    tE = aE;
}

// Alias table of the list of d entries with weights weight(j) (d * w_j and W
// must fit T) and capacity W > 0; idx (d uint32) and pre (d T) are scratch;
// store(j, thr, alias) receives each entry's threshold (<= W) and alias
// position.  Every thread of the block must call it.
template <typename T, int NT, typename Weight, typename Store>
__device__ void block_alias(uint32_t d, T W, Weight weight, uint32_t *idx, T *pre, Store store) {
    const int tid = threadIdx.x;
    uint32_t nl = 0, nh = 0;
    T Arun = 0, Prun = 0;
    for (uint32_t base = 0; base < d; base += NT) {
        const uint32_t j = base + tid;
        const bool valid = j < d;
        const T q = valid ? (T)weight(j) * (T)d : (T)0;
        const bool light = valid && q < W, heavy = valid && !light;
        const T D = light ? W - q : (T)0, E = heavy ? q - W : (T)0;
        // light and heavy counts packed in one 64-bit lane (low, high word)
        uint64_t ic = light ? 1ull : (heavy ? 1ull << 32 : 0ull), tc;
        T iD = D, iE = E, tD, tE;
        block_scan3<T, NT>(ic, iD, iE, tc, tD, tE);
        const uint32_t il = (uint32_t)ic, ih = (uint32_t)(ic >> 32);
        const uint32_t tl = (uint32_t)tc, th = (uint32_t)(tc >> 32);
        if (light) {
            const uint32_t r = nl + il - 1;
            idx[r] = j;
            pre[r] = Arun + iD - D;          // exclusive A_i
        } else if (heavy) {
            const uint32_t r = nh + ih - 1;
            idx[d - 1 - r] = j;
            pre[d - 1 - r] = Prun + iE;      // inclusive P_k
        }
        nl += tl;
        nh += th;
        Arun += tD;
        Prun += tE;
    }
    __syncthreads();   // the split is visible to the whole block
    const T Ptot = Prun;
    {
        const uint32_t cl = (nl + NT - 1) / NT;
        const uint32_t i0 = tid * cl, i1 = min(nl, i0 + cl);
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
                store(j, (T)weight(j) * (T)d, idx[d - 1 - k]);
            }
        }
    }
    {
        const uint32_t ch = (nh + NT - 1) / NT;
        const uint32_t k0 = tid * ch, k1 = min(nh, k0 + ch);
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
                if (Pk < Ptot) {
                    const T Ai = i < nl ? pre[i] : Ptot;
                    store(j, W + Pk - Ai, idx[d - 1 - (k + 1)]);
                } else {
                    store(j, W, j);
                }
            }
        }
    }
    __syncthreads();   // idx / pre are reused by the block's next list
}

// The blocks that share a pass: a whole launch, or a run of its blocks when
// passes that do not depend on each other share one.
struct GridPart {
    uint32_t block, blocks;
};
__device__ __forceinline__ GridPart whole_grid() { return GridPart{blockIdx.x, gridDim.x}; }

// ------------------------------------------------------------ short lists --
// Lists of at most kShortList entries, most lists of a power-law graph, go to
// groups of 8, 16 or 32 lanes, an entry per lane, so one warp builds four, two
// or one of them at a time.  A warp per list leaves most lanes idle: the
// passes over 1M lists of mean length 16 were bound by the instructions of
// their half-empty warps, not by the ~60 bytes an entry moves.  Measured there (us):
// k_slots 174 -> 79, k_sigma_alias 428 -> 195 with the alias's fields filled in
// the same pass (the fill 169 -> 107), k_rank_warp 372 -> 154, k_min_alias with
// the short lists' slot and pick records 780 + 283 + 172 -> 525 + 177 + 108,
// k_owner 72 -> 27.
constexpr uint32_t kShortList = 32;

// Walks every vertex v < n: a warp takes TILE consecutive records and hands
// their lists of 1..kShortList entries to small(G, v, rec, j, valid) -- a
// group of G.value lanes per list, lane j of it entry j when valid; all 32
// lanes call, groups without a list with valid false -- and empty ones to
// empty(v, rec), one lane each; and, of TILE records a stride apart (so that
// long lists which lie together spread over the warps), the longer lists one
// by one to large(v, rec), the whole warp each.
// The walk is shared by the blocks of `grid`.
template <int TILE, typename Small, typename Empty, typename Large>
__device__ __forceinline__ void for_lists(GridPart grid, uint32_t n, const uint4 *rec, Small small, Empty empty,
                                          Large large) {
    const int lane = threadIdx.x & 31;
    const uint64_t tiles = ((uint64_t)n + TILE - 1) / TILE;
    const uint64_t warps = (uint64_t)grid.blocks * (blockDim.x >> 5);
    for (uint64_t t = (uint64_t)grid.block * (blockDim.x >> 5) + (threadIdx.x >> 5); t < tiles; t += warps) {
        const uint64_t v0 = t * TILE, vs = t + (uint64_t)lane * tiles;
        const bool here = lane < TILE && v0 + lane < n;
        const uint4 r = here ? rec[v0 + lane] : make_uint4(0u, 0u, 0u, 0u);
        const uint4 rs = lane < TILE && vs < n ? rec[vs] : make_uint4(0u, 0u, 0u, 0u);
        if (here && r.y == 0) empty((uint32_t)(v0 + lane), r);
        auto pass = [&](auto G, uint32_t mask) {
            constexpr int g = decltype(G)::value;
            while (mask) {   // warp-uniform
                int src = -1;
#pragma unroll
                for (int k = 0; k < 32 / g; ++k) {   // group k takes the mask's next list
                    if (lane / g == k && mask) src = __ffs(mask) - 1;
                    mask &= mask - 1;
                }
                const int from = src < 0 ? 0 : src;
                uint4 q;
                q.x = __shfl_sync(0xffffffffu, r.x, from);
                q.y = __shfl_sync(0xffffffffu, r.y, from);
                q.z = __shfl_sync(0xffffffffu, r.z, from);
                q.w = __shfl_sync(0xffffffffu, r.w, from);
                const uint32_t j = lane & (g - 1);
                small(G, (uint32_t)(v0 + from), q, j, src >= 0 && j < q.y);
            }
        };
        pass(std::integral_constant<int, 8>{}, __ballot_sync(0xffffffffu, r.y >= 1 && r.y <= 8));
        pass(std::integral_constant<int, 16>{}, __ballot_sync(0xffffffffu, r.y > 8 && r.y <= 16));
        pass(std::integral_constant<int, 32>{}, __ballot_sync(0xffffffffu, r.y > 16 && r.y <= kShortList));
        for (uint32_t mask = __ballot_sync(0xffffffffu, rs.y > kShortList); mask; mask &= mask - 1) {
            const int src = __ffs(mask) - 1;
            uint4 q;
            q.x = __shfl_sync(0xffffffffu, rs.x, src);
            q.y = __shfl_sync(0xffffffffu, rs.y, src);
            q.z = __shfl_sync(0xffffffffu, rs.z, src);
            q.w = __shfl_sync(0xffffffffu, rs.w, src);
            large((uint32_t)(t + (uint64_t)src * tiles), q);
        }
    }
}

// Lists above kHubList entries get 1,024 threads (hub_blocks(n) blocks walk
// them), their splits in up to kHubSmemList entries of shared memory: with 256
// the longest list's chain of rounds was the whole pass (d_max 15,000, us:
// sigma 255 -> 109 + 89 for the lists up to kHubList, MOSS-4Min 525 -> 197 +
// 147; the passes that a graph's largest degree rules out are not launched).
constexpr uint32_t kHubList = 2048;
constexpr int kHubThreads = 1024;
constexpr uint32_t kHubSmemList = 16384;   // 192 KB at 12 bytes an entry
inline unsigned hub_blocks(uint32_t n) {
    const uint64_t chunks = ((uint64_t)n + kHubThreads - 1) / kHubThreads, sms = (uint64_t)current_sms();
    return (unsigned)(chunks < sms ? chunks : sms);
}

// records per warp: enough lists to fill the groups, but a warp for every
// scheduler first
template <typename F>
inline void with_tile(uint32_t n, F f) {
    if (n >= (1u << 18)) f(std::integral_constant<int, 32>{});
    else f(std::integral_constant<int, 8>{});
}
// blocks of THREADS threads that cover n records in tiles, at most per_sm an SM
inline unsigned tile_blocks(uint32_t n, int tile, int threads, int sms, int per_sm) {
    const uint64_t tiles = ((uint64_t)n + tile - 1) / tile, b = (tiles + threads / 32 - 1) / (threads / 32);
    const uint64_t cap = (uint64_t)sms * per_sm;
    return (unsigned)(b < 1 ? 1 : (b < cap ? b : cap));
}

// inclusive sum over the lanes of a group of G
template <int G>
__device__ __forceinline__ uint64_t group_scan(uint64_t x, uint32_t j) {
#pragma unroll
    for (int d = 1; d < G; d <<= 1) {
        const uint64_t t = __shfl_up_sync(0xffffffffu, x, d, G);
        if (j >= (uint32_t)d) x += t;
    }
    return x;
}

// The alias table of a list held by a group of G lanes, lane j with q_j = w_j d
// (closed form as above): the prefixes of deficits and excesses stay in the
// lanes and, being monotone over them, are searched there by shuffles.
template <int G>
__device__ __forceinline__ void group_alias(bool valid, uint64_t q, uint64_t W, uint32_t j, uint64_t &thr,
                                            uint32_t &alias) {
    const int lane = threadIdx.x & 31;
    const bool light = valid && q < W, heavy = valid && !light;
    const uint32_t group = G == 32 ? 0xffffffffu : (1u << (G & 31)) - 1u;
    const uint32_t heavies = __ballot_sync(0xffffffffu, heavy) >> (lane & ~(G - 1)) & group;
    const uint64_t D = light ? W - q : 0;
    const uint64_t A = group_scan<G>(D, j) - D;                  // exclusive deficits
    const uint64_t P = group_scan<G>(heavy ? q - W : 0, j);      // inclusive excesses
    const uint64_t total = __shfl_sync(0xffffffffu, P, G - 1, G);
    // light: the first lane whose P reaches A; heavy: the first whose A exceeds P
    uint32_t at = 0;
#pragma unroll
    for (int step = G / 2; step > 0; step >>= 1) {
        const uint64_t Pe = __shfl_sync(0xffffffffu, P, at + step - 1, G);
        const uint64_t Ae = __shfl_sync(0xffffffffu, A, at + step - 1, G);
        if (light ? Pe < A : Ae <= P) at += step;
    }
    const uint64_t Aat = __shfl_sync(0xffffffffu, A, at, G);
    if (light) {
        thr = q;
        alias = __ffs(heavies >> at << at) - 1;
    } else if (P < total) {
        // the first light there or after has the same A (nothing in between
        // adds a deficit); without one A ends at the total
        thr = W + P - (Aat > P ? Aat : total);
        alias = __ffs(heavies & ~((2u << j) - 1u)) - 1;
    } else {
        thr = W;
        alias = j;
    }
}

// Calls body(v) for every vertex v < n whose record passes pred, one vertex at
// a time for the whole block (body is block-cooperative).  Blocks take chunks
// of CH <= NT vertices and test a chunk's records in parallel, so a block
// touches n / gridDim records rather than one by one; a small CH spreads
// frequent qualifying vertices over more blocks.  Chunk c holds the vertices
// c + j C (j < CH, C = ceil(n / CH) chunks): vertices that are close in id
// fall into different chunks, so a graph whose long lists sit together (one
// loaded in degree order) still spreads them over the blocks.
template <int NT, int CH = NT, typename Pred, typename Body>
__device__ __forceinline__ void for_each_vertex(GridPart grid, uint32_t n, const uint4 *rec, Pred pred, Body body) {
    static_assert(CH <= NT, "chunk larger than the block");
    __shared__ uint32_t found[CH];
    __shared__ uint32_t nfound;
    const uint64_t chunks = ((uint64_t)n + CH - 1) / CH;
    for (uint64_t c = grid.block; c < chunks; c += grid.blocks) {
        if (threadIdx.x == 0) nfound = 0;
        __syncthreads();
        const uint64_t v = c + (uint64_t)threadIdx.x * chunks;
        if (threadIdx.x < CH && v < n && pred(rec[v])) found[atomicAdd(&nfound, 1u)] = (uint32_t)v;
        __syncthreads();
        const uint32_t cnt = nfound;
        for (uint32_t k = 0; k < cnt; ++k) body(found[k]);
        __syncthreads();
    }
}

}  // namespace moss
