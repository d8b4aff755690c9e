// moss_sampler.cuh -- one sample of each method on the device: random words,
// vertex draw, sigma draw(s), uniform list picks, edge probes, class.  Shared
// by the sampling kernels of moss_sample.cu (sample ids in order) and
// moss_group.cu (sample ids grouped by the vertex they draw); every translation
// unit that includes it holds its own copy of the class tables
// (upload_luts_here).
#pragma once

#include "moss_internal.cuh"

namespace moss {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kLut = 1024;
// hub-pair bits behind the filter, per method (MOSS-4, T-5, Path-5, MOSS-4Min):
// measured on the 34M-edge graph against the same build without them, 5e8
// samples per call, T-5 -7.5%, Path-5 -16%, MOSS-4Min -27%, MOSS-4 +0.8% (its
// three probes hold few hub pairs)
constexpr bool kHubProbes[kMethods] = {false, true, true, true};

__device__ uint8_t g_lut4[64];
__device__ uint8_t g_lut5[1024];
__device__ uint8_t g_lutc[4096];   // c(s) of MOSS-4Min by (edge mask << 6 | order bits)

__device__ __forceinline__ uint4 ld4(const uint4 *p) { return __ldg(p); }
__device__ __forceinline__ uint2 ld2(const uint2 *p) { return __ldg(p); }
__device__ __forceinline__ uint32_t ld1(const uint32_t *p) { return __ldg(p); }

// Probe modes of the sampler instances: kPmPlain (list search, or the hashed
// edge set with one-level vertex tables), kPmFilter (the edge filter in front
// of the set: L2 hints and hub-pair bits) and kPmStream (the set with
// two-level vertex tables, which fit the L1: the scattered loads of lists,
// slot records and buckets skip L1 allocation, so the heavy level's records,
// read evict-last, stay there and those draws cost no L2 request).
// kPmGroup is kPmFilter for samples grouped by their first vertex v
// (moss_group.cu): its neighbours in the group read v's slot records again, so
// those are not read evict-first.
constexpr int kPmPlain = 0, kPmFilter = 1, kPmStream = 2, kPmGroup = 3, kPmBatch = 4;
constexpr uint32_t kStreamHeavy = 4096;   // heavy columns (32 B each) that kPmStream keeps in L1
__host__ __device__ constexpr bool behind_filter(int pm) { return pm == kPmFilter || pm == kPmGroup; }

// How a sample's pairs walk the edge set: in rounds over all of them, one bucket
// each; by lanes, each lane its own next pair, from the first bucket on; or the
// home buckets of all of them together and the full ones' pairs by lanes.
//   Without the filter, a set of two slots an edge sends 14% of the pairs past
// their home bucket, and with another round over all pairs nearly every p has
// some lane waiting.  1.7e7 samples, ms, rounds -> home then lanes: power-law
// graph of 4M entries T-5 0.79 -> 0.74, Path-5 1.02 -> 0.88, mesh of 4M 0.82 ->
// 0.74 and 1.13 -> 1.00; roomier sets 0-1% either way, and the redraws, which
// would spill, stay with rounds.
//   Behind the filter few pairs reach the set.  Grouped samples go by lanes (the
// 34M-edge step 70.4 ms, 73.2 with the home buckets first).  Ungrouped ones by
// lanes / in rounds, ms: Path-5 1.02 / 1.05 (7M edges, degree order), 1.19 / 1.24
// (4M), but T-5 1.94 / 1.80 (34M edges), 1.04 / 1.00 (4M), MOSS-4Min 0.99 / 0.95
// (7M).  Batches (kPmBatch, otherwise as kPmPlain) keep the rounds: 13.7 ms for
// 256 graphs, 13.9 with the home buckets first.
constexpr int kRounds = 0, kLanes = 1, kHomeThenLanes = 2;
__host__ __device__ constexpr int walk_of(int pm, int method, int stage = 0) {
    if (behind_filter(pm) || pm == kPmBatch)
        return kHubProbes[method] && (pm != kPmFilter || method == 2) ? kLanes : kRounds;
    return stage == 1 || stage == 2 ? kRounds : kHomeThenLanes;
}

// a vertex record without L1 allocation
__device__ __forceinline__ uint4 ld4_na(const uint4 *p) {
    uint4 r;
    asm("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
    return r;
}

// a list entry (neighbour id) in mode PM
template <int PM>
__device__ __forceinline__ uint32_t ldc(const uint32_t *p) {
    if (PM != kPmStream) return __ldg(p);
    uint32_t r;
    asm("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(r) : "l"(p));
    return r;
}

struct Pick {
    uint32_t pos;   // position in N_v
    uint32_t id;    // the vertex
    uint32_t twin;  // position of v in N_id
    uint32_t off;   // N_id = col[off .. off + deg)
    uint32_t deg;
};

// one 32-byte sector in a single 256-bit load (32-byte aligned)
struct alignas(32) Sector {
    uint4 lo, hi;
};
__device__ __forceinline__ Sector ld8(const uint4 *p) {
    Sector r;
    asm("ld.global.nc.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(r.lo.x), "=r"(r.lo.y), "=r"(r.lo.z), "=r"(r.lo.w), "=r"(r.hi.x), "=r"(r.hi.y), "=r"(r.hi.z),
          "=r"(r.hi.w)
        : "l"(p));
    return r;
}

// The same load without L1 allocation (scattered records in kPmStream)
__device__ __forceinline__ Sector ld8_na(const uint4 *p) {
    Sector r;
    asm("ld.global.nc.L1::no_allocate.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(r.lo.x), "=r"(r.lo.y), "=r"(r.lo.z), "=r"(r.lo.w), "=r"(r.hi.x), "=r"(r.hi.y), "=r"(r.hi.z),
          "=r"(r.hi.w)
        : "l"(p));
    return r;
}

// ... and kept in L1 as long as possible (heavy-level vertex records in kPmStream)
__device__ __forceinline__ Sector ld8_keep(const uint4 *p) {
    Sector r;
    asm("ld.global.nc.L1::evict_last.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(r.lo.x), "=r"(r.lo.y), "=r"(r.lo.z), "=r"(r.lo.w), "=r"(r.hi.x), "=r"(r.hi.y), "=r"(r.hi.z),
          "=r"(r.hi.w)
        : "l"(p));
    return r;
}

// The same load marked evict-first in L2, for the per-slot records (sigma
// slot records, MOSS-4Min pick records): they are the largest and least
// densely used tables of a sampler, so with the working set at the size of
// the L2 they are the ones to give up first, which keeps the denser edge
// hash, neighbour lists and vertex alias records resident.
__device__ __forceinline__ Sector ld8_first(const uint4 *p) {
    uint64_t pol;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    Sector r;
    asm("ld.global.nc.L2::cache_hint.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], %9;"
        : "=r"(r.lo.x), "=r"(r.lo.y), "=r"(r.lo.z), "=r"(r.lo.w), "=r"(r.hi.x), "=r"(r.hi.y), "=r"(r.hi.z),
          "=r"(r.hi.w)
        : "l"(p), "l"(pol));
    return r;
}
__device__ __forceinline__ Sector ld8_first_na(const uint4 *p) {
    uint64_t pol;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    Sector r;
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], %9;"
        : "=r"(r.lo.x), "=r"(r.lo.y), "=r"(r.lo.z), "=r"(r.lo.w), "=r"(r.hi.x), "=r"(r.hi.y), "=r"(r.hi.z),
          "=r"(r.hi.w)
        : "l"(p), "l"(pol));
    return r;
}

// a scattered 32-byte record (bucket, MOSS-4Min slot record) in mode PM
template <int PM>
__device__ __forceinline__ Sector ld8s(const uint4 *p) {
    return behind_filter(PM) ? ld8_first(p) : (PM == kPmStream ? ld8_na(p) : ld8(p));
}
// a per-slot record (sigma slot, MOSS-4Min pick) in mode PM: evict-first in
// L2 unless the samples are grouped by its list
template <int PM>
__device__ __forceinline__ Sector ld8p(const uint4 *p) {
    if (PM == kPmGroup) return ld8(p);
    return PM == kPmStream ? ld8_first_na(p) : ld8_first(p);
}

struct VertexPick {
    uint32_t v;
    uint4 rec;      // v's vertex record (vert, or mvert for MOSS-4Min)
};

// WeightRandomVertex(V, .) through a vertex alias table whose 32-byte column
// records carry the alias's vertex record: one load, plus the column's own
// record only when the column keeps the draw.  The table has two levels: the
// level word picks the light one (columns nh..n-1) when it is below the
// level's bound, else the heavy one (columns 0..nh-1: the few vertices that
// carry almost all the weight, a table small enough to stay cached).  Behind
// the edge filter a light record is read evict-first, since that table is as
// large as the L2 and drawn uniformly, so a line is rarely read twice; in
// kPmStream a heavy record is kept in L1.
// The level word (word lw of the sample) is generated only for a table with
// a heavy level (uniform across the launch).
template <int PM, int RNG>
__device__ __forceinline__ VertexPick draw_vertex(const DevGraph &g, int l, const uint4 *vrec, uint64_t seed,
                                                  uint64_t s, uint32_t lw, uint64_t xc, uint64_t xt) {
    const uint32_t nh = g.nheavy[l];
    bool light = true;
    if (nh != 0) light = sample_word<RNG>(seed, (uint32_t)l, s, lw) < g.tlight[l];
    const uint32_t c = (light ? nh : 0u) + word_index32(xc, light ? g.n - nh : nh);
    const uint4 *rec = g.seed[l] + 2 * (uint64_t)c;
    const Sector r = PM == kPmFilter ? (light ? ld8_first(rec) : ld8(rec))
                                     : (PM == kPmStream ? (light ? ld8_na(rec) : ld8_keep(rec)) : ld8(rec));
    // {T lo, T hi, alias, self} {alias's record}
    const uint64_t T = ((uint64_t)r.lo.y << 32) | r.lo.x;
    if (xt < T) return VertexPick{r.lo.w, PM == kPmStream && light ? ld4_na(vrec + r.lo.w) : ld4(vrec + r.lo.w)};
    return VertexPick{r.lo.z, r.hi};
}

// The neighbour half of a slot record (col, nb, off): a neighbour with 2^16
// or more neighbours keeps its twin in off and its list in vert[].
__device__ __forceinline__ Pick unpack_pick(const uint4 *vert, uint32_t pos, uint32_t id, uint32_t nb, uint32_t off) {
    if (nb != kSlotHub) return Pick{pos, id, nb & (kSlotDegLimit - 1), off, nb >> 16};
    const uint4 r = ld4(vert + id);
    return Pick{pos, id, off, r.x, r.y};
}

// WeightRandomVertex(N_v, sigma^(v)) through the list's alias table: one
// 32-byte slot record holds the column's pick and its alias's, each with the
// picked neighbour's list and twin
template <int PM>
__device__ __forceinline__ Pick draw_sigma(const uint4 *slot, const uint4 *vert, uint32_t ov, uint32_t dv, uint32_t Sv,
                                           uint64_t xc, uint64_t xt) {
    const uint32_t j = word_index32(xc, dv);
    const Sector rec = ld8p<PM>(slot + 2 * (uint64_t)(ov + j));   // {col, nb, thr, alias} {off, alias col, nb, off}
    const bool keep = word_index32(xt, Sv) < rec.lo.z;
    return unpack_pick(vert, keep ? j : rec.lo.w, keep ? rec.lo.x : rec.hi.y, keep ? rec.lo.y : rec.hi.z,
                       keep ? rec.hi.x : rec.hi.w);
}

// the pick of position p of N_v from its own half of the slot record
__device__ __forceinline__ Pick slot_pick(const uint4 *slot, const uint4 *vert, uint32_t ov, uint32_t p) {
    const Sector rec = ld8(slot + 2 * (uint64_t)(ov + p));
    return unpack_pick(vert, p, rec.lo.x, rec.lo.y, rec.hi.x);
}

__device__ __forceinline__ uint32_t skip1(uint32_t j, uint32_t e) { return j < e ? j : j + 1; }

__device__ __forceinline__ uint32_t skip2(uint32_t j, uint32_t e1, uint32_t e2) {
    const uint32_t lo = min(e1, e2), hi = max(e1, e2);
    j += (j >= lo);
    j += (j >= hi);
    return j;
}

// Membership tests (a_p, b_p) in E for P pairs, advanced in lock step so the
// P searches of a sample overlap in memory.  Each pair searches the shorter
// of the two sorted lists.  Returns bit p set when the pair is an edge.
template <int P>
__device__ __forceinline__ uint32_t probe_pairs(const uint32_t *col, const uint4 (&ra)[P], const uint4 (&rb)[P],
                                                const uint32_t (&a)[P], const uint32_t (&b)[P]) {
    uint32_t lo[P], len[P], key[P];
    uint32_t found = 0;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const bool use_a = ra[p].y <= rb[p].y;
        lo[p] = use_a ? ra[p].x : rb[p].x;
        len[p] = use_a ? ra[p].y : rb[p].y;
        key[p] = use_a ? b[p] : a[p];
    }
    bool any = true;
    while (any) {
        any = false;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            if (len[p] > 0) {
                const uint32_t half = len[p] >> 1;
                const uint32_t val = ld1(col + lo[p] + half);
                if (val == key[p]) {
                    found |= 1u << p;
                    len[p] = 0;
                } else if (val < key[p]) {
                    lo[p] += half + 1;
                    len[p] -= half + 1;
                } else {
                    len[p] = half;
                }
                any |= len[p] > 0;
            }
        }
    }
    return found;
}

// whether a bucket holds an edge key
__device__ __forceinline__ bool holds(const Sector &e, uint64_t key) {
    const uint32_t lo = (uint32_t)key, hi = (uint32_t)(key >> 32);
    return (e.lo.x == lo && e.lo.y == hi) || (e.lo.z == lo && e.lo.w == hi) || (e.hi.x == lo && e.hi.y == hi) ||
           (e.hi.z == lo && e.hi.w == hi);
}

// The pairs of `pending` in the set from bucket `first` after their home on, each
// lane its own next one: where few pairs are left, at different p in the lanes
// of a warp, the warp makes as many rounds of dependent loads as its busiest
// lane has buckets to see, not one for every p.  Returns the pairs found.
template <int P, int PM>
__device__ __forceinline__ uint32_t probe_lanes(const DevGraph &g, const uint32_t (&a)[P], const uint32_t (&b)[P],
                                                uint32_t pending, uint32_t first) {
    uint32_t found = 0, step = first;
    while (pending != 0) {   // (a set has two buckets at least: hash_mask >= 1)
        const uint32_t p = __ffs(pending) - 1;
        uint32_t x = a[0], y = b[0];
#pragma unroll
        for (int q = 1; q < P; ++q) {
            x = p == q ? a[q] : x;
            y = p == q ? b[q] : y;
        }
        const uint64_t key = edge_key(x, y);
        const Sector e = ld8s<PM>(g.hash + 2 * (uint64_t)((edge_bucket(key, g.hash_shift) + step) & g.hash_mask));
        const bool hit = holds(e, key);
        const bool last = hit || (e.hi.z == 0xffffffffu && e.hi.w == 0xffffffffu) || step == g.hash_mask;
        found |= (uint32_t)hit << p;
        pending &= ~((uint32_t)last << p);
        step = last ? first : step + 1;
    }
    return found;
}

// Membership tests through the hashed edge set: one 32-byte bucket load per
// pair in the common case, all P loads issued together.  kPmFilter (behind
// the filter): the filter rules out most pairs; the set is far larger than the
// L2 and a bucket is rarely read twice, so buckets are read evict-first,
// which keeps the filter, lists and hub slot records resident.  With HUB,
// the ends' rank-table entries come first (one 8-byte load per vertex, all
// together), and a pair of two hubs is answered by one bit of the hubs'
// adjacency bitmap, loaded beside the other pairs' filter words.
template <int P, int PM, bool HUB, int WALK>
__device__ __forceinline__ uint32_t probe_hash(const DevGraph &g, const uint32_t (&a)[P], const uint32_t (&b)[P]) {
    uint32_t found = 0, pending = (1u << P) - 1u;
    if (g.filter) {   // warp-uniform: only pairs the filter cannot rule out go to the set
        uint32_t hubpair = 0, bit[P];
        if (behind_filter(PM) && HUB && g.hub_rank) {   // warp-uniform
            uint2 ea[P], eb[P];
#pragma unroll
            for (int p = 0; p < P; ++p) {
                ea[p] = ld2(g.hub_rank + (a[p] >> 5));
                eb[p] = ld2(g.hub_rank + (b[p] >> 5));
            }
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const uint32_t ia = hub_index(ea[p], a[p]), ib = hub_index(eb[p], b[p]);
                bit[p] = ia * g.hubs + ib;
                if (ia != kNoHub && ib != kNoHub) hubpair |= 1u << p;
            }
        }
        uint32_t word[P];
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const uint64_t h = filter_hash(edge_key(a[p], b[p]));
            const bool hub = hubpair >> p & 1u;
            word[p] = ld1(hub ? g.hub_bits + (bit[p] >> 5) : g.filter + (h >> g.filter_shift));
            if (!hub) bit[p] = (uint32_t)h;
        }
#pragma unroll
        for (int p = 0; p < P; ++p) {
            if (hubpair >> p & 1u) {
                found |= (word[p] >> (bit[p] & 31u) & 1u) << p;
                pending &= ~(1u << p);
            } else {
                const uint32_t m = filter_mask(bit[p]);
                if ((word[p] & m) != m) pending &= ~(1u << p);
            }
        }
        if constexpr (WALK == kLanes) return found | probe_lanes<P, PM>(g, a, b, pending, 0);
    }
    if constexpr (WALK != kHomeThenLanes) {
        uint32_t bk[P];
#pragma unroll
        for (int p = 0; p < P; ++p) bk[p] = edge_bucket(edge_key(a[p], b[p]), g.hash_shift);
        for (uint32_t it = 0; pending != 0 && it <= g.hash_mask; ++it) {
#pragma unroll
            for (int p = 0; p < P; ++p) {
                if (pending >> p & 1u) {
                    const Sector e = ld8s<PM>(g.hash + 2 * (uint64_t)bk[p]);
                    if (holds(e, edge_key(a[p], b[p]))) {
                        found |= 1u << p;
                        pending &= ~(1u << p);
                    } else if (e.hi.z == 0xffffffffu && e.hi.w == 0xffffffffu) {   // last slot empty
                        pending &= ~(1u << p);
                    } else {
                        bk[p] = (bk[p] + 1) & g.hash_mask;
                    }
                }
            }
        }
        return found;
    } else {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            if (pending >> p & 1u) {
                const uint64_t key = edge_key(a[p], b[p]);
                const Sector e = ld8s<PM>(g.hash + 2 * (uint64_t)edge_bucket(key, g.hash_shift));
                const bool hit = holds(e, key);
                found |= (uint32_t)hit << p;
                if (hit || (e.hi.z == 0xffffffffu && e.hi.w == 0xffffffffu)) pending &= ~(1u << p);
            }
        }
        return found | probe_lanes<P, PM>(g, a, b, pending, 1);
    }
}

struct Sample {
    uint32_t v[5];
    int cls;
};

// Each sampler in two parts: the draw of its first vertex v (first_vertex)
// and, given v and its record, everything after it (rest_*).

// the level word of the vertex draw of each method
__host__ __device__ constexpr uint32_t level_word(int method) { return method == 1 ? 7 : (method == 2 ? 14 : 6); }

template <int METHOD, int RNG, int PM>
__device__ __forceinline__ VertexPick first_vertex(const DevGraph &g, uint64_t seed, uint64_t s) {
    const Words2 x01 = sample_words2<RNG>(seed, METHOD, s, 0);
    return draw_vertex<PM, RNG>(g, METHOD, METHOD == 3 ? g.mvert : g.vert, seed, s, level_word(METHOD), x01.x[0],
                                x01.x[1]);
}

template <int RNG, bool HASH, int PM>
__device__ __forceinline__ Sample rest_moss4(const DevGraph &g, const uint8_t *lut, uint64_t seed, uint64_t s,
                                             const VertexPick &pv) {
    Sample out;
    const uint32_t v = pv.v;
    const uint4 vr = pv.rec;
    const Words2 x23 = sample_words2<RNG>(seed, 0, s, 1);
    const Pick pu = draw_sigma<PM>(g.slot, g.vert, vr.x, vr.y, vr.z, x23.x[0], x23.x[1]);
    const Words2 x45 = sample_words2<RNG>(seed, 0, s, 2);
    const uint32_t jw = skip1(word_index32(x45.x[0], vr.y - 1), pu.pos);
    const uint32_t w = ldc<PM>(g.col + vr.x + jw);
    const uint32_t jr = skip1(word_index32(x45.x[1], pu.deg - 1), pu.twin);
    const uint32_t r = ldc<PM>(g.col + pu.off + jr);
    out.v[0] = v; out.v[1] = pu.id; out.v[2] = w; out.v[3] = r; out.v[4] = 0;
    if (r == pu.id || r == w) {
        out.cls = 0;
        return out;
    }
    // unknown pairs: v-r, u-w, w-r
    const uint32_t A[3] = {v, pu.id, w}, B[3] = {r, w, r};
    uint32_t f;
    if (HASH) {
        f = probe_hash<3, PM, kHubProbes[0], walk_of(PM, 0)>(g, A, B);
    } else {
        const uint4 ur = make_uint4(pu.off, pu.deg, 0u, 0u), wr = ld4(g.vert + w), rr = ld4(g.vert + r);
        const uint4 ra[3] = {vr, ur, wr}, rb[3] = {rr, wr, rr};
        f = probe_pairs<3>(g.col, ra, rb, A, B);
    }
    // pair bits (0,1)(0,2)(0,3)(1,2)(1,3)(2,3); known: v-u, v-w, u-r
    const uint32_t mask = 0x1u | 0x2u | ((f & 1u) << 2) | (((f >> 1) & 1u) << 3) | 0x10u | (((f >> 2) & 1u) << 5);
    out.cls = lut[mask];
    return out;
}

template <int RNG, bool HASH, int PM = kPmPlain>
__device__ __forceinline__ Sample sample_moss4(const DevGraph &g, const uint8_t *lut, uint64_t seed, uint64_t s) {
    return rest_moss4<RNG, HASH, PM>(g, lut, seed, s, first_vertex<0, RNG, PM>(g, seed, s));
}

template <int RNG, bool HASH, int PM>
__device__ __forceinline__ Sample rest_t5(const DevGraph &g, const uint8_t *lut, uint64_t seed, uint64_t s,
                                          const VertexPick &pv) {
    Sample out;
    const uint32_t v = pv.v;
    const uint4 vr = pv.rec;
    const Words2 x23 = sample_words2<RNG>(seed, 1, s, 1);
    const Pick pu = draw_sigma<PM>(g.slot, g.vert, vr.x, vr.y, vr.z, x23.x[0], x23.x[1]);
    const Words2 x45 = sample_words2<RNG>(seed, 1, s, 2);
    const uint32_t jw = skip1(word_index32(x45.x[0], vr.y - 1), pu.pos);
    const uint32_t jr = skip2(word_index32(x45.x[1], vr.y - 2), pu.pos, jw);
    const uint32_t w = ldc<PM>(g.col + vr.x + jw);
    const uint32_t r = ldc<PM>(g.col + vr.x + jr);
    const uint32_t jt = skip1(word_index32(sample_word<RNG>(seed, 1, s, 6), pu.deg - 1), pu.twin);
    const uint32_t t = ldc<PM>(g.col + pu.off + jt);
    out.v[0] = v; out.v[1] = pu.id; out.v[2] = w; out.v[3] = r; out.v[4] = t;
    if (t == w || t == r) {
        out.cls = 0;
        return out;
    }
    // unknown pairs: u-w, u-r, w-r, v-t, w-t, r-t
    const uint32_t A[6] = {pu.id, pu.id, w, v, w, r}, B[6] = {w, r, r, t, t, t};
    uint32_t f;
    if (HASH) {
        f = probe_hash<6, PM, kHubProbes[1], walk_of(PM, 1)>(g, A, B);
    } else {
        const uint4 ur = make_uint4(pu.off, pu.deg, 0u, 0u);
        const uint4 wr = ld4(g.vert + w), rr = ld4(g.vert + r), tr = ld4(g.vert + t);
        const uint4 ra[6] = {ur, ur, wr, vr, wr, rr}, rb[6] = {wr, rr, rr, tr, tr, tr};
        f = probe_pairs<6>(g.col, ra, rb, A, B);
    }
    // pair bits (0,1)(0,2)(0,3)(0,4)(1,2)(1,3)(1,4)(2,3)(2,4)(3,4)
    // known: v-u (0), v-w (1), v-r (2), u-t (6)
    uint32_t mask = 0x1u | 0x2u | 0x4u | 0x40u;
    mask |= ((f >> 0) & 1u) << 4;   // u-w
    mask |= ((f >> 1) & 1u) << 5;   // u-r
    mask |= ((f >> 2) & 1u) << 7;   // w-r
    mask |= ((f >> 3) & 1u) << 3;   // v-t
    mask |= ((f >> 4) & 1u) << 8;   // w-t
    mask |= ((f >> 5) & 1u) << 9;   // r-t
    out.cls = lut[mask];
    return out;
}

template <int RNG, bool HASH, int PM = kPmPlain>
__device__ __forceinline__ Sample sample_t5(const DevGraph &g, const uint8_t *lut, uint64_t seed, uint64_t s) {
    return rest_t5<RNG, HASH, PM>(g, lut, seed, s, first_vertex<1, RNG, PM>(g, seed, s));
}

// ------------------------------------------------------------- MOSS-4Min --

// order bits of the four roles for the c(s) table: bit b set when the first
// role of pair b ((0,1),(0,2),(0,3),(1,2),(1,3),(2,3)) is above the second;
// key[] holds the order keys (d_x << 32) | x
__device__ __forceinline__ uint32_t order_bits(const uint64_t (&key)[4]) {
    return (uint32_t)(key[0] > key[1]) | (uint32_t)(key[0] > key[2]) << 1 | (uint32_t)(key[0] > key[3]) << 2 |
           (uint32_t)(key[1] > key[2]) << 3 | (uint32_t)(key[1] > key[3]) << 4 | (uint32_t)(key[2] > key[3]) << 5;
}

// count slot of a MOSS-4Min hit: 4-cycles 0..3, diamonds 4..9, 4-cliques
// 10..21 by c; kSlots (not counted) for collisions and the other classes
__device__ __forceinline__ int min_slot(int cls, uint32_t c) {
    if (cls == 3 && c >= 1 && c <= 4) return (int)c - 1;
    if (cls == 5 && c >= 1 && c <= 6) return 4 + (int)c - 1;
    if (cls == 6 && c >= 1 && c <= 12) return 10 + (int)c - 1;
    return kSlots;
}

template <int RNG, bool HASH, int PM>
__device__ __forceinline__ Sample rest_min(const DevGraph &g, const uint8_t *lut, const uint8_t *lutc, uint64_t seed,
                                           uint64_t s, const VertexPick &pv) {
    Sample out;
    const uint32_t v = pv.v;
    const uint4 mv = pv.rec;                           // {off, d_v, Gamma-check_v}
    const uint64_t Gv = ((uint64_t)mv.w << 32) | mv.z;
    // WeightRandomVertex(N_v, sigma-check^(v)): from a list with
    // Gamma-check_v < 2^32, one pick record carries the draw and both
    // possible picks; otherwise (or when a field overflows 16 bits) the slot
    // record, and the alias position's when the column does not keep the draw
    const Words2 x23 = sample_words2<RNG>(seed, 3, s, 1);
    const uint32_t j = word_index32(x23.x[0], mv.y);
    const uint64_t y = word_index(x23.x[1], Gv);
    uint4 sb;   // {off_u, d_u, d_{v,u}, d_{u,v}}
    uint32_t u;
    Sector pk;
    pk.hi.w = kSlotHub;
    if (mv.w == 0) pk = ld8p<PM>(g.mpick + 2 * (uint64_t)(mv.x + j));
    if (pk.hi.w != kSlotHub) {
        const bool keep = y < pk.lo.x;
        const uint32_t dd = keep ? pk.lo.w : pk.hi.z;
        u = keep ? pk.lo.y : pk.hi.x;
        sb = make_uint4(keep ? pk.lo.z : pk.hi.y, keep ? (pk.hi.w & 0xffffu) : (pk.hi.w >> 16), dd & 0xffffu,
                        dd >> 16);
    } else {
        constexpr int pm = PM == kPmStream ? kPmStream : kPmPlain;
        Sector ms = ld8s<pm>(g.mslot + 2 * (uint64_t)(mv.x + j));
        if (!(y < (((uint64_t)ms.lo.y << 32) | ms.lo.x))) ms = ld8s<pm>(g.mslot + 2 * (uint64_t)(mv.x + ms.lo.z));
        sb = ms.hi;
        u = ms.lo.w;
    }
    const Words2 x45 = sample_words2<RNG>(seed, 3, s, 2);
    const uint2 we = ld2(g.rlist + mv.x + word_index32(x45.x[0], sb.z));   // w in N_{v,u}
    const uint2 re = ld2(g.rlist + sb.x + word_index32(x45.x[1], sb.w));   // r in N_{u,v}
    const uint32_t w = we.x, r = re.x;
    out.v[0] = v; out.v[1] = u; out.v[2] = w; out.v[3] = r; out.v[4] = 0;
    if (r == u || r == w) {
        out.cls = 0;
        return out;
    }
    // unknown pairs: v-r, u-w, w-r
    const uint32_t A[3] = {v, u, w}, B[3] = {r, w, r};
    uint32_t f;
    if (HASH) {
        f = probe_hash<3, PM, kHubProbes[3], walk_of(PM, 3)>(g, A, B);
    } else {
        const uint4 vr = make_uint4(mv.x, mv.y, 0u, 0u), ur = make_uint4(sb.x, sb.y, 0u, 0u);
        const uint4 wr = ld4(g.vert + w), rr = ld4(g.vert + r);
        const uint4 ra[3] = {vr, ur, wr}, rb[3] = {rr, wr, rr};
        f = probe_pairs<3>(g.col, ra, rb, A, B);
    }
    // known: v-u, v-w, u-r
    const uint32_t mask = 0x1u | 0x2u | ((f & 1u) << 2) | (((f >> 1) & 1u) << 3) | 0x10u | (((f >> 2) & 1u) << 5);
    out.cls = lut[mask];
    // c(s) from the table (zero for the classes MOSS-4Min does not count)
    const uint64_t key[4] = {((uint64_t)mv.y << 32) | v, ((uint64_t)sb.y << 32) | u, ((uint64_t)we.y << 32) | w,
                             ((uint64_t)re.y << 32) | r};
    out.v[4] = lutc[mask << 6 | order_bits(key)];
    return out;
}

template <int RNG, bool HASH, int PM = kPmPlain>
__device__ __forceinline__ Sample sample_min(const DevGraph &g, const uint8_t *lut, const uint8_t *lutc, uint64_t seed,
                                             uint64_t s) {
    return rest_min<RNG, HASH, PM>(g, lut, lutc, seed, s, first_vertex<3, RNG, PM>(g, seed, s));
}

// Path-5 fallback: u from tau^(v), w from mu^(v,u) (Sec. 5.1.4).  The
// prefix of the tau weights w_i (S - w_i), w_i = d_x - 1, is S ACC[p] - sq[p],
// so u is the last position whose prefix is <= y, found by binary search
// (the same position a scan of the running sum gives); w by the search of
// ACC with u's interval removed.
__device__ __noinline__ void path5_fallback(const uint32_t *acc, const uint64_t *sq, uint32_t v, uint4 vr,
                                            uint64_t x12, uint64_t x13, uint32_t &iu, uint32_t &iw) {
    const uint32_t o = vr.x, d = vr.y, S = vr.z;
    const uint32_t wl = S - ld1(acc + o + d - 1);
    const uint64_t Q = __ldg(sq + o + d - 1) + (uint64_t)wl * wl;
    const uint64_t G = (uint64_t)S * S - Q;
    const uint64_t y = word_index(x12, G);
    {
        uint32_t lo = 0, len = d;   // first p with prefix(p) > y
        while (len > 0) {
            const uint32_t half = len >> 1, p = lo + half;
            const uint64_t f = (uint64_t)S * ld1(acc + o + p) - __ldg(sq + o + p);
            if (f <= y) {
                lo = p + 1;
                len -= half + 1;
            } else {
                len = half;
            }
        }
        iu = lo - 1;
    }
    const uint32_t au = ld1(acc + o + iu);
    const uint32_t wu = (iu + 1 < d ? ld1(acc + o + iu + 1) : S) - au;
    uint64_t y2 = word_index(x13, (uint64_t)(S - wu));
    if (y2 >= au) y2 += wu;
    // last i with ACC[i] <= y2
    uint32_t lo = 0, len = d;
    while (len > 0) {
        const uint32_t half = len >> 1;
        if ((uint64_t)ld1(acc + o + lo + half) <= y2) { lo += half + 1; len -= half + 1; } else { len = half; }
    }
    iw = lo - 1;
}

// Path-5 in stages, so that the rare paths do not set the register budget
// of the common one: STAGE 0 takes the first attempt and returns kDeferred
// when it collides (the main launch); STAGE 1 the second attempt of such a
// sample, again kDeferred when it collides; STAGE 2 the fallback of a sample
// whose two attempts collided; STAGE 3 all three in turn.  The draws depend
// only on the sample id, so the stages give the sample the same result as
// STAGE 3.
constexpr int kDeferred = 254;

template <int RNG, bool HASH, int STAGE, int PM>
__device__ __forceinline__ Sample rest_path5(const DevGraph &g, const uint8_t *lut, uint64_t seed, uint64_t s,
                                             const VertexPick &pv) {
    Sample out;
    const uint32_t v = pv.v;
    const uint4 vr = pv.rec;
    Pick pu, pw;
    bool collide = true;
    if (STAGE == 0 || STAGE == 3) {
        const Words2 x45 = sample_words2<RNG>(seed, 2, s, 2);
        const Words2 x67 = sample_words2<RNG>(seed, 2, s, 3);
        pu = draw_sigma<PM>(g.slot, g.vert, vr.x, vr.y, vr.z, x45.x[0], x45.x[1]);
        pw = draw_sigma<PM>(g.slot, g.vert, vr.x, vr.y, vr.z, x67.x[0], x67.x[1]);
        collide = pu.pos == pw.pos;
        if (STAGE == 0 && collide) {
            out.cls = kDeferred;
            return out;
        }
    }
    if (STAGE == 1 || (STAGE == 3 && collide)) {
        const Words2 x89 = sample_words2<RNG>(seed, 2, s, 4);
        const Words2 x1011 = sample_words2<RNG>(seed, 2, s, 5);
        pu = draw_sigma<PM>(g.slot, g.vert, vr.x, vr.y, vr.z, x89.x[0], x89.x[1]);
        pw = draw_sigma<PM>(g.slot, g.vert, vr.x, vr.y, vr.z, x1011.x[0], x1011.x[1]);
        collide = pu.pos == pw.pos;
        if (STAGE == 1 && collide) {
            out.cls = kDeferred;
            return out;
        }
    }
    if (STAGE == 2 || (STAGE == 3 && collide)) {
        const Words2 x1213 = sample_words2<RNG>(seed, 2, s, 6);
        uint32_t iu, iw;
        path5_fallback(g.acc, g.sq, v, vr, x1213.x[0], x1213.x[1], iu, iw);
        pu = slot_pick(g.slot, g.vert, vr.x, iu);
        pw = slot_pick(g.slot, g.vert, vr.x, iw);
    }
    const uint32_t u = pu.id, w = pw.id;
    const Words2 x23 = sample_words2<RNG>(seed, 2, s, 1);
    const uint32_t r = ldc<PM>(g.col + pu.off + skip1(word_index32(x23.x[0], pu.deg - 1), pu.twin));
    const uint32_t t = ldc<PM>(g.col + pw.off + skip1(word_index32(x23.x[1], pw.deg - 1), pw.twin));
    out.v[0] = v; out.v[1] = u; out.v[2] = w; out.v[3] = r; out.v[4] = t;
    if (t == u || r == w || t == r) {
        out.cls = 0;
        return out;
    }
    // unknown pairs: v-r, v-t, u-w, u-t, w-r, r-t
    const uint32_t A[6] = {v, v, u, u, w, r}, B[6] = {r, t, w, t, r, t};
    uint32_t f;
    if (HASH) {
        f = probe_hash<6, PM, kHubProbes[2], walk_of(PM, 2, STAGE)>(g, A, B);
    } else {
        const uint4 ur = make_uint4(pu.off, pu.deg, 0u, 0u), wr = make_uint4(pw.off, pw.deg, 0u, 0u);
        const uint4 rr = ld4(g.vert + r), tr = ld4(g.vert + t);
        const uint4 ra[6] = {vr, vr, ur, ur, wr, rr}, rb[6] = {rr, tr, wr, tr, rr, tr};
        f = probe_pairs<6>(g.col, ra, rb, A, B);
    }
    // known: v-u (0), v-w (1), u-r (5), w-t (8)
    uint32_t mask = 0x1u | 0x2u | 0x20u | 0x100u;
    mask |= ((f >> 0) & 1u) << 2;   // v-r
    mask |= ((f >> 1) & 1u) << 3;   // v-t
    mask |= ((f >> 2) & 1u) << 4;   // u-w
    mask |= ((f >> 3) & 1u) << 6;   // u-t
    mask |= ((f >> 4) & 1u) << 7;   // w-r
    mask |= ((f >> 5) & 1u) << 9;   // r-t
    out.cls = lut[mask];
    return out;
}

template <int RNG, bool HASH, int STAGE, int PM = kPmPlain>
__device__ __forceinline__ Sample sample_path5(const DevGraph &g, const uint8_t *lut, uint64_t seed, uint64_t s) {
    return rest_path5<RNG, HASH, STAGE, PM>(g, lut, seed, s, first_vertex<2, RNG, PM>(g, seed, s));
}

// The block's counts (its warps' histograms) added to the launch's sums, which
// are zero before it: whole numbers, so any order of the blocks gives the same.
// With a row per block and a kernel to add up the rows, an estimate of 5e6
// samples on a 2M-edge mesh took 448 us (440 like this), one of 1e4 on 8k edges
// 40.7 (39.1): a block's 22 adds go beside other blocks' samples.
template <int WARPS>
__device__ __forceinline__ void add_sums(const uint32_t (&hist)[WARPS][kSlots], uint64_t *sums) {
    if (threadIdx.x < kSlots) {
        uint64_t sum = 0;
        for (int w = 0; w < WARPS; ++w) sum += hist[w][threadIdx.x];
        if (sum) atomicAdd(reinterpret_cast<unsigned long long *>(sums) + threadIdx.x, (unsigned long long)sum);
    }
}

// the class tables of this translation unit on the current device
inline void upload_luts_here(const uint8_t *lut4, const uint8_t *lut5, const uint8_t *lutc) {
    cudaMemcpyToSymbol(g_lut4, lut4, 64);
    cudaMemcpyToSymbol(g_lut5, lut5, 1024);
    cudaMemcpyToSymbol(g_lutc, lutc, 4096);
}

}  // namespace

}  // namespace moss
