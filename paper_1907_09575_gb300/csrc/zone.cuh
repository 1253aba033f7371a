// Dense zones: the top labels of long rows of U as bit blocks.
//
// In degree order the highest labels are the hubs, and most of a long row
// lies among them: at RMAT scale 20 the entries with one of the top 2,048
// labels are 73 % of all table probes, one label in ten or more being present
// in the rows that are probed.  There a probe per entry is the wrong form:
// the row's stretch of 2,048 labels as 64 words of bits, one load of two
// words a lane, tests them all against the pivot's bits with two ANDs.
//
// Zone q is the labels [n - 2048 (q + 1), n - 2048 q).  A row of more than
// kZoneMinRow entries has blocks for zones 0 .. nz-1, nz the number of
// leading zones with at least kZoneMinCount of its entries (kZoneMinCount2
// beyond the first).  zrow[r] = {first block << kZoneNzBits | nz, the edge where the zoned entries begin};
// a task (i, j) of a pivot with more than kZoneMinPivot entries then has its
// tail cut at that edge and holds zrow[i].x: the zone kernel counts the
// rest.  Blocks that do not fit the capacity are left out
// (the row then stays a list).
#pragma once
#include "common.cuh"

namespace tc {

constexpr int kZoneLabels = 2048;
constexpr int kZoneWords = kZoneLabels / 32;
constexpr int kZoneNzBits = 5;        // of a task's zone word: the number of zones; above them the first block
constexpr int kZoneMax = (1 << kZoneNzBits) - 1;
#ifndef TC_ZONE_MIN_COUNT
#define TC_ZONE_MIN_COUNT 24
#endif
#ifndef TC_ZONE_MIN_COUNT2
#define TC_ZONE_MIN_COUNT2 32
#endif
constexpr int kZoneMinCount = TC_ZONE_MIN_COUNT;     // entries of zone 0 ...
constexpr int kZoneMinCount2 = TC_ZONE_MIN_COUNT2;   // ... and of a further one
constexpr int kZoneMinRow = 32;
constexpr int kMidMaxOutdeg = 256;    // largest pivot row that one warp counts
constexpr int kZoneMinPivot = 64;
constexpr int kZoneTasks = 248;       // tasks of one unit of the zone kernel: a label's hits fit a byte

// Block capacity of a graph of up to m edges: 2 B an edge (measured need: 0.6
// B an edge on a Chung-Lu graph to 1.3 B on RMAT scale 20); block 0 stands
// for none.  No zones, and no pivots of more than 64 entries for single warps,
// up to 2^19 edges: there a count is as long as its longest unit, which eight
// warps share, and the further launches cost what they save (kept RMAT graphs,
// totals: 2^17 pairs 30 us as CTA units, 52 by warps with zones; 2^18 47 and
// 69; 2^19 63 and 76; 2^20 106 and 92; 2^21 196 and 121).
// A graph preprocessed in one launch has them by its pairs, which the host
// knows before its edges: zcap, not m, says whether a graph has zones.
inline bool zones_at(int64_t m) { return m > (1ll << 19); }
inline int64_t zone_capacity(int64_t m) { return zones_at(m) ? m / 128 : 0; }   // x 256 B: below 2^32

// One warp makes the blocks of row r: adj[rb, rb + d), sorted, d >
// kZoneMinRow.  buf: kZoneWords words of the warp's shared memory.  nblocks
// counts the blocks taken (from 1).
__device__ __forceinline__ void zone_row(const int32_t* adj, int64_t rb, int d, int64_t r, int64_t n,
                                         uint2* zrow, uint32_t* zbits, uint32_t* zowner, int64_t cap,
                                         unsigned* nblocks, uint32_t* buf) {
    const int lane = threadIdx.x & 31;
    // leading zones with enough entries, from the row's end
    int nz = 0, split = d;
    for (int c = d; nz < kZoneMax;) {
        const int64_t low = n - (int64_t)kZoneLabels * (nz + 1);
        int count = 0;
        while (true) {
            const int p = c - count - 1 - lane;
            const int in = __popc(__ballot_sync(0xffffffffu, p >= 0 && adj[rb + max(p, 0)] >= low));
            count += in;
            if (in < 32) break;
        }
        if (count < (nz == 0 ? kZoneMinCount : kZoneMinCount2)) break;
        c -= count;
        split = c;
        ++nz;
        if (c == 0 || low <= 0) break;
    }
    if (nz == 0) return;
    unsigned at = 0;
    if (lane == 0) at = 1 + atomicAdd(nblocks, (unsigned)nz);
    at = __shfl_sync(0xffffffffu, at, 0);
    if ((int64_t)at + nz > cap) return;
    int c = d;
    for (int q = 0; q < nz; ++q) {
        const int64_t low = n - (int64_t)kZoneLabels * (q + 1);
        __syncwarp();
        buf[lane] = 0;
        buf[lane + 32] = 0;
        __syncwarp();
        while (true) {
            const int p = c - 1 - lane;
            const int64_t b = p >= 0 ? adj[rb + p] - low : -1;
            if (b >= 0) atomicOr(&buf[b >> 5], 1u << (b & 31));
            const int in = __popc(__ballot_sync(0xffffffffu, b >= 0));
            c -= in;
            if (in < 32) break;
        }
        __syncwarp();
        reinterpret_cast<uint2*>(zbits + (size_t)(at + q) * kZoneWords)[lane] = reinterpret_cast<uint2*>(buf)[lane];
    }
    if (lane == 0) {
        zowner[at] = (uint32_t)r;
        zrow[r] = make_uint2(at << kZoneNzBits | (unsigned)nz, (uint32_t)(rb + split));
    }
}

// The entries of edge e's tail (len of them) left to the list, and *z the
// zone task, for a pivot with (big) or without enough entries.
__device__ __forceinline__ int zone_cut(uint2 zr, bool big, int64_t e, int len, uint32_t* z) {
    if (!big || (zr.x & (unsigned)kZoneMax) == 0 || len <= 0) {
        *z = 0;
        return len;
    }
    *z = zr.x;
    return (int)max64((int64_t)zr.y - e - 1, 0);
}

// ---------------------------------------------------------------------------
// Which units a pivot of dp entries and nt tasks becomes: `small` ones (flat,
// k_light's second part), `large` ones (a CTA each) and `wide` ones, which
// k_light's first part counts with a table per warp (dp <= kMidMaxOutdeg) and
// the zone kernel visits (more than kZoneMinPivot entries, in a graph with
// zones; those above kMidMaxOutdeg are large as well).  A pivot of few
// entries is wide when its tasks make a table worth its building: about
// 600 instructions against 45 more a warp's step of the flat search.
#ifndef TC_FLAT_WORK
#define TC_FLAT_WORK 1024
#endif
constexpr int64_t kFlatWork = TC_FLAT_WORK;
static_assert(kFlatWork / 64 >= 16, "a wide pivot of few entries has at least 16 tasks");

struct UnitRule {
    int small_max, mid_max;   // mid_max 0: no wide pivots but the zones' own
    int merge_max;            // pivots of at most this many entries get no table
    int warp_tasks, cta_tasks, wide_tasks, slice;
    int zones;                // 0: no zones, or not used (lists are read whole), and no wide pivots
};

// MERGE: the rule has a merge_max (the one preprocessing plans for has none).
template <bool MERGE>
__host__ __device__ __forceinline__ void unit_split(const UnitRule& r, bool zoned, int64_t dp, int64_t nt,
                                                    int64_t& small, int64_t& large, int64_t& wide) {
    small = large = wide = 0;
    if (dp <= 0 || nt <= 0) return;
    const bool tabled = dp <= r.small_max && (!MERGE || dp > r.merge_max) && dp * nt >= kFlatWork;
    const bool mid = dp <= r.mid_max && (dp > kZoneMinPivot || tabled);
    if (mid || (zoned && dp > kZoneMinPivot)) wide = (nt + r.wide_tasks - 1) / r.wide_tasks;
    if (mid) return;
    if (dp <= r.small_max) small = (nt + r.warp_tasks - 1) / r.warp_tasks;
    else large = ((dp + r.slice - 1) / r.slice) * ((nt + r.cta_tasks - 1) / r.cta_tasks);
}

}  // namespace tc
