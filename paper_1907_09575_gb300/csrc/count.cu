// tc_count: Eq. 1 / Eq. 2 by the paper's <j,i,k> map-based enumeration.
//
// For a pivot j the row U_j (the labels k > j adjacent to j) is put in a
// shared-memory table once; every task (i,j) of j -- an edge of U whose row
// U_i continues after j -- then probes the table with each entry of U_i
// after j.  Each hit k is one triangle {i, j, k} counted at edge (i, j)
// (Eq. 1 sums exactly the k > j with u_ik = u_jk = 1).
//
// Tables (Section 5.2, "Modifying the hashing routine for sparser vertices"):
// a bitmap over [min U_j, max U_j] when that label span fits (collision
// free); else, for slices of at most kTagMaxEntries entries, a tag table
// (one slot per label hash holding the rest of the hashed label and the
// entry's rank: one load decides a probe exactly); else buckets of 4 slots
// with bucket = k AND (buckets - 1) (tc_tuning.table_mode = 1 forces
// buckets everywhere).  A probe outside [min U_j, max U_j] cannot hit --
// the per-probe form of the early exit of Section 5.2: a bitmap lookup
// clamps it onto a guard bit that is always clear, a bucket lookup rejects
// it before reading the table, a tag lookup finds no equal tag.
//
// Work: units (graph, pivot, slice of U_j, range of tasks), heaviest pivots
// first, popped by persistent kernels; units may come from many graphs at once
// (the batched form), each graph reached through a view table.  Pivots above
// 256 entries are CTA units (k_count: a shared table, slices of <= 4096
// entries); k_light counts the others, with a table per warp (65 to 256
// entries, or few entries and many tasks) or by searching the row; in small
// graphs that have CTA units k_count takes all, warp units after them.  Tails that
// lie among the top labels of long rows are counted as bits (zone.cu).  Tiles
// of host-resident graphs and table_mode 1 take k_count's other instances,
// where pivots of up to 64 entries are warp units with a private table.
//
// Per-vertex counts (t[v] = triangles through v): a task's hits credit i once,
// per-entry hit counters credit k once per unit, j is credited once per unit.
#include <algorithm>
#include <memory>

#include "common.cuh"
#include "tc_internal.cuh"

namespace tc {
namespace {

#ifndef TC_TLOW32
#define TC_TLOW32 1            // per-task credit into 32-bit counters when they cannot overflow
#endif
#ifndef TC_LARGE_MINB
#define TC_LARGE_MINB 4        // CTAs per SM the CTA kernel's registers must allow
#endif

constexpr int kGrab = 4;          // warp units popped per queue access ...
constexpr int kGrabMin = 8;       // ... when every warp gets this many or more, else one
constexpr int kEmpty = -1;
#ifndef TC_UNROLL
#define TC_UNROLL 4
#endif
constexpr int kUnroll = TC_UNROLL;   // independent loads in flight per lane
#ifndef TC_PV_BRANCHLESS
#define TC_PV_BRANCHLESS 1     // per-vertex bitmap probe: 1 computes the rank on every lane
#endif

// warp unit table region: 128 hash slots, or a 128-word bitmap (4095 labels
// and the guard bit)
// plus its 128 16-bit rank prefixes
constexpr int kSmallBitWords = 128;
constexpr int kSmallRegionWords = kSmallBitWords + kSmallBitWords / 2;
// CTA unit table region (32-bit words): hash slots <= 2 * slice <= 8192, or a
// bitmap of kBitWords words (kBitWords * 32 labels) plus 16-bit prefixes
#ifndef TC_REGION_WORDS
#define TC_REGION_WORDS 8192
#endif
constexpr int kRegionWords = TC_REGION_WORDS;
constexpr int kBitWords = (kRegionWords * 2 / 3) & ~31;
static_assert(kBitWords + kBitWords / 2 <= kRegionWords, "bitmap + prefix fit the region");

__device__ __forceinline__ int64_t shfl64(int64_t v, int src) {
    return __shfl_sync(0xffffffffu, v, src);
}

__device__ __forceinline__ int warp_incl_scan_i32(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The rows a launch counts and where their tails sit: all rows at their
// place for a device-resident graph; for one tile of a host-resident graph
// the rows [i0, i1) of its row block, whose entries start `shift` entries
// into the tile's row buffer.
struct TaskWindow {
    int i0, i1;
    int64_t shift;
};

// *p += 1 in shared memory when h is set: one predicated reduction, no
// branch around it.  p must point into shared memory; when h is 0 the
// address is formed but never accessed, so it may lie outside the array.
__device__ __forceinline__ void add_if(unsigned* p, unsigned h) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %1, 0;\n\t@q red.shared.add.u32 [%0], 1;\n\t}"
                 ::"r"(a), "r"(h) : "memory");
}

// bits [lo, hi) of a 32-bit mask, 0 <= lo <= hi <= 32
__device__ __forceinline__ unsigned bit_range(int lo, int hi) {
    const unsigned up = (hi >= 32) ? 0xffffffffu : ((1u << hi) - 1u);
    const unsigned dn = (lo >= 32) ? 0xffffffffu : ((1u << lo) - 1u);
    return up & ~dn;
}

// ---------------------------------------------------------------------------
// Tables for one pivot slice S = U_j[rb, re) (sorted labels lo..hi).
//
// Bitmap (the direct, collision-free case of Section 5.2): bit k - lo is set
// for k in S.  Membership is one shared load and a shift.  The rank of a hit
// among S -- its position in the slice, used to credit per-vertex counts --
// is the 16-bit prefix popcount of the words before it plus a popcount.
//
// Hash (labels too spread for a bitmap): 4-slot buckets, bucket = k AND
// (buckets - 1) (the paper's AND hash), overflow to the next bucket; the
// occupied slots of a bucket are a prefix, so an empty last slot ends a miss.
// Both return a counter index for per-vertex credit (rank or slot), or -1.
// A probe of -1 (a lane past the end of a tail) is a miss in every table:
// the bitmap clamps it onto the guard bit, the others fail the window test.
// ---------------------------------------------------------------------------
struct BitTab {
    const unsigned* bm;
    const unsigned short* pre;
    int lo, hi;
    // labels outside [lo, hi] are clamped onto bit hi - lo + 1, which the
    // table keeps clear: no range test, no branch
    __device__ __forceinline__ unsigned offset(int k) const {
        return min((unsigned)(k - lo), (unsigned)(hi - lo + 1));
    }
    template <bool PV>
    __device__ __forceinline__ int find(int k) const {
        const unsigned d = offset(k);
        const unsigned w = bm[d >> 5];
        if (!((w >> (d & 31)) & 1u)) return -1;
        if (!PV) return 0;
        return (int)pre[d >> 5] + __popc(w & ((1u << (d & 31)) - 1u));
    }
    __device__ __forceinline__ unsigned bit(int k) const {
        const unsigned d = offset(k);
        return (bm[d >> 5] >> (d & 31)) & 1u;
    }
    // membership and rank without a branch on the membership: the rank is
    // read for every probe (the guard bit's word has a prefix too), and only
    // the credit is predicated on the hit
    __device__ __forceinline__ void probe_credit(int k, unsigned* cnt, unsigned& mine) const {
        const unsigned d = offset(k);
        const unsigned w = bm[d >> 5];
        // bit d & 31 moved to the top: the sign is the hit, and the popc
        // counts the bits up to and including it
        const unsigned x = w << (~d & 31u);
        mine += x >> 31;
        const int r1 = (int)pre[d >> 5] + __popc(x);
        add_if(&cnt[r1 - 1], x >> 31);
    }
    // hit counters by rank (rank < slice <= 4096): one word each, so hits on
    // neighbouring entries never share an atomic's word
    __device__ __forceinline__ void credit(unsigned* cnt, int r) const { atomicAdd(&cnt[r], 1u); }
    __device__ __forceinline__ unsigned credited(const unsigned* cnt, int r) const { return cnt[r]; }
};

struct HashTab {
    const int* tab;
    unsigned bmask;
    int lo, hi;
    template <bool PV>
    __device__ __forceinline__ int find(int k) const {
        if ((unsigned)(k - lo) > (unsigned)(hi - lo)) return -1;
        unsigned b = (unsigned)k & bmask;
        while (true) {
            const int4 v = reinterpret_cast<const int4*>(tab)[b];
            if (v.x == k) return (int)(4 * b);
            if (v.y == k) return (int)(4 * b + 1);
            if (v.z == k) return (int)(4 * b + 2);
            if (v.w == k) return (int)(4 * b + 3);
            if (v.w == kEmpty) return -1;
            b = (b + 1) & bmask;
        }
    }
    __device__ __forceinline__ unsigned bit(int k) const { return find<false>(k) >= 0; }
    // hit counters by slot (up to twice the slice): 16 bits each, two a
    // word (a counter never exceeds the tasks of a unit, below 2^16 by the
    // unit size cap)
    __device__ __forceinline__ void credit(unsigned* cnt, int r) const {
        atomicAdd(&cnt[r >> 1], 1u << ((r & 1) << 4));
    }
    __device__ __forceinline__ unsigned credited(const unsigned* cnt, int r) const {
        return (cnt[r >> 1] >> ((r & 1) << 4)) & 0xffffu;
    }
};

// Tag table, for slices of at most kTagMaxEntries entries whose labels are
// too spread for the bitmap: p = k * kTagMul (mod 2^32) is a bijection of
// the label; its top b bits pick one of 2^b slots (per-vertex: about 8 an
// entry, 1024 to 8192; totals only: 8192, the whole table region) and the
// slot keeps the low 32 - b bits of p (the tag) with the entry's rank in
// the bits above, below bit 31, so one 32-bit load decides membership
// exactly and gives the rank.  A slot two entries map to holds kTagMulti;
// those entries go to a second table of 2048 slots (another multiplier,
// 21-bit tags) beside the hit counters, and an entry that collides there
// too is found by a binary search of the sorted slice.
constexpr int kTagMaxEntries = 1024;                 // ranks below 2^10 in the second table
constexpr int kTagSlots = 8192;                      // first table: at most 13 index bits
constexpr int kTagSlots2 = 2048, kTag2Shift = 21;    // second table: 11 index bits, 21 tag bits
constexpr unsigned kTag2Mask = (1u << kTag2Shift) - 1u;
static_assert(kTagMaxEntries <= (1 << (31 - kTag2Shift)), "ranks fit both tables below bit 31");
static_assert(kTagSlots <= kRegionWords, "the first table fills at most the region");
static_assert(kTagMaxEntries + kTagSlots2 <= kRegionWords / 2, "counters and second table share the counters' space");
#ifndef TC_TAG_SUB
#define TC_TAG_SUB 1024        // entries of a tag table; a longer slice is probed in sub-slices
#endif
constexpr int kTagSub = TC_TAG_SUB;
static_assert(kTagSub >= 1 && kTagSub <= kTagMaxEntries, "a sub-slice fits the tables");
constexpr unsigned kTagMul = 0x9E3779B1u, kTagMul2 = 0x85EBCA77u;
constexpr unsigned kTagEmpty = 0xffffffffu, kTagMulti = 0xfffffffeu;

struct TagTab {
    const unsigned* t1;        // 2^(32 - s1) words
    const unsigned* t2;        // kTagSlots2 words
    const int32_t* row;        // the sorted slice in device memory
    int dp;
    int s1;                    // tag bits of the first table
    unsigned m1;               // (1 << s1) - 1
    __device__ int slow(int k) const {
        const unsigned p = (unsigned)k * kTagMul2;
        const unsigned w = t2[p >> kTag2Shift];
        if (w != kTagMulti) return ((w & (0x80000000u | kTag2Mask)) == (p & kTag2Mask)) ? (int)(w >> kTag2Shift) : -1;
        int a = 0, b = dp;
        while (a < b) {
            const int c = (a + b) >> 1;
            if (__ldg(row + c) < k) a = c + 1; else b = c;
        }
        return (a < dp && __ldg(row + a) == k) ? a : -1;
    }
    template <bool PV>
    __device__ __forceinline__ int find(int k) const {
        const unsigned p = (unsigned)k * kTagMul;
        const unsigned w = t1[p >> s1];
        if (w == kTagMulti) return slow(k);
        return ((w & (0x80000000u | m1)) == (p & m1)) ? (int)(w >> s1) : -1;
    }
    __device__ __forceinline__ unsigned bit(int k) const { return find<false>(k) >= 0; }
    __device__ __forceinline__ void probe_credit(int k, unsigned* cnt, unsigned& mine) const {
        const unsigned p = (unsigned)k * kTagMul;
        const unsigned w = t1[p >> s1];
        unsigned h = (w & (0x80000000u | m1)) == (p & m1);
        int r = (int)(w >> s1);
        if (w == kTagMulti) {
            r = slow(k);
            h = r >= 0;
        }
        mine += h;
        add_if(&cnt[r], h);
    }
    __device__ __forceinline__ void credit(unsigned* cnt, int r) const { atomicAdd(&cnt[r], 1u); }
    __device__ __forceinline__ unsigned credited(const unsigned* cnt, int r) const { return cnt[r]; }
};

__device__ __forceinline__ void tag_insert2(unsigned* t2, int k, int q) {
    const unsigned p = (unsigned)k * kTagMul2;
    unsigned* s = t2 + (p >> kTag2Shift);
    if (atomicCAS(s, kTagEmpty, ((unsigned)q << kTag2Shift) | (p & kTag2Mask)) != kTagEmpty) atomicExch(s, kTagMulti);
}

// The tag table of one warp, for a pivot of at most kMidEntries entries: the
// same on the 31 bits of a label (labels are below 2^31 - 1, and the -1 of a
// lane without a probe becomes 2^31 - 1: a miss), which leaves room for the
// rank beside the longer tags of smaller tables.
constexpr int kMidEntries = kMidMaxOutdeg;           // 256: ranks of 8 bits
constexpr int kMidSlotBits = 10, kMidSlots = 1 << kMidSlotBits;
constexpr int kMidSlot2Bits = 8, kMidSlots2 = 1 << kMidSlot2Bits;
constexpr int kMidTag = 31 - kMidSlotBits, kMidTag2 = 31 - kMidSlot2Bits;
static_assert(kMidEntries <= (1 << (31 - kMidTag2)), "ranks fit both tables below bit 31");
constexpr unsigned kMid31 = 0x7fffffffu;

struct MidTab {
    const unsigned* t1;
    const unsigned* t2;
    const int32_t* row;
    int dp;
    __device__ int slow(int k) const {
        const unsigned p = ((unsigned)k * kTagMul2) & kMid31;
        const unsigned w = t2[p >> kMidTag2];
        if (w != kTagMulti)
            return ((w ^ p) & (0x80000000u | ((1u << kMidTag2) - 1u))) == 0 ? (int)(w >> kMidTag2) : -1;
        int a = 0, b = dp;
        while (a < b) {
            const int c = (a + b) >> 1;
            if (__ldg(row + c) < k) a = c + 1; else b = c;
        }
        return (a < dp && __ldg(row + a) == k) ? a : -1;
    }
    template <bool PV>
    __device__ __forceinline__ int find(int k) const {
        const unsigned p = ((unsigned)k * kTagMul) & kMid31;
        const unsigned w = t1[p >> kMidTag];
        if (w == kTagMulti) return slow(k);
        return ((w ^ p) & (0x80000000u | ((1u << kMidTag) - 1u))) == 0 ? (int)(w >> kMidTag) : -1;
    }
    __device__ __forceinline__ unsigned bit(int k) const { return find<false>(k) >= 0; }
    __device__ __forceinline__ void probe_credit(int k, unsigned* cnt, unsigned& mine) const {
        const int r = find<true>(k);
        mine += r >= 0;
        add_if(&cnt[r], r >= 0);
    }
    __device__ __forceinline__ void credit(unsigned* cnt, int r) const { atomicAdd(&cnt[r], 1u); }
    __device__ __forceinline__ unsigned credited(const unsigned* cnt, int r) const { return cnt[r]; }
};

__device__ __forceinline__ void hash_insert(int* tab, unsigned bmask, int k) {
    unsigned b = (unsigned)k & bmask;
    while (true) {
#pragma unroll
        for (int w = 0; w < 4; ++w)
            if (atomicCAS(&tab[4 * b + w], kEmpty, k) == kEmpty) return;
        b = (b + 1) & bmask;
    }
}

__device__ __forceinline__ unsigned hash_buckets(int dp) {
    unsigned b = 1;
    while (4 * b < 2u * (unsigned)dp) b <<= 1;   // load factor <= 1/2
    return b;
}


template <class Tab>
struct has_probe_credit {
    template <class U>
    static constexpr bool check(decltype(&U::probe_credit)) { return true; }
    template <class U>
    static constexpr bool check(...) { return false; }
    static constexpr bool value = check<Tab>(nullptr);
};

template <bool PV, class Tab>
__device__ __forceinline__ void probe_one(const Tab& T, int k, unsigned* cnt, unsigned& mine) {
    if constexpr (!PV) {
        mine += T.bit(k);
    } else if constexpr (TC_PV_BRANCHLESS && has_probe_credit<Tab>::value) {
        T.probe_credit(k, cnt, mine);
    } else {
        const int r = T.template find<PV>(k);
        if (r >= 0) {
            ++mine;
            T.credit(cnt, r);
        }
    }
}

// ---------------------------------------------------------------------------
// One warp walks one long tail (>= 32 entries with per-vertex counts, >= 64
// for totals only) adj[st, st+L): lane q of a
// step reads entry q, kUnroll steps a round.  Returns the task's hits (the
// same in all lanes) with per-vertex counts, else 0.
//
// Per-vertex: the next round's entries are loaded before this round is
// probed, so a tail of up to 2 * 32 * kUnroll entries waits on memory about
// once.  Totals only: unchecked full rounds, then a checked last one -- the
// lighter probe leaves no latency worth the extra registers to hide.
// ---------------------------------------------------------------------------
template <bool PV, class Tab>
__device__ __forceinline__ unsigned warp_walk_tail(int64_t st, int L, const int32_t* __restrict__ adj,
                                                   const Tab& T, unsigned* cnt, uint64_t& hits) {
    const int lane = threadIdx.x & 31;
    const int32_t* __restrict__ p = adj + st + lane;
    unsigned mine = 0;
    if constexpr (PV) {
        int k[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) k[u] = (32 * u + lane < L) ? __ldg(p + 32 * u) : -1;
        for (int q0 = 0; q0 < L; q0 += 32 * kUnroll) {
            const int q1 = q0 + 32 * kUnroll;
            int kn[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) kn[u] = (q1 + 32 * u + lane < L) ? __ldg(p + q1 + 32 * u) : -1;
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) probe_one<PV>(T, k[u], cnt, mine);   // -1: a miss
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) k[u] = kn[u];
        }
        hits += mine;
        return __reduce_add_sync(0xffffffffu, mine);
    } else {
        int q0 = 0;
        for (; q0 + 32 * kUnroll <= L; q0 += 32 * kUnroll) {
            int k[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) k[u] = __ldg(p + q0 + 32 * u);
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) probe_one<PV>(T, k[u], cnt, mine);
        }
        if (q0 < L) {
            int k[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const int q = q0 + 32 * u + lane;
                k[u] = (q < L) ? __ldg(p + q0 + 32 * u) : -1;
            }
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) probe_one<PV>(T, k[u], cnt, mine);   // -1: a miss
        }
        hits += mine;
        return 0;
    }
}

// A task's hits (i's share of its triangles, at most C(|U_i|, 2)): into the
// 32-bit counters tlow when the caller provides them (the largest row keeps
// that share below 2^32; half the bytes of the 64-bit accumulator, so more
// of the scattered atomics stay in L2), else into tnew.
__device__ __forceinline__ void credit_task(unsigned long long* tnew, unsigned* tlow, int i, unsigned c) {
    if (tlow)
        atomicAdd(&tlow[i], c);
    else
        atomicAdd(&tnew[i], (unsigned long long)c);
}

__device__ __forceinline__ int64_t off_at(const GraphView& G, int64_t v) {
    return G.off64 ? static_cast<const int64_t*>(G.off)[v]
                   : (int64_t) static_cast<const int32_t*>(G.off)[v];
}

// WHOLE: the length of a task's tail with what the zones hold of it
template <bool WHOLE>
__device__ __forceinline__ int tail_length(const GraphView& G, const Task& t) {
    if (WHOLE && t.zone) return (int)(off_at(G, (int64_t)t.i + 1) - (int64_t)t.start);
    return t.len;
}

// ---------------------------------------------------------------------------
// One warp takes up to 32 tasks [tb, min(tb+32, t1)).
//
// Long tails (>= kShort entries) are either walked right away (defer == null) or
// appended to the CTA's queue of long tasks (their index relative to t0), to
// be shared out one task per warp later.  Short tails are concatenated: lane
// q of a step reads entry q of the concatenation; its owner is the number of
// short tasks starting at or before the step's first position, plus those
// starting inside the step before q (a ballot and a warp OR-reduce), minus
// one; the short tasks' start - prefix are compacted into s_base by rank, so
// the address is s_base[owner] + q.
// PV: lane s keeps the hit ballot of step s (a group's short tails total at
// most 31 * 32 entries, so 31 steps); a short task, which spans at most two
// steps, takes its hits from their popcounts over its positions at the end.
// Each task's hits go once to tnew[i]; per-entry hits to the counters cnt.
// ---------------------------------------------------------------------------
template <bool PV, bool WIN, bool WHOLE, class Tab>
__device__ __forceinline__ void warp_probe_group(const GraphView& G, const Task* __restrict__ tasks, int64_t tb, int64_t t1,
                                                 const int32_t* __restrict__ adj, const Tab& T,
                                                 unsigned* cnt, unsigned long long* tnew, unsigned* tlow,
                                                 int64_t* s_base, int64_t t0, unsigned short* defer,
                                                 int* ndefer, uint64_t& hits, uint64_t& probes,
                                                 const TaskWindow& win) {
    const int lane = threadIdx.x & 31;
    const int64_t t = tb + lane;
    const bool valid = t < t1;
    int64_t start = 0;
    int len = 0, i = 0;
    if (valid) {
        const Task tk = tasks[t];
        start = tk.start;
        len = tail_length<WHOLE>(G, tk);
        i = tk.i;
        if (WIN) {
            // a tile of a host-resident graph: rows outside its block wait
            // for another tile; tails are read from the tile's row buffer
            if (i < win.i0 || i >= win.i1) len = 0;
            start -= win.shift;
        }
    }
    unsigned c = 0;
    const unsigned le = (2u << lane) - 1u;   // bits 0..lane

    // long tails
    // tails shorter than kShort are concatenated across the lanes: 32 with
    // per-vertex counts (a short task then spans at most two steps), 64
    // for totals only (measured: the per-vertex short path costs more per
    // step than the longer walk of tails of 32-63 entries)
    constexpr int kShort = PV ? 32 : 64;
    const bool lg = valid && len >= kShort;
    unsigned longm = __ballot_sync(0xffffffffu, lg);
    if (defer) {
        if (longm) {
            int slot = 0;
            if (lane == 0) slot = atomicAdd(ndefer, __popc(longm));
            slot = __shfl_sync(0xffffffffu, slot, 0);
            if (lg) defer[slot + __popc(longm & (le >> 1))] = (unsigned short)(t - t0);
        }
    } else {
        while (longm) {
            const int o = __ffs(longm) - 1;
            longm &= longm - 1;
            const int64_t st = shfl64(start, o);
            const int L = __shfl_sync(0xffffffffu, len, o);
            probes += (uint64_t)L;
            const unsigned ch = warp_walk_tail<PV>(st, L, adj, T, cnt, hits);
            if (PV && lane == o) c += ch;
        }
    }

    // short tails, concatenated
    const int slen = (valid && len < kShort) ? len : 0;
    const int incl = warp_incl_scan_i32(slen);
    const int excl = incl - slen;
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    const bool sv = slen > 0;
    const unsigned shortm = __ballot_sync(0xffffffffu, sv);
    if (sv) s_base[__popc(shortm & (le >> 1))] = start - excl;
    __syncwarp();
    probes += (uint64_t)total;
    unsigned step_hits = 0;   // PV: the hit ballot of step `lane`
    for (int q0 = 0; q0 < total; q0 += 32 * kUnroll) {
        int k[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int qb = q0 + 32 * u;
            const unsigned before = __ballot_sync(0xffffffffu, sv && excl <= qb);
            const int d = excl - qb;
            const unsigned head = (sv && d > 0 && d < 32) ? (1u << d) : 0u;
            const unsigned M = __reduce_or_sync(0xffffffffu, head);
            const int o = __popc(before) - 1 + __popc(M & le);
            const int q = qb + lane;
            k[u] = (q < total) ? __ldg(&adj[s_base[o] + q]) : -1;
        }
        int r[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) r[u] = T.template find<PV>(k[u]);   // -1 (past the end): a miss
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const bool hit = r[u] >= 0;
            hits += hit ? 1 : 0;
            if (PV) {
                const unsigned hm = __ballot_sync(0xffffffffu, hit);
                if (lane == (q0 >> 5) + u) step_hits = hm;
                if (hit) T.credit(cnt, r[u]);
            }
        }
    }
    if (PV && total > 0) {
        const int s0 = excl >> 5, b0 = excl & 31;
        const unsigned h0 = __shfl_sync(0xffffffffu, step_hits, s0);
        const unsigned h1 = __shfl_sync(0xffffffffu, step_hits, (s0 + 1) & 31);
        if (sv) {
            c += __popc(h0 & bit_range(b0, min(b0 + slen, 32)));
            if (b0 + slen > 32) c += __popc(h1 & bit_range(0, b0 + slen - 32));
        }
    }
    __syncwarp();   // s_base is rewritten by the warp's next group
    if (PV && valid && c) credit_task(tnew, tlow, i, c);
}

// Per-warp running total of hits bound for one counter (a graph's total, or
// a component's total), flushed when the warp moves to a unit whose hits go
// elsewhere (and at the end).  Every triangle found at pivot j lies in j's
// component, so the pivot decides the counter.
__device__ __forceinline__ unsigned long long* unit_target(const GraphView& G, const Unit& U) {
    return G.comp ? G.comp_totals + G.comp[U.j] : G.total;
}

struct GraphAcc {
    unsigned long long* target = nullptr;
    uint64_t hits = 0;
    __device__ __forceinline__ void to(unsigned long long* t) {
        if (t == target) return;
        flush();
        target = t;
    }
    __device__ __forceinline__ void flush() {
        const uint64_t s = warp_sum_u64(hits);
        if ((threadIdx.x & 31) == 0 && target && s) atomicAdd(target, (unsigned long long)s);
        hits = 0;
    }
};

// ---------------------------------------------------------------------------
// Warp unit: a pivot with |U_j| <= 64 processed by one warp with a private
// table (a bitmap of <= 4095 labels, or 128 hash slots).
// ---------------------------------------------------------------------------
template <bool PV, bool WIN>
__device__ __forceinline__ void warp_unit(const GraphView& G, const Unit& U, unsigned* region,
                                          unsigned* cnt, int64_t* s_base, bool hash_only,
                                          unsigned* tlow, uint64_t& hits, uint64_t& probes, uint64_t& staged) {
    const int lane = threadIdx.x & 31;
    const int64_t rb = off_at(G, U.j), re = off_at(G, U.j + 1);
    const int dp = (int)(re - rb);
    const int lo = G.adj[rb], hi = G.adj[re - 1];
    const int mine = (lane < dp) ? G.adj[rb + lane] : 0;
    const int mine2 = (lane + 32 < dp) ? G.adj[rb + 32 + lane] : 0;
    const bool bitmap = !hash_only && (int64_t)hi - lo + 1 < 32 * kSmallBitWords;   // labels + guard bit
    uint64_t uh = 0;
    if (PV)
        for (int s = lane; s < kSmallTable / 2; s += 32) cnt[s] = 0;
    if (bitmap) {
        const int words = ((hi - lo + 1) >> 5) + 1;
        for (int s = lane; s < words; s += 32) region[s] = 0;
        __syncwarp();
        if (lane < dp) atomicOr(&region[(mine - lo) >> 5], 1u << ((mine - lo) & 31));
        if (lane + 32 < dp) atomicOr(&region[(mine2 - lo) >> 5], 1u << ((mine2 - lo) & 31));
        __syncwarp();
        unsigned short* pre = reinterpret_cast<unsigned short*>(region + kSmallBitWords);
        if (PV) {
            // prefix popcounts of the (at most 128) words, 4 per lane
            int a[4], sum = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int wi = lane * 4 + q;
                a[q] = (wi < words) ? __popc(region[wi]) : 0;
                sum += a[q];
            }
            int run = warp_incl_scan_i32(sum) - sum;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int wi = lane * 4 + q;
                if (wi < words) pre[wi] = (unsigned short)run;
                run += a[q];
            }
        }
        __syncwarp();
        const BitTab T{region, pre, lo, hi};
        for (int64_t tb = U.t0; tb < U.t1; tb += 32)
            warp_probe_group<PV, WIN, false>(G, G.tasks, tb, U.t1, G.adj, T, cnt, G.tnew, tlow, s_base, U.t0, nullptr,
                                      nullptr, uh, probes, TaskWindow{G.i0, G.i1, G.tail_shift});
        __syncwarp();
        if (PV) {
            if (lane < dp) {
                const unsigned h = T.credited(cnt, lane);
                if (h) atomicAdd(&G.tnew[mine], (unsigned long long)h);
            }
            if (lane + 32 < dp) {
                const unsigned h = T.credited(cnt, lane + 32);
                if (h) atomicAdd(&G.tnew[mine2], (unsigned long long)h);
            }
        }
    } else {
        int* tab = reinterpret_cast<int*>(region);
        const unsigned bmask = hash_buckets(dp) - 1u;
        for (int s = lane; s < kSmallTable; s += 32) tab[s] = kEmpty;
        __syncwarp();
        if (lane < dp) hash_insert(tab, bmask, mine);
        if (lane + 32 < dp) hash_insert(tab, bmask, mine2);
        __syncwarp();
        const HashTab T{tab, bmask, lo, hi};
        for (int64_t tb = U.t0; tb < U.t1; tb += 32)
            warp_probe_group<PV, WIN, false>(G, G.tasks, tb, U.t1, G.adj, T, cnt, G.tnew, tlow, s_base, U.t0, nullptr,
                                      nullptr, uh, probes, TaskWindow{G.i0, G.i1, G.tail_shift});
        __syncwarp();
        if (PV)
            for (int s = lane; s < kSmallTable; s += 32) {
                const unsigned h = T.credited(cnt, s);
                if (h) atomicAdd(&G.tnew[tab[s]], (unsigned long long)h);
            }
    }
    staged += (uint64_t)dp;
    hits += uh;
    if (PV) {
        uh = warp_sum_u64(uh);
        if (lane == 0 && uh) atomicAdd(&G.tnew[G.jbase + U.j], (unsigned long long)uh);
    }
    __syncwarp();
}

// ---------------------------------------------------------------------------
// CTA unit: a slice of a larger pivot with its table shared by the CTA.
// Phase A: warps take groups of 32 tasks from a shared counter, probe the
// short tails and queue the long ones; phase B: warps pop one long task at a
// time, with later tasks' records already loading and the next tail
// prefetched into L2 while the current tail is walked.
// ---------------------------------------------------------------------------
template <bool PV, bool WIN, bool WHOLE, class Tab>
__device__ __forceinline__ void cta_probe_unit(const GraphView& G, const Unit& U, const Tab& T,
                                               unsigned* cnt, int* s_ctl, int64_t* s_base,
                                               unsigned short* s_long, unsigned* tlow, uint64_t& uh,
                                               uint64_t& probes) {
    // s_ctl: [0] next group, [1] deferred long tasks, [2] next long task
    const int lane = threadIdx.x & 31;
    const Task* __restrict__ tasks = G.tasks;
    const int32_t* __restrict__ adj = G.adj;
    while (true) {
        int g = 0;
        if (lane == 0) g = atomicAdd(&s_ctl[0], 1);
        g = __shfl_sync(0xffffffffu, g, 0);
        const int64_t tb = U.t0 + (int64_t)g * 32;
        if (tb >= U.t1) break;
        warp_probe_group<PV, WIN, WHOLE>(G, tasks, tb, U.t1, adj, T, cnt, G.tnew, tlow, s_base, U.t0, s_long,
                                  &s_ctl[1], uh, probes, TaskWindow{G.i0, G.i1, G.tail_shift});
    }
    __syncthreads();
    const int nlong = s_ctl[1];
    auto pop = [&]() {
        int v = 0;
        if (lane == 0) v = atomicAdd(&s_ctl[2], 1);
        return __shfl_sync(0xffffffffu, v, 0);
    };
    // deferred tasks passed the window in phase A; only their tails move
    const int64_t shift = WIN ? G.tail_shift : 0;
    auto record = [&](int x) {
        Task t;
        t.len = 0;
        if (x < nlong) {
            t = tasks[U.t0 + s_long[x]];
            t.len = tail_length<WHOLE>(G, t);
            t.start -= shift;
        }
        return t;
    };
    // the next task's tail is prefetched into L2 while this one is walked
    auto prefetch_tail = [&](const Task& t) {
        if (32 * lane < t.len) asm volatile("prefetch.global.L2 [%0];" ::"l"(adj + t.start + 32 * lane));
    };
    if constexpr (!PV) {
        // records two tasks ahead: the record load of task x+2 overlaps the
        // walk of task x, and the prefetch of x+1's tail waits on nothing
        int x = pop(), x1 = pop();
        Task cur = record(x), nxt = record(x1);
        while (x < nlong) {
            const int x2 = pop();
            const Task nn = record(x2);
            prefetch_tail(nxt);
            probes += (uint64_t)cur.len;
            warp_walk_tail<PV>(cur.start, cur.len, adj, T, cnt, uh);
            x = x1;
            x1 = x2;
            cur = nxt;
            nxt = nn;
        }
    } else {
        // one task ahead (a third record would spill the per-vertex kernel;
        // written out, as the helpers above cost it registers too)
        int x = pop();
        Task cur;
        cur.len = 0;
        if (x < nlong) {
            cur = tasks[U.t0 + s_long[x]];
            cur.len = tail_length<WHOLE>(G, cur);
            cur.start -= shift;
        }
        while (x < nlong) {
            const int xn = pop();
            Task nxt;
            nxt.len = 0;
            if (xn < nlong) {
                nxt = tasks[U.t0 + s_long[xn]];
                nxt.len = tail_length<WHOLE>(G, nxt);
                nxt.start -= shift;
                if (32 * lane < nxt.len)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(adj + nxt.start + 32 * lane));
            }
            probes += (uint64_t)cur.len;
            const unsigned ch = warp_walk_tail<PV>(cur.start, cur.len, adj, T, cnt, uh);
            if (lane == 0 && ch) credit_task(G.tnew, tlow, cur.i, ch);
            x = xn;
            cur = nxt;
        }
    }
}

// BUCKETS: the instance for tc_tuning.table_mode = 1, every slice in
// 4-slot buckets; otherwise a bitmap when the slice's label span fits, else
// tag tables.  The two are separate instances because the bucket code,
// compiled into the default kernel, slowed its bitmap walk (2 %).
template <bool PV, bool WIN, bool BUCKETS>
__device__ __forceinline__ void cta_unit(const GraphView& G, const Unit& U, int slice_max,
                                         unsigned* region, unsigned* cnt, int* s_ctl,
                                         int64_t* s_base, unsigned short* s_long,
                                         unsigned* s_wsum, unsigned* tlow, uint64_t& hits, uint64_t& probes) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t rb = off_at(G, U.j) + (int64_t)U.slice * slice_max;
    const int64_t re = min64(off_at(G, U.j + 1), rb + slice_max);
    const int dp = (int)(re - rb);
    const int lo = G.adj[rb], hi = G.adj[re - 1];
    const bool bitmap = !BUCKETS && (int64_t)hi - lo + 1 < 32ll * kBitWords;   // labels + guard bit
    uint64_t uh = 0;
    // counters: by rank (< dp) for bitmaps and tag tables, by 16-bit slot
    // for buckets
    if (PV)
        for (int s = threadIdx.x; s < (BUCKETS ? kRegionWords / 2 : dp); s += blockDim.x) cnt[s] = 0;
    if (bitmap) {
        const int words = ((hi - lo + 1) >> 5) + 1;
        for (int s = threadIdx.x; s < words; s += blockDim.x) region[s] = 0;
        __syncthreads();
        for (int q = threadIdx.x; q < dp; q += blockDim.x) {
            const int k = G.adj[rb + q] - lo;
            atomicOr(&region[k >> 5], 1u << (k & 31));
        }
        __syncthreads();
        unsigned short* pre = reinterpret_cast<unsigned short*>(region + kBitWords);
        if (PV) {
            // prefix popcounts over the words: each thread a contiguous run
            const int per = (words + blockDim.x - 1) / blockDim.x;
            const int w0 = threadIdx.x * per;
            int sum = 0;
            for (int q = 0; q < per; ++q)
                if (w0 + q < words) sum += __popc(region[w0 + q]);
            const int inc = warp_incl_scan_i32(sum);
            if (lane == 31) s_wsum[w] = (unsigned)inc;
            __syncthreads();
            int before = 0;
            for (int q = 0; q < w; ++q) before += (int)s_wsum[q];
            int run = before + inc - sum;
            for (int q = 0; q < per; ++q)
                if (w0 + q < words) {
                    pre[w0 + q] = (unsigned short)run;
                    run += __popc(region[w0 + q]);
                }
            __syncthreads();
        }
        const BitTab T{region, pre, lo, hi};
        cta_probe_unit<PV, WIN, false>(G, U, T, cnt, s_ctl, s_base, s_long, tlow, uh, probes);
        __syncthreads();
        if (PV)
            for (int r = threadIdx.x; r < dp; r += blockDim.x) {
                const unsigned h = T.credited(cnt, r);
                if (h) atomicAdd(&G.tnew[G.adj[rb + r]], (unsigned long long)h);
            }
    } else if (!BUCKETS) {
        // tag tables over sub-slices of at most kTagMaxEntries entries, the
        // unit's tasks probing each in turn (a slice that long and that
        // spread is rare: none in RMAT scale 26)
        for (int sb = 0; sb < dp; sb += kTagSub) {
            const int sd = min(dp - sb, kTagSub);
            const int64_t sr = rb + sb;
            // the second table sits past the counters the slice can use (for
            // totals only, where the counters are); a barrier first, as the
            // counters were just cleared (or the last pass just read them)
            unsigned* t2 = cnt + (PV ? kTagMaxEntries : 0);
            __syncthreads();
            if (sb > 0) {
                if (threadIdx.x == 0) {
                    s_ctl[0] = 0;
                    s_ctl[1] = 0;
                    s_ctl[2] = 0;
                }
                if (PV)
                    for (int s = threadIdx.x; s < kTagMaxEntries; s += blockDim.x) cnt[s] = 0;
            }
            // index bits: with per-vertex counts 2^b1 >= 8 * sd, 10..13 (the
            // rank then fits below bit 31; less to clear a unit), for totals
            // only 13 (fewer shared slots: measured faster each way)
            int b1 = PV ? 10 : 13;
            while (b1 < 13 && (1 << b1) < 8 * sd) ++b1;
            const int s1 = 32 - b1;
            const unsigned m1 = (1u << s1) - 1u;
            for (int s = threadIdx.x; s < (1 << b1); s += blockDim.x) region[s] = kTagEmpty;
            for (int s = threadIdx.x; s < kTagSlots2; s += blockDim.x) t2[s] = kTagEmpty;
            __syncthreads();
            for (int q = threadIdx.x; q < sd; q += blockDim.x) {
                const int k = G.adj[sr + q];
                const unsigned p = (unsigned)k * kTagMul;
                unsigned* slot = region + (p >> s1);
                if (atomicCAS(slot, kTagEmpty, ((unsigned)q << s1) | (p & m1)) != kTagEmpty) {
                    // a shared slot: this entry and the one displaced (if still
                    // there) move to the second table
                    const unsigned old = atomicExch(slot, kTagMulti);
                    tag_insert2(t2, k, q);
                    if (old != kTagMulti) {
                        const int q2 = (int)(old >> s1);
                        tag_insert2(t2, G.adj[sr + q2], q2);
                    }
                }
            }
            __syncthreads();
            const TagTab T{region, t2, G.adj + sr, sd, s1, m1};
            cta_probe_unit<PV, WIN, false>(G, U, T, cnt, s_ctl, s_base, s_long, tlow, uh, probes);
            __syncthreads();
            if (PV)
                for (int r = threadIdx.x; r < sd; r += blockDim.x) {
                    const unsigned h = T.credited(cnt, r);
                    if (h) atomicAdd(&G.tnew[G.adj[sr + r]], (unsigned long long)h);
                }
        }
    } else {
        int* tab = reinterpret_cast<int*>(region);
        const unsigned buckets = hash_buckets(dp);
        const unsigned bmask = buckets - 1u;
        for (int s = threadIdx.x; s < 4 * (int)buckets; s += blockDim.x) tab[s] = kEmpty;
        __syncthreads();
        for (int q = threadIdx.x; q < dp; q += blockDim.x) hash_insert(tab, bmask, G.adj[rb + q]);
        __syncthreads();
        const HashTab T{tab, bmask, lo, hi};
        cta_probe_unit<PV, WIN, BUCKETS && !WIN>(G, U, T, cnt, s_ctl, s_base, s_long, tlow, uh, probes);
        __syncthreads();
        if (PV)
            for (int s = threadIdx.x; s < 4 * (int)buckets; s += blockDim.x) {
                const unsigned h = T.credited(cnt, s);
                if (h) atomicAdd(&G.tnew[tab[s]], (unsigned long long)h);
            }
    }
    hits += uh;
    if (PV) {
        // j's credit: each warp adds its share (no barrier at the unit's end)
        uh = warp_sum_u64(uh);
        if (lane == 0 && uh) atomicAdd(&G.tnew[G.jbase + U.j], (unsigned long long)uh);
    }
}

// ---------------------------------------------------------------------------
// The count kernel: persistent CTAs first pop CTA units (heaviest first),
// then each warp pops warp units until both queues are empty.  Units may
// belong to different graphs (the batched form): each carries its graph's
// index into the view table, and hits are added to that graph's total.
//
// Dynamic shared memory: per-warp bases (nw x 32 int64) | table region
// (kRegionWords words; warp units use 192-word slices of it) | hit counters
// (PV: kRegionWords/2 words, a tag table's second table past the first
// kTagMaxEntries of them; totals only: the second table alone) | long-task
// queue (unit_tasks x 16 bit).
// ---------------------------------------------------------------------------
// SMALL: the warps' units (pivots of up to 64 entries) as well, each with a
// table; BUCKETS and WIN instances always take them.
template <bool PV, bool WIN, bool BUCKETS, bool SMALL>
__global__ void __launch_bounds__(256, TC_LARGE_MINB)
    k_count(const GraphView* __restrict__ views, const Unit* __restrict__ large, int64_t nlarge,
            const Unit* __restrict__ small, int64_t nsmall, int slice_max, int grab, unsigned* tlow,
            unsigned long long* __restrict__ ctr) {
    extern __shared__ __align__(16) unsigned smem[];
    __shared__ long long s_unit;
    __shared__ int s_ctl[4];
    __shared__ unsigned s_wsum[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int64_t* s_base = reinterpret_cast<int64_t*>(smem) + 32 * w;
    unsigned* region = smem + 64 * nw;
    unsigned* cnt = region + kRegionWords;
    unsigned short* s_long =
        reinterpret_cast<unsigned short*>(cnt + (PV ? kRegionWords / 2 : kTagSlots2));
    __shared__ unsigned long long s_work[6];   // units, tasks, staged for [warp, CTA] units
    if (threadIdx.x < 6) s_work[threadIdx.x] = 0;
    GraphAcc acc;
    uint64_t probes = 0;

    // CTA units
    while (true) {
        if (threadIdx.x == 0) {
            s_unit = (long long)atomicAdd(&ctr[CTR_LARGE_HEAD], 1ull);
            s_ctl[0] = 0;
            s_ctl[1] = 0;
            s_ctl[2] = 0;
        }
        __syncthreads();
        const long long u = s_unit;
        if (u >= nlarge) break;
        const Unit U = large[u];
        const GraphView G = views[U.g];
        acc.to(unit_target(G, U));
        cta_unit<PV, WIN, BUCKETS>(G, U, slice_max, region, cnt, s_ctl, s_base, s_long, s_wsum,
                                   tlow, acc.hits, probes);
        if (threadIdx.x == 0) {
            s_work[1] += 1;
            s_work[3] += (unsigned long long)(U.t1 - U.t0);
            s_work[5] += (unsigned long long)min64(
                off_at(G, U.j + 1) - off_at(G, U.j) - (int64_t)U.slice * slice_max, slice_max);
        }
        __syncthreads();
    }
    if (lane == 0 && probes) atomicAdd(&ctr[CTR_PROBES + 1], (unsigned long long)probes);
    probes = 0;

    // warp units, each warp on its own slice of the region
    unsigned* wregion = region + w * kSmallRegionWords;
    unsigned* wcnt = cnt + w * (kSmallTable / 2);
    uint64_t staged = 0;
    while (SMALL) {
        long long u0 = 0;
        if (lane == 0) u0 = (long long)atomicAdd(&ctr[CTR_SMALL_HEAD], (unsigned long long)grab);
        u0 = __shfl_sync(0xffffffffu, u0, 0);
        if (u0 >= nsmall) break;
        const int64_t u1 = min64(u0 + grab, nsmall);
        for (int64_t u = u0; u < u1; ++u) {
            const Unit U = small[u];
            const GraphView G = views[U.g];
            acc.to(unit_target(G, U));
            warp_unit<PV, WIN>(G, U, wregion, wcnt, s_base, BUCKETS, tlow, acc.hits,
                                 probes, staged);
            if (lane == 0) {
                atomicAdd(&s_work[0], 1ull);
                atomicAdd(&s_work[2], (unsigned long long)(U.t1 - U.t0));
            }
        }
    }
    acc.flush();
    if (lane == 0) {
        if (probes) atomicAdd(&ctr[CTR_PROBES + 0], (unsigned long long)probes);
        if (staged) atomicAdd(&s_work[4], (unsigned long long)staged);
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        const int k = threadIdx.x;
        atomicAdd(&ctr[CTR_UNITS + k], s_work[k]);
        atomicAdd(&ctr[CTR_TASKS + k], s_work[2 + k]);
        atomicAdd(&ctr[CTR_STAGED + k], s_work[4 + k]);
    }
}

// ---------------------------------------------------------------------------
// Pivots of kZoneMinPivot+1 .. kMidEntries entries, the units of the zone
// kernel (at most 248 tasks), one warp each.  What the zones leave of such a
// pivot's tails is little -- at RMAT scale 20 about 15 entries of each of 220
// tasks -- and a CTA spent more on a unit's chain of loads and barriers (4 us
// of table building) than on its probes; a warp with a table of its own needs
// no barrier, and 32 of them on an SM hide one another's loads.  The table is
// a bitmap (672 words and their rank prefixes) or, for a wider span, 1,024
// tag slots with 256 more for the entries that share one.
//
// Dynamic shared memory of a warp: bases (32 int64) | table (kMidSlots words)
// | second table (kMidSlots2) | hit counters (PV: kMidEntries).
// ---------------------------------------------------------------------------
constexpr int kMidThreads = 256;
constexpr int kMidBitWords = (kMidSlots * 2 / 3) & ~31;
constexpr int kLightMinBlocks = 4;
constexpr size_t mid_warp_words(bool pv) { return 64 + kMidSlots + kMidSlots2 + (pv ? kMidEntries : 0); }

constexpr size_t light_smem(bool pv) { return sizeof(unsigned) * mid_warp_words(pv) * (kMidThreads / 32); }

constexpr int kFlatUnits = 4;
static_assert(kFlatUnits * kSmallMaxOutdeg <= kMidEntries, "the units' counters fit the pivot counters of a warp");
constexpr int kFlatWindow = 2048;   // concatenated entries whose tasks' starts are marked at once
struct __align__(16) FlatWarp {   // one warp's shared memory while it counts warp units
    int64_t t0[kFlatUnits];   // per unit: first task less the tasks of earlier units
    const int32_t* adj[kFlatUnits];
    unsigned heads[kFlatWindow / 32];   // bit q: a task's entries start at q
    int row[kFlatUnits * kSmallMaxOutdeg];   // the pivots' rows, filled up with the largest int
    int end[kFlatUnits];      // tasks up to and including the unit's
    unsigned rb[kFlatUnits];
    int j[kFlatUnits], g[kFlatUnits];
    unsigned base[32];        // per task with a tail: its entries' place less their position
    int unit[32];             // its unit
};

template <bool PV, class Tab>
__device__ __forceinline__ void mid_probe(const GraphView& G, const Unit& U, const Tab& T, unsigned* cnt,
                                          int64_t* s_base, unsigned* tlow, int64_t rb, int dp, uint64_t& hits,
                                          uint64_t& probes) {
    const int lane = threadIdx.x & 31;
    uint64_t uh = 0;
    for (int64_t tb = U.t0; tb < U.t1; tb += 32)
        warp_probe_group<PV, false, false>(G, G.tasks, tb, U.t1, G.adj, T, cnt, G.tnew, tlow, s_base, U.t0, nullptr, nullptr,
                                    uh, probes, TaskWindow{0, 0, 0});
    hits += uh;
    __syncwarp();
    if (PV) {
        for (int r = lane; r < dp; r += 32) {
            const unsigned h = T.credited(cnt, r);
            if (h) atomicAdd(&G.tnew[G.adj[rb + r]], (unsigned long long)h);
        }
        uh = warp_sum_u64(uh);
        if (lane == 0 && uh) atomicAdd(&G.tnew[U.j], (unsigned long long)uh);
    }
}

// Pivots of at most kSmallMaxOutdeg entries (warp units), without tables: the
// tasks of up to kFlatUnits units are dealt to the lanes 32 at a time whatever
// their pivots, their tails concatenated, and each entry is looked up by a
// branchless binary search of its own pivot's row in shared memory (the
// list-based traversal of Section 3.1, a lane a probe).  Such a unit holds
// some hundred probes: as a table of its own, built, probed and flushed, it
// took 600-1,000 instructions whatever its size (G(n,p) of 1.6e6 edges:
// 141,601 units, 146 us).  An entry's task is the number of task starts up to
// it, counted in a bit mask of the starts.  Few units at a time: a hub's are
// hundreds of times longer than others.  Per-vertex: hits on the pivots'
// entries count in shared memory (adding each to its vertex's accumulator
// made the hubs' a bottleneck: RMAT scale 20 0.7 -> 2.3 ms).
template <bool PV>
__device__ __forceinline__ void flat_units(const GraphView* __restrict__ views, const Unit* __restrict__ small,
                                           long long u0, int n, FlatWarp& S, unsigned* cnt, unsigned* tlow,
                                           GraphAcc& acc, unsigned long long* work) {
    const int lane = threadIdx.x & 31;
    const unsigned le = (2u << lane) - 1u;
    int nt = 0, dp = 0;
    Unit U{};
    __syncwarp();   // the last batch's reads of S are done
    if (lane < n) {
        U = small[u0 + lane];
        const GraphView& V = views[U.g];
        const int64_t rb = off_at(V, U.j);
        dp = (int)(off_at(V, U.j + 1) - rb);
        nt = (int)(U.t1 - U.t0);
        S.adj[lane] = V.adj;
        S.rb[lane] = (unsigned)rb;
        S.j[lane] = U.j;
        S.g[lane] = U.g;
    }
    const int uend = warp_incl_scan_i32(nt);
    const int N = __shfl_sync(0xffffffffu, uend, 31);
    if (lane < kFlatUnits) {
        S.end[lane] = lane < n ? uend : 0x7fffffff;
        S.t0[lane] = U.t0 - (uend - nt);
    }
    const int g0 = __shfl_sync(0xffffffffu, U.g, 0);
    const bool one_graph = __all_sync(0xffffffffu, lane >= n || U.g == g0);
    const bool wide_rows = __any_sync(0xffffffffu, dp > 16);
    const int32_t* __restrict__ adj0 = views[g0].adj;
    // hits may go to one counter as they come, without a task's share of them
    const bool bulk = !PV && one_graph && !views[g0].comp;
    if (bulk) acc.to(views[g0].total);
    __syncwarp();
#pragma unroll
    for (int o = 0; o < kFlatUnits; ++o) {
        if (o >= n) break;
        const int d = __shfl_sync(0xffffffffu, dp, o);
        const int32_t* a = S.adj[o] + S.rb[o];
        int* r = S.row + o * kSmallMaxOutdeg;
        r[lane] = lane < d ? a[lane] : 0x7fffffff;
        r[lane + 32] = lane + 32 < d ? a[lane + 32] : 0x7fffffff;
        if (PV) {
            cnt[o * kSmallMaxOutdeg + lane] = 0;
            cnt[o * kSmallMaxOutdeg + lane + 32] = 0;
        }
    }
    __syncwarp();
    unsigned nprobes = 0;
    for (int x0 = 0; x0 < N; x0 += 32) {
        const int x = x0 + lane;
        // this lane's task and its unit: the first that ends after x
        int o = 0;
#pragma unroll
        for (int step = kFlatUnits / 2; step > 0; step >>= 1)
            if (S.end[o + step - 1] <= x) o += step;
        o = min(o, n - 1);
        int len = 0, i = 0;
        unsigned start = 0;
        if (x < N) {
            const Task t = views[S.g[o]].tasks[S.t0[o] + x];
            start = t.start;
            len = t.len;
            i = t.i;
        }
        const int incl = warp_incl_scan_i32(len), excl = incl - len;
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        const unsigned on = __ballot_sync(0xffffffffu, len > 0);
        if (len > 0) {
            const int at = __popc(on & (le >> 1));
            S.base[at] = start - (unsigned)excl;
            S.unit[at] = o;
        }
        nprobes += (unsigned)total;
        unsigned c = 0;
        for (int w0 = 0; w0 < total; w0 += kFlatWindow) {
            S.heads[lane] = 0;
            S.heads[lane + 32] = 0;
            __syncwarp();
            if (len > 0 && excl >= w0 && excl < w0 + kFlatWindow)
                atomicOr(&S.heads[(excl - w0) >> 5], 1u << (excl & 31));
            int seen = __popc(__ballot_sync(0xffffffffu, len > 0 && excl < w0)) - 1;
            __syncwarp();
            const int w1 = min(total, w0 + kFlatWindow);
            for (int q0 = w0; q0 < w1; q0 += 32 * kUnroll) {
                static_assert(kUnroll == 4, "four words of starts a round");
                const uint4 H = *reinterpret_cast<const uint4*>(&S.heads[(q0 - w0) >> 5]);
                const unsigned M[4] = {H.x, H.y, H.z, H.w};
                int k[kUnroll], p[kUnroll];
#pragma unroll
                for (int u = 0; u < kUnroll; ++u) {
                    const int q = q0 + 32 * u + lane;
                    const int w = seen + __popc(M[u] & le);
                    seen += __popc(M[u]);
                    k[u] = -1;
                    p[u] = 0;
                    if (q < w1) {
                        const int un = S.unit[w];
                        const int32_t* __restrict__ a = one_graph ? adj0 : S.adj[un];
                        k[u] = __ldg(a + (S.base[w] + (unsigned)q));
                        p[u] = un * kSmallMaxOutdeg;
                    }
                }
                // the last entry <= k
                if (wide_rows) {
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u)
                        if (S.row[p[u] + 32] <= k[u]) p[u] += 32;
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u)
                        if (S.row[p[u] + 16] <= k[u]) p[u] += 16;
                }
#pragma unroll
                for (int s = 8; s > 0; s >>= 1) {
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u)
                        if (S.row[p[u] + s] <= k[u]) p[u] += s;
                }
#pragma unroll
                for (int u = 0; u < kUnroll; ++u) {
                    const bool hit = S.row[p[u]] == k[u];
                    if (PV && hit) atomicAdd(&cnt[p[u]], 1u);
                    if (bulk) {
                        acc.hits += hit ? 1 : 0;
                    } else {
                        const unsigned hm = __ballot_sync(0xffffffffu, hit);
                        if (hm) {   // each task takes its hits of these 32
                            const int qb = q0 + 32 * u;
                            const int b0 = max(excl - qb, 0), b1 = min(incl - qb, 32);
                            if (b0 < b1) c += __popc(hm & bit_range(b0, b1));
                        }
                    }
                }
            }
            __syncwarp();
        }
        if (!bulk) {
            // credits: per task, and per unit for its pivot and total
            const GraphView& V = views[S.g[o]];
            if (PV && c) credit_task(V.tnew, tlow, i, c);
            const int csum = warp_incl_scan_i32((int)c);
            const int o_next = __shfl_down_sync(0xffffffffu, o, 1);
            const bool seg_end = x < N && (lane == 31 || x + 1 == N || o_next != o);
            const unsigned ends = __ballot_sync(0xffffffffu, seg_end);
            const unsigned below = ends & (le >> 1);
            const int prev = __shfl_sync(0xffffffffu, csum, below ? 31 - __clz(below) : 0);
            const unsigned h = (unsigned)(csum - (below ? prev : 0));
            if (seg_end && h) {
                if (PV) atomicAdd(&V.tnew[S.j[o]], (unsigned long long)h);
                atomicAdd(V.comp ? V.comp_totals + V.comp[S.j[o]] : V.total, (unsigned long long)h);
            }
        }
        __syncwarp();   // base and unit are rewritten by the next 32 tasks
    }
    if (PV) {
        for (int q = lane; q < n * kSmallMaxOutdeg; q += 32) {
            const unsigned h = cnt[q];
            if (h) atomicAdd(&views[S.g[q / kSmallMaxOutdeg]].tnew[S.row[q]], (unsigned long long)h);
        }
    }
    const unsigned staged = __reduce_add_sync(0xffffffffu, (unsigned)dp);
    if (lane == 0) {
        work[0] += (unsigned)n;
        work[1] += (unsigned)N;
        work[2] += nprobes;
        work[3] += staged;
    }
}

static_assert(sizeof(FlatWarp) <= sizeof(unsigned) * (64 + kMidSlots + kMidSlots2) && mid_warp_words(true) % 4 == 0 &&
                  mid_warp_words(false) % 4 == 0, "one region, 16-byte aligned, for both parts");

template <bool PV>
__global__ void __launch_bounds__(kMidThreads, kLightMinBlocks)
    k_light(const GraphView* __restrict__ views, const Unit* __restrict__ units, int64_t nunits,
            int mid_max, const Unit* __restrict__ small, int64_t nsmall, int grab, unsigned* tlow,
            unsigned long long* __restrict__ ctr) {
    extern __shared__ __align__(16) unsigned smem[];
    __shared__ unsigned long long s_work[kMidThreads / 32][4];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned* mine = smem + (size_t)w * mid_warp_words(PV);
    int64_t* s_base = reinterpret_cast<int64_t*>(mine);
    unsigned* tab = mine + 64;
    unsigned* t2 = tab + kMidSlots;
    unsigned* cnt = t2 + kMidSlots2;
    if (lane < 4) s_work[w][lane] = 0;
    GraphAcc acc;
    uint64_t probes = 0, staged = 0;
    unsigned long long nu = 0, nt = 0;
    // The first of a list's units are dealt to the warps, the rest popped: a
    // queue head serves its atomics one after the other, about 3 ns each, and a
    // pop of each list and one more to find it empty were most of a count of some
    // thousand units of 16 tasks (RMAT of 65,536 pairs and vertices: 30 us, 18
    // dealt).  Warp units are dealt only where no warp has wide ones before them.
    const long long all = (long long)gridDim.x * (kMidThreads / 32), me = (long long)w * gridDim.x + blockIdx.x;
    auto pop = [&](int head, long long n, long long dealt, int step) {
        if (dealt >= n) return n;
        long long u = 0;
        if (lane == 0) u = (long long)atomicAdd(&ctr[head], (unsigned long long)step);
        return dealt + __shfl_sync(0xffffffffu, u, 0);
    };
    for (long long u = me; u < nunits; u = pop(CTR_MID_HEAD, nunits, all, 1)) {
        const Unit U = units[u];
        const GraphView G = views[U.g];
        const int64_t rb = off_at(G, U.j);
        const int64_t d = off_at(G, U.j + 1) - rb;
        if (d > mid_max) continue;   // a CTA unit
        const int dp = (int)d;
        acc.to(unit_target(G, U));
        const int lo = G.adj[rb], hi = G.adj[rb + dp - 1];
        if (PV)
            for (int q = lane; q < dp; q += 32) cnt[q] = 0;
        if ((int64_t)hi - lo + 1 < 32ll * kMidBitWords) {   // labels + guard bit
            const int words = ((hi - lo + 1) >> 5) + 1;
            for (int q = lane; q < words; q += 32) tab[q] = 0;
            __syncwarp();
            for (int q = lane; q < dp; q += 32) {
                const int k = G.adj[rb + q] - lo;
                atomicOr(&tab[k >> 5], 1u << (k & 31));
            }
            __syncwarp();
            unsigned short* pre = reinterpret_cast<unsigned short*>(tab + kMidBitWords);
            if (PV) {
                int before = 0;   // prefix popcounts, 32 words at a time
                for (int q0 = 0; q0 < words; q0 += 32) {
                    const int c = q0 + lane < words ? __popc(tab[q0 + lane]) : 0;
                    const int inc = warp_incl_scan_i32(c);
                    if (q0 + lane < words) pre[q0 + lane] = (unsigned short)(before + inc - c);
                    before += __shfl_sync(0xffffffffu, inc, 31);
                }
                __syncwarp();
            }
            const BitTab T{tab, pre, lo, hi};
            mid_probe<PV>(G, U, T, cnt, s_base, tlow, rb, dp, acc.hits, probes);
        } else {
            for (int q = lane; q < kMidSlots + kMidSlots2; q += 32) tab[q] = kTagEmpty;
            __syncwarp();
            for (int q = lane; q < dp; q += 32) {
                const int k = G.adj[rb + q];
                const unsigned p = ((unsigned)k * kTagMul) & kMid31;
                unsigned* slot = tab + (p >> kMidTag);
                const unsigned word = ((unsigned)q << kMidTag) | (p & ((1u << kMidTag) - 1u));
                if (atomicCAS(slot, kTagEmpty, word) != kTagEmpty) {
                    // a shared slot: this entry and the one displaced (if
                    // still there) move to the second table
                    const unsigned old = atomicExch(slot, kTagMulti);
                    for (int h = 0; h < 2; ++h) {
                        if (h == 1 && old == kTagMulti) break;
                        const int qq = h == 0 ? q : (int)(old >> kMidTag);
                        const unsigned p2 = ((unsigned)G.adj[rb + qq] * kTagMul2) & kMid31;
                        unsigned* s2 = t2 + (p2 >> kMidTag2);
                        if (atomicCAS(s2, kTagEmpty, ((unsigned)qq << kMidTag2) | (p2 & ((1u << kMidTag2) - 1u))) !=
                            kTagEmpty)
                            atomicExch(s2, kTagMulti);
                    }
                }
            }
            __syncwarp();
            const MidTab T{tab, t2, G.adj + rb, dp};
            mid_probe<PV>(G, U, T, cnt, s_base, tlow, rb, dp, acc.hits, probes);
        }
        staged += (uint64_t)dp;
        nu += 1;
        nt += (unsigned long long)(U.t1 - U.t0);
        __syncwarp();   // the table is rebuilt by the next unit
    }
    if (lane == 0 && nu) {
        atomicAdd(&ctr[CTR_UNITS + 1], nu);
        atomicAdd(&ctr[CTR_TASKS + 1], nt);
        atomicAdd(&ctr[CTR_PROBES + 1], (unsigned long long)probes);
        atomicAdd(&ctr[CTR_STAGED + 1], (unsigned long long)staged);
    }
    // the warp units
    FlatWarp& S = *reinterpret_cast<FlatWarp*>(mine);
    const long long dealt = nunits == 0 ? all * grab : 0;
    for (long long u0 = dealt ? me * grab : pop(CTR_SMALL_HEAD, nsmall, 0, grab); u0 < nsmall;
         u0 = pop(CTR_SMALL_HEAD, nsmall, dealt, grab))
        flat_units<PV>(views, small, u0, (int)min64(grab, nsmall - u0), S, cnt, tlow, acc, s_work[w]);
    acc.flush();
    __syncwarp();
    if (lane < 4 && s_work[w][0]) {
        const int slot = lane == 0 ? CTR_UNITS : lane == 1 ? CTR_TASKS : lane == 2 ? CTR_PROBES : CTR_STAGED;
        atomicAdd(&ctr[slot], s_work[w][lane]);
    }
}

// per-vertex counts in original ids: the 64-bit accumulator plus, when used,
// the 32-bit per-task shares
__global__ void k_gather_pv(const unsigned long long* __restrict__ tnew, const unsigned* __restrict__ tlow,
                            const int32_t* __restrict__ perm, int64_t n,
                            uint64_t* __restrict__ out) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t x = perm[v];
        out[v] = tnew[x] + (tlow ? (uint64_t)tlow[x] : 0ull);
    }
}

__global__ void k_copy_total(const unsigned long long* __restrict__ ctr, uint64_t* __restrict__ out) {
    *out = ctr[CTR_TOTAL];
}

// ---------------------------------------------------------------------------
// Work units over one or many graphs.  Vertex v of the concatenation of the
// graphs (vpre = prefix of vertex counts) is visited in reverse order, so
// the last graph's heaviest pivots come first (batches list their graphs by
// ascending size, so the largest graph leads).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int find_graph(const int64_t* __restrict__ vpre, int num, int64_t v) {
    int lo = 0, hi = num - 1;   // largest g with vpre[g] <= v
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (vpre[mid] <= v) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__global__ void k_unit_counts(const GraphView* __restrict__ views, const int64_t* __restrict__ vpre,
                              int num, int64_t V, UnitRule rule, int32_t* __restrict__ cs,
                              int32_t* __restrict__ cl, int32_t* __restrict__ cz) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < V;
         x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = V - 1 - x;
        const int g = find_graph(vpre, num, v);
        const GraphView& G = views[g];
        const int64_t j = v - vpre[g];
        int64_t a, b, c;
        unit_split<true>(rule, rule.zones && G.zrow != nullptr, off_at(G, j + 1) - off_at(G, j),
                         G.loff[j + 1] - G.loff[j], a, b, c);
        cs[x] = (int32_t)a;
        cl[x] = (int32_t)b;
        if (cz) cz[x] = (int32_t)c;
    }
}

__global__ void k_unit_fill(const GraphView* __restrict__ views, const int64_t* __restrict__ vpre,
                            int num, int64_t V, UnitRule rule,
                            const int64_t* __restrict__ ps, const int64_t* __restrict__ pl,
                            const int64_t* __restrict__ pz, Unit* __restrict__ us, Unit* __restrict__ ul,
                            Unit* __restrict__ uz) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < V;
         x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = V - 1 - x;
        const int g = find_graph(vpre, num, v);
        const GraphView& G = views[g];
        const int64_t j = v - vpre[g];
        const int64_t dp = off_at(G, j + 1) - off_at(G, j);
        const int64_t a = G.loff[j], b = G.loff[j + 1];
        int64_t ns, nl, nw;
        unit_split<true>(rule, rule.zones && G.zrow != nullptr, dp, b - a, ns, nl, nw);
        if (nw > 0) {
            int64_t p = pz[x];
            for (int64_t t = a; t < b; t += rule.wide_tasks)
                uz[p++] = Unit{(int32_t)j, 0, g, 0, t, min64(t + rule.wide_tasks, b)};
        }
        if (ns > 0) {
            int64_t p = ps[x];
            for (int64_t t = a; t < b; t += rule.warp_tasks)
                us[p++] = Unit{(int32_t)j, 0, g, 0, t, min64(t + rule.warp_tasks, b)};
        } else if (nl > 0) {
            const int64_t slices = (dp + rule.slice - 1) / rule.slice;
            int64_t p = pl[x];
            for (int64_t t = a; t < b; t += rule.cta_tasks)
                for (int64_t s = 0; s < slices; ++s)
                    ul[p++] = Unit{(int32_t)j, (int32_t)s, g, 0, t, min64(t + rule.cta_tasks, b)};
        }
    }
}

}  // namespace

UnitRule unit_rule(const tc_tuning& t, bool win, bool zones) {
    UnitRule r;
    r.small_max = t.small_max_outdeg;
    r.merge_max = t.merge_max_outdeg;
    r.mid_max = win || t.table_mode == 1 || !zones ? 0 : kMidMaxOutdeg;
    r.warp_tasks = t.warp_unit_tasks;
    r.cta_tasks = t.cta_unit_tasks;
    r.wide_tasks = kZoneTasks;
    r.slice = t.slice_max;
    r.zones = !win && t.table_mode != 1 && zones;
    return r;
}

tc_tuning clamp_tuning(const tc_tuning& t) {
    tc_tuning tt = t;
    tt.slice_max = std::min(tt.slice_max, kRegionWords / 2);   // a hashed slice needs 2 slots per entry
    return tt;
}

void plan_units(UnitPlan& P, const GraphView* views_dev, const int64_t* vpre_dev, int num, int64_t V,
                const UnitRule& rule, Alloc& al, cudaStream_t st) {
    const unsigned G = (unsigned)(num_sms() * 8);
    P.V = V;
    P.num = num;
    P.views = views_dev;
    P.vpre = vpre_dev;
    P.rule = rule;
    P.cs = Buf<int32_t>(al, (size_t)std::max<int64_t>(V, 1));
    P.cl = Buf<int32_t>(al, (size_t)std::max<int64_t>(V, 1));
    if (rule.zones) P.cz = Buf<int32_t>(al, (size_t)std::max<int64_t>(V, 1));
    P.ps = Buf<int64_t>(al, (size_t)(V + 1));
    P.pl = Buf<int64_t>(al, (size_t)(V + 1));
    if (rule.zones) P.pz = Buf<int64_t>(al, (size_t)(V + 1));
    if (V > 0) {
        Prof prof_("k_unit_counts", st);
        k_unit_counts<<<grid_for(V, 256, G), 256, 0, st>>>(views_dev, vpre_dev, num, V, rule, P.cs.get(), P.cl.get(),
                                                           P.cz.get());
    }
    TC_LAUNCH_CHECK();
    exclusive_scan2_i32_to_i64(P.cs.get(), P.ps.get(), P.ps.get() + V, P.cl.get(), P.pl.get(), P.pl.get() + V, V,
                               al, st);
    if (rule.zones) exclusive_scan_i32_to_i64(P.cz.get(), P.pz.get(), V, P.pz.get() + V, al, st);
}

UnitLists fill_units(UnitPlan& P, int64_t ns, int64_t nl, int64_t nz, Alloc& al, cudaStream_t st) {
    const unsigned G = (unsigned)(num_sms() * 8);
    UnitLists L;
    L.bytes = sizeof(Unit) * (size_t)std::max<int64_t>(ns + nl + nz, 1);
    L.mem = al.get(L.bytes);
    L.large = static_cast<Unit*>(L.mem);
    L.small = L.large + nl;
    L.zone = L.small + ns;
    L.nlarge = nl;
    L.nsmall = ns;
    L.nzone = nz;
    L.mid_max = P.rule.mid_max;
    if (P.V > 0) {
        {
            Prof prof_("k_unit_fill", st);
            k_unit_fill<<<grid_for(P.V, 256, G), 256, 0, st>>>(P.views, P.vpre, P.num, P.V, P.rule, P.ps.get(),
                                                               P.pl.get(), P.pz.get(), L.small, L.large, L.zone);
        }
        TC_LAUNCH_CHECK();
    }
    P.cs.release();
    P.cl.release();
    P.cz.release();
    P.ps.release();
    P.pl.release();
    P.pz.release();
    return L;
}

UnitLists build_unit_lists(const GraphView* views_dev, const int64_t* vpre_dev, int num, int64_t V,
                           const UnitRule& rule, Alloc& al, cudaStream_t st) {
    UnitPlan P;
    plan_units(P, views_dev, vpre_dev, num, V, rule, al, st);
    int64_t ns = 0, nl = 0, nz = 0;
    TC_CUDA(cudaMemcpyAsync(&ns, P.ps.get() + V, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    if (rule.zones) TC_CUDA(cudaMemcpyAsync(&nz, P.pz.get() + V, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    TC_CUDA(cudaMemcpyAsync(&nl, P.pl.get() + V, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    TC_CUDA(cudaStreamSynchronize(st));
    return fill_units(P, ns, nl, nz, al, st);
}

void adopt_units(tc_graph* g, const UnitLists& L, const tc_tuning& tt) {
    if (g->units_mem) g->alloc.put(g->units_mem, g->units_bytes);
    g->units_mem = L.mem;
    g->units_bytes = L.bytes;
    g->small_units = L.small;
    g->large_units = L.large;
    g->zone_units = L.zone;
    g->n_zone = L.nzone;
    g->n_small = L.nsmall;
    g->n_large = L.nlarge;
    g->units_tuning = tt;
    g->stats.small_units = L.nsmall;
    g->stats.large_units = L.nlarge;
}

UnitLists units_of(const tc_graph* g) {
    UnitLists L;
    L.large = g->large_units;
    L.small = g->small_units;
    L.zone = g->zone_units;
    L.nlarge = g->n_large;
    L.nsmall = g->n_small;
    L.nzone = g->n_zone;
    L.zones = g->zcap > 0;
    L.mid_max = unit_rule(g->units_tuning, false, L.zones).mid_max;
    return L;
}

size_t count_smem_bytes(bool pv, int threads, int unit_tasks) {
    return sizeof(int64_t) * 32 * (size_t)(threads / 32) +
           sizeof(unsigned) * (size_t)(kRegionWords + (pv ? kRegionWords / 2 : kTagSlots2)) +
           sizeof(unsigned short) * (size_t)unit_tasks;
}

using CountKernel = void (*)(const GraphView*, const Unit*, int64_t, const Unit*, int64_t, int, int, unsigned*,
                            unsigned long long*);

// the count kernel instance for a launch: per-vertex or totals; the CTA units
// alone (k_light takes the rest), or the warps' units as well: in graphs
// without zones that have CTA units, in the instance that counts one tile of
// a host-resident graph (a window of rows) and in the bucket form for
// table_mode 1
CountKernel count_kernel(bool pv, bool win, bool buckets, bool small) {
    if (buckets) return win ? (pv ? k_count<true, true, true, true> : k_count<false, true, true, true>)
                            : (pv ? k_count<true, false, true, true> : k_count<false, false, true, true>);
    if (win) return pv ? k_count<true, true, false, true> : k_count<false, true, false, true>;
    if (small) return pv ? k_count<true, false, false, true> : k_count<false, false, false, true>;
    return pv ? k_count<true, false, false, false> : k_count<false, false, false, false>;
}

CountLaunch prepare_count(const UnitLists& L, const tc_tuning& t, bool pv, bool win) {
    CountLaunch c;
    c.threads = t.cta_threads;
    c.smem = count_smem_bytes(pv, c.threads, t.cta_unit_tasks);
    c.pv = pv;
    c.buckets = t.table_mode == 1;
    c.win = win;
    // a graph with CTA units but no wide ones is small: one kernel for all,
    // unless its short rows are to be searched
    c.light = !c.win && !c.buckets && (L.nzone > 0 || L.nlarge == 0 || t.merge_max_outdeg > 0);
    auto kern = count_kernel(pv, c.win, c.buckets, !c.light);
    TC_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c.smem));
    int per_sm = 0;
    TC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, c.threads, c.smem));
    per_sm = std::max(per_sm, 1);
    const int64_t warps = (int64_t)num_sms() * per_sm * (c.threads / 32);
    c.grab = L.nsmall < kGrabMin * warps ? 1 : kGrab;
    const int64_t warp_units = c.light ? 0 : L.nsmall;
    const int64_t want = L.nlarge + (warp_units + c.grab * (c.threads / 32) - 1) / (c.grab * (c.threads / 32));
    if (c.light) {
        TC_CUDA(cudaFuncSetAttribute(pv ? k_light<true> : k_light<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)light_smem(pv)));
    }
    c.grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)num_sms() * per_sm, want));
    return c;
}

void launch_count_raw(const CountLaunch& c, const GraphView* views_dev, const UnitLists& L,
                      const tc_tuning& t, unsigned long long* ctr, cudaStream_t st, unsigned* tlow, bool profile) {
    if (L.nlarge + (c.light ? 0 : L.nsmall) > 0) {
        const std::unique_ptr<Prof> prof(profile ? new Prof("k_count", st) : nullptr);
        auto kern = count_kernel(c.pv, c.win, c.buckets, !c.light);
        kern<<<c.grid, c.threads, c.smem, st>>>(views_dev, L.large, L.nlarge, L.small, L.nsmall, t.slice_max, c.grab,
                                                tlow, ctr);
        TC_LAUNCH_CHECK();
    }
    if (c.light && L.nzone + L.nsmall > 0) {
        // as many warp units at a time as leave every warp a turn; up to
        // kFlatUnits a warp, where they are dealt, so that nothing is popped
        const int64_t warps = (int64_t)num_sms() * kLightMinBlocks * (kMidThreads / 32);
        const int grab = (int)std::max<int64_t>(
            1, std::min<int64_t>(kFlatUnits, (L.nsmall + (L.nzone == 0 ? warps - 1 : 0)) / warps));
        const int64_t items = L.nzone + (L.nsmall + grab - 1) / grab;
        const unsigned blocks = (unsigned)std::min<int64_t>((items + kMidThreads / 32 - 1) / (kMidThreads / 32),
                                                            (int64_t)num_sms() * kLightMinBlocks);
        const std::unique_ptr<Prof> prof(profile ? new Prof("k_light", st) : nullptr);
        auto kern = c.pv ? k_light<true> : k_light<false>;
        kern<<<blocks, kMidThreads, light_smem(c.pv), st>>>(views_dev, L.zone, L.nzone, L.mid_max, L.small, L.nsmall,
                                                            grab, tlow, ctr);
        TC_LAUNCH_CHECK();
    }
}

void launch_count(const GraphView* views_dev, const UnitLists& L, const tc_tuning& t, bool pv,
                  unsigned long long* ctr, cudaStream_t st, bool profile, unsigned* tlow, bool win) {
    launch_count_raw(prepare_count(L, t, pv, win), views_dev, L, t, ctr, st, tlow, profile);
}

void build_units(tc_graph* g, const tc_tuning& t, cudaStream_t st) {
    const tc_tuning tt = clamp_tuning(t);
    Alloc& al = g->alloc;
    Buf<int64_t> vpre(al, 2);
    const int64_t hv[2] = {0, g->n};
    TC_CUDA(cudaMemcpyAsync(vpre.get(), hv, sizeof(hv), cudaMemcpyHostToDevice, st));
    UnitLists L = build_unit_lists(g->view, vpre.get(), 1, g->n, unit_rule(tt, false, g->zcap > 0), al, st);
    adopt_units(g, L, tt);
}

void count_components(tc_graph* g, const tc_tuning& t, uint64_t* comp_totals_dev,
                      cudaStream_t st) {
    const tc_tuning tt = clamp_tuning(size_tuning(t, g->plan_m));
    if (!tuning_equal(tt, g->units_tuning)) build_units(g, tt, st);
    // counters and component totals lie next to each other
    TC_CUDA(cudaMemsetAsync(g->counters, 0,
                            (size_t)(reinterpret_cast<char*>(g->comp_totals + g->num_comps) -
                                     reinterpret_cast<char*>(g->counters)), st));
    const UnitLists L = units_of(g);
    launch_count(g->view_comp, L, tt, false, g->counters, st, true, nullptr);
    launch_zone(g->view_comp, L, false, g->counters, st, nullptr, true);
    g->zone_probes = L.nzone > 0 ? g->covered : 0;
    TC_CUDA(cudaMemcpyAsync(comp_totals_dev, g->comp_totals, sizeof(uint64_t) * (size_t)g->num_comps,
                            cudaMemcpyDeviceToDevice, st));
}

void count(tc_graph* g, const tc_tuning& t, uint64_t* total_dev, uint64_t* per_vertex_dev,
           cudaStream_t st) {
    // the unit lists are a cache of the tuning they were built for
    const tc_tuning tt = clamp_tuning(size_tuning(t, g->plan_m));
    if (!tuning_equal(tt, g->units_tuning)) build_units(g, tt, st);
    const bool pv = per_vertex_dev != nullptr;
    // the counters, and with per-vertex counts the accumulators behind them
    TC_CUDA(cudaMemsetAsync(g->counters, 0, pv ? g->zero_bytes : sizeof(unsigned long long) * CTR_COUNT, st));
    // a task's share is at most C(max |U_i|, 2): 32-bit counters when that fits
    const uint64_t dmax = (uint64_t)g->stats.max_outdeg;
    const bool tlow32 = TC_TLOW32 && pv && g->n > 0 && dmax * (dmax - (dmax > 0)) / 2 < (1ull << 32);
    if (tlow32 && !g->tlow_in_arena) {
        if (!g->tlow) {
            g->tlow_bytes = sizeof(unsigned) * (size_t)g->n;
            g->tlow = static_cast<unsigned*>(g->alloc.get(g->tlow_bytes));
        }
        TC_CUDA(cudaMemsetAsync(g->tlow, 0, g->tlow_bytes, st));
    }
    const UnitLists L = units_of(g);
    launch_count(g->view, L, tt, pv, g->counters, st, true, tlow32 ? g->tlow : nullptr);
    launch_zone(g->view, L, pv, g->counters, st, tlow32 ? g->tlow : nullptr, true);
    g->zone_probes = L.nzone > 0 ? g->covered : 0;
    if (pv && g->n > 0) {
        {
            Prof prof_("k_gather_pv", st);
            k_gather_pv<<<grid_for(g->n, 256, num_sms() * 8), 256, 0, st>>>(
                reinterpret_cast<const unsigned long long*>(g->tnew), tlow32 ? g->tlow : nullptr, g->perm, g->n, per_vertex_dev);
        }
        TC_LAUNCH_CHECK();
    }
    if (total_dev) {
        {
            Prof prof_("k_copy_total", st);
            k_copy_total<<<1, 1, 0, st>>>(g->counters, total_dev);
        }
        TC_LAUNCH_CHECK();
    }
}

}  // namespace tc
