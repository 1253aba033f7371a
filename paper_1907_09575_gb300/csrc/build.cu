// tc_preprocess in one persistent kernel, for graphs of up to kBuildMaxPairs
// pairs: the steps a1-a6 of Section 5.3 as phases of a cooperative grid,
// separated by grid-wide barriers.
//
// Run as separate kernels the steps of a small graph take 24-36 launches,
// a dozen memsets and copies and two host round trips, each of them longer
// than its work (RMAT scale 14: 405 us a step, of which the kernels' own
// work was about a third).  As phases they cost a barrier (1-2 us) each, and
// what one phase knows need not be written out for the next:
//
//   insert    pair -> canonical key -> hash set; the pair that inserts a key
//             is marked in a bit mask (the set is never compacted) and
//             counts both degrees
//   relabel   stable LSD counting passes on the degree, 8 bits each, as many
//             as the largest degree has digits; the last writes the labels
//   orient    marked pairs -> (row, column) and the pair's place in its row
//             (the value the row counter's atomic returns: the scatter below
//             needs no atomics)
//   offsets   exclusive scan of the row lengths
//   scatter   columns into their rows
//   sort      each row where it lies; an entry with entries after it is a
//             <j,i,k> task of its column: its place among that pivot's tasks
//             is taken here by one atomic
//   tasks     scan of the task counts, then the task records, without atomics
//   units     work units for the default tuning
//
// The set's memory is reused for the oriented pairs.  Graphs of at most
// kBuildOnePairs pairs run all phases in one launch with arrays sized by the
// pair count; larger ones stop after the degrees (the host then sizes the
// arena by the edge count) and before the units.
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "tc_internal.cuh"

namespace tc {
namespace {

constexpr int kBT = 512;                  // threads of a block
constexpr int kBlocksPerSm = 2;           // 64 registers a thread: the row sort's network
constexpr int kBW = kBT / 32;
constexpr int kBItems = 4;                // independent pairs or edges in flight a thread
constexpr int kTileN = kBT * kBItems;     // entries of one tile of a scan or a counting pass
constexpr int kMedRow = 32;               // longer rows are sorted one warp a row ...
constexpr int kLongRow = 1024;            // ... and beyond this one block a row
constexpr int kMaxRow = 8192;             // d^2 <= 2m: no row of 2^24 edges passes 5,793
constexpr long kBarrierSpins = 1l << 23;
constexpr uint64_t kNoKey = ~0ull;        // keys use 2b <= 62 bits

constexpr int kTaskCopies = 8;
constexpr int kMaxChunks = 512;           // blocks that split the vertices among them

// What the phases count, read back by the host.
struct Tally {
    unsigned bar[2];         // barrier arrivals of the first and the second launch
    int err;                 // 1 bad id, 2 pair across components, 4 barrier wait, 8 row too long
    int maxdeg, maxout;
    int nmed, nlong;         // listed rows
    int med_head;
    unsigned long long m, tasks, probes, probes_ijk;
    long long nsmall, nlarge, nzone;
    unsigned long long covered;
    unsigned nblocks, pad;
};

struct BuildArgs {
    const int32_t* src;
    const int32_t* dst;
    const int64_t* vpre;     // components, or null
    int64_t P, n;
    int num_comps, off64;
    int phase0, phase1;      // phases [phase0, phase1) of kPhase*
    int64_t chunk;           // vertices of one block, a multiple of 32
    int nchunks;
    Tally* tally;
    uint64_t* table;
    uint64_t cap;
    uint32_t* first;         // bit e: pair e inserted its key
    int32_t* deg;            // by id
    int32_t* degn;           // by label
    int32_t* dplus;          // row lengths
    int32_t* tcur;           // tasks of each pivot, counted in `tcopies` arrays by the task's row;
    int tcopies;             // then the first slot of each copy's tasks
    uint32_t *ord0, *ord1;   // vertices between the relabel's passes; later the listed rows
    unsigned* hist;          // nchunks x 256
    long long* sums;         // 5 x nchunks
    uint2* pairs;            // oriented pairs (in the table's memory)
    uint32_t* place;         // place of a pair in its row; later of an edge among its pivot's tasks
    uint32_t* row;           // row of each edge
    void* off;
    int32_t* adj;
    int32_t* perm;
    int64_t* loff;
    Task* tasks;
    int32_t* comp;
    uint2* zrow;             // dense zones (zcap > 0)
    uint32_t *zbits, *zowner;
    int64_t zcap;
    GraphView view, view_comp;
    GraphView *view_at, *view_comp_at;
    Unit *large, *wide;      // the small units follow the wide ones
    UnitRule rule;
};

enum : int { kPhaseInsert = 0, kPhaseGraph = 1, kPhaseUnits = 2, kPhaseEnd = 3 };

__device__ __forceinline__ uint64_t mix64b(uint64_t x) {   // splitmix64's finaliser
    x ^= x >> 30;
    x *= 0xbf58476d1ce4e5b9ull;
    x ^= x >> 27;
    x *= 0x94d049bb133111ebull;
    x ^= x >> 31;
    return x;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Barrier over the (co-resident) grid.  The wait is bounded: past the bound
// the block sets error bit 4 and the kernel returns.
struct Grid {
    Tally* t;
    unsigned* bar;
    unsigned goal;
    __device__ bool sync() {
        __shared__ int ok;
        __syncthreads();
        if (threadIdx.x == 0) {
            goal += gridDim.x;
            __threadfence();
            atomicAdd(bar, 1u);
            long spins = 0;
            ok = 1;
            while ((int)(ld_acquire(bar) - goal) < 0)
                if (++spins > kBarrierSpins) {
                    atomicOr(&t->err, 4);
                    ok = 0;
                    break;
                }
            __threadfence();
        }
        __syncthreads();
        return ok != 0;
    }
};

__device__ __forceinline__ int64_t row_begin(const BuildArgs& a, int64_t r) {
    return a.off64 ? static_cast<const int64_t*>(a.off)[r] : (int64_t) static_cast<const int32_t*>(a.off)[r];
}

__device__ __forceinline__ int comp_index(const int64_t* vpre, int num, int64_t v) {
    int lo = 0, hi = num - 1;   // largest c with vpre[c] <= v
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (vpre[mid] <= v) lo = mid; else hi = mid - 1;
    }
    return lo;
}

template <class T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ int warp_max(int v) { return __reduce_max_sync(0xffffffffu, v); }

// Exclusive scan of one value per thread over the block; *total = the sum.
__device__ long long block_scan(long long v, long long* total) {
    __shared__ long long ws[kBW];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    long long before = 0, all = 0;
#pragma unroll
    for (int q = 0; q < kBW; ++q) {
        if (q < w) before += ws[q];
        all += ws[q];
    }
    __syncthreads();
    *total = all;
    return before + inc - v;
}

// Sum of x[0 .. count) over the block (every thread gets it).
__device__ long long block_sum(const long long* x, int count) {
    long long s = 0, total;
    for (int q = threadIdx.x; q < count; q += kBT) s += x[q];
    block_scan(s, &total);
    return total;
}

// --- insert -----------------------------------------------------------------
__device__ void phase_clear(const BuildArgs& a) {
    const int64_t T = (int64_t)gridDim.x * kBT, t = (int64_t)blockIdx.x * kBT + threadIdx.x;
    ulonglong2* tab = reinterpret_cast<ulonglong2*>(a.table);   // cap is even
    for (int64_t i = t; i < (int64_t)(a.cap >> 1); i += T) tab[i] = make_ulonglong2(kNoKey, kNoKey);
    for (int64_t i = t; i < a.n; i += T) {
        a.deg[i] = 0;
        a.dplus[i] = 0;
    }
    for (int64_t i = t; i < a.tcopies * a.n; i += T) a.tcur[i] = 0;
}

__device__ void phase_insert(const BuildArgs& a, int bits) {
    const int64_t T = (int64_t)gridDim.x * kBT, t = (int64_t)blockIdx.x * kBT + threadIdx.x;
    const int lane = threadIdx.x & 31;
    unsigned long long* table = reinterpret_cast<unsigned long long*>(a.table);
    unsigned long long mine = 0;
    int err = 0;
    for (int64_t base = 0; base < a.P; base += kBItems * T) {
        int32_t lo[kBItems], hi[kBItems];
        unsigned long long prev[kBItems];
        uint64_t slot[kBItems];
#pragma unroll
        for (int u = 0; u < kBItems; ++u) {
            const int64_t e = base + u * T + t;
            lo[u] = hi[u] = 0;
            if (e < a.P) {
                const int32_t x = a.src[e], y = a.dst[e];
                lo[u] = min(x, y);
                hi[u] = max(x, y);
            }
        }
#pragma unroll
        for (int u = 0; u < kBItems; ++u) {
            if (lo[u] < 0 || (int64_t)hi[u] >= a.n) {
                if (base + u * T + t < a.P) err |= 1;
                lo[u] = hi[u] = 0;
            }
            prev[u] = 0;
            if (lo[u] != hi[u]) {
                const unsigned long long key = ((unsigned long long)lo[u] << bits) | (unsigned)hi[u];
                slot[u] = __umul64hi(mix64b(key), a.cap);
                prev[u] = atomicCAS(&table[slot[u]], kNoKey, key);
            }
        }
        // collisions of all the pairs in flight advance together; the set
        // (capacity >= 2 pairs) never fills, bounded all the same
        uint64_t probe = 0;
        bool more = true;
        while (more && probe++ < a.cap) {
            more = false;
#pragma unroll
            for (int u = 0; u < kBItems; ++u) {
                const unsigned long long key = ((unsigned long long)lo[u] << bits) | (unsigned)hi[u];
                if (lo[u] != hi[u] && prev[u] != kNoKey && prev[u] != key) {
                    slot[u] = slot[u] + 1 == a.cap ? 0 : slot[u] + 1;
                    prev[u] = atomicCAS(&table[slot[u]], kNoKey, key);
                    more = true;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kBItems; ++u) {
            const bool first = lo[u] != hi[u] && prev[u] == kNoKey;
            if (first) {
                atomicAdd(&a.deg[lo[u]], 1);
                atomicAdd(&a.deg[hi[u]], 1);
                ++mine;
                if (a.num_comps > 0 && comp_index(a.vpre, a.num_comps, lo[u]) !=
                                           comp_index(a.vpre, a.num_comps, hi[u]))
                    err |= 2;
            }
            const unsigned b = __ballot_sync(0xffffffffu, first);
            const int64_t e0 = base + u * T + t - lane;
            if (lane == 0 && e0 < a.P) a.first[e0 >> 5] = b;
        }
    }
    mine = warp_sum(mine);
    if (lane == 0 && mine) atomicAdd(&a.tally->m, mine);
    if (err) atomicOr(&a.tally->err, err);
}

// --- relabel: stable counting passes on the degree ----------------------------
__device__ void relabel_count(const BuildArgs& a, int pass, const uint32_t* in) {
    if ((int)blockIdx.x >= a.nchunks) return;
    __shared__ unsigned h[256];
    if (threadIdx.x < 256) h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t c0 = (int64_t)blockIdx.x * a.chunk, c1 = min64(c0 + a.chunk, a.n);
    int mx = 0;
    for (int64_t p = c0 + threadIdx.x; p < c1; p += kBT) {
        const int d = a.deg[in ? in[p] : p];
        mx = max(mx, d);
        atomicAdd(&h[(d >> (8 * pass)) & 255], 1u);
    }
    if (pass == 0) {
        mx = warp_max(mx);
        if ((threadIdx.x & 31) == 0 && mx) atomicMax(&a.tally->maxdeg, mx);
    }
    __syncthreads();
    if (threadIdx.x < 256) a.hist[(size_t)blockIdx.x * 256 + threadIdx.x] = h[threadIdx.x];
}

// out = the vertices by this digit, or (last pass) perm and degn by label
__device__ void relabel_scatter(const BuildArgs& a, int pass, const uint32_t* in, uint32_t* out, bool last) {
    if ((int)blockIdx.x >= a.nchunks) return;
    __shared__ unsigned base[256], half[2][256], whole[2][256], wsum[8];
    __shared__ unsigned short wcnt[kBW][256];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    {
        // digit d: the entries of earlier blocks, and all entries of lower digits
        const int d = threadIdx.x & 255, part = threadIdx.x >> 8;
        unsigned before = 0, all = 0;
#pragma unroll 8
        for (int c = part; c < a.nchunks; c += 2) {
            const unsigned x = a.hist[(size_t)c * 256 + d];
            all += x;
            if (c < (int)blockIdx.x) before += x;
        }
        half[part][d] = before;
        whole[part][d] = all;
        __syncthreads();
        if (part == 0) {
            const unsigned c = whole[0][d] + whole[1][d];
            unsigned inc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) wsum[w] = inc;
            base[d] = inc - c + half[0][d] + half[1][d];
        }
        __syncthreads();
        if (part == 0)
            for (int q = 0; q < w; ++q) base[d] += wsum[q];
    }
    const int64_t c0 = (int64_t)blockIdx.x * a.chunk, c1 = min64(c0 + a.chunk, a.n);
    for (int64_t t0 = c0; t0 < c1; t0 += kTileN) {
        for (int q = threadIdx.x; q < kBW * 256; q += kBT) (&wcnt[0][0])[q] = 0;
        __syncthreads();
        uint32_t v[kBItems];
        int dg[kBItems], dig[kBItems];
        unsigned rank[kBItems];
#pragma unroll
        for (int r = 0; r < kBItems; ++r) {
            const int64_t p = t0 + w * 32 * kBItems + r * 32 + lane;
            v[r] = p < c1 ? (in ? in[p] : (uint32_t)p) : 0u;
            dg[r] = p < c1 ? a.deg[v[r]] : -1;
        }
#pragma unroll
        for (int r = 0; r < kBItems; ++r) {
            const bool valid = dg[r] >= 0;
            const int d = valid ? (dg[r] >> (8 * pass)) & 255 : 0;
            dig[r] = d;
            unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const bool bit = (d >> b) & 1;
                const unsigned bal = __ballot_sync(0xffffffffu, bit);
                peers &= bit ? bal : ~bal;
            }
            const unsigned prior = valid ? wcnt[w][d] : 0u;
            __syncwarp();
            if (valid) {
                rank[r] = prior + __popc(peers & ((1u << lane) - 1u));
                if (lane == __ffs(peers) - 1) wcnt[w][d] = (unsigned short)(prior + __popc(peers));
            }
            __syncwarp();
        }
        __syncthreads();
        unsigned total = 0;
        if (threadIdx.x < 256) {
#pragma unroll
            for (int q = 0; q < kBW; ++q) {
                const unsigned c = wcnt[q][threadIdx.x];
                wcnt[q][threadIdx.x] = (unsigned short)total;
                total += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kBItems; ++r)
            if (dg[r] >= 0) {
                const unsigned at = base[dig[r]] + wcnt[w][dig[r]] + rank[r];
                if (last) {
                    a.perm[v[r]] = (int32_t)at;
                    a.degn[at] = dg[r];
                    if (a.comp) a.comp[at] = comp_index(a.vpre, a.num_comps, v[r]);
                } else {
                    out[at] = v[r];
                }
            }
        __syncthreads();
        if (threadIdx.x < 256) base[threadIdx.x] += total;
    }
}

// --- orient -----------------------------------------------------------------
__device__ void phase_orient(const BuildArgs& a) {
    const int64_t T = (int64_t)gridDim.x * kBT, t = (int64_t)blockIdx.x * kBT + threadIdx.x;
    const int lane = threadIdx.x & 31;
    for (int64_t base = t; base - lane < a.P; base += kBItems * T) {
        unsigned lo[kBItems], hi[kBItems], at[kBItems];
        bool on[kBItems];
#pragma unroll
        for (int u = 0; u < kBItems; ++u) {
            const int64_t e = base + u * T;
            on[u] = e < a.P && ((a.first[e >> 5] >> lane) & 1u);
            lo[u] = hi[u] = 0;
            if (on[u]) {
                lo[u] = (unsigned)a.src[e];
                hi[u] = (unsigned)a.dst[e];
            }
        }
#pragma unroll
        for (int u = 0; u < kBItems; ++u)
            if (on[u]) {
                const unsigned x = (unsigned)a.perm[lo[u]], y = (unsigned)a.perm[hi[u]];
                lo[u] = min(x, y);
                hi[u] = max(x, y);
            }
#pragma unroll
        for (int u = 0; u < kBItems; ++u)
            if (on[u]) at[u] = (unsigned)atomicAdd(&a.dplus[lo[u]], 1);
#pragma unroll
        for (int u = 0; u < kBItems; ++u)
            if (on[u]) {
                a.pairs[base + u * T] = make_uint2(lo[u], hi[u]);
                a.place[base + u * T] = at[u];
            }
    }
}

// --- offsets ----------------------------------------------------------------
__device__ void offsets_sum(const BuildArgs& a) {
    if ((int)blockIdx.x >= a.nchunks) return;
    const int64_t c0 = (int64_t)blockIdx.x * a.chunk, c1 = min64(c0 + a.chunk, a.n);
    long long s = 0;
    unsigned long long probes = 0, ijk = 0;
    int mx = 0;
    for (int64_t r = c0 + threadIdx.x; r < c1; r += kBT) {
        if (a.zcap > 0) a.zrow[r] = make_uint2(0, 0);
        const long long d = a.dplus[r], din = a.degn[r] - d;
        s += d;
        mx = max(mx, (int)d);
        probes += (unsigned long long)(d * (d - 1) / 2);
        ijk += (unsigned long long)(din * d);
    }
    long long total;
    block_scan(s, &total);
    if (threadIdx.x == 0) a.sums[blockIdx.x] = total;
    mx = warp_max(mx);
    probes = warp_sum(probes);
    ijk = warp_sum(ijk);
    if ((threadIdx.x & 31) == 0) {
        if (mx) atomicMax(&a.tally->maxout, mx);
        if (probes) atomicAdd(&a.tally->probes, probes);
        if (ijk) atomicAdd(&a.tally->probes_ijk, ijk);
    }
}

// lists r in list[] (one atomic a warp)
__device__ __forceinline__ void list_rows(bool on, int64_t r, uint32_t* list, int* count) {
    const int lane = threadIdx.x & 31;
    const unsigned b = __ballot_sync(0xffffffffu, on);
    if (!b) return;
    int at = 0;
    if (lane == 0) at = atomicAdd(count, __popc(b));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (on) list[at + __popc(b & ((1u << lane) - 1u))] = (uint32_t)r;
}

__device__ void offsets_write(const BuildArgs& a) {
    if ((int)blockIdx.x >= a.nchunks) return;
    const int64_t c0 = (int64_t)blockIdx.x * a.chunk, c1 = min64(c0 + a.chunk, a.n);
    long long carry = block_sum(a.sums, blockIdx.x);
    for (int64_t t0 = c0; t0 < c1; t0 += kTileN) {
        int d[kBItems];
        long long s = 0, total;
        const int64_t r0 = t0 + (int64_t)threadIdx.x * kBItems;
#pragma unroll
        for (int q = 0; q < kBItems; ++q) {
            d[q] = r0 + q < c1 ? a.dplus[r0 + q] : 0;
            s += d[q];
        }
        long long run = carry + block_scan(s, &total);
        carry += total;
#pragma unroll
        for (int q = 0; q < kBItems; ++q) {
            if (r0 + q < c1) {
                if (a.off64) static_cast<int64_t*>(a.off)[r0 + q] = run;
                else static_cast<int32_t*>(a.off)[r0 + q] = (int32_t)run;
            }
            run += d[q];
            list_rows(d[q] > kMedRow && d[q] <= kLongRow, r0 + q, a.ord0, &a.tally->nmed);
            list_rows(d[q] > kLongRow, r0 + q, a.ord1, &a.tally->nlong);
        }
    }
    if ((int)blockIdx.x == a.nchunks - 1 && threadIdx.x == 0) {
        if (a.off64) static_cast<int64_t*>(a.off)[a.n] = carry;
        else static_cast<int32_t*>(a.off)[a.n] = (int32_t)carry;
    }
}

__device__ void phase_scatter(const BuildArgs& a) {
    const int64_t T = (int64_t)gridDim.x * kBT, t = (int64_t)blockIdx.x * kBT + threadIdx.x;
    const int lane = threadIdx.x & 31;
    for (int64_t base = t; base - lane < a.P; base += kBItems * T) {
        uint2 p[kBItems];
        int64_t at[kBItems];
        bool on[kBItems];
#pragma unroll
        for (int u = 0; u < kBItems; ++u) {
            const int64_t e = base + u * T;
            on[u] = e < a.P && ((a.first[e >> 5] >> lane) & 1u);
            if (on[u]) {
                p[u] = a.pairs[e];
                at[u] = a.place[e];
            }
        }
#pragma unroll
        for (int u = 0; u < kBItems; ++u)
            if (on[u]) at[u] += row_begin(a, p[u].x);
#pragma unroll
        for (int u = 0; u < kBItems; ++u)
            if (on[u]) a.adj[at[u]] = (int32_t)p[u].y;
    }
}

// The counter that takes row i's task at pivot j.  A hub is a column of up to
// a fifteenth of all rows, and the atomics on one counter are served one after
// the other (about 7 ns each when the value comes back: RMAT scale 20, with
// 64,599 edges at one vertex, spent 454 us of its sort there), so the rows
// are dealt out over tcopies counters.
__device__ __forceinline__ int64_t task_counter(const BuildArgs& a, uint32_t i, uint32_t j) {
    return (int64_t)(i & (unsigned)(a.tcopies - 1)) * a.n + j;
}

// --- sort -------------------------------------------------------------------
// A row's sorted entry x at edge e, with `more` when entries follow it: the
// column, the row, and (a task) its place among the tasks of pivot x.
__device__ __forceinline__ void put_entry(const BuildArgs& a, int64_t e, uint32_t x, uint32_t r, bool more) {
    a.adj[e] = (int32_t)x;
    a.row[e] = r;
    if (more) a.place[e] = (uint32_t)atomicAdd(&a.tcur[task_counter(a, r, x)], 1);
}

// Rows of at most W entries, 32 / W of them at a time: W lanes a row, a
// bitonic network of shuffles.  `todo`: the lanes whose row (begin rb,
// length d, label r0 + lane) is of this class.
template <int W>
__device__ __forceinline__ void sort_rows_sub(const BuildArgs& a, unsigned todo, int64_t rb, int d, int64_t r0) {
    const int lane = threadIdx.x & 31, q = lane & (W - 1);
    while (todo) {
        int from = -1;
#pragma unroll
        for (int s = 0; s < 32 / W; ++s) {
            const int b = __ffs(todo) - 1;
            if (todo) todo &= todo - 1;
            if (s == lane / W) from = b;
        }
        const int64_t b = __shfl_sync(0xffffffffu, rb, max(from, 0));
        int len = __shfl_sync(0xffffffffu, d, max(from, 0));
        if (from < 0) len = 0;
        uint32_t x = q < len ? (uint32_t)a.adj[b + q] : 0xffffffffu;
#pragma unroll
        for (int k = 2; k <= W; k <<= 1)
#pragma unroll
            for (int j = k >> 1; j > 0; j >>= 1) {
                const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
                x = (((q & k) == 0) == ((q & j) == 0)) ? min(x, y) : max(x, y);
            }
        if (q < len) put_entry(a, b + q, x, (uint32_t)(r0 + from), q + 1 < len);
    }
}

// One row of at most 32 * E entries by one warp: lane l sorts with entries
// l*E .. l*E+E-1 in registers, then the row goes through the warp's shared
// memory (32 * E words and a word of padding every 32) to be written out
// coalesced.
template <int E>
__device__ __forceinline__ void sort_row_warp(const BuildArgs& a, int64_t rb, int d, uint32_t r, uint32_t* buf) {
    const int lane = threadIdx.x & 31;
    uint32_t x[E];
#pragma unroll
    for (int q = 0; q < E; ++q) x[q] = q * 32 + lane < d ? (uint32_t)a.adj[rb + q * 32 + lane] : 0xffffffffu;
#pragma unroll
    for (int k = 2; k <= 32 * E; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j < E) {
#pragma unroll
                for (int q = 0; q < E; ++q)
                    if ((q & j) == 0) {
                        const bool up = ((lane * E + q) & k) == 0;
                        const uint32_t lo = min(x[q], x[q | j]), hi = max(x[q], x[q | j]);
                        x[q] = up ? lo : hi;
                        x[q | j] = up ? hi : lo;
                    }
            } else {
                const int lj = j / E;
#pragma unroll
                for (int q = 0; q < E; ++q) {
                    const uint32_t y = __shfl_xor_sync(0xffffffffu, x[q], lj);
                    const bool up = ((lane * E + q) & k) == 0;
                    x[q] = (((lane & lj) == 0) == up) ? min(x[q], y) : max(x[q], y);
                }
            }
        }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < E; ++q) {
        const int p = lane * E + q;
        buf[p + (p >> 5)] = x[q];
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < E; ++q) {
        const int p = q * 32 + lane;
        if (p < d) put_entry(a, rb + p, buf[p + (p >> 5)], r, p + 1 < d);
    }
}

__device__ void phase_sort(const BuildArgs& a, uint32_t* smem) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // rows beyond kLongRow: a block each, bitonic in shared memory
    const int nlong = a.tally->nlong, nmed = a.tally->nmed;
    for (int x = blockIdx.x; x < nlong; x += gridDim.x) {
        const uint32_t r = a.ord1[x];
        const int64_t rb = row_begin(a, r);
        const int d = (int)(row_begin(a, (int64_t)r + 1) - rb);
        if (d > kMaxRow) {
            if (threadIdx.x == 0) atomicOr(&a.tally->err, 8);
            continue;
        }
        int N = 2 * kLongRow;
        while (N < d) N <<= 1;
        for (int q = threadIdx.x; q < N; q += kBT) smem[q] = q < d ? (uint32_t)a.adj[rb + q] : 0xffffffffu;
        __syncthreads();
        for (int k = 2; k <= N; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int h = threadIdx.x; h < N / 2; h += kBT) {
                    const int q = ((h & ~(j - 1)) << 1) | (h & (j - 1));   // the lower of the pair
                    const uint32_t lo = smem[q], hi = smem[q | j];
                    if ((lo > hi) == ((q & k) == 0)) {
                        smem[q] = hi;
                        smem[q | j] = lo;
                    }
                }
                __syncthreads();
            }
        for (int q = threadIdx.x; q < d; q += kBT) put_entry(a, rb + q, smem[q], r, q + 1 < d);
        __syncthreads();
    }
    // rows of kMedRow+1 .. kLongRow: a warp each, taken from the list
    uint32_t* buf = smem + w * (kLongRow + 32);
    while (true) {
        int x = 0;
        if (lane == 0) x = atomicAdd(&a.tally->med_head, 1);
        x = __shfl_sync(0xffffffffu, x, 0);
        if (x >= nmed) break;
        const uint32_t r = a.ord0[x];
        const int64_t rb = row_begin(a, r);
        const int d = (int)(row_begin(a, (int64_t)r + 1) - rb);
        if (d <= 64) sort_row_warp<2>(a, rb, d, r, buf);
        else if (d <= 128) sort_row_warp<4>(a, rb, d, r, buf);
        else if (d <= 256) sort_row_warp<8>(a, rb, d, r, buf);
        else if (d <= 512) sort_row_warp<16>(a, rb, d, r, buf);
        else sort_row_warp<32>(a, rb, d, r, buf);
    }
    // the rest: `per` neighbouring rows a warp at a time, few enough that
    // every warp gets some (a warp's rows wait for one another's loads)
    const int64_t warps = (int64_t)gridDim.x * kBW;
    int per = 32;
    while (per > 2 && a.n < 2 * per * warps) per >>= 1;
    for (int64_t r0 = ((int64_t)blockIdx.x * kBW + w) * per; r0 < a.n; r0 += warps * per) {
        const int64_t r = r0 + lane;
        int64_t rb = 0;
        int d = 0;
        if (lane < per && r < a.n) {
            rb = row_begin(a, r);
            d = (int)(row_begin(a, r + 1) - rb);
        }
        if (d == 1) a.row[rb] = (uint32_t)r;
        sort_rows_sub<8>(a, __ballot_sync(0xffffffffu, d > 1 && d <= 8), rb, d, r0);
        sort_rows_sub<16>(a, __ballot_sync(0xffffffffu, d > 8 && d <= 16), rb, d, r0);
        sort_rows_sub<32>(a, __ballot_sync(0xffffffffu, d > 16 && d <= 32), rb, d, r0);
    }
}

// --- tasks and units ----------------------------------------------------------
__device__ void tasks_sum(const BuildArgs& a) {
    if ((int)blockIdx.x >= a.nchunks) return;
    const int64_t c0 = (int64_t)blockIdx.x * a.chunk, c1 = min64(c0 + a.chunk, a.n);
    long long t = 0, us = 0, ul = 0, uz = 0, total;
    for (int64_t r = c0 + threadIdx.x; r < c1; r += kBT) {
        long long nt = 0;
        int64_t x, y, z;
        for (int c = 0; c < a.tcopies; ++c) nt += a.tcur[c * a.n + r];
        unit_split<false>(a.rule, a.zcap > 0, a.dplus[r], nt, x, y, z);
        t += nt;
        us += x;
        ul += y;
        uz += z;
    }
    long long* s = a.sums + a.nchunks;   // the row sums may still be read by slower blocks
    block_scan(t, &total);
    if (threadIdx.x == 0) s[blockIdx.x] = total;
    block_scan(us, &total);
    if (threadIdx.x == 0) {
        s[a.nchunks + blockIdx.x] = total;
        if (total) atomicAdd(reinterpret_cast<unsigned long long*>(&a.tally->nsmall), (unsigned long long)total);
    }
    block_scan(ul, &total);
    if (threadIdx.x == 0) {
        s[2 * a.nchunks + blockIdx.x] = total;
        if (total) atomicAdd(reinterpret_cast<unsigned long long*>(&a.tally->nlarge), (unsigned long long)total);
    }
    block_scan(uz, &total);
    if (threadIdx.x == 0) {
        s[3 * a.nchunks + blockIdx.x] = total;
        if (total) atomicAdd(reinterpret_cast<unsigned long long*>(&a.tally->nzone), (unsigned long long)total);
    }
}

// --- zones: the bit blocks of the listed rows, a warp each --------------------
__device__ void phase_zones(const BuildArgs& a, uint32_t* smem) {
    if (a.zcap == 0) return;
    const int w = threadIdx.x >> 5;
    uint32_t* buf = smem + w * kZoneWords;
    const int nmed = a.tally->nmed, all = nmed + a.tally->nlong;
    for (int x = blockIdx.x * kBW + w; x < all; x += gridDim.x * kBW) {
        const uint32_t r = x < nmed ? a.ord0[x] : a.ord1[x - nmed];
        const int64_t rb = row_begin(a, r);
        zone_row(a.adj, rb, (int)(row_begin(a, (int64_t)r + 1) - rb), r, a.n, a.zrow, a.zbits, a.zowner, a.zcap,
                 &a.tally->nblocks, buf);
    }
}

__device__ void tasks_offsets(const BuildArgs& a) {
    if ((int)blockIdx.x >= a.nchunks) return;
    const int64_t c0 = (int64_t)blockIdx.x * a.chunk, c1 = min64(c0 + a.chunk, a.n);
    long long carry = block_sum(a.sums + a.nchunks, blockIdx.x);
    for (int64_t t0 = c0; t0 < c1; t0 += kBT) {
        const int64_t r = t0 + threadIdx.x;
        int d[kTaskCopies];
        long long s = 0, total;
#pragma unroll
        for (int c = 0; c < kTaskCopies; ++c) {
            d[c] = r < c1 && c < a.tcopies ? a.tcur[c * a.n + r] : 0;
            s += d[c];
        }
        long long run = carry + block_scan(s, &total);
        carry += total;
        if (r < c1) {
            // the first slots, with the pivot's part in the zones in the top bit
            const int32_t big = a.zcap > 0 && a.dplus[r] > kZoneMinPivot ? (int32_t)0x80000000 : 0;
            a.loff[r] = run;
#pragma unroll
            for (int c = 0; c < kTaskCopies; ++c)
                if (c < a.tcopies) {
                    a.tcur[c * a.n + r] = (int32_t)run | big;
                    run += d[c];
                }
        }
    }
    if ((int)blockIdx.x == a.nchunks - 1 && threadIdx.x == 0) {
        a.loff[a.n] = carry;
        a.tally->tasks = (unsigned long long)carry;
    }
}

__device__ void tasks_write(const BuildArgs& a) {
    const int64_t T = (int64_t)gridDim.x * kBT, t = (int64_t)blockIdx.x * kBT + threadIdx.x;
    const int64_t m = row_begin(a, a.n);
    unsigned long long cut = 0;
    for (int64_t base = t; base < m; base += kBItems * T) {
        uint32_t i[kBItems], j[kBItems], at[kBItems];
        int len[kBItems];
        int32_t slot[kBItems];
        uint2 zr[kBItems];
#pragma unroll
        for (int u = 0; u < kBItems; ++u) {
            const int64_t e = base + u * T;
            if (e < m) {
                i[u] = a.row[e];
                j[u] = (uint32_t)a.adj[e];
                at[u] = a.place[e];   // not set for a row's last entry: unused there
            }
        }
#pragma unroll
        for (int u = 0; u < kBItems; ++u) {
            const int64_t e = base + u * T;
            len[u] = 0;
            if (e < m) {
                len[u] = (int)(row_begin(a, (int64_t)i[u] + 1) - e - 1);
                slot[u] = a.tcur[task_counter(a, i[u], j[u])];
                zr[u] = a.zcap > 0 ? a.zrow[i[u]] : make_uint2(0, 0);
            }
        }
#pragma unroll
        for (int u = 0; u < kBItems; ++u)
            if (len[u] > 0) {
                Task x;
                x.start = (uint32_t)(base + u * T + 1);
                x.len = zone_cut(zr[u], slot[u] < 0, base + u * T, len[u], &x.zone);
                x.i = (int32_t)i[u];
                cut += (unsigned)(len[u] - x.len);
                a.tasks[(int64_t)(slot[u] & 0x7fffffff) + at[u]] = x;
            }
    }
    cut = warp_sum(cut);
    if ((threadIdx.x & 31) == 0 && cut) atomicAdd(&a.tally->covered, cut);
}

__device__ __forceinline__ void put_unit(const BuildArgs& a, Unit* small_at, int64_t j, bool small, long long at, int64_t q,
                                         int64_t slices, int64_t t0, int64_t t1) {
    Unit u;
    u.j = (int32_t)j;
    u.g = 0;
    u.pad = 0;
    if (small) {
        u.slice = 0;
        u.t0 = t0 + q * a.rule.warp_tasks;
        u.t1 = min64(u.t0 + a.rule.warp_tasks, t1);
        small_at[at + q] = u;
    } else {
        u.slice = (int32_t)(q % slices);
        u.t0 = t0 + q / slices * a.rule.cta_tasks;
        u.t1 = min64(u.t0 + a.rule.cta_tasks, t1);
        a.large[at + q] = u;
    }
}

// Units in descending label order (heaviest pivots first): a pivot's place is
// what the labels above it take.  A hub may have thousands of units: those of
// a pivot with more than kBItems are written by the whole warp.
__device__ void phase_units(const BuildArgs& a) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.view_at = a.view;
        *a.view_comp_at = a.view_comp;
    }
    if ((int)blockIdx.x >= a.nchunks) return;
    const int lane = threadIdx.x & 31;
    const int64_t c0 = (int64_t)blockIdx.x * a.chunk, c1 = min64(c0 + a.chunk, a.n);
    long long cs = block_sum(a.sums + 2 * a.nchunks, blockIdx.x);
    long long cl = block_sum(a.sums + 3 * a.nchunks, blockIdx.x);
    long long cz = block_sum(a.sums + 4 * a.nchunks, blockIdx.x);
    const long long ns = a.tally->nsmall, nl = a.tally->nlarge, nz = a.tally->nzone;
    for (int64_t t0 = c0; t0 < c1; t0 += kBT) {
        const int64_t j = t0 + threadIdx.x;
        int64_t us = 0, ul = 0, uz = 0;
        long long ts, tl, tz;
        int64_t b0 = 0, b1 = 0, slices = 1;
        if (j < c1) {
            const int64_t dp = row_begin(a, j + 1) - row_begin(a, j);
            b0 = a.loff[j];
            b1 = a.loff[j + 1];
            unit_split<false>(a.rule, a.zcap > 0, dp, b1 - b0, us, ul, uz);
            slices = (dp + a.rule.slice - 1) / a.rule.slice;
        }
        const long long xs = cs + block_scan(us, &ts), xl = cl + block_scan(ul, &tl);
        const long long az = nz - uz - (cz + block_scan(uz, &tz));
        cs += ts;
        cl += tl;
        cz += tz;
        const bool small = us > 0;
        const long long count = us + ul;
        const long long at = small ? ns - xs - us : nl - xl - ul;
        if (count > 0 && count <= kBItems)
            for (int64_t q = 0; q < count; ++q) put_unit(a, a.wide + nz, j, small, at, q, slices, b0, b1);
        unsigned many = __ballot_sync(0xffffffffu, count > kBItems);
        while (many) {
            const int o = __ffs(many) - 1;
            many &= many - 1;
            const long long c = __shfl_sync(0xffffffffu, count, o), p = __shfl_sync(0xffffffffu, at, o);
            const int64_t x0 = __shfl_sync(0xffffffffu, b0, o), x1 = __shfl_sync(0xffffffffu, b1, o);
            const int64_t s = __shfl_sync(0xffffffffu, slices, o), jj = __shfl_sync(0xffffffffu, j, o);
            const bool sm = __shfl_sync(0xffffffffu, (int)small, o);
            for (int64_t q = lane; q < c; q += 32) put_unit(a, a.wide + nz, jj, sm, p, q, s, x0, x1);
        }
        unsigned zoned = __ballot_sync(0xffffffffu, uz > 0);
        while (zoned) {
            const int o = __ffs(zoned) - 1;
            zoned &= zoned - 1;
            const long long c = __shfl_sync(0xffffffffu, uz, o), p = __shfl_sync(0xffffffffu, az, o);
            const int64_t x0 = __shfl_sync(0xffffffffu, b0, o), x1 = __shfl_sync(0xffffffffu, b1, o);
            const int64_t jj = __shfl_sync(0xffffffffu, j, o);
            for (int64_t q = lane; q < c; q += 32)
                a.wide[p + q] =
                    Unit{(int32_t)jj, 0, 0, 0, x0 + q * a.rule.wide_tasks, min64(x0 + (q + 1) * a.rule.wide_tasks, x1)};
        }
    }
}

__global__ void __launch_bounds__(kBT, kBlocksPerSm) k_build(const __grid_constant__ BuildArgs a, int bits) {
    extern __shared__ __align__(16) uint32_t smem[];
    Grid grid{a.tally, &a.tally->bar[a.phase0 == kPhaseInsert ? 0 : 1], 0};
    if (a.phase0 == kPhaseInsert) {
        phase_clear(a);
        if (!grid.sync()) return;
        phase_insert(a, bits);
        if (a.phase1 > kPhaseGraph && !grid.sync()) return;
    }
    if (a.phase0 <= kPhaseGraph && a.phase1 > kPhaseGraph) {
        const uint32_t* in = nullptr;
        uint32_t *out = a.ord0, *other = a.ord1;
        int passes = 1;
        for (int p = 0; p < passes; ++p) {
            relabel_count(a, p, in);
            if (!grid.sync()) return;
            if (p == 0)
                while (passes < 4 && (a.tally->maxdeg >> (8 * passes)) != 0) ++passes;
            relabel_scatter(a, p, in, out, p == passes - 1);
            if (!grid.sync()) return;
            in = out;
            out = other;
            other = const_cast<uint32_t*>(in);
        }
        phase_orient(a);
        if (!grid.sync()) return;
        offsets_sum(a);
        if (!grid.sync()) return;
        offsets_write(a);
        if (!grid.sync()) return;
        phase_scatter(a);
        if (!grid.sync()) return;
        phase_sort(a, smem);
        if (!grid.sync()) return;
        tasks_sum(a);
        phase_zones(a, smem);
        if (!grid.sync()) return;
        tasks_offsets(a);
        if (!grid.sync()) return;
        tasks_write(a);
    }
    if (a.phase1 > kPhaseUnits) phase_units(a);
}

size_t pad256(size_t x) { return (x + 255) & ~size_t(255); }

constexpr size_t kBuildSmem = sizeof(uint32_t) * (size_t)kBW * (kLongRow + 32);
static_assert(kBuildSmem >= sizeof(uint32_t) * kMaxRow, "a long row fits the warps' buffers");

}  // namespace

bool build_takes(int64_t P, int64_t n) { return P > 0 && P <= kBuildMaxPairs && n <= kBuildMaxPairs; }

void build_graph(tc_graph* g, const int32_t* src, const int32_t* dst, int64_t P, uint32_t flags,
                 const int64_t* vpre_host, int32_t num_comps, cudaStream_t st) {
    Alloc& al = g->alloc;
    const int64_t n = g->n;
    const bool one = P <= kBuildOnePairs && !g->lean;
    tc_tuning def;
    tuning_defaults(&def);

    // scratch in one block: the tally, the vertex arrays, the set (its memory
    // then holds the oriented pairs, their places and the edges' rows)
    const int64_t nchunks = std::min<int64_t>(std::max<int64_t>((n + 2 * kBT - 1) / (2 * kBT), 1),
                                              std::min<int64_t>(kMaxChunks, (int64_t)num_sms() * kBlocksPerSm));
    BuildArgs a{};
    a.chunk = ((n + nchunks - 1) / nchunks + 31) / 32 * 32;
    a.nchunks = (int)std::max<int64_t>(1, (n + a.chunk - 1) / std::max<int64_t>(a.chunk, 1));
    a.cap = 2 * (uint64_t)std::max<int64_t>(P, 512);
    const size_t nv = (size_t)std::max<int64_t>(n, 1);
    a.tcopies = g->lean ? 1 : n <= (1ll << 21) ? kTaskCopies : n <= (1ll << 22) ? 4 : 1;
    size_t need = 0;
    auto take = [&](size_t bytes) {
        const size_t at = need;
        need += pad256(bytes);
        return at;
    };
    const size_t o_tally = take(sizeof(Tally)), o_vpre = take(8 * (size_t)(num_comps + 1));
    const size_t o_hist = take(4 * 256 * (size_t)a.nchunks), o_sums = take(8 * 5 * (size_t)a.nchunks);
    const size_t o_deg = take(4 * nv), o_degn = take(4 * nv), o_dplus = take(4 * nv), o_tcur = take(4 * nv * (size_t)a.tcopies);
    const size_t o_ord0 = take(4 * nv), o_ord1 = take(4 * nv);
    const size_t o_first = take(4 * (size_t)((P + 31) / 32));
    const size_t o_table = take(8 * (size_t)a.cap);
    Buf<char> scratch(al, need);
    char* s = scratch.get();
    a.tally = reinterpret_cast<Tally*>(s + o_tally);
    a.hist = reinterpret_cast<unsigned*>(s + o_hist);
    a.sums = reinterpret_cast<long long*>(s + o_sums);
    a.deg = reinterpret_cast<int32_t*>(s + o_deg);
    a.degn = reinterpret_cast<int32_t*>(s + o_degn);
    a.dplus = reinterpret_cast<int32_t*>(s + o_dplus);
    a.tcur = reinterpret_cast<int32_t*>(s + o_tcur);
    a.ord0 = reinterpret_cast<uint32_t*>(s + o_ord0);
    a.ord1 = reinterpret_cast<uint32_t*>(s + o_ord1);
    a.first = reinterpret_cast<uint32_t*>(s + o_first);
    a.table = reinterpret_cast<uint64_t*>(s + o_table);
    a.pairs = reinterpret_cast<uint2*>(a.table);
    a.place = reinterpret_cast<uint32_t*>(a.pairs + P);
    a.row = a.place + P;
    a.src = src;
    a.dst = dst;
    a.P = P;
    a.n = n;
    a.num_comps = num_comps;
    TC_CUDA(cudaMemsetAsync(a.tally, 0, sizeof(Tally), st));
    if (num_comps > 0) {
        a.vpre = reinterpret_cast<const int64_t*>(s + o_vpre);
        // pageable source: the copy is staged before the call returns
        TC_CUDA(cudaMemcpyAsync(s + o_vpre, vpre_host, sizeof(int64_t) * (size_t)(num_comps + 1),
                                cudaMemcpyHostToDevice, st));
    }

    Tally h{};
    auto read_tally = [&]() {
        TC_CUDA(cudaMemcpyAsync(&h, a.tally, sizeof(Tally), cudaMemcpyDeviceToHost, st));
        TC_CUDA(cudaStreamSynchronize(st));
        if (h.err & 1) TC_FAIL(TC_EINVAL, "tc_preprocess: a vertex id lies outside [0, n)");
        if (h.err & 2) TC_FAIL(TC_EINVAL, "tc_preprocess_components: a pair joins two components");
        if (h.err & 4) TC_FAIL(TC_ETIMEOUT, "tc_preprocess: a grid barrier wait ran past its bound");
        if (h.err & 8) TC_FAIL(TC_EUNSUPPORTED, "tc_preprocess: a row of U exceeds the row sort's bound");
    };
    // co-resident blocks: one thread an entry of the larger side, at most
    // kBlocksPerSm a multiprocessor
    const unsigned blocks = (unsigned)std::min<int64_t>(
        std::max<int64_t>((std::max(P, n) + kBT - 1) / kBT, a.nchunks), (int64_t)num_sms() * kBlocksPerSm);
    TC_CUDA(cudaFuncSetAttribute(k_build, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBuildSmem));
    auto launch = [&](int p0, int p1) {
        a.phase0 = p0;
        a.phase1 = p1;
        int bits = g->bits;
        void* args[] = {&a, &bits};
        Prof prof_("k_build", st);
        TC_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_build), dim3(blocks), dim3(kBT), args,
                                            kBuildSmem, st));
    };

    const bool off64 = (flags & TC_OFFSETS_64) != 0;   // m < 2^31 - 1 here
    a.off64 = off64 ? 1 : 0;
    int64_t cap_m = P;   // one launch: arrays sized by the pairs
    if (!one) {
        launch(kPhaseInsert, kPhaseGraph);
        read_tally();
        cap_m = (int64_t)h.m;
    }
    g->plan_m = cap_m;
    const tc_tuning tt = clamp_tuning(size_tuning(def, cap_m));
    graph_arena(g, cap_m, g->lean ? 0 : zone_capacity(cap_m), off64, num_comps);
    a.off = g->off;
    a.adj = g->adj;
    a.perm = g->perm;
    a.loff = g->loff;
    a.tasks = g->tasks;
    a.comp = g->comp;
    a.zrow = g->zrow;
    a.zbits = g->zbits;
    a.zowner = g->zowner;
    a.zcap = g->zcap;
    graph_views(g, &a.view, &a.view_comp);
    a.view_at = g->view;
    a.view_comp_at = g->view_comp;
    a.rule = unit_rule(tt, false, g->zcap > 0);
    UnitLists L;
    auto take_units = [&](int64_t nl, int64_t rest) {
        L.bytes = sizeof(Unit) * (size_t)std::max<int64_t>(nl + rest, 1);
        L.mem = al.get(L.bytes);
        a.large = L.large = static_cast<Unit*>(L.mem);
        a.wide = L.zone = L.large + nl;
        // the graph owns them from here on, whatever fails next
        adopt_units(g, L, tt);
    };
    if (one) {
        // A large pivot has over kSmallMaxOutdeg of the edges and one slice
        // (d^2 <= 2m).  Of the others each has a unit, small or wide, and at
        // most one more for each full unit of tasks; the large ones with
        // zones are wide as well.
        static_assert(2 * kBuildOnePairs <= (int64_t)kMaxSlice * kMaxSlice, "one slice a pivot");
        const int64_t nl = P / kSmallMaxOutdeg + P / a.rule.cta_tasks + 1;
        take_units(nl, std::min(n, P) + P / a.rule.warp_tasks + 2 * (P / a.rule.wide_tasks) + P / kMidMaxOutdeg + 1);
        launch(kPhaseInsert, kPhaseEnd);
        read_tally();
    } else {
        launch(kPhaseGraph, kPhaseUnits);
        read_tally();
        take_units((int64_t)h.nlarge, (int64_t)(h.nsmall + h.nzone));
        launch(kPhaseUnits, kPhaseEnd);
    }
    g->small_units = g->zone_units + h.nzone;
    g->n_small = h.nsmall;
    g->n_large = h.nlarge;
    g->n_zone = h.nzone;
    g->covered = h.covered;
    g->zone_blocks = h.nblocks;
    g->m = (int64_t)h.m;
    g->n_tasks = (int64_t)h.tasks;
    g->stats.m = g->m;
    g->stats.max_deg = h.maxdeg;
    g->stats.max_outdeg = h.maxout;
    g->stats.tasks = (int64_t)h.tasks;
    g->stats.probes = h.probes;
    g->stats.probes_ijk = h.probes_ijk;
    g->stats.offset_bytes = off64 ? 8 : 4;
    g->stats.small_units = h.nsmall;
    g->stats.large_units = h.nlarge;
    g->stats.device_bytes = (int64_t)(g->arena_bytes + g->units_bytes);
}

}  // namespace tc
