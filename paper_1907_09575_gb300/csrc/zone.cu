// The zone kernel (see zone.cuh): the part of the count whose tails lie in
// the dense zones, as ANDs of bit blocks.
//
// A unit is a pivot j and up to 248 of its tasks, counted by one warp.  The
// tasks that have blocks are listed in shared memory by descending number of
// zones, so the tasks of zone q are a prefix.  For each zone the pivot's 64
// words sit in registers, two a lane (its own block, or built from its
// entries), and eight tasks at a time load their 256-byte blocks, AND and
// count.
//
// Totals only: a Harley-Seal tree of carry-save adders (published as such in
// Warren, Hacker's Delight, section 5-1) over the words, one popc for 16
// words: population counts issue at an eighth of the rate of the logic.
// Per-vertex counts: the same adders run down each bit column of the eight
// tasks' words -- bit b of the planes is the number of tasks that hit label b
// -- so that the credit of the third vertex, one shared-memory atomic per hit
// in the list kernel, is three logic operations per word of 32 labels; a
// task's own hits are two popcs a lane and its share of a reduction.  Planes are
// transposed into bytes once a unit and zone and added to the labels'
// accumulators.
#include <algorithm>

#include "common.cuh"
#include "tc_internal.cuh"

namespace tc {
namespace {

constexpr int kZT = 256;           // threads of a block
constexpr int kZW = kZT / 32;
constexpr int kPlanes = 8;         // a label's hits in one unit: at most kZoneTasks
static_assert(kZoneTasks < (1 << kPlanes) && kZoneTasks % 8 == 0, "planes hold a unit's hits");
constexpr int kZoneSlots = 256;    // a unit's tasks, eight a lane
constexpr int kFlushBits = 12;     // labels hit per lane up to which planes are read bit by bit
constexpr int kFlushStride = 33;   // words between the rows of the transposed counts

struct ZoneWarp {                  // one warp's shared memory
    uint32_t task[kZoneSlots];
    uint32_t hits[kZoneSlots];
    uint32_t words[kZoneWords];
    uint32_t flush[16 * kFlushStride];
};

__device__ __forceinline__ int64_t zoff(const GraphView& G, int64_t v) {
    return G.off64 ? static_cast<const int64_t*>(G.off)[v] : (int64_t) static_cast<const int32_t*>(G.off)[v];
}

__device__ __forceinline__ uint64_t zsum(uint64_t v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// full adder of three bit vectors: s = the sum bits, returns the carries
__device__ __forceinline__ uint32_t csa(uint32_t& s, uint32_t a, uint32_t b) {
    const uint32_t carry = (s & a) | (s & b) | (a & b);
    s ^= a ^ b;
    return carry;
}

// planes += the bits of x[0..7] (one word column of eight tasks)
__device__ __forceinline__ void add_planes(uint32_t (&p)[kPlanes], const uint32_t (&x)[8]) {
    const uint32_t t0 = csa(p[0], x[0], x[1]), t1 = csa(p[0], x[2], x[3]);
    const uint32_t t2 = csa(p[0], x[4], x[5]), t3 = csa(p[0], x[6], x[7]);
    const uint32_t f0 = csa(p[1], t0, t1), f1 = csa(p[1], t2, t3);
    uint32_t c = csa(p[2], f0, f1);
#pragma unroll
    for (int k = 3; k < kPlanes; ++k) {
        const uint32_t o = p[k] & c;
        p[k] ^= c;
        c = o;
    }
}

// 8 x 8 bit transposes of the four byte columns: byte c of p[k] becomes the
// eight plane bits of bit 8c + k
__device__ __forceinline__ void transpose_planes(uint32_t (&p)[kPlanes]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t t = ((p[i] >> 4) ^ p[i + 4]) & 0x0f0f0f0fu;
        p[i + 4] ^= t;
        p[i] ^= t << 4;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if ((i & 2) == 0) {
            const uint32_t t = ((p[i] >> 2) ^ p[i + 2]) & 0x33333333u;
            p[i + 2] ^= t;
            p[i] ^= t << 2;
        }
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
        const uint32_t t = ((p[i] >> 1) ^ p[i + 1]) & 0x55555555u;
        p[i + 1] ^= t;
        p[i] ^= t << 1;
    }
}

// a lane's running population count of a stream of words
struct HarleySeal {
    uint32_t ones = 0, twos = 0, fours = 0, eights = 0;
    unsigned sixteens = 0;
    __device__ __forceinline__ void add(const uint32_t (&x)[16]) {
        const uint32_t a0 = csa(ones, x[0], x[1]), a1 = csa(ones, x[2], x[3]);
        const uint32_t a2 = csa(ones, x[4], x[5]), a3 = csa(ones, x[6], x[7]);
        const uint32_t a4 = csa(ones, x[8], x[9]), a5 = csa(ones, x[10], x[11]);
        const uint32_t a6 = csa(ones, x[12], x[13]), a7 = csa(ones, x[14], x[15]);
        const uint32_t b0 = csa(twos, a0, a1), b1 = csa(twos, a2, a3);
        const uint32_t b2 = csa(twos, a4, a5), b3 = csa(twos, a6, a7);
        const uint32_t c0 = csa(fours, b0, b1), c1 = csa(fours, b2, b3);
        sixteens += __popc(csa(eights, c0, c1));
    }
    __device__ __forceinline__ uint64_t take() {
        const uint64_t s = 16ull * sixteens + 8 * __popc(eights) + 4 * __popc(fours) + 2 * __popc(twos) + __popc(ones);
        ones = twos = fours = eights = sixteens = 0;
        return s;
    }
};

template <bool PV>
__global__ void __launch_bounds__(kZT, PV ? 3 : 4)
    k_zone(const GraphView* __restrict__ views, const Unit* __restrict__ units, int64_t nunits, unsigned* tlow,
           unsigned long long* __restrict__ ctr) {
    __shared__ __align__(16) ZoneWarp warps[kZW];
    const int lane = threadIdx.x & 31;
    ZoneWarp& S = warps[threadIdx.x >> 5];
    HarleySeal hs;
    unsigned long long* target = nullptr;
    uint64_t total = 0;
    while (true) {
        long long u = 0;
        if (lane == 0) u = (long long)atomicAdd(&ctr[CTR_ZONE_HEAD], 1ull);
        u = __shfl_sync(0xffffffffu, u, 0);
        if (u >= nunits) break;
        const Unit U = units[u];
        const GraphView G = views[U.g];
        unsigned long long* to = G.comp ? G.comp_totals + G.comp[U.j] : G.total;
        if (to != target) {
            if (!PV) total += hs.take();
            total = zsum(total);
            if (lane == 0 && total) atomicAdd(target, (unsigned long long)total);
            total = 0;
            target = to;
        }
        // the unit's tasks with blocks, by descending number of zones
        uint32_t zt[kZoneSlots / 32];
        int nz = 0;
#pragma unroll
        for (int s = 0; s < kZoneSlots / 32; ++s) {
            const int64_t t = U.t0 + s * 32 + lane;
            zt[s] = t < U.t1 ? G.tasks[t].zone : 0u;
            nz = max(nz, (int)(zt[s] & (unsigned)kZoneMax));
        }
        nz = __reduce_max_sync(0xffffffffu, nz);
        if (nz == 0) continue;
        __syncwarp();   // the last unit's reads of S are done
        int ntask = 0, upto = 0;   // lane q: tasks with more than q zones
        for (int v = nz; v > 0; --v) {
#pragma unroll
            for (int s = 0; s < kZoneSlots / 32; ++s) {
                const bool on = (int)(zt[s] & (unsigned)kZoneMax) == v;
                const unsigned b = __ballot_sync(0xffffffffu, on);
                if (on) S.task[ntask + __popc(b & ((1u << lane) - 1u))] = (zt[s] >> kZoneNzBits) * (uint32_t)(4 * kZoneWords);
                ntask += __popc(b);
            }
            if (lane == v - 1) upto = ntask;
        }
        if (PV)
            for (int t = lane; t < kZoneSlots; t += 32) S.hits[t] = 0;
        const int64_t rb = zoff(G, U.j);
        const uint2 zp = G.zrow[U.j];
        int64_t cursor = (zp.x & (unsigned)kZoneMax) ? (int64_t)zp.y : zoff(G, U.j + 1);
        for (int q = 0; q < nz; ++q) {
            const int64_t low = G.n - (int64_t)kZoneLabels * (q + 1);
            if (U.j >= low + kZoneLabels - 1) break;   // the pivot's entries lie above this zone
            uint2 piv;
            if (q < (int)(zp.x & (unsigned)kZoneMax)) {
                piv = __ldg(reinterpret_cast<const uint2*>(G.zbits + ((size_t)(zp.x >> kZoneNzBits) + q) * kZoneWords) + lane);
            } else {
                __syncwarp();
                S.words[lane] = 0;
                S.words[lane + 32] = 0;
                __syncwarp();
                while (true) {
                    const int64_t p = cursor - 1 - lane;
                    const int64_t b = p >= rb ? G.adj[p] - low : -1;
                    if (b >= 0) atomicOr(&S.words[b >> 5], 1u << (b & 31));
                    const int in = __popc(__ballot_sync(0xffffffffu, b >= 0));
                    cursor -= in;
                    if (in < 32) break;
                }
                __syncwarp();
                piv = reinterpret_cast<uint2*>(S.words)[lane];
            }
            if (!__any_sync(0xffffffffu, (piv.x | piv.y) != 0)) continue;
            const int nq = __shfl_sync(0xffffffffu, upto, q);
            __syncwarp();
            const char* __restrict__ zb = reinterpret_cast<const char*>(G.zbits + q * kZoneWords) + 8 * lane;
            uint32_t px[kPlanes], py[kPlanes];
#pragma unroll
            for (int k = 0; k < kPlanes; ++k) px[k] = py[k] = 0;
            auto fetch = [&](int t, uint2 (&w)[8]) {
                uint32_t a[8];
                *reinterpret_cast<uint4*>(a) = *reinterpret_cast<const uint4*>(&S.task[t]);
                *reinterpret_cast<uint4*>(a + 4) = *reinterpret_cast<const uint4*>(&S.task[t + 4]);
                if (t + 8 <= nq) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) w[k] = __ldg(reinterpret_cast<const uint2*>(zb + a[k]));
                } else {   // the prefix ends inside these eight: the others count nothing
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        w[k] = t + k < nq ? __ldg(reinterpret_cast<const uint2*>(zb + a[k])) : make_uint2(0, 0);
                }
            };
            auto count8 = [&](int t, const uint2 (&w)[8]) {
                uint32_t x[8], y[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    x[k] = w[k].x & piv.x;
                    y[k] = w[k].y & piv.y;
                }
                if constexpr (PV) {
                    // the tasks' hits, two 16-bit sums a register, added up by
                    // halving: after two exchanges each lane holds one pair of
                    // tasks' sums over four lanes, after three more over all
                    // (redux takes 9 cycles of the SM each: 4 of them for the
                    // eight tasks were a quarter of the kernel's time)
                    unsigned r[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        r[k] = (unsigned)(__popc(x[2 * k]) + __popc(y[2 * k])) +
                               ((unsigned)(__popc(x[2 * k + 1]) + __popc(y[2 * k + 1])) << 16);
                    const bool up = lane & 16, odd = lane & 8;
                    const unsigned a0 = (up ? r[2] : r[0]) + __shfl_xor_sync(0xffffffffu, up ? r[0] : r[2], 16);
                    const unsigned a1 = (up ? r[3] : r[1]) + __shfl_xor_sync(0xffffffffu, up ? r[1] : r[3], 16);
                    unsigned v = (odd ? a1 : a0) + __shfl_xor_sync(0xffffffffu, odd ? a0 : a1, 8);
                    v += __shfl_xor_sync(0xffffffffu, v, 4);
                    v += __shfl_xor_sync(0xffffffffu, v, 2);
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                    if ((lane & 7) < 2) S.hits[t + 2 * (lane >> 3) + (lane & 1)] += (lane & 1) ? v >> 16 : v & 0xffffu;
                    add_planes(px, x);
                    add_planes(py, y);
                } else {
                    const uint32_t z[16] = {x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7],
                                            y[0], y[1], y[2], y[3], y[4], y[5], y[6], y[7]};
                    hs.add(z);
                }
            };
            // (fetching the next eight before these are counted was slower: the
            // warps of the SM hide the loads, and the copies cost issue slots)
            for (int t = 0; t < nq; t += 8) {
                uint2 w[8];
                fetch(t, w);
                count8(t, w);
            }
            if constexpr (PV) {
                uint32_t ux = px[0], uy = py[0];
#pragma unroll
                for (int k = 1; k < kPlanes; ++k) {
                    ux |= px[k];
                    uy |= py[k];
                }
                unsigned long long* acc = G.tnew + low;
                if (__reduce_max_sync(0xffffffffu, (unsigned)(__popc(ux) + __popc(uy))) <= kFlushBits) {
                    // few labels hit: bit by bit
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        uint32_t m = h ? uy : ux;
                        while (m) {
                            const int b = __ffs(m) - 1;
                            m &= m - 1;
                            unsigned c = 0;
#pragma unroll
                            for (int k = 0; k < kPlanes; ++k) c += (((h ? py[k] : px[k]) >> b) & 1u) << k;
                            atomicAdd(&acc[64 * lane + 32 * h + b], (unsigned long long)c);
                        }
                    }
                    __syncwarp();
                } else {
                    transpose_planes(px);
                    transpose_planes(py);
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        S.flush[k * kFlushStride + lane] = px[k];
                        S.flush[(8 + k) * kFlushStride + lane] = py[k];
                    }
                    __syncwarp();
                    // word s of the zone: lane l takes bit l, counted by lane s / 2
                    const unsigned char* bytes = reinterpret_cast<const unsigned char*>(S.flush) +
                                                 (lane & 7) * kFlushStride * 4 + (lane >> 3);
#pragma unroll 16
                    for (int s = 0; s < kZoneWords; ++s) {
                        const unsigned h = bytes[(s & 1) * 8 * kFlushStride * 4 + (s >> 1) * 4];
                        if (h) atomicAdd(&acc[s * 32 + lane], (unsigned long long)h);
                    }
                }
            }
        }
        if constexpr (PV) {
            __syncwarp();
            uint64_t mine = 0;
            for (int t = lane; t < ntask; t += 32) {
                const unsigned h = S.hits[t];
                if (h) {
                    const uint32_t i = G.zowner[S.task[t] / (uint32_t)(4 * kZoneWords)];
                    if (tlow) atomicAdd(&tlow[i], h);
                    else atomicAdd(&G.tnew[i], (unsigned long long)h);
                    mine += h;
                }
            }
            total += mine;
            mine = zsum(mine);
            if (lane == 0 && mine) atomicAdd(&G.tnew[U.j], (unsigned long long)mine);
        }
    }
    if (!PV) total += hs.take();
    total = zsum(total);
    if (lane == 0 && total) atomicAdd(target, (unsigned long long)total);
}

// zrow and the blocks of every row of a graph whose rows are sorted
template <class OffT>
__global__ void __launch_bounds__(256) k_zone_rows(const OffT* __restrict__ off, const int32_t* __restrict__ adj,
                                                   int64_t n, uint2* __restrict__ zrow, uint32_t* zbits,
                                                   uint32_t* zowner, int64_t cap, unsigned* nblocks) {
    __shared__ __align__(8) uint32_t buf[8][kZoneWords];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // 32 neighbouring rows a warp at a time, fewer where that leaves warps
    // without: a dense graph has few rows, all of them long (K_8000: 5.8 ms with
    // 32 a warp, 0.25)
    const int64_t warps = (int64_t)gridDim.x * 8;
    int per = 32;
    while (per > 1 && n < 2 * per * warps) per >>= 1;
    for (int64_t r0 = ((int64_t)blockIdx.x * 8 + w) * per; r0 < n; r0 += warps * per) {
        const int64_t r = r0 + lane;
        int64_t rb = 0;
        int d = 0;
        if (lane < per && r < n) {
            rb = (int64_t)off[r];
            d = (int)((int64_t)off[r + 1] - rb);
            zrow[r] = make_uint2(0, 0);
        }
        __syncwarp();
        unsigned on = __ballot_sync(0xffffffffu, d > kZoneMinRow);
        while (on) {
            const int o = __ffs(on) - 1;
            on &= on - 1;
            zone_row(adj, __shfl_sync(0xffffffffu, rb, o), __shfl_sync(0xffffffffu, d, o), r0 + o, n, zrow, zbits,
                     zowner, cap, nblocks, buf[w]);
        }
    }
}

// the tasks' tails whole again (a graph that leaves the device)
template <class OffT>
__global__ void k_zone_restore(const OffT* __restrict__ off, Task* __restrict__ tasks, int64_t count) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count;
         t += (int64_t)gridDim.x * blockDim.x) {
        tasks[t].len = (int32_t)((int64_t)off[tasks[t].i + 1] - (int64_t)tasks[t].start);
        tasks[t].zone = 0;
    }
}

}  // namespace

void zone_rows(const tc_graph* g, unsigned* nblocks, cudaStream_t st) {
    Prof prof_("k_zone_rows", st);
    const unsigned blocks = (unsigned)(num_sms() * 8);
    if (g->off64)
        k_zone_rows<int64_t><<<blocks, 256, 0, st>>>(static_cast<const int64_t*>(g->off), g->adj, g->n, g->zrow,
                                                     g->zbits, g->zowner, g->zcap, nblocks);
    else
        k_zone_rows<int32_t><<<blocks, 256, 0, st>>>(static_cast<const int32_t*>(g->off), g->adj, g->n, g->zrow,
                                                     g->zbits, g->zowner, g->zcap, nblocks);
    TC_LAUNCH_CHECK();
}

void zone_restore(const tc_graph* g, cudaStream_t st) {
    if (g->zcap == 0 || g->n_tasks == 0) return;
    const unsigned blocks = grid_for(g->n_tasks, 256, (int64_t)num_sms() * 8);
    if (g->off64)
        k_zone_restore<int64_t><<<blocks, 256, 0, st>>>(static_cast<const int64_t*>(g->off), g->tasks, g->n_tasks);
    else
        k_zone_restore<int32_t><<<blocks, 256, 0, st>>>(static_cast<const int32_t*>(g->off), g->tasks, g->n_tasks);
    TC_LAUNCH_CHECK();
}

void launch_zone(const GraphView* views_dev, const UnitLists& L, bool pv, unsigned long long* ctr, cudaStream_t st,
                 unsigned* tlow, bool profile) {
    if (L.nzone == 0 || !L.zones) return;
    const unsigned blocks =
        (unsigned)std::min<int64_t>((L.nzone + kZW - 1) / kZW, (int64_t)num_sms() * (pv ? 3 : 4));
    auto go = [&]() {
        if (pv) k_zone<true><<<blocks, kZT, 0, st>>>(views_dev, L.zone, L.nzone, tlow, ctr);
        else k_zone<false><<<blocks, kZT, 0, st>>>(views_dev, L.zone, L.nzone, tlow, ctr);
    };
    if (profile) {
        Prof prof_("k_zone", st);
        go();
    } else {
        go();
    }
    TC_LAUNCH_CHECK();
}

}  // namespace tc
