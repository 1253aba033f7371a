// Stable LSD radix sort of 64-bit keys on a bit range, 8-bit digits.
//
// One kernel first counts every digit position of every key (LSD passes only
// permute keys, so all passes' global digit counts are known up front).  Then
// each pass is one kernel: a tile of kTile keys, taken in launch order from a
// tile counter, is ranked stably in registers (warp w owns a contiguous
// segment; the lanes holding the same digit are found with one ballot per
// digit bit, and a running per-warp counter orders the rounds);
// the tile publishes its digit counts and finds, per digit, how many keys
// earlier tiles hold by looking back over their published counts (decoupled
// look-back: a tile that has its inclusive prefix publishes it, so the walk
// stops there); it then permutes its keys into digit order in shared memory
// and writes each digit run out contiguously.  Look-back waits are bounded:
// past the bound the pass records an error and the sort reports TC_ETIMEOUT.
#include "common.cuh"

namespace tc {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
#ifndef TC_SWEEP_ITEMS
#define TC_SWEEP_ITEMS 26
#endif
constexpr int kItems = TC_SWEEP_ITEMS;     // keys per thread
constexpr int kTile = kThreads * kItems;   // 6656 keys per tile
constexpr int kSeg = kTile / kWarps;       // 832 keys per warp segment
static_assert(kItems % 2 == 0 && kTile < 65536, "ranks two to a register, places in 16 bits");
static_assert(kSeg == 32 * kItems, "a warp's segment is one key a lane and register");
constexpr int kRadix = 256;

__device__ __forceinline__ unsigned digit_of(uint64_t k, int shift, unsigned mask) {
    return (unsigned)(k >> shift) & mask;
}

constexpr int kMaxPasses = 8;
constexpr unsigned long long kFlagAgg = 1ull << 62;
constexpr unsigned long long kFlagPre = 2ull << 62;
constexpr unsigned long long kValMask = (1ull << 62) - 1ull;
constexpr long kSpinLimit = 1l << 24;
#ifndef TC_LOOK
#define TC_LOOK 4
#endif
constexpr int kLook = TC_LOOK;

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Waits until the status word *q carries a flag (top two bits), at most
// `limit` polls; true with the word in v, false when the bound ran out.
__device__ __forceinline__ bool wait_published(const unsigned long long* q, unsigned long long& v,
                                               long limit) {
    v = ld_relaxed(q);
    long spins = 0;
    while ((v >> 62) == 0) {
        if (++spins > limit) return false;
        __nanosleep(32);
        v = ld_relaxed(q);
    }
    return true;
}

// One warp waits, bounded, on a word nothing publishes: the look-back's wait
// running out, error bit 4 set, the kernel returning.
__global__ void k_wait_selftest(const unsigned long long* word, long limit, int* err) {
    unsigned long long v;
    if (!wait_published(word, v, limit) && threadIdx.x == 0) atomicOr(err, 4);
}

// Global digit counts of every pass: hist[pass][digit], bits [lo, hi).  An
// atomic in shared memory per key and digit, of the constant 1 (a variable
// count takes a slower form: 3.3 times the kernel's time); kHistKeys keys'
// loads in flight a thread.  A ballot and a shuffle a digit, to count lanes
// that agree with the first as one, took 2.7 times as long on the keys of
// graphs, so only a warp of equal keys is counted at once.
constexpr int kHistKeys = 4;
__global__ void __launch_bounds__(kThreads) k_digit_hist(const uint64_t* __restrict__ keys,
                                                         int64_t count, int lo, int npass, int hi,
                                                         unsigned long long* __restrict__ hist) {
    __shared__ unsigned h[kMaxPasses][kRadix];
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < kMaxPasses * kRadix; i += kThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    const uint64_t top = hi < 64 ? (1ull << hi) - 1ull : ~0ull;
    for (int64_t base = blockIdx.x * (int64_t)kThreads; base < count; base += kHistKeys * stride) {
        uint64_t k[kHistKeys];
        bool valid[kHistKeys], equal[kHistKeys];
#pragma unroll
        for (int u = 0; u < kHistKeys; ++u) {
            const int64_t idx = base + u * stride + threadIdx.x;
            valid[u] = idx < count;
            k[u] = idx < count ? (keys[idx] & top) >> lo : 0;
        }
#pragma unroll
        for (int u = 0; u < kHistKeys; ++u) {
            const uint64_t k0 = __shfl_sync(0xffffffffu, k[u], 0);
            equal[u] = __all_sync(0xffffffffu, valid[u] && k[u] == k0);
        }
        for (int p = 0; p < npass; ++p) {
#pragma unroll
            for (int u = 0; u < kHistKeys; ++u) {
                const unsigned d = (unsigned)k[u] & 255u;
                if (equal[u]) {
                    if (lane == 0) atomicAdd(&h[p][d], 32u);
                } else if (valid[u]) {
                    atomicAdd(&h[p][d], 1u);
                }
                k[u] >>= 8;
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < npass * kRadix; i += kThreads) {
        const unsigned c = (&h[0][0])[i];
        if (c) atomicAdd(&hist[i], (unsigned long long)c);
    }
}

// hist[pass][digit] -> exclusive prefix over digits, per pass: one block of
// kRadix threads per pass, a thread per digit.
__global__ void __launch_bounds__(kRadix) k_digit_offsets(unsigned long long* __restrict__ hist, int npass) {
    __shared__ unsigned long long wsum[kRadix / 32];
    const int p = blockIdx.x;
    if (p >= npass) return;
    unsigned long long* h = hist + (size_t)p * kRadix;
    const int d = threadIdx.x, lane = d & 31, w = d >> 5;
    const unsigned long long c = h[d];
    unsigned long long inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    unsigned long long before = 0;
    for (int q = 0; q < w; ++q) before += wsum[q];
    h[d] = before + inc - c;
}

// One pass, 8-bit digits (fewer in a last pass: the masked bits read as 0).
//
// What bounds it is instructions and the look-back: 16 B of traffic a key is
// 2.5 ms of a 2^30-key pass; staged in shared memory, ranked there and looked
// back one tile at a time the pass took 7.2 ms, 170 instructions for every 32
// keys.  So a key stays with its thread from the load to its place in the tile
// (in registers but for 116 bytes: three blocks an SM leave 80 a thread; warp w
// holds a contiguous segment, a row of 32 keys a register), its rank beside it,
// two to a register; a digit's place in the output is one 64-bit word, to which
// the key's place in the tile is added; the look-back reads kLook tiles' words
// at a time, and the keys move to their places before it starts (2^30 keys: 7.2
// -> 5.7 ms; 1, 2, 4, 8 words: 6.0, 5.9, 5.7, 5.8).  Larger tiles share out a
// tile's fixed work -- counters, scan, look-back -- further: 16, 24, 26, 28 keys
// a thread 4.9, 4.6, 4.5, 4.5 ms (the first at four blocks an SM, the others at
// three).  The last tile is filled up with keys of the highest digit, which end
// up behind its own and are not written.
#ifndef TC_SWEEP_MINB
#define TC_SWEEP_MINB 3
#endif
__global__ void __launch_bounds__(kThreads, TC_SWEEP_MINB) k_onesweep(const uint64_t* __restrict__ in,
                                                                      uint64_t* __restrict__ out, int64_t count,
                                                                      int shift, int nbits,
                                                                      const unsigned long long* __restrict__ goff,
                                                                      unsigned long long* status,
                                                                      unsigned* tile_ctr, int* err) {
    __shared__ uint64_t stage[kTile];
    __shared__ unsigned short wcnt[kWarps][kRadix];
    __shared__ unsigned wsum[kWarps];
    __shared__ unsigned long long s_out[kRadix];
    __shared__ int s_tile;
    if (threadIdx.x == 0) s_tile = (int)atomicAdd(tile_ctr, 1u);
    for (int i = threadIdx.x; i < kWarps * kRadix / 2; i += kThreads) reinterpret_cast<unsigned*>(&wcnt[0][0])[i] = 0;
    __syncthreads();
    const int tile = s_tile;
    const int valid_in_tile = (int)min64((int64_t)kTile, count - (int64_t)tile * kTile);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const unsigned mask = (1u << nbits) - 1u;
    const int seg = w * kSeg + lane;
    const uint64_t* __restrict__ mine = in + (int64_t)tile * kTile + seg;
    uint64_t key[kItems];
    unsigned rank[kItems / 2];
#pragma unroll
    for (int r = 0; r < kItems; ++r) key[r] = seg + r * 32 < valid_in_tile ? mine[r * 32] : ~0ull;
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        const unsigned d = digit_of(key[r], shift, mask);
        unsigned peers = 0xffffffffu;   // the lanes with this digit, a ballot a bit
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const bool bit = (d >> b) & 1u;
            const unsigned bal = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? bal : ~bal;
        }
        const unsigned below = peers & lt, prior = wcnt[w][d];
        const unsigned x = prior + __popc(below);
        rank[r / 2] = (r & 1) ? rank[r / 2] | x << 16 : x;
        __syncwarp();
        if (below == 0) wcnt[w][d] = (unsigned short)(prior + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    // digit d = threadIdx.x: the warps' keys before each other's, the tile's
    // count, published; then the keys of digit d in earlier tiles
    unsigned tot = 0;
    {
        const int d = threadIdx.x;
        unsigned c[kWarps];
#pragma unroll
        for (int q = 0; q < kWarps; ++q) c[q] = wcnt[q][d];
#pragma unroll
        for (int q = 0; q < kWarps; ++q) tot += c[q];
        unsigned long long* my = status + (size_t)tile * kRadix + d;
        st_relaxed(my, (tile == 0 ? kFlagPre : kFlagAgg) | (unsigned long long)tot);
        // start of the digit in the tile, and of each warp's share of it
        unsigned inc = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) wsum[w] = inc;
        __syncthreads();
        unsigned start = inc - tot;
#pragma unroll
        for (int q = 0; q < kWarps; ++q)
            if (q < w) start += wsum[q];
        unsigned run = start;
#pragma unroll
        for (int q = 0; q < kWarps; ++q) {
            wcnt[q][d] = (unsigned short)run;
            run += c[q];
        }
        __syncthreads();
        // the keys move to their places in the tile while the look-back's
        // first status words are on their way
        unsigned long long excl = 0;
#pragma unroll
        for (int r = 0; r < kItems; ++r)
            stage[wcnt[w][digit_of(key[r], shift, mask)] + ((r & 1) ? rank[r / 2] >> 16 : rank[r / 2] & 0xffffu)] =
                key[r];
        if (tile > 0) {
            // kLook status words at a time: each costs a trip to L2
            bool more = true;
            for (int p = tile - 1; more && p >= 0; p -= kLook) {
                unsigned long long v[kLook];
#pragma unroll
                for (int k = 0; k < kLook; ++k)
                    v[k] = p - k >= 0 ? ld_relaxed(status + (size_t)(p - k) * kRadix + d) : kFlagPre;
#pragma unroll
                for (int k = 0; k < kLook; ++k) {
                    if (!more) break;
                    if ((v[k] >> 62) == 0 &&
                        !wait_published(status + (size_t)(p - k) * kRadix + d, v[k], kSpinLimit)) {
                        atomicOr(err, 4);
                        more = false;
                        break;
                    }
                    excl += v[k] & kValMask;
                    more = (v[k] >> 62) != 2;
                }
            }
            st_relaxed(my, kFlagPre | (excl + tot));
        }
        s_out[d] = goff[d] + excl - start;   // place in the output of the tile's entry 0, were it of digit d
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const int p = k * kThreads + threadIdx.x;
        if (p < valid_in_tile) {
            const uint64_t kk = stage[p];
            out[s_out[digit_of(kk, shift, mask)] + (unsigned)p] = kk;
        }
    }
}

}  // namespace

void radix_sort_u64(uint64_t** keys, uint64_t** alt, int64_t count, int lo, int hi, Alloc& al,
                    cudaStream_t st, int* err_dev) {
    if (count <= 1 || hi <= lo) return;
    const int64_t ntiles = (count + kTile - 1) / kTile;
    const int npass = (hi - lo + 7) / 8;
    // [hist: kMaxPasses x 256 u64][tile counters: kMaxPasses u32][error flag]
    Buf<unsigned long long> hist(al, (size_t)kMaxPasses * kRadix + 8);
    Buf<unsigned long long> status(al, (size_t)ntiles * kRadix);
    unsigned* ctrs = reinterpret_cast<unsigned*>(hist.get() + (size_t)kMaxPasses * kRadix);
    int* err = err_dev ? err_dev : reinterpret_cast<int*>(ctrs + kMaxPasses);
    TC_CUDA(cudaMemsetAsync(hist.get(), 0, sizeof(unsigned long long) * ((size_t)kMaxPasses * kRadix + 8), st));
    {
        Prof prof_("k_digit_hist", st);
        k_digit_hist<<<grid_for(count, kThreads, (int64_t)num_sms() * 8), kThreads, 0, st>>>(
            *keys, count, lo, npass, hi, hist.get());
    }
    TC_LAUNCH_CHECK();
    {
        Prof prof_("k_digit_offsets", st);
        k_digit_offsets<<<npass, kRadix, 0, st>>>(hist.get(), npass);
    }
    TC_LAUNCH_CHECK();
    for (int p = 0; p < npass; ++p) {
        const int shift = lo + 8 * p;
        const int nbits = min(8, hi - shift);
        TC_CUDA(cudaMemsetAsync(status.get(), 0, sizeof(unsigned long long) * (size_t)ntiles * kRadix, st));
        {
            Prof prof_("k_onesweep", st);
            k_onesweep<<<(unsigned)ntiles, kThreads, 0, st>>>(*keys, *alt, count, shift, nbits,
                                                              hist.get() + (size_t)p * kRadix,
                                                              status.get(), ctrs + p, err);
        }
        TC_LAUNCH_CHECK();
        uint64_t* t = *keys;
        *keys = *alt;
        *alt = t;
    }
    if (err_dev) return;   // the caller reads the flag at its next synchronisation
    int herr = 0;
    TC_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st));
    TC_CUDA(cudaStreamSynchronize(st));
    if (herr) TC_FAIL(TC_ETIMEOUT, "radix sort: a look-back wait ran past its bound");
}

}  // namespace tc

namespace tc {

bool selftest_wait_timeout(long limit, Alloc& al, cudaStream_t st) {
    Buf<unsigned long long> w(al, 2);   // [0] the word nothing publishes, [1] error flag
    TC_CUDA(cudaMemsetAsync(w.get(), 0, 2 * sizeof(unsigned long long), st));
    k_wait_selftest<<<1, 32, 0, st>>>(w.get(), limit, reinterpret_cast<int*>(w.get() + 1));
    TC_LAUNCH_CHECK();
    int err = 0;
    TC_CUDA(cudaMemcpyAsync(&err, w.get() + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
    TC_CUDA(cudaStreamSynchronize(st));
    return (err & 4) != 0;
}

}  // namespace tc
