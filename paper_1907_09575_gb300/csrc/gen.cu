// Device RMAT input generator (synthetic inputs only; not the counting method).
//
// An independent implementation of the integer RMAT stream defined by the
// host generator: counter-based splitmix64 draws (Steele, Lea and Flood,
// OOPSLA 2014), one 32-bit half per recursion level against the cumulative
// a, a+b, a+b+c thresholds, a seeded bijective scramble x -> ((x*A mod 2^s)
// xor B) * C mod 2^s, and rejection of ids >= n (64 attempts, then the
// self-loop (0,0)).  Equal output for equal (seed, scale, n, pair index).
#include <algorithm>

#include "common.cuh"
#include "tc_internal.cuh"

namespace tc {
namespace {

constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;
constexpr uint64_t kTagPairs = 0x524D4154ull;  // "RMAT"
constexpr uint64_t kTagScramble = 0x5343524Dull;  // "SCRM"
constexpr int kAttempts = 64;

__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__host__ __device__ __forceinline__ uint64_t draw(uint64_t key, uint64_t ctr) {
    return mix64(key + (ctr + 1ull) * kGamma);
}

// One attempt at pair e: the two scrambled ids (below 2^scale <= 2^31, so all
// but the draws is 32-bit arithmetic); false when one of them is >= n.
struct RmatShape {
    uint64_t key;
    uint32_t A, B, C, n, t1, t2, t3;
    int scale;
};

__device__ __forceinline__ bool rmat_attempt(const RmatShape& J, uint64_t e, int attempt, uint32_t& u, uint32_t& v) {
    const uint32_t mask = (1u << J.scale) - 1u;
    uint64_t z = J.key + ((e * kAttempts + (uint64_t)attempt) * (uint64_t)((J.scale + 1) / 2) + 1ull) * kGamma;
    u = v = 0;
    for (int l = 0; l < J.scale; l += 2) {
        const uint64_t h = mix64(z);
        z += kGamma;
        const uint32_t r0 = (uint32_t)h, r1 = (uint32_t)(h >> 32);
        u = 2 * u + (r0 >= J.t2);
        v = 2 * v + ((r0 >= J.t1 && r0 < J.t2) || r0 >= J.t3);
        if (l + 1 < J.scale) {
            u = 2 * u + (r1 >= J.t2);
            v = 2 * v + ((r1 >= J.t1 && r1 < J.t2) || r1 >= J.t3);
        }
    }
    u = ((((u * J.A) & mask) ^ J.B) * J.C) & mask;
    v = ((((v * J.A) & mask) ^ J.B) * J.C) & mask;
    return u < J.n && v < J.n;
}

__global__ void k_rmat(RmatShape J, int64_t e0, int64_t count, int32_t* __restrict__ src, int32_t* __restrict__ dst) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t u = 0, v = 0;
        int a = 0;
        while (a < kAttempts && !rmat_attempt(J, (uint64_t)(e0 + i), a, u, v)) ++a;
        src[i] = a < kAttempts ? (int32_t)u : 0;
        dst[i] = a < kAttempts ? (int32_t)v : 0;
    }
}

// Many RMAT requests at once: pair x of the concatenation belongs to the
// request r with ppre[r] <= x < ppre[r+1]; its ids are offset by vpre[r].
//
// Bound by the draws' arithmetic.  A request's n is rarely a power of two, so
// an attempt succeeds about six times in ten, and 32 lanes that wait for the
// last of them make four to five attempts a pair.  So a warp owns a stretch of
// pairs and a lane whose pair is done takes the stretch's next one.
__global__ void __launch_bounds__(256) k_rmat_multi(const RmatJob* __restrict__ jobs,
                                                    const int64_t* __restrict__ ppre, int nreq, int64_t total,
                                                    int64_t stretch, int32_t* __restrict__ src,
                                                    int32_t* __restrict__ dst) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t next = warp * stretch;
    const int64_t end = min64(next + stretch, total);
    int64_t x = 0, first = 0, last = 0;   // the lane's pair; its request's pairs [first, last)
    int64_t vbase = 0;
    RmatShape J{};
    bool busy = false;
    int attempt = 0;
    while (true) {
        const unsigned idle = __ballot_sync(0xffffffffu, !busy);
        if (!busy) {
            x = next + __popc(idle & ((1u << lane) - 1u));
            busy = x < end;
            attempt = 0;
            if (busy && (x < first || x >= last)) {
                int lo = 0, hi = nreq - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (ppre[mid] <= x) lo = mid; else hi = mid - 1;
                }
                const RmatJob& K = jobs[lo];
                J = RmatShape{K.key, (uint32_t)K.A, (uint32_t)K.B, (uint32_t)K.C, (uint32_t)K.n, K.t1, K.t2, K.t3,
                              K.scale};
                vbase = K.vbase;
                first = ppre[lo];
                last = ppre[lo + 1];
            }
        }
        next += __popc(idle);
        if (!__any_sync(0xffffffffu, busy)) break;
        if (busy) {
            uint32_t u, v;
            const bool ok = rmat_attempt(J, (uint64_t)(x - first), attempt, u, v);
            if (ok || ++attempt == kAttempts) {
                src[x] = (int32_t)(vbase + (ok ? u : 0u));
                dst[x] = (int32_t)(vbase + (ok ? v : 0u));
                busy = false;
            }
        }
    }
}

}  // namespace

RmatJob make_rmat_job(uint64_t seed, int scale, int64_t n, uint32_t t1, uint32_t t2, uint32_t t3,
                      int64_t vbase) {
    RmatJob J;
    J.key = mix64(seed * kGamma + kTagPairs);
    const uint64_t ks = mix64(seed * kGamma + kTagScramble);
    const uint64_t mask = (1ull << scale) - 1ull;
    J.A = (draw(ks, 0) | 1ull) & mask;
    J.B = draw(ks, 1) & mask;
    J.C = (draw(ks, 2) | 1ull) & mask;
    J.n = n;
    J.vbase = vbase;
    J.scale = scale;
    J.t1 = t1;
    J.t2 = t2;
    J.t3 = t3;
    return J;
}

void generate_rmat_multi(const RmatJob* jobs_dev, const int64_t* ppre_dev, int nreq, int64_t total,
                         int32_t* src, int32_t* dst, cudaStream_t st) {
    if (total <= 0) return;
    {
        Prof prof_("k_rmat_multi", st);
        // as many warps as the device runs at once, a whole number of rounds each
        const int64_t warps = std::min<int64_t>((total + 31) / 32, (int64_t)num_sms() * 64);
        const int64_t stretch = (total + warps - 1) / warps;
        k_rmat_multi<<<grid_for(32 * ((total + stretch - 1) / stretch), 256), 256, 0, st>>>(
            jobs_dev, ppre_dev, nreq, total, stretch, src, dst);
    }
    TC_LAUNCH_CHECK();
}

}  // namespace tc

using namespace tc;

extern "C" tc_status tc_generate_rmat(uint64_t seed, int32_t scale, int64_t n, int64_t e0,
                                      int64_t count, uint32_t t1, uint32_t t2, uint32_t t3,
                                      int32_t* src_dev, int32_t* dst_dev, void* stream) {
    clear_error();
    if (scale < 1 || scale > 31) {
        set_error("tc_generate_rmat: scale outside [1, 31]");
        return TC_EINVAL;
    }
    if (n < 1 || n > (1ll << scale) || e0 < 0 || count < 0 || (count > 0 && (!src_dev || !dst_dev))) {
        set_error("tc_generate_rmat: bad n, e0, count or output pointer");
        return TC_EINVAL;
    }
    if (!(t1 <= t2 && t2 <= t3)) {
        set_error("tc_generate_rmat: thresholds must be non-decreasing");
        return TC_EINVAL;
    }
    if (count == 0) return TC_OK;
    const uint64_t key = mix64(seed * kGamma + kTagPairs);
    const uint64_t ks = mix64(seed * kGamma + kTagScramble);
    const uint64_t mask = (1ull << scale) - 1ull;
    const uint64_t A = (draw(ks, 0) | 1ull) & mask;
    const uint64_t B = draw(ks, 1) & mask;
    const uint64_t C = (draw(ks, 2) | 1ull) & mask;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    {
        Prof prof_("k_rmat", st);
        const RmatShape J{key, (uint32_t)A, (uint32_t)B, (uint32_t)C, (uint32_t)n, t1, t2, t3, scale};
        k_rmat<<<grid_for(count, 256, (int64_t)num_sms() * 16), 256, 0, st>>>(J, e0, count, src_dev, dst_dev);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("tc_generate_rmat: launch failed: %s", cudaGetErrorString(e));
        return TC_ECUDA;
    }
    return TC_OK;
}
