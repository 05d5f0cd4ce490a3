// Critical value lambda(alpha, h, N/n) of the boundary (Eq. 4) by simulation.
//
// The paper obtains lambda "by simulation" of the limiting MOSUM process
// (Section 2.3; the one printed value, 2.39, is for alpha = 0.05, h/n = 0.5,
// N/n = 2 in Section 4.3).  Here every warp simulates one path: a Brownian
// motion W on a grid of G steps per unit time up to T = N/n, Gaussian
// increments of variance 1/G, and the statistic
//     sup_{t in [1, T]} |W(t) - W(t - h) - h W(1)| / sqrt(log+ t)
// over the grid points t = i/G, i = G..T*G.  lambda is the (1 - alpha)
// empirical quantile over the paths.
//
// Random numbers: per path a SplitMix64 stream (Steele, Lea and Flood, 2014)
// started from (seed, path), two 53-bit uniforms per normal, Box-Muller
// (sqrt(-2 ln u1) cos(2 pi u2), u1 in (0, 1]).  The stream advances by a
// fixed increment per draw, so any step's normal can be drawn on its own.
//
// What bounds it: the normals.  In FP64 (one thread per path, the lagged
// W(t - h) rebuilt by a second pass over the stream) 1e5 paths of 1816 steps
// took 52.6 ms, nearly all of it FP64 issue.  Here the normals come from
// lambda_fixed.cuh (integer arithmetic) and W is a 64-bit fixed-point word with steps of
// 2^-frac (2^-56 at T = 1.8; a double is finer only for |W| below a sixteenth), which
// sums without further rounding: against 113-bit arithmetic,
// over 150 such paths, the statistic is off by 7.2e-17 on average and 2.2e-16 at
// most; in FP64 by 6.6e-16 and 4.8e-15.  Fixed-point sums do not
// depend on their order, so a warp takes one path, 64 steps at a time: every lane
// draws two, a prefix sum over the warp gives W, and the last h G of them
// stay in a shared-memory ring for W(t - h): 3.5 ms, bound by the integer
// pipe (4.3 before the quantile was taken on the device, the logarithm's sum kept in one
// word and the additions of the 64-bit products folded into the multiplies).
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "bfm_internal.cuh"
#include "lambda_fixed.cuh"

namespace bfm {
namespace {

using fixedpt::Count;

constexpr uint64_t kGolden = 0x9E3779B97F4A7C15ull;  // SplitMix64 increment
constexpr int kWarps = 4;                             // paths at a time per block
constexpr int kPer = 2;                               // consecutive steps of a lane
constexpr int kSteps = 32 * kPer;                     // steps of a warp at a time
constexpr double kE = 2.718281828459045235360287;
constexpr size_t kMaxRingBytes = 200 * 1024;          // rings of a block
// Up to here two blocks share an SM (228 KB, 4 KB of each for the tables and the system).
// Beyond, four warps an SM wait on one another's draws, and drawing the lagged steps again at
// full occupancy is the faster: 20000 paths, h = 1, T = 1.8, ring against second draw: G = 2000
// 1.67 and 2.07 ms, 3000 2.77 and 2.96, 4000 5.51 and 3.84, 6000 8.12 and 5.61.  With no
// more paths than one block per SM takes, the ring stays ahead (200 paths, G = 6000:
// 457 and 578 us).
constexpr size_t kTwoRingBytes = 110 * 1024;

struct LambdaParams {
    int G, nsteps, ih, reps;
    int ie;                // last step with log+ (i / G) = 1
    int ring;              // ring slots per warp (a multiple of kSteps, >= ih + kSteps), 0: no ring
    int frac;              // fraction bits of W
    uint64_t seed, sd, h;  // sd: sqrt(2 / G) 2^63; h times 2^64 (h = 1 as 0)
    double* stats;
};

__device__ __forceinline__ uint64_t splitmix_mix(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// The increment of W (2^-frac steps) whose two draws follow the stream state s.
__device__ __forceinline__ int64_t increment(uint64_t s, const LambdaParams& P, const uint64_t* ln, const uint32_t* rec) {
    const uint64_t n = (splitmix_mix(s + kGolden) >> 11) + 1, f = splitmix_mix(s + 2 * kGolden) >> 11;
    bool neg;
    const uint64_t z = fixedpt::normal_q59(n, f, ln, rec, neg);     // 2^59 |z| / sqrt(2), |z| <= 8.6
    const uint64_t q = fixedpt::mulhi(z, P.sd);                     // 2^58 |z| / sqrt(G); sd < 1.5 2^63, z < 2^62
    const int sh = 58 - P.frac;                                     // >= 2
    const int64_t d = (int64_t)((q + (1ull << (sh - 1))) >> sh);
    return neg ? -d : d;
}

__device__ __forceinline__ int64_t warp_scan(int64_t v, int lane) {  // inclusive sums over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t t = __shfl_up_sync(~0u, v, o);
        v += lane >= o ? t : 0;
    }
    return v;
}

// The k-th smallest (from 0) of n values >= 0 into v[n]: their bits order as the values
// do, and one block fixes eleven of them at a time from the top, counting the values
// that share the bits fixed so far, until one value is left.  A host nth_element took
// 0.9 ms for 1e5 values.  Short calls are the sum of the steps' latencies: the counts
// of a lane are summed without bank conflicts and the digit is found by all lanes of a
// warp.  A call of ten paths of two steps: 215 us with one lane's search and all six
// rounds, 195 so (and 197 with the quantile on the host); 1e6 paths 2.03 and 1.95 ms.
constexpr int kSelThreads = 1024, kSelBits = 11;
__global__ void __launch_bounds__(kSelThreads) kth_smallest(double* v, int n, int k) {
    constexpr int kEach = (1 << kSelBits) / 32;  // counts of a lane
    __shared__ int hist[1 << kSelBits];
    __shared__ int s_digit, s_below, s_count;
    auto bits = [&](Count i) { return (uint64_t)__double_as_longlong(v[i]); };
    uint64_t prefix = 0;
    for (int top = 64; top > 0; top -= kSelBits) {
        const int shift = top > kSelBits ? top - kSelBits : 0, width = top - shift;
        for (int i = threadIdx.x; i < (1 << kSelBits); i += kSelThreads) hist[i] = 0;
        __syncthreads();
#pragma unroll 4
        for (Count i = threadIdx.x; i < (Count)n; i += kSelThreads) {
            const uint64_t u = bits(i);
            if (top == 64 || (u >> top) == (prefix >> top)) atomicAdd(&hist[(int)((u >> shift) & ((1u << width) - 1u))], 1);
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
            int sum = 0;
#pragma unroll 8
            for (int i = 0; i < kEach; ++i) sum += hist[lane * kEach + ((i + lane) & (kEach - 1))];
            int below = 0;  // values in the lanes before, then in the owner's digits before
            auto scan = [&](int x) {  // sums over the lanes up to this one
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(~0u, x, o);
                    x += lane >= o ? t : 0;
                }
                return x;
            };
            below = scan(sum) - sum;
            const int owner = __ffs(__ballot_sync(~0u, k >= below && k < below + sum)) - 1;
            below = __shfl_sync(~0u, below, owner);
            // the owner's 64 digits, two a lane
            const int d = owner * kEach + 2 * lane, c0 = hist[d], c1 = hist[d + 1];
            const int b0 = below + scan(c0 + c1) - (c0 + c1), b1 = b0 + c0;
            if (k >= b0 && k < b1 + c1) {
                const bool up = k >= b1;
                s_digit = up ? d + 1 : d;
                s_below = up ? b1 : b0;
                s_count = up ? c1 : c0;
            }
        }
        __syncthreads();
        prefix |= (uint64_t)s_digit << shift;
        k -= s_below;
        if (s_count == 1) {  // the value with this prefix
#pragma unroll 4
            for (Count i = threadIdx.x; i < (Count)n; i += kSelThreads)
                if ((bits(i) >> shift) == (prefix >> shift)) v[n] = v[i];
            return;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) v[n] = __longlong_as_double((long long)prefix);
}

// One path per warp.  kRing: W(t - h) from the ring; otherwise (h G too long for two
// blocks per SM) rebuilt from the stream by a second draw of the lagged steps.
template <bool kRing>
__global__ void __launch_bounds__(32 * kWarps)
    lambda_paths(const __grid_constant__ fixedpt::LogTable tab, const LambdaParams P) {
    __shared__ uint64_t s_ln[256];
    __shared__ uint32_t s_rec[256];
    extern __shared__ __align__(16) int64_t s_ring[];
    for (int i = threadIdx.x; i < 256; i += 32 * kWarps) {
        s_ln[i] = tab.ln[i];
        s_rec[i] = fixedpt::log_recip((uint32_t)i);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t* ring = s_ring + warp * P.ring;
    const double unit = ldexp(1.0, -P.frac);
    for (int64_t r = (int64_t)blockIdx.x * kWarps + warp; r < P.reps; r += (int64_t)gridDim.x * kWarps) {
        // stream of path r (one discarded draw after seeding); step i uses draws 2i - 1 and 2i
        const uint64_t s0 = P.seed * 0xA0761D6478BD642Full + (uint64_t)r * 0xE7037ED1A0B428DBull + 1ull + kGolden;
        uint64_t st = s0 + 2 * kPer * kGolden * (uint64_t)lane;
        int64_t base = 0, hw1 = 0;  // W before the block of steps, h W(1)
        int64_t lbase = 0;          // !kRing: W(t - h) before the block
        uint64_t best = 0;
        int pos = 0;                // ring slot of the block's first step
        if (kRing) {
            __syncwarp();  // the previous path's reads
            if (lane == 0) ring[P.ring - 1] = 0;  // W(0), the slot before step 1
        }
        for (Count i0 = 1; i0 <= (Count)P.nsteps; i0 += kSteps) {
            const Count i = i0 + kPer * lane;  // this lane's steps i, i + 1
            int64_t W[kPer];
            {
                const int64_t d0 = increment(st, P, s_ln, s_rec), d1 = increment(st + 2 * kGolden, P, s_ln, s_rec);
                W[1] = base + warp_scan(d0 + d1, lane);
                W[0] = W[1] - d1;
            }
            st += 2 * kSteps * kGolden;
            base = __shfl_sync(~0u, W[1], 31);
            int64_t lag[kPer] = {0, 0};
            if (kRing) {
                *reinterpret_cast<longlong2*>(ring + pos + kPer * lane) = make_longlong2(W[0], W[1]);
                __syncwarp();
#pragma unroll
                for (int u = 0; u < kPer; ++u) {
                    int s = pos + kPer * lane + u - P.ih;
                    s += s < 0 ? P.ring : 0;
                    lag[u] = ring[s];  // steps before the ring's first lap are not used (i < G)
                }
                pos += kSteps;
                pos = pos == P.ring ? 0 : pos;
                __syncwarp();
            } else if (i0 + kSteps - 1 > (Count)P.ih) {
                int64_t d[kPer];  // the lagged steps
#pragma unroll
                for (int u = 0; u < kPer; ++u) {
                    const int j = (int)(i + u - (Count)P.ih);
                    d[u] = j >= 1 ? increment(s0 + 2 * kGolden * (uint64_t)(j - 1), P, s_ln, s_rec) : 0;
                }
                lag[1] = lbase + warp_scan(d[0] + d[1], lane);
                lag[0] = lag[1] - d[1];
                lbase = __shfl_sync(~0u, lag[1], 31);
            }
            if (i0 + kSteps - 1 >= (Count)P.G) {
                if (i0 <= (Count)P.G) {  // W(1) is in this block
                    const int at = (int)((Count)P.G - i0);
                    const int64_t w1 = __shfl_sync(~0u, (at & 1) ? W[1] : W[0], at >> 1);
                    const uint64_t a = (uint64_t)(w1 < 0 ? -w1 : w1), ha = P.h ? __umul64hi(a, P.h) : a;
                    hw1 = w1 < 0 ? -(int64_t)ha : (int64_t)ha;
                }
#pragma unroll
                for (int u = 0; u < kPer; ++u)
                    if (i + u >= (Count)P.G && i + u <= (Count)P.nsteps) {
                        const int64_t z = W[u] - lag[u] - hw1;
                        uint64_t v = (uint64_t)(z < 0 ? -z : z);
                        if (v > best) {  // the boundary's factor, at least 1, only lowers it
                            if (i + u > (Count)P.ie) v = (uint64_t)((double)v / sqrt(log((double)(i + u) / (double)P.G)));
                            best = v > best ? v : best;
                        }
                    }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const uint64_t t = __shfl_xor_sync(~0u, best, o);
            best = t > best ? t : best;
        }
        if (lane == 0) P.stats[r] = (double)best * unit;
    }
}

const fixedpt::LogTable& log_table() {
    static fixedpt::LogTable t;
    static std::once_flag once;
    std::call_once(once, [] {
        for (uint32_t i = 0; i < 256; ++i) t.ln[i] = fixedpt::log_entry(i);
    });
    return t;
}

template <bool kRing>
cudaError_t launch_paths(const LambdaParams& P, size_t smem, int sms, cudaStream_t st) {
    auto* fn = lambda_paths<kRing>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxRingBytes);
    int per = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, 32 * kWarps, smem);
    if (e != cudaSuccess) return e;
    const int64_t want = ((int64_t)P.reps + kWarps - 1) / kWarps, most = (int64_t)sms * (per < 1 ? 1 : per);
    fn<<<(unsigned)(want < most ? want : most), 32 * kWarps, smem, st>>>(log_table(), P);
    return cudaGetLastError();
}

}  // namespace
}  // namespace bfm

using namespace bfm;

extern "C" bfm_status bfm_lambda(double alpha, double h, double T, int G, int reps, uint64_t seed,
                                 double* lambda_out, double* stats_host, void* stream) {
    if (!(alpha > 0.0 && alpha < 1.0) || !(h > 0.0 && h <= 1.0) || !(T > 1.0) || G < 1 || reps < 1 ||
        !lambda_out) {
        set_error("bfm_lambda: needs 0 < alpha < 1, 0 < h <= 1, T > 1, G >= 1, reps >= 1 and lambda_out");
        return BFM_EINVAL;
    }
    const int nsteps = (int)std::llround(T * (double)G);
    const int ih = (int)std::llround(h * (double)G);
    if (ih < 1 || nsteps < G) {
        set_error("bfm_lambda: h * G rounds to 0 or T * G to fewer than G steps");
        return BFM_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    double* d_stats = nullptr;
    cudaError_t e = cudaMallocAsync(&d_stats, sizeof(double) * ((size_t)reps + 1), st);
    if (e != cudaSuccess) return cuda_fail(e, "bfm_lambda: cudaMallocAsync");
    LambdaParams P{};
    P.G = G;
    P.nsteps = nsteps;
    P.ih = ih;
    P.reps = reps;
    P.ie = (int)std::min<double>(std::floor(kE * (double)G), 2147483647.0);
    while ((double)P.ie / (double)G > kE) --P.ie;
    while (P.ie < nsteps && (double)(P.ie + 1) / (double)G <= kE) ++P.ie;
    // |W| stays below 13 sqrt(T) (13 standard deviations) and |W - Wlag - h W(1)| below
    // three times that: the integer part holds 40 sqrt(T)
    P.frac = 62 - (int)std::ceil(std::log2(40.0 * std::sqrt(T)));
    P.seed = seed;
    P.sd = (uint64_t)std::ldexp(std::sqrt(2.0 / (double)G), 63);
    P.h = h < 1.0 ? (uint64_t)std::ldexp(h, 64) : 0ull;
    P.stats = d_stats;
    const int64_t slots = ((int64_t)ih + 2 * kSteps - 1) / kSteps * kSteps;
    int dev = 0, sms = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) {
        cudaFreeAsync(d_stats, st);
        return cuda_fail(e, "bfm_lambda: device attributes");
    }
    const bool ring = (size_t)slots * kWarps * 8 <= (reps <= kWarps * sms ? kMaxRingBytes : kTwoRingBytes);
    P.ring = ring ? (int)slots : 0;
    e = ring ? launch_paths<true>(P, (size_t)slots * kWarps * 8, sms, st) : launch_paths<false>(P, 0, sms, st);
    // (1 - alpha) empirical quantile: the ceil((1 - alpha) reps)-th smallest
    long q = (long)std::ceil((1.0 - alpha) * (double)reps) - 1;
    q = q < 0 ? 0 : (q >= reps ? reps - 1 : q);
    if (e == cudaSuccess) {
        kth_smallest<<<1, kSelThreads, 0, st>>>(d_stats, reps, (int)q);
        e = cudaGetLastError();
    }
    double lambda = 0.0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&lambda, d_stats + reps, sizeof lambda, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && stats_host)
        e = cudaMemcpyAsync(stats_host, d_stats, sizeof(double) * (size_t)reps, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaFreeAsync(d_stats, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "bfm_lambda: simulation");
    *lambda_out = lambda;
    return BFM_OK;
}
