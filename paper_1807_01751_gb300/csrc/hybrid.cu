// Hybrid form of the general path (BFM_ALGO_HYBRID): one thread per pixel for
// the per-date scan, the tensor cores for every contraction over dates.
//
// A CTA owns 512 pixels (four 128-pixel M-tiles = four TMEM lane sets) and
// runs one per SM, so that one copy of the basis tables, 48 KB of stages and
// a residual ring of floor(h_frac n_hist) slots for all 512 pixels share the
// SM's shared memory.  The M-tiles work in two groups of two, each a pipeline
// of its own over work blocks of 256 pixels: eight pixel warps that own 32
// pixels each (the pixel's TMEM lane is its thread's lane), a warp that issues
// the 2-D TMA boxes of Y (128 pixels x 8 float or 16 int16 dates, one per
// M-tile and stage) and a warp that issues the tensor-core work.  Per work
// block (Section 2.1, Eq. 3-6, Algorithm 1 with missing values masked):
//
//   A   history, 16 dates per chunk: each pixel thread writes its row of the
//       chunk's A operands into TMEM -- the 0/1 validity mask as fp16 and the
//       masked y as tf32 -- and the MMA warp accumulates
//         G  += mask x [basis hi | basis lo]   (the 3 + 6k masked basis sums
//                                               of bfm::Basis, fp16, N = 32)
//         b  += y x [x hi | x lo]              (X'My, tf32, N = 16)
//       The pixel thread reads G and b, forms the Gram matrix (identities of
//       gram_from_sums), FP32 Cholesky with the rank test of the other forms,
//       beta0 = G^-1 X'My, and writes beta0 (scaled by a power of two, split
//       fp16 hi + lo) as an A operand.
//   B'  history again (from L2): yhat0 = X beta0 in TMEM pieces of 32 dates
//       (fp16 MMA, B = the regressors hi and lo read MN-major); the thread
//       forms r0 = y - yhat0 at valid dates, s0 = sum r0^2, and writes r0
//       (scaled, fp16 hi + lo) as an A operand for c += r0 x [x hi | x lo]
//       (X'M r0, the refinement step).  It also notes the date of the oldest
//       history observation of its first MOSUM window.  Then delta = G^-1 c,
//       beta = beta0 + delta, sigma-hat^2 = (s0 - delta'c) / (n_p - K)
//       (Algorithm 1 step 5), and delta is written as a further A operand.
//   C   dates from the earliest window start of the block to N: yhat = X
//       (beta0 + delta) in TMEM pieces; residuals r = y - yhat; history dates
//       of the first window fill the ring, monitoring dates slide the window
//       (Eq. 3) and test MO against the boundary of Eq. 4: the exact test
//       runs only on stages whose largest |MO| reaches the boundary at the
//       stage's first position (the boundary grows with the position), and
//       only until the first crossing.
//
// Precision: the Gram sums use the basis split into fp16 hi + lo (22 bits);
// X'My uses tf32 y (beta0 is only the start of the refinement); r0 and the
// coefficients are split hi + lo with per-pixel power-of-two scales, and the
// regressors of the fitted values, scaled by 2^12, three ways (hi, mid, lo),
// so that the fitted values carry ~22 bits of beta0 and of delta separately
// and lose no more to the regressors: the float rounding of an intercept or
// trend would otherwise enter every residual of a window alike.
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <vector>

#include "bfm_internal.cuh"
#include "ptx.cuh"
#include "simt_seg.cuh"
#include "stage.cuh"

namespace bfm {

__device__ unsigned int g_bfm_hybrid_err = 0;  // bit 0: a bounded wait gave up

cudaError_t hybrid_read_clear_errors(cudaStream_t s, unsigned int* bits) {
    unsigned int v = 0;
    cudaError_t e = cudaMemcpyFromSymbolAsync(&v, g_bfm_hybrid_err, sizeof v, 0, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    const unsigned int zero = 0;
    e = cudaMemcpyToSymbolAsync(g_bfm_hybrid_err, &zero, sizeof zero, 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    *bits = v;
    return e;
}

namespace {

using namespace stage;

constexpr int kMT = 4;                    // 128-pixel M-tiles per CTA
constexpr int kPx = 128 * kMT;            // pixels per CTA tile
constexpr int kCons = 4 * kMT;            // pixel warps, four per M-tile
constexpr int kBoxPx = 128;               // TMA box width (one M-tile)
constexpr int kBoxBytes = 4096;
constexpr int kStages = 3;                // stages in flight per group
// The M-tiles of a CTA work in two groups, each with its own producer and MMA warp,
// stages and barriers: the four pixel warps of a scheduler then belong to two
// pipelines, and one computes while the other waits for a stage, an MMA or a solve.
// With all four M-tiles in one group the kernel issued on 58 % of its cycles, with two
// groups 68 %: 7.50 -> 6.70 ms (float) and 7.63 -> 6.91 ms (int16) on 8.4 Mi pixels of 414
// dates, 193 -> 167 us on 250k pixels of 256; with whole chunks and groups in loops of
// their own, without bounds checks, 6.48 ms, 6.49 ms and 154 us, and with the ring
// addressed directly 6.30, 6.41 and 154.  One M-tile per group (24 warps, 80
// registers) was slower at every size but the smallest.
constexpr int kGrp = 2;                       // M-tiles per group
constexpr int kGroups = kMT / kGrp;
constexpr int kGrpWarps = 4 * kGrp;           // pixel warps of a group
constexpr int kGrpPx = 128 * kGrp;            // pixels of a group
constexpr int kStageBytes = kGrp * kBoxBytes; // a stage: kGrp boxes
constexpr int kProdWarp = kCons;              // first of kGroups TMA producer warps
constexpr int kMmaWarp = kCons + kGroups;     // first of kGroups MMA warps (it owns TMEM)
constexpr int kThreads = 32 * (kCons + 2 * kGroups);
// Stages the loads of one group may lead those of the other.  Every date of a large
// scene is on a page of its own, and when the groups drift apart the CTA's loads touch
// more pages than its address translations cover: on the 8.4 Mi-pixel scene 10.1 ms
// without a limit (int16 13.0), 9.4 at 32 stages (15.4), 6.7 (6.95) at 1 to 8, float also
// at 16.  Scenes of under 0.5 GB run alike with any limit.
constexpr int kLead = 4;
constexpr uint32_t kTmemCols = 512;
constexpr uint64_t kWaitNs = 2000000000ull;
constexpr size_t kSmemCap = 232448;       // opt-in dynamic shared memory per block

// TMEM columns within an M-tile's 128 (the phases reuse them in turn):
//   pass A : G sums [0, 32), X'My [32, 48), A buffers 2 x (mask 8 | y 16) [48, 96)
//   pass B': c [0, 16), beta0 coefficients (24) [16, 40), r0 buffers 2 x (hi 8 | lo 8) [40, 72),
//            fitted-value pieces 2 x 16 [72, 104), the basis sums kept for the second solve [104, 128)
//   pass C : beta0 coefficients [16, 40), delta coefficients (24) [40, 64), pieces 2 x 32 [64, 128)
constexpr uint32_t kColG = 0, kColB = 32, kColA = 48, kColC = 0, kColB0 = 16, kColR = 40, kColY0 = 72, kColDl = 40,
                   kColY = 64;
// Pass B' keeps the pixel's basis sums (up to 21) in [104, 128), free until pass C, for the
// second solve, so that they do not occupy registers through the pass.
constexpr uint32_t kColS = 104;
// Coefficient operands: 24 columns per set, A_hi (K = 32: 16 columns) then A_lo (K = 16: 8 columns).
constexpr uint32_t kCoefLo = 16;
// The regressors of the fitted-value table are scaled by 2^12 before their three-way fp16 split.
constexpr float kYScale = 4096.f, kInvYScale = 1.f / 4096.f;

template <typename T>
struct Dt {
    static constexpr int G = kBoxBytes / (kBoxPx * (int)sizeof(T));  // dates per stage: 8 float, 16 int16
};

struct HybridParams {
    uint64_t wait_ns;            // bound of the pixel warps' stage waits (bfm_stage_wait_limit)
    const uint32_t* mask;
    int64_t m, mask_words;
    int N, n, hmax, npad;
    double h_frac;
    const unsigned char* tabs;   // design tables (hybrid_tables), npad dates
    float lam2, c_over_s, inv_s;
    int32_t* brk;
    float* mean;
    float* sigma;
    float* beta;
    uint8_t* status;
    float* maxmo;
};

// Byte offsets of the design tables in global memory for npad dates.
__host__ __device__ inline size_t tab_gram_lo(int npad) { return (size_t)npad * 48; }
__host__ __device__ inline size_t tab_x(int npad) { return (size_t)npad * 96; }
__host__ __device__ inline size_t tab_yhat(int npad) { return (size_t)npad * 160; }
__host__ __device__ inline size_t tab_yhat_bytes(int npad) { return (size_t)npad * 48 + 128; }
__host__ __device__ inline size_t tab_bytes(int npad) { return tab_yhat(npad) + tab_yhat_bytes(npad); }

struct HLayout {
    size_t gh, gl, xt, yh, stages, ring, bars, total;
};

// One tile of a batched launch (bfm_batch): its tensor map, parameters and
// first 512-pixel work block within its group.
struct HybBatchTile {
    CUtensorMap tm;  // 64-byte aligned type
    HybridParams P;
    int64_t block0;
};

// The batch side of a launch: the group's tiles (device memory), its work
// blocks and the shared-memory layout that holds the largest tables and ring
// among them.
struct HybBatch {
    const HybBatchTile* tiles;
    int ntiles;
    int64_t blocks;
    HLayout lo;
};

__host__ __device__ inline size_t up1024(size_t x) { return (x + 1023) & ~(size_t)1023; }

// Shared memory: Gram table hi and lo and the tf32 regressor table over the
// history (16-date chunks), the fitted-value table over all npad dates, the
// stages, the ring [hmax][kPx], barriers and a few words.
__host__ __device__ inline HLayout hyb_layout(int n, int npad, int hmax) {
    const size_t nh16 = (size_t)((n + 15) & ~15);
    HLayout L{};
    L.gh = 0;
    L.gl = L.gh + nh16 / 8 * 384;
    L.xt = L.gl + nh16 / 8 * 384;
    L.yh = L.xt + nh16 / 4 * 256;
    L.stages = L.yh + tab_yhat_bytes(npad);  // every part so far is a multiple of 128 bytes
    L.ring = L.stages + (size_t)kStages * kMT * kBoxBytes;
    L.bars = L.ring + (size_t)hmax * kPx * 4;
    // The bound that decides whether a call takes this form counts the tables in full
    // (256 bytes more), rounds the stages up to 1024 and adds 176 bytes; the barriers
    // (kBarBytes) fit in what that leaves: yh ends 384 or 896 bytes above a multiple
    // of 1024, so the three together are 560 bytes or more.
    L.total = up1024(L.yh + tab_yhat_bytes(npad) + 256) + (size_t)kStages * kMT * kBoxBytes + (size_t)hmax * kPx * 4 + 176;
    return L;
}

// Barriers: per group 2 kStages + 10, then two for the batch's tables; the TMEM address,
// the abort flag, a byte per pixel warp and a word per producer.
constexpr int kGrpBars = 2 * kStages + 10;
constexpr size_t kBarBytes = (size_t)(kGroups * kGrpBars + 2) * 8 + 8 + kCons + 4 * kGroups;
static_assert(kBarBytes <= 560, "the barriers fit the slack of hyb_layout's bound");

__device__ __forceinline__ float obs_y(float raw, bool& ok) {
    ok = !isnan(raw);
    return raw;
}
__device__ __forceinline__ float obs_y(int16_t raw, bool& ok) {
    ok = raw != (int16_t)-32768;
    return (float)raw;
}

// 2^(T - e) for v = 1.x * 2^e (so |v| * scale lies in [2^T, 2^(T+1))); 1 for
// zero, subnormal, infinite or NaN v.
__device__ __forceinline__ float pow2_scale(float v, int T) {
    const int e = (__float_as_int(v) >> 23) & 0xff;
    if (e == 0 || e == 0xff) return 1.f;
    int r = 254 + T - e;
    r = r < 1 ? 1 : (r > 254 ? 254 : r);
    return __int_as_float(r << 23);
}

__device__ __forceinline__ uint32_t h2bits(__half lo, __half hi) {
    return (uint32_t)__half_as_ushort(lo) | ((uint32_t)__half_as_ushort(hi) << 16);
}

// x = hi + lo exactly in float, hi the fp16 rounding of x; lo is rounded to fp16 by the caller.
__device__ __forceinline__ void split_h(float x, __half& hi, float& lo) {
    hi = __float2half_rn(x);
    lo = x - __half2float(hi);
}

// Coefficient A operands (fp16) for the fitted-value table, whose K rows are
// the regressors' three-way split [hi; mid; lo] (rows 24..31 are read from the
// next date group and meet zeros here): A_hi = [c_hi | c_hi | c_hi | 0]
// (K = 32, words 0..15) and A_lo = [c_lo | c_lo] (K = 16, words 16..23), so
// that the products cover c_hi (hi + mid + lo) + c_lo (hi + mid).  Returns in
// rep the value the products represent, c_hi + c_lo, in float.
template <int K>
__device__ __forceinline__ void coef_words(const float (&c)[K], float scale, uint32_t (&w)[24], float (&rep)[K]) {
    __half hi[8], lo[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if (i < K) {
            float l;
            split_h(c[i] * scale, hi[i], l);
            lo[i] = __float2half_rn(l);
            rep[i < K ? i : 0] = __half2float(hi[i]) + __half2float(lo[i]);
        } else {
            hi[i] = __float2half_rn(0.f);
            lo[i] = hi[i];
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        w[j] = h2bits(hi[2 * j], hi[2 * j + 1]);
        w[4 + j] = w[j];
        w[8 + j] = w[j];
        w[12 + j] = 0u;
        w[16 + j] = h2bits(lo[2 * j], lo[2 * j + 1]);
        w[20 + j] = w[16 + j];
    }
}

__device__ __forceinline__ void coef_store(uint32_t taddr, const uint32_t (&w)[24]) {
    uint32_t a[16], b[8];
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = w[i];
#pragma unroll
    for (int i = 0; i < 8; ++i) b[i] = w[16 + i];
    ptx::tmem_st16(taddr, a);
    ptx::tmem_st8(taddr + kCoefLo, b);
}

// Bounded wait that also ends when the CTA aborts; false when it gave up.
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag,
                                         uint64_t limit_ns) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = ptx::globaltimer_ns();
    while (true) {
        if (ptx::mbar_try_wait_hint(bar, parity, 20000u)) return true;
        if (*abort_flag || ptx::globaltimer_ns() - t0 > limit_ns) return false;
    }
}

__device__ __forceinline__ void raise_abort(volatile uint32_t* abort_flag) {
    if (!*abort_flag) {
        *abort_flag = 1u;
        atomicOr(&g_bfm_hybrid_err, 1u);
    }
}

// Validity of one observation of this thread's pixel: the in-band marker
// (float NaN, int16 -32768) and, with an explicit mask, the pixel's mask bit:
// bit u of `bits` for date u of the group of 8 at hand.  `in_range` false
// makes the date invalid.
template <typename T, bool kMask>
struct Obs {
    uint32_t bits = 0u;
    __device__ __forceinline__ bool valid(T raw, int u, bool in_range) const {
        bool ok;
        (void)obs_y(raw, ok);
        ok = ok && in_range;
        if (kMask) ok = ok && ((bits >> u) & 1u) != 0u;
        return ok;
    }
    // value (0 when invalid) and validity
    __device__ __forceinline__ float value(T raw, int u, bool in_range, bool& ok) const {
        const float y = obs_y(raw, ok);
        ok = ok && in_range;
        if (kMask) ok = ok && ((bits >> u) & 1u) != 0u;
        return y;
    }
};

// Eight dates of a stage into registers: ahead of a wait (for a buffer, for a TMEM load),
// so that the two latencies overlap.
template <typename T>
__device__ __forceinline__ void load8(const T* st, T (&raw)[8]) {
#pragma unroll
    for (int u = 0; u < 8; ++u) raw[u] = st[u * kBoxPx];
}

// Pass A, 8 dates from d8: masked y as tf32 bits, the 0/1 mask as 4 fp16
// pairs (even date in the low half), and max |y|.
template <bool kFull, typename T, bool kMask>
__device__ __forceinline__ void pass_a8(const Obs<T, kMask>& ob, const T (&raw)[8], int d8, int n, uint32_t* yv,
                                        uint32_t* mk, float& ymax) {
    float vf[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        bool ok;
        float y = ob.value(raw[u], u, kFull || d8 + u < n, ok);
        y = ok ? y : 0.f;
        ymax = fmaxf(ymax, fabsf(y));
        yv[u] = __float_as_uint(y);
        vf[u] = ok ? 1.f : 0.f;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const __half2 h = __floats2half2_rn(vf[2 * j], vf[2 * j + 1]);
        mk[j] = *reinterpret_cast<const uint32_t*>(&h);
    }
}

// Pass B', 8 dates from d8: r0 = y - yhat0 (0 where invalid), s0 += r0^2,
// r0 * s_r split into fp16 hi (11 leading bits) + lo as 4 + 4 packed pairs;
// with kScan, the date of valid rank `rem` (counted down) becomes wdate.
template <bool kFull, bool kScan, typename T, bool kMask>
__device__ __forceinline__ void pass_b8(const Obs<T, kMask>& ob, const T (&raw)[8], int d8, int n, const float* yh,
                                        float inv_sb, float s_r, float& ss0, uint32_t* hw, uint32_t* lw, int& rem,
                                        int& wdate) {
    float hi[8], lo[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        bool ok;
        const float y = ob.value(raw[u], u, kFull || d8 + u < n, ok);
        const float r = ok ? fmaf(-yh[u], inv_sb, y) : 0.f;
        ss0 = fmaf(r, r, ss0);
        const float rs = r * s_r;
        hi[u] = __uint_as_float(__float_as_uint(rs) & 0xFFFFE000u);
        lo[u] = rs - hi[u];
        if (kScan) wdate = (ok && rem == 0) ? d8 + u : wdate;
        rem -= ok ? 1 : 0;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const __half2 h = __floats2half2_rn(hi[2 * j], hi[2 * j + 1]);
        const __half2 l = __floats2half2_rn(lo[2 * j], lo[2 * j + 1]);
        hw[j] = *reinterpret_cast<const uint32_t*>(&h);
        lw[j] = *reinterpret_cast<const uint32_t*>(&l);
    }
}

// The ring is addressed by 32-bit shared-memory addresses, so that a slot needs no
// address arithmetic of its own.
__device__ __forceinline__ float ring_ld(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void ring_st(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v)); }
constexpr uint32_t kSlot = kPx * 4;  // bytes from slot to slot

// State of the monitoring scan of one pixel.
struct Mon {
    uint32_t slot = 0;    // address of the next residual's ring slot
    uint32_t beg = 0;     // of the first slot
    uint32_t end = 0;     // behind h_p slots
    uint32_t fill_end = 0;  // behind h_p - 1 slots: the first window's history part
    int wdate = 0;        // date of the first window's oldest history observation
    int cnt = 0;          // valid monitoring observations so far
    float inv_sb = 1.f;
    float W = 0.f;        // window sum of h_p residuals
    float blk = 0.f;      // sum of W over this stretch's valid monitoring positions
    float amax = 0.f;     // largest |W| seen in this stretch (a bound for the boundary pre-test)
    float wmax = -INFINITY, wmin = INFINITY;  // extreme W over the monitoring positions
};

// History dates [d8, d8 + 8) before n: the first window's residuals into the ring.
template <typename T, bool kMask>
__device__ __forceinline__ void mon_hist8(const Obs<T, kMask>& ob, const T (&raw)[8], int d8, const float* yh,
                                          Mon& mo) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        bool ok;
        const float y = ob.value(raw[u], u, true, ok);
        const float r = fmaf(-yh[u], mo.inv_sb, y);
        const bool take = ok && d8 + u >= mo.wdate && mo.slot < mo.fill_end;
        if (take) ring_st(mo.slot, r);
        mo.slot += take ? kSlot : 0u;
        mo.W += take ? r : 0.f;
    }
}

// One monitoring date: the window gains r and loses the ring slot it replaces.
template <bool kExt>
__device__ __forceinline__ void mon_step(bool ok, float r, Mon& mo) {
    const float old = ring_ld(mo.slot);
    if (ok) ring_st(mo.slot, r);
    const uint32_t ns = mo.slot + (ok ? kSlot : 0u);
    mo.slot = ns == mo.end ? mo.beg : ns;
    mo.W += ok ? r - old : 0.f;
    mo.cnt += ok ? 1 : 0;
    mo.blk += ok ? mo.W : 0.f;
    mo.amax = fmaxf(mo.amax, fabsf(mo.W));
    if (kExt) {
        mo.wmax = ok ? fmaxf(mo.wmax, mo.W) : mo.wmax;
        mo.wmin = ok ? fminf(mo.wmin, mo.W) : mo.wmin;
    }
}

// Eight monitoring dates, all in [n, N).
template <bool kExt, typename T, bool kMask>
__device__ __forceinline__ void mon8(const Obs<T, kMask>& ob, const T (&raw)[8], const float* yh, Mon& mo,
                                     float (&Wu)[8]) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        bool ok;
        const float y = ob.value(raw[u], u, true, ok);
        mon_step<kExt>(ok, fmaf(-yh[u], mo.inv_sb, y), mo);
        Wu[u] = mo.W;
    }
}

// Dates [d8, d8 + 8) that hold n (or N): history dates fill the ring, later ones are monitored.
template <typename T, bool kMask>
__device__ __forceinline__ void mon_mixed8(const Obs<T, kMask>& ob, const T (&raw)[8], int d8, int n, int N,
                                        const float* yh, Mon& mo, float (&Wu)[8], bool ext) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int d = d8 + u;
        bool ok;
        const float y = ob.value(raw[u], u, d < N, ok);
        const float r = fmaf(-yh[u], mo.inv_sb, y);
        if (d < n) {
            const bool take = ok && d >= mo.wdate && mo.slot < mo.fill_end;
            if (take) ring_st(mo.slot, r);
            mo.slot += take ? kSlot : 0u;
            mo.W += take ? r : 0.f;
        } else if (ext) {
            mon_step<true>(ok, r, mo);
        } else {
            mon_step<false>(ok, r, mo);
        }
        Wu[u] = mo.W;
    }
}

// kBatch: the work blocks of several tiles (Bt; tmap and P are unused but for
// P.wait_ns), the tables of a block's tile loaded by the MMA warp when its
// previous block belonged to another tile; otherwise the blocks of one tile.
template <int KH, typename T, bool kMask, bool kBatch>
__global__ void __launch_bounds__(kThreads, 1)
    hybrid_kernel(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ HybridParams P,
                  const HybBatch Bt) {
    using B = Basis<KH>;
    constexpr int K = B::K, NBR = B::NBR;
    constexpr int G = Dt<T>::G;         // dates per stage
    extern __shared__ __align__(1024) unsigned char smem[];
    const HLayout Lo = kBatch ? Bt.lo : hyb_layout(P.n, P.npad, P.hmax);
    unsigned char* s_gh = smem + Lo.gh;
    unsigned char* s_gl = smem + Lo.gl;
    unsigned char* s_xt = smem + Lo.xt;
    unsigned char* s_yh = smem + Lo.yh;
    unsigned char* stages = smem + Lo.stages;
    float* ring = reinterpret_cast<float*>(smem + Lo.ring);
    // (the shuffle tells the compiler that the warp index is uniform)
    const int tid = threadIdx.x, warp = __shfl_sync(~0u, tid >> 5, 0), lane = tid & 31;
    // the group this warp works for
    const int g = warp < kCons ? warp / kGrpWarps : (warp - kCons) % kGroups;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Lo.bars);
    uint64_t* full = bars + g * kGrpBars;   // [kStages] stage landed
    uint64_t* empty = full + kStages;       // [kStages] stage released by the group's pixel warps
    uint64_t* afull = empty + kStages;      // [2] A buffer written by the pixel warps
    uint64_t* aempty = afull + 2;           // [2] MMAs reading the A buffer done
    uint64_t* yfull = aempty + 2;           // [2] fitted-value piece computed
    uint64_t* yempty = yfull + 2;           // [2] fitted-value piece read by the pixel warps
    uint64_t* accd = yempty + 2;            // sums complete: pass A, then pass B' (two phases per block)
    uint64_t* coefb = accd + 1;             // coefficient operands written: beta0, then delta with the window
                                            // starts published (two phases per block)
    uint64_t* tabb = bars + kGroups * kGrpBars; // batch: a tile's tables landed
    uint64_t* tabfree = tabb + 1;           // batch: the MMAs of every group's earlier blocks done
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(tabfree + 1);
    volatile uint32_t* abort_flag = s_tmem + 1;
    unsigned char* s_dstart = reinterpret_cast<unsigned char*>(s_tmem + 2);  // [kCons] window start / 8 by pixel warp
    volatile int* s_pos = reinterpret_cast<volatile int*>(s_dstart + kCons);  // [kGroups] stage each producer is at

    if constexpr (!kBatch) {
        const int npad = P.npad;
        const size_t nh16 = (size_t)((P.n + 15) & ~15);
        auto copy = [&](unsigned char* dst, size_t src_off, size_t bytes) {
            const uint4* s = reinterpret_cast<const uint4*>(P.tabs + src_off);
            uint4* d = reinterpret_cast<uint4*>(dst);
            for (size_t i = tid; i < bytes / 16; i += kThreads) d[i] = __ldg(s + i);
        };
        copy(s_gh, 0, nh16 / 8 * 384);
        copy(s_gl, tab_gram_lo(npad), nh16 / 8 * 384);
        copy(s_xt, tab_x(npad), nh16 / 4 * 256);
        copy(s_yh, tab_yhat(npad), tab_yhat_bytes(npad));
    }
    if (tid == 0) {
        for (int t = 0; t < kGroups; ++t) {
            uint64_t* b0 = bars + t * kGrpBars;  // in the order of the pointers above
            const int wpt = kGrpWarps;
            for (int s = 0; s < kStages; ++s) {
                ptx::mbar_init(b0 + s, 1);
                ptx::mbar_init(b0 + kStages + s, wpt);
            }
            b0 += 2 * kStages;
            for (int b = 0; b < 2; ++b) {
                ptx::mbar_init(b0 + b, wpt);
                ptx::mbar_init(b0 + 2 + b, 1);
                ptx::mbar_init(b0 + 4 + b, 1);
                ptx::mbar_init(b0 + 6 + b, wpt);
            }
            ptx::mbar_init(b0 + 8, 1);
            ptx::mbar_init(b0 + 9, wpt);
        }
        ptx::mbar_init(tabb, 1);
        ptx::mbar_init(tabfree, kGroups);
        for (int t = 0; t < kGroups; ++t) s_pos[t] = 0;
        *abort_flag = 0u;
        ptx::fence_mbar_init();
    }
    if (warp == kMmaWarp) ptx::tmem_alloc(s_tmem, kTmemCols);
    ptx::fence_async_smem();  // tables written by the threads, read by the tensor cores
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = *s_tmem;

    // Work blocks.  One tile: the pixels of a group, block u of the scene to CTA u % grid,
    // group (u / grid) % N, so that a scene of few blocks spreads over the SMs first.
    // Batch: 512 pixels of a tile, a part to each group (the groups share the tile's
    // tables).
    const int64_t nwork = kBatch ? Bt.blocks : (P.m + kGrpPx - 1) / kGrpPx;
    const int64_t wb0 = (int64_t)blockIdx.x + (kBatch ? 0 : (int64_t)gridDim.x * g);
    const int64_t wstep = kBatch ? (int64_t)gridDim.x : (int64_t)gridDim.x * kGroups;
    auto locate = [&](int64_t wb, int& ti, int64_t& px0) {
        if constexpr (kBatch) {
            int lo = 0, hi = Bt.ntiles - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (Bt.tiles[mid].block0 <= wb)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            ti = lo;
            px0 = (wb - Bt.tiles[lo].block0) * kPx + g * kGrpPx;
        } else {
            ti = 0;
            px0 = wb * kGrpPx;
        }
    };
    // the group's earliest window start, a multiple of the stage's dates
    auto dstart = [&]() -> int {
        const volatile uint32_t* w = reinterpret_cast<const volatile uint32_t*>(s_dstart + kGrpWarps * g);
        uint32_t v = w[0];
#pragma unroll
        for (int i = 1; i < kGrp; ++i) v = __vminu4(v, w[i]);
        const uint32_t a = min(v & 0xffu, (v >> 8) & 0xffu), b = min((v >> 16) & 0xffu, v >> 24);
        return (int)min(a, b) * 8 / G * G;
    };

    if (warp >= kProdWarp && warp < kMmaWarp) {
        // ---------------- TMA producer: passes A, B' over the history, C from the window start
        if (lane == 0) {
            if constexpr (!kBatch) ptx::prefetch_tmap(&tmap);
            const uint64_t keep = l2_evict_last(), normal = l2_evict_normal(), drop = l2_evict_first();
            unsigned char* const st0 = stages + g * (kStages * kStageBytes);
            int slot = 0;
            uint32_t lap = 0;  // laps of the ring completed
            bool ok = true;
            // pos: the stage in the order of blocks, passes and dates.  Waiting for the other
            // group only keeps the loads together: it ends by itself after 20 us.
            auto issue = [&](const CUtensorMap* tm, int64_t px0, int d0, uint64_t pol, int pos) -> bool {
                s_pos[g] = pos;
                if (s_pos[g ^ 1] < pos - kLead) {
                    const uint64_t t0 = ptx::globaltimer_ns();
                    while (s_pos[g ^ 1] < pos - kLead && !*abort_flag && ptx::globaltimer_ns() - t0 < 20000) __nanosleep(50);
                }
                if (lap && !wait_released(empty + slot, (lap - 1u) & 1u, abort_flag, kWaitNs)) {
                    raise_abort(abort_flag);
                    return false;
                }
                if (*abort_flag) return false;
                ptx::mbar_arrive_expect_tx(full + slot, (uint32_t)kStageBytes);
#pragma unroll
                for (int i = 0; i < kGrp; ++i)
                    tma_box(st0 + slot * kStageBytes + i * kBoxBytes, tm, full + slot, (int)(px0 + i * kBoxPx), d0, pol);
                if (++slot == kStages) {
                    slot = 0;
                    ++lap;
                }
                return true;
            };
            int cur = -1, pos0 = 0;
            for (int64_t wb = wb0; wb < nwork && ok; wb += wstep) {
                int ti;
                int64_t px0;
                locate(wb, ti, px0);
                const CUtensorMap* tm = &tmap;
                if constexpr (kBatch) {
                    tm = &Bt.tiles[ti].tm;
                    if (ti != cur) ptx::fence_tmap_acquire(tm);  // a map in global memory
                    cur = ti;
                }
                const HybridParams& Q = kBatch ? Bt.tiles[ti].P : P;
                const int n = Q.n, N = Q.N;
                const int nsh = (n + G - 1) / G, per_block = 2 * nsh + (N + G - 1) / G;
                if (px0 >= Q.m) {
                    pos0 += per_block;
                    s_pos[g] = pos0;
                    continue;
                }
                for (int d0 = 0; d0 < n && ok; d0 += G) ok = issue(tm, px0, d0, keep, pos0 + d0 / G);
                for (int d0 = 0; d0 < n && ok; d0 += G) {
                    // the block's first coefb phase is seen before the last stage of pass B'
                    // is issued: the second phase cannot complete without that stage
                    if (d0 + G >= n && !wait_bar(coefb, 0u, abort_flag, kWaitNs)) {
                        raise_abort(abort_flag);
                        ok = false;
                        break;
                    }
                    ok = issue(tm, px0, d0, drop, pos0 + nsh + d0 / G);
                }
                if (!ok) break;
                if (!wait_bar(coefb, 1u, abort_flag, kWaitNs)) {
                    raise_abort(abort_flag);
                    break;
                }
                for (int d0 = dstart(); d0 < N && ok; d0 += G) ok = issue(tm, px0, d0, normal, pos0 + 2 * nsh + d0 / G);
                pos0 += per_block;
            }
            s_pos[g] = INT_MAX;
            // copies still in flight land before the CTA's shared memory is released
            for (int i = 0; i < kStages; ++i) {
                const uint32_t uses = lap + (i < slot ? 1u : 0u);
                if (uses) ptx::mbar_wait_bounded(full + i, (uses - 1u) & 1u, kWaitNs);
            }
        }
        __syncwarp();
    } else if (warp >= kMmaWarp) {
        // ---------------- tensor-core issuer of the group
        if (lane == 0) {
            const uint32_t id_g = ptx::idesc_f16(128, 32, false), id_c = ptx::idesc_f16(128, 16, false);
            const uint32_t id_x = ptx::idesc_tf32(128, 16);
            const uint32_t id_y16 = ptx::idesc_f16(128, 16, true), id_y32 = ptx::idesc_f16(128, 32, true);
            uint32_t cc = 0, pc = 0;
            uint32_t nacc = 0;  // commits on accd
            bool ok = true;
            // fitted values into piece buffer pc & 1: 16 dates of beta0 in pass B', 32 dates of
            // beta0 + delta in pass C.  Per coefficient set: A_hi x rows 0..15, A_hi x rows 16..31,
            // A_lo x rows 0..15 of the table (rows 16..31 start 256 bytes on).
            auto piece = [&](int d0, bool pass_c) -> bool {
                const uint32_t b = pc & 1u;
                if (pc >= 2 && !wait_bar(yempty + b, ((pc >> 1) - 1) & 1u, abort_flag, kWaitNs)) return false;
                ptx::tc_fence_after();
                const uint64_t y01 = ptx::smem_desc(s_yh + (size_t)(d0 / 8) * 384, 128, 384);
                const uint64_t y23 = ptx::smem_desc(s_yh + (size_t)(d0 / 8) * 384 + 256, 128, 384);
                const uint32_t idy = pass_c ? id_y32 : id_y16;
#pragma unroll
                for (int i = 0; i < kGrp; ++i) {
                    const uint32_t base = tmem + 128u * (uint32_t)(g * kGrp + i);
                    const uint32_t dcol = pass_c ? base + kColY + 32u * b : base + kColY0 + 16u * b;
                    ptx::mma_f16_ta(dcol, base + kColB0, y01, idy, false);
                    ptx::mma_f16_ta(dcol, base + kColB0 + 8, y23, idy, true);
                    ptx::mma_f16_ta(dcol, base + kColB0 + kCoefLo, y01, idy, true);
                    if (pass_c) {
                        ptx::mma_f16_ta(dcol, base + kColDl, y01, idy, true);
                        ptx::mma_f16_ta(dcol, base + kColDl + 8, y23, idy, true);
                        ptx::mma_f16_ta(dcol, base + kColDl + kCoefLo, y01, idy, true);
                    }
                }
                ptx::mma_commit(yfull + b);
                ++pc;
                return true;
            };
            auto wait_a = [&]() -> bool {
                const uint32_t b = cc & 1u;
                if (!wait_bar(afull + b, (cc >> 1) & 1u, abort_flag, kWaitNs)) return false;
                ptx::tc_fence_after();
                return true;
            };
            int cur = -1;
            uint32_t tpar = 0, fpar = 0;
            bool tab_pending = false;  // a table copy not seen to land
            for (int64_t wb = wb0; wb < nwork && ok; wb += wstep) {
                int ti;
                int64_t px0;
                locate(wb, ti, px0);
                const HybridParams& Q = kBatch ? Bt.tiles[ti].P : P;
                const int n = Q.n, N = Q.N;
                const int nck = (n + 15) / 16;  // 16-date chunks of the history
                if constexpr (kBatch) {
                    if (ti != cur) {
                        // the MMAs of every group's earlier blocks have read the previous
                        // tile's tables before the first MMA warp replaces them
                        if (cur >= 0) ptx::mma_commit(tabfree);
                        if (g == 0) {
                            if (cur >= 0) {
                                if (!(ok = wait_bar(tabfree, fpar, abort_flag, kWaitNs))) break;
                                fpar ^= 1u;
                            }
                            const int npad = Q.npad;
                            const uint32_t bg = (uint32_t)((n + 15) & ~15) / 8 * 384,
                                           bx = (uint32_t)((n + 15) & ~15) / 4 * 256;
                            const uint32_t by = (uint32_t)tab_yhat_bytes(npad);
                            ptx::mbar_arrive_expect_tx(tabb, 2 * bg + bx + by);
                            ptx::bulk_g2s(s_gh, Q.tabs, bg, tabb);
                            ptx::bulk_g2s(s_gl, Q.tabs + tab_gram_lo(npad), bg, tabb);
                            ptx::bulk_g2s(s_xt, Q.tabs + tab_x(npad), bx, tabb);
                            ptx::bulk_g2s(s_yh, Q.tabs + tab_yhat(npad), by, tabb);
                            tab_pending = true;
                        }
                        if (!(ok = wait_bar(tabb, tpar, abort_flag, kWaitNs))) break;
                        tab_pending = false;
                        tpar ^= 1u;
                        cur = ti;
                    }
                }
                if (px0 >= Q.m) continue;
                // pass A: masked basis sums and X'My
                for (int c = 0; c < nck && ok; ++c) {
                    if (!(ok = wait_a())) break;
                    const uint32_t b = cc & 1u;
                    const uint64_t gh = ptx::smem_desc(s_gh + (size_t)(2 * c) * 384, 384, 128);
                    const uint64_t gl = ptx::smem_desc(s_gl + (size_t)(2 * c) * 384, 384, 128);
                    const uint64_t x0 = ptx::smem_desc(s_xt + (size_t)(4 * c) * 256, 256, 128);
                    const uint64_t x1 = ptx::smem_desc(s_xt + (size_t)(4 * c + 2) * 256, 256, 128);
#pragma unroll
                    for (int i = 0; i < kGrp; ++i) {
                        const uint32_t base = tmem + 128u * (uint32_t)(g * kGrp + i), a = base + kColA + 24u * b;
                        ptx::mma_f16_ta(base + kColG, a, gh, id_g, c > 0);
                        ptx::mma_f16_ta(base + kColG, a, gl, id_g, true);
                        ptx::mma_tf32_ta(base + kColB, a + 8, x0, id_x, c > 0);
                        ptx::mma_tf32_ta(base + kColB, a + 16, x1, id_x, true);
                    }
                    ptx::mma_commit(aempty + b);
                    ++cc;
                }
                if (!ok) break;
                ptx::mma_commit(accd);
                ++nacc;
                // pass B': fitted values of beta0, refinement sums X'M r0
                if (!(ok = wait_bar(coefb, 0u, abort_flag, kWaitNs))) break;
                ptx::tc_fence_after();
                for (int c = 0; c < 2 && c < nck && ok; ++c) ok = piece(16 * c, false);
                for (int c = 0; c < nck && ok; ++c) {
                    if (!(ok = wait_a())) break;
                    const uint32_t b = cc & 1u;
                    const uint64_t gh = ptx::smem_desc(s_gh + (size_t)(2 * c) * 384, 384, 128);
                    const uint64_t gl = ptx::smem_desc(s_gl + (size_t)(2 * c) * 384, 384, 128);
#pragma unroll
                    for (int i = 0; i < kGrp; ++i) {
                        const uint32_t base = tmem + 128u * (uint32_t)(g * kGrp + i), a = base + kColR + 16u * b;
                        ptx::mma_f16_ta(base + kColC, a, gh, id_c, c > 0);
                        ptx::mma_f16_ta(base + kColC, a + 8, gh, id_c, true);
                        ptx::mma_f16_ta(base + kColC, a, gl, id_c, true);
                    }
                    ptx::mma_commit(aempty + b);
                    ++cc;
                    // the pixel warps read chunk c's fitted values before they wrote its A operands
                    if (c + 2 < nck) ok = piece(16 * (c + 2), false);
                }
                if (!ok) break;
                ptx::mma_commit(accd);
                ++nacc;
                // pass C: fitted values of beta0 + delta from the group's earliest window start
                if (!(ok = wait_bar(coefb, 1u, abort_flag, kWaitNs))) break;
                ptx::tc_fence_after();
                for (int d0 = dstart(); d0 < N && ok; d0 += 32) ok = piece(d0, true);
            }
            if (!ok) raise_abort(abort_flag);
            // a table copy in flight lands before the CTA's shared memory is released
            if (g == 0 && tab_pending) ptx::mbar_wait_bounded(tabb, tpar, kWaitNs);
            // every MMA issued has completed before the tensor memory is released
            ptx::mma_commit(accd);
            ptx::mbar_wait_bounded(accd, nacc & 1u, kWaitNs);
        }
        __syncwarp();
    } else {
        // ---------------- pixel warps
        const int w = warp, q = w & 3;
        const int pl = 32 * w + lane;                       // ring column of the pixel
        const uint32_t tl = (uint32_t)(32 * q) << 16;       // TMEM lane field of this warp
        const uint32_t tcol = tmem + 128u * (uint32_t)(w >> 2);  // this M-tile's columns
        const int gp = pl % kGrpPx;                         // pixel within the group's block
        const uint32_t ring_a = ptx::smem_u32(ring + pl);
        const T* sbase =
            reinterpret_cast<const T*>(stages + g * (kStages * kStageBytes) + (gp >> 7) * kBoxBytes) + (pl & 127);
        const float qnan = __int_as_float(0x7fc00000);
        bool bad = false;
        int cslot = 0;
        uint32_t cphase = 0;
        uint32_t cc = 0, pc = 0;
        // Wait for the next stage and return this thread's column in it.  Fast path:
        // one look at the barrier and a warp vote; the bounded wait (which also ends
        // on the abort flag) only when some lane finds the stage not yet landed.  A
        // bound below 1 us (a test of the failure path) makes that look a
        // non-blocking one and the only one.  A warp whose wait gives up raises the
        // abort flag and is `bad` from then on (warp-uniform): it may finish reading
        // the chunk it is in, whose contents no longer matter (its pixels end as
        // TIMEOUT), but it releases no stage, so the producer never refills a slot
        // whose copy may still be in flight.
        const bool test_mode = P.wait_ns < 1000u;
        auto acquire = [&]() -> const T* {
            const int slot = cslot;
            bool ok = !test_mode && ptx::mbar_try_wait(full + slot, cphase);
            if (!__all_sync(~0u, ok)) {
                if (!ok)
                    ok = test_mode ? ptx::mbar_test_wait(full + slot, cphase)
                                   : wait_bar(full + slot, cphase, abort_flag, P.wait_ns);
                if (__any_sync(~0u, !ok)) {
                    if (lane == 0) raise_abort(abort_flag);
                    bad = true;
                }
            }
            return sbase + slot * (kStageBytes / (int)sizeof(T));
        };
        auto release = [&]() {
            __syncwarp();
            if (lane == 0 && !bad) mbar_arrive(empty + cslot);
            const int ns = cslot + 1;
            cphase ^= ns == kStages ? 1u : 0u;
            cslot = ns == kStages ? 0 : ns;
        };
        auto wait_w = [&](uint64_t* bar, uint32_t parity) -> bool {  // warp-uniform bounded wait
            bool ok = ptx::mbar_try_wait(bar, parity);
            if (!__all_sync(~0u, ok)) {
                if (!ok) ok = wait_bar(bar, parity, abort_flag, kWaitNs);
                if (__any_sync(~0u, !ok)) {
                    if (lane == 0) raise_abort(abort_flag);
                    bad = true;
                    return false;
                }
            }
            return true;
        };
        auto arrive = [&](uint64_t* bar) {  // after this warp's TMEM accesses
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar);
        };
        auto write_unfitted = [&](const HybridParams& Q, int64_t p, int st) {
            Q.brk[p] = -1;
            Q.mean[p] = qnan;
            Q.sigma[p] = qnan;
#pragma unroll
            for (int a = 0; a < K; ++a) Q.beta[(size_t)a * Q.m + p] = qnan;
            Q.status[p] = (uint8_t)st;
            if (Q.maxmo) Q.maxmo[p] = qnan;
        };

        int64_t wb = wb0;
        for (; wb < nwork; wb += wstep) {
            int ti;
            int64_t px0;
            locate(wb, ti, px0);
            const HybridParams& Q = kBatch ? Bt.tiles[ti].P : P;
            const int n = Q.n, N = Q.N, hmax = Q.hmax;
            const int nck = (n + 15) / 16;  // 16-date chunks of the history
            const int64_t m = Q.m;
            if (px0 >= m) continue;
            const int64_t p = px0 + gp;
            const bool active = p < m;
            Obs<T, kMask> ob;
            // the warp's 32 pixels share one mask word per date
            const int64_t wcol = (px0 + gp) >> 5;
            MaskBits mb{kMask ? Q.mask + wcol : nullptr, (size_t)Q.mask_words, kMask && wcol < Q.mask_words ? N : 0};

            // ---- pass A: A operands of the masked basis sums and X'My
            float ymax = 0.f;
            if (kMask) mb.open(0, lane);
            // whole chunks carry no bounds checks; the last dates of a history that ends
            // within a chunk go through the same code with them
            auto chunk_a = [&](int c, auto full_c) {
                constexpr bool full = decltype(full_c)::value;
                const uint32_t b = cc & 1u;
                if (kMask && (c & 1) == 0) mb.next(16 * c, lane);
                uint32_t yv[16], mk[8];
                const T* stg = nullptr;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int d8 = 16 * c + 8 * h;
                    if (full || d8 < n) {  // warp-uniform: the dates exist
                        if (h == 0 || G == 8) stg = acquire();
                        const T* st = stg + (G == 16 ? h * 8 * kBoxPx : 0);
                        if (kMask) ob.bits = mb.cur >> (d8 & 31);
                        T raw[8];
                        load8(st, raw);
                        pass_a8<full>(ob, raw, d8, n, yv + 8 * h, mk + 4 * h, ymax);
                        if (G == 8 || h == 1 || (!full && d8 + 8 >= n)) release();
                    } else {
#pragma unroll
                        for (int u = 0; u < 8; ++u) yv[8 * h + u] = 0u;
#pragma unroll
                        for (int j = 0; j < 4; ++j) mk[4 * h + j] = 0u;
                    }
                }
                if (bad || (cc >= 2 && !wait_w(aempty + b, ((cc >> 1) - 1) & 1u))) return;
                ptx::tc_fence_after();
                const uint32_t a = tl + tcol + kColA + 24u * b;
                ptx::tmem_st8(a, mk);
                ptx::tmem_st16(a + 8, yv);
                ptx::tmem_wait_st();
                arrive(afull + b);
                ++cc;
            };
            const int nwhole = n / 16;
            for (int c = 0; c < nwhole && !bad; ++c) chunk_a(c, std::true_type{});
            if (nwhole < nck && !bad) chunk_a(nwhole, std::false_type{});
            if (bad) break;
            if (!wait_w(accd, 0u)) break;
            ptx::tc_fence_after();
            float S[NBR], Bv[K];
            {
                float v32[32], v16[16];
                ptx::tmem_ld32(tl + tcol + kColG, v32);
                ptx::tmem_ld16(tl + tcol + kColB, v16);
#pragma unroll
                for (int i = 0; i < NBR; ++i) S[i] = v32[i];
#pragma unroll
                for (int a = 0; a < K; ++a) Bv[a] = v16[a] + v16[8 + a];
            }
            const int np = (int)S[0];  // basis row 0 is 1: the count of valid history dates
            {
                uint32_t w16[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) w16[i] = i < NBR ? __float_as_uint(S[i]) : 0u;
                ptx::tmem_st16(tl + tcol + kColS, w16);
                if constexpr (NBR > 16) {
                    uint32_t w8[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) w8[i] = 16 + i < NBR ? __float_as_uint(S[16 + i]) : 0u;
                    ptx::tmem_st8(tl + tcol + kColS + 16, w8);
                }
            }
            float b0[K];
            bool nonsingular;
            {
                float Gm[K][K], Lc[K][K], dinv[K];
                gram_from_sums<KH>(S, Gm);
                nonsingular = cholesky<K>(Gm, Lc, dinv);
                chol_solve<K>(Lc, dinv, Bv, b0);
            }
            // operand scales (powers of two): |beta0| * s_b < 2^13; |r0| <= max|y| + sum|beta0|
            // (|x_i| <= 1 with the centred trend), so |r0| * s_r < 2^13
            float s_b, s_r;
            {
                float bm = 0.f, bs = 0.f;
#pragma unroll
                for (int a = 0; a < K; ++a) {
                    bm = fmaxf(bm, fabsf(b0[a]));
                    bs += fabsf(b0[a]);
                }
                s_b = pow2_scale(bm, 12);
                s_r = pow2_scale(ymax + bs, 12);
                if (!(bs < INFINITY)) {  // a singular pixel: keep every operand finite
                    s_b = 1.f;
                    s_r = 1.f;
#pragma unroll
                    for (int a = 0; a < K; ++a) b0[a] = 0.f;
                }
            }
            const float inv_sb = 1.f / s_b, inv_sr = 1.f / s_r;
            const float inv_fit = inv_sb * kInvYScale;  // the fitted values come out scaled by s_b 2^12
            {
                uint32_t wv[24];
                float rep[K];
                coef_words<K>(b0, s_b, wv, rep);
                coef_store(tl + tcol + kColB0, wv);
                ptx::tmem_wait_st();
                arrive(coefb);
            }
            const bool fit = np > K && nonsingular;
            int hp = (int)floor(Q.h_frac * (double)np);
            hp = hp < 1 ? 1 : (hp > np ? np : hp);
            if (!fit) hp = 1;  // keeps the ring arithmetic in range; nothing of it is used
            hp = hp > hmax ? hmax : hp;  // n_p <= n_hist, so this never binds: the ring holds hmax slots
            const int wq = fit ? np - hp + 1 : np;  // 0-based valid rank of the first window's oldest history obs

            // ---- pass B': r0 = y - yhat0, s0, A operands of X'M r0, the window's start date
            float ss0 = 0.f;
            int rem = wq, wdate = n;
            if (kMask) mb.open(0, lane);
            auto chunk_b = [&](int c, auto full_c) {
                constexpr bool full = decltype(full_c)::value;
                if (kMask && (c & 1) == 0) mb.next(16 * c, lane);
                if (!wait_w(yfull + (pc & 1u), (pc >> 1) & 1u)) return;
                ptx::tc_fence_after();
                uint32_t yq[2][8];
                ptx::tmem_ld8_issue(tl + tcol + kColY0 + 16u * (pc & 1u), yq[0]);
                ptx::tmem_ld8_issue(tl + tcol + kColY0 + 16u * (pc & 1u) + 8u, yq[1]);
                const uint32_t b = cc & 1u;
                uint32_t hw[8], lw[8];
                const T* stg = nullptr;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int d8 = 16 * c + 8 * h;
                    if (full || d8 < n) {
                        if (h == 0 || G == 8) stg = acquire();
                        const T* st = stg + (G == 16 ? h * 8 * kBoxPx : 0);
                        if (kMask) ob.bits = mb.cur >> (d8 & 31);
                        T raw[8];
                        load8(st, raw);
                        if (h == 0) {
                            ptx::tmem_wait_ld8(yq[0]);
                            ptx::tmem_wait_ld8(yq[1]);
                            arrive(yempty + (pc & 1u));
                            ++pc;
                        }
                        float yh[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) yh[u] = __uint_as_float(yq[h][u]);
                        // a pixel may reach its window's start among these dates (after it, rem < 0)
                        if (!full || __any_sync(~0u, (unsigned)rem < 8u))
                            pass_b8<full, true>(ob, raw, d8, n, yh, inv_fit, s_r, ss0, hw + 4 * h, lw + 4 * h, rem, wdate);
                        else
                            pass_b8<full, false>(ob, raw, d8, n, yh, inv_fit, s_r, ss0, hw + 4 * h, lw + 4 * h, rem, wdate);
                        if (G == 8 || h == 1 || (!full && d8 + 8 >= n)) release();
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            hw[4 * h + j] = 0u;
                            lw[4 * h + j] = 0u;
                        }
                    }
                }
                if (bad || (cc >= 2 && !wait_w(aempty + b, ((cc >> 1) - 1) & 1u))) return;
                ptx::tc_fence_after();
                const uint32_t a = tl + tcol + kColR + 16u * b;
                ptx::tmem_st8(a, hw);
                ptx::tmem_st8(a + 8, lw);
                ptx::tmem_wait_st();
                arrive(afull + b);
                ++cc;
            };
            for (int c = 0; c < nwhole && !bad; ++c) chunk_b(c, std::true_type{});
            if (nwhole < nck && !bad) chunk_b(nwhole, std::false_type{});
            if (bad) break;
            if (!wait_w(accd, 1u)) break;
            ptx::tc_fence_after();
            float cr[K];
            {
                float v16[16];
                ptx::tmem_ld16(tl + tcol + kColC, v16);
#pragma unroll
                for (int a = 0; a < K; ++a) cr[a] = v16[a] * inv_sr;
            }
            float dl[K];
            {
                float S2[NBR];
                {
                    float v16[16];
                    ptx::tmem_ld16(tl + tcol + kColS, v16);
#pragma unroll
                    for (int i = 0; i < 16 && i < NBR; ++i) S2[i] = v16[i];
                    if constexpr (NBR > 16) {
                        float v8[8];
                        ptx::tmem_ld8(tl + tcol + kColS + 16, v8);
#pragma unroll
                        for (int i = 16; i < NBR; ++i) S2[i] = v8[i - 16];
                    }
                }
                float Gm[K][K], Lc[K][K], dinv[K];
                gram_from_sums<KH>(S2, Gm);
                cholesky<K>(Gm, Lc, dinv);
                chol_solve<K>(Lc, dinv, cr, dl);
            }
            float dc = 0.f;
#pragma unroll
            for (int a = 0; a < K; ++a) dc = fmaf(dl[a], cr[a], dc);
            const float sig = sqrtf(fmaxf(ss0 - dc, 0.f) / (float)(np - K));
            const bool degenerate = !(sig > kDegenerateRatio * ymax) || ymax == 0.f;
            // beta of the centred trend: beta0 as the MMAs see it (c_hi + c_lo of its coefficient
            // words, unscaled; read back rather than kept in registers through pass B') plus delta.
            // The TMEM loads are warp-collective, so every lane takes them, before any branch.
            float bt[K];
            {
                float wh[8], wl[8];
                ptx::tmem_ld8(tl + tcol + kColB0, wh);
                ptx::tmem_ld8(tl + tcol + kColB0 + kCoefLo, wl);
#pragma unroll
                for (int a = 0; a < K; ++a) {
                    const uint32_t uh = __float_as_uint(wh[a >> 1]), ul = __float_as_uint(wl[a >> 1]);
                    const float h = __half2float(__ushort_as_half((unsigned short)((a & 1) ? uh >> 16 : uh)));
                    const float l = __half2float(__ushort_as_half((unsigned short)((a & 1) ? ul >> 16 : ul)));
                    bt[a] = (h + l) * inv_sb + dl[a];
                }
            }
            // outputs known now (the rest after the monitoring scan)
            if (active) {
                if (np <= K) {
                    write_unfitted(Q, p, BFM_PX_INSUFFICIENT_HISTORY);
                } else if (!nonsingular) {
                    write_unfitted(Q, p, BFM_PX_SINGULAR);
                } else {
                    Q.sigma[p] = sig;
                    // -> raw parameterisation of Eq. 2
                    Q.beta[p] = fmaf(-bt[1], Q.c_over_s, bt[0]);
                    Q.beta[(size_t)m + p] = bt[1] * Q.inv_s;
#pragma unroll
                    for (int a = 2; a < K; ++a) Q.beta[(size_t)a * m + p] = bt[a];
                }
            }
            {
                float dfin[K];
#pragma unroll
                for (int a = 0; a < K; ++a) dfin[a] = (fit && isfinite(dl[a])) ? dl[a] : 0.f;
                uint32_t wv[24];
                float rep[K];
                coef_words<K>(dfin, s_b, wv, rep);
                coef_store(tl + tcol + kColDl, wv);
            }
            // the warp's earliest window start, for the producer and the MMA warp (n / 8 <= 224)
            {
                const unsigned v = active && wdate < n ? (unsigned)wdate : (unsigned)n;
                const unsigned wmn = __reduce_min_sync(~0u, v);
                if (lane == 0) s_dstart[w] = (unsigned char)(wmn >> 3);
            }
            ptx::tmem_wait_st();
            arrive(coefb);
            if (!wait_w(coefb, 1u)) break;
            const int ds = dstart();

            // ---- pass C: window fill from the history, then the monitoring scan
            const float inv_scale = (fit && !degenerate) ? 1.f / (sig * sqrtf((float)np)) : 0.f;
            const float inv2 = inv_scale * inv_scale;
            const float lam2 = Q.lam2, lam2ln2 = lam2 * kLn2f, blg = lam2ln2 * log2_fast((float)np);
            float* const maxmo = Q.maxmo;
            const float jlimf = (float)floor(kEuler * (double)np);  // J / n_p <= e  <=>  J <= jlim
            Mon mo{};
            mo.beg = mo.slot = ring_a;
            mo.end = ring_a + (uint32_t)hp * kSlot;
            mo.fill_end = mo.end - kSlot;
            mo.wdate = wdate;
            mo.inv_sb = inv_fit;
            ring_st(mo.fill_end, 0.f);  // the first monitoring step finds h_p - 1 residuals
            int brk = -1;
            float sh = 0.f, sl = 0.f;
            const T* stg = nullptr;
            if (kMask) mb.open(ds, lane);
            // the values and fitted values of the dates [d8, d8 + 8); a stage or a piece of
            // fitted values is handed back behind its last group (end8, and here)
            auto begin8 = [&](int d8, T (&raw)[8], float (&yh)[8]) -> bool {
                const int off = d8 - ds;
                if (kMask) {
                    if ((off & 31) == 0) mb.next(d8, lane);
                    ob.bits = mb.cur >> (off & 31);
                }
                if ((off & 31) == 0 && !wait_w(yfull + (pc & 1u), (pc >> 1) & 1u)) return false;
                ptx::tc_fence_after();
                uint32_t yq[8];
                ptx::tmem_ld8_issue(tl + tcol + kColY + 32u * (pc & 1u) + (uint32_t)(off & 31), yq);
                if (off % G == 0) stg = acquire();
                load8(stg + (off % G) * kBoxPx, raw);  // dates of the stage are rows of kBoxPx elements
                ptx::tmem_wait_ld8(yq);
#pragma unroll
                for (int u = 0; u < 8; ++u) yh[u] = __uint_as_float(yq[u]);
                if ((off & 31) == 24 || d8 + 8 >= N) {
                    arrive(yempty + (pc & 1u));
                    ++pc;
                }
                return true;
            };
            auto end8 = [&](int d8) {
                if (((d8 - ds) % G) + 8 == G || d8 + 8 >= N) release();
            };
            // the boundary grows with the position: a stretch whose largest |MO| stays
            // within the boundary at its first position J0 holds no crossing (lowered by
            // 1e-6 relative, so that rounding of the boundary never hides a crossing)
            auto test8 = [&](int d8, int J0, const T (&raw)[8], const float (&Wu)[8]) {
                comp_add(sh, sl, mo.blk);
                if (brk < 0) {
                    const float Jf0 = (float)J0;
                    const float b2f = (Jf0 > jlimf ? fmaf(lam2ln2, log2_fast(Jf0), -blg) : lam2) * 0.999999f;
                    if (fmaf(mo.amax * mo.amax, inv2, -b2f) > 0.f) {
                        float Jc = Jf0;
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const int d = d8 + u;
                            if (d >= n && ob.valid(raw[u], u, d < N)) {
                                const float b2 = Jc > jlimf ? fmaf(lam2ln2, log2_fast(Jc), -blg) : lam2;
                                if (brk < 0 && fmaf(Wu[u] * Wu[u], inv2, -b2) > 0.f) brk = d;
                                Jc += 1.f;
                            }
                        }
                    }
                }
            };
            // eight dates that hold n or N
            auto mixed = [&](int d8) -> bool {
                T raw[8];
                float yh[8], Wu[8];
                if (!begin8(d8, raw, yh)) return false;
                const int J0 = np + 1 + mo.cnt;
                mo.blk = 0.f;
                mo.amax = 0.f;
                mon_mixed8(ob, raw, d8, n, N, yh, mo, Wu, maxmo != nullptr);
                test8(d8, J0, raw, Wu);
                end8(d8);
                return true;
            };
            auto monitor8 = [&](int d8, auto ext_c) -> bool {
                T raw[8];
                float yh[8], Wu[8];
                if (!begin8(d8, raw, yh)) return false;
                const int J0 = np + 1 + mo.cnt;
                mo.blk = 0.f;
                mo.amax = 0.f;
                mon8<decltype(ext_c)::value>(ob, raw, yh, mo, Wu);
                test8(d8, J0, raw, Wu);
                end8(d8);
                return true;
            };
            int d8 = ds;
            for (; d8 + 8 <= n && !bad; d8 += 8) {
                T raw[8];
                float yh[8];
                if (!begin8(d8, raw, yh)) break;
                mon_hist8(ob, raw, d8, yh, mo);
                end8(d8);
            }
            if (d8 < n && !bad && mixed(d8)) d8 += 8;
            if (maxmo)
                for (; d8 + 8 <= N && !bad && monitor8(d8, std::true_type{}); d8 += 8) {}
            else
                for (; d8 + 8 <= N && !bad && monitor8(d8, std::false_type{}); d8 += 8) {}
            if (d8 < N && !bad) mixed(d8);
            if (bad) break;
            if (!active) continue;

            const int Np = np + mo.cnt;
            if (fit) {
                if (degenerate) {
                    Q.status[p] = BFM_PX_DEGENERATE;
                    Q.brk[p] = -1;
                    Q.mean[p] = 0.f;
                    if (maxmo) maxmo[p] = 0.f;
                } else if (Np == np) {
                    Q.status[p] = BFM_PX_NO_MONITOR;
                    Q.brk[p] = -1;
                    Q.mean[p] = qnan;
                    if (maxmo) maxmo[p] = qnan;
                } else {
                    Q.status[p] = BFM_PX_OK;
                    Q.brk[p] = brk;
                    Q.mean[p] = (sh + sl) * inv_scale / (float)(Np - np);
                    // largest |MO| (positive on an exact tie of opposite signs)
                    if (maxmo) maxmo[p] = (mo.wmax >= -mo.wmin ? mo.wmax : mo.wmin) * inv_scale;
                }
            }
        }
        if (bad) {
            // a wait gave up: mark this thread's unfinished pixels
            for (; wb < nwork; wb += wstep) {
                int ti;
                int64_t px0;
                locate(wb, ti, px0);
                const HybridParams& Q = kBatch ? Bt.tiles[ti].P : P;
                const int64_t p = px0 + gp;
                if (p < Q.m) write_unfitted(Q, p, BFM_PX_TIMEOUT);
            }
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, kTmemCols);
    }
}

template <int KH, typename T, bool kMask>
bfm_status launch_one(const CUtensorMap& tm, const HybridParams& P, int grid, size_t smem, cudaStream_t st) {
    auto* fn = hybrid_kernel<KH, T, kMask, false>;
    // the opt-in maximum, not this launch's size: launches of other sizes (other
    // scenes, other host threads) never find a smaller limit in place
    const cudaError_t ea = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemCap);
    if (ea != cudaSuccess) return cuda_fail(ea, "bfm_monitor (hybrid): shared memory attribute");
    fn<<<grid, kThreads, smem, st>>>(tm, P, HybBatch{});
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "bfm_monitor (hybrid): launch");
    return BFM_OK;
}

template <int KH>
bfm_status launch_kh(const CUtensorMap& tm, const HybridParams& P, int dtype, int grid, size_t smem,
                     cudaStream_t st) {
    if (dtype == BFM_F32)
        return P.mask ? launch_one<KH, float, true>(tm, P, grid, smem, st)
                      : launch_one<KH, float, false>(tm, P, grid, smem, st);
    return P.mask ? launch_one<KH, int16_t, true>(tm, P, grid, smem, st)
                  : launch_one<KH, int16_t, false>(tm, P, grid, smem, st);
}

int hyb_hmax(int n_hist, double h_frac) {
    int h = (int)std::floor(h_frac * (double)n_hist);
    return h < 1 ? 1 : (h > n_hist ? n_hist : h);
}

int hyb_npad(int N) { return (N + 31) / 32 * 32 + 32; }

}  // namespace

// Design tables of the hybrid form for npad = hyb_npad(N) dates (zero beyond N):
//   Gram hi, Gram lo: the 3 + 6k basis functions (bfm::Basis order) split fp16
//     hi + lo, K-major over dates, three 8-row groups per 8-date group:
//     (t/8)*384 + (r/8)*128 + (r%8)*16 + (t%8)*2 (an MMA with N = 32 reads its
//     fourth row group from the next date group: accumulator columns 24..31,
//     which nothing reads);
//   X: the K regressors as tf32 hi (rows 0..7) and lo = x - hi (rows 8..15),
//     K-major over dates: (t/4)*256 + (r/8)*128 + (r%8)*16 + (t%4)*4;
//   fitted values: the K regressors times 2^12 split three ways into fp16 hi
//     (rows 0..7), mid (8..15) and lo (16..23), read MN-major:
//     (t/8)*384 + (r/8)*128 + (r%8)*16 + (t%8)*2, plus one row group of zeros
//     at the end (rows 24..31 of the last group are read from it and meet zero
//     coefficients).
void hybrid_tables(const bfm_design_s& d, const std::vector<double>& rows, std::vector<unsigned char>& out) {
    const int npad = hyb_npad(d.N), nbr = 3 + 6 * d.k, K = d.K;
    out.assign(tab_bytes(npad), 0);
    unsigned char* gh = out.data();
    unsigned char* gl = out.data() + tab_gram_lo(npad);
    unsigned char* xt = out.data() + tab_x(npad);
    unsigned char* yh = out.data() + tab_yhat(npad);
    for (int t = 0; t < d.N; ++t) {
        for (int r = 0; r < nbr; ++r) {
            const double v = rows[(size_t)t * d.NB + r];
            const __half hi = __double2half(v);
            const __half lo = __double2half(v - (double)__half2float(hi));
            const size_t o = (size_t)(t / 8) * 384 + (size_t)(r / 8) * 128 + (size_t)(r % 8) * 16 + (size_t)(t % 8) * 2;
            std::memcpy(gh + o, &hi, 2);
            std::memcpy(gl + o, &lo, 2);
        }
        for (int r = 0; r < K; ++r) {
            const double v = rows[(size_t)t * d.NB + r];
            // tf32 keeps the top 10 stored mantissa bits: hi by truncation, lo exact in float
            uint32_t bits;
            const float vf = (float)v;
            std::memcpy(&bits, &vf, 4);
            bits &= 0xFFFFE000u;
            float hif;
            std::memcpy(&hif, &bits, 4);
            const float lof = (float)(v - (double)hif);
            std::memcpy(xt + (size_t)(t / 4) * 256 + (size_t)(r % 8) * 16 + (size_t)(t % 4) * 4, &hif, 4);
            std::memcpy(xt + (size_t)(t / 4) * 256 + 128 + (size_t)(r % 8) * 16 + (size_t)(t % 4) * 4, &lof, 4);
            const double vs = v * (double)kYScale;
            const __half h1 = __double2half(vs);
            const double r1 = vs - (double)__half2float(h1);
            const __half h2 = __double2half(r1);
            const __half h3 = __double2half(r1 - (double)__half2float(h2));
            const size_t oy = (size_t)(t / 8) * 384 + (size_t)(r % 8) * 16 + (size_t)(t % 8) * 2;
            std::memcpy(yh + oy, &h1, 2);
            std::memcpy(yh + oy + 128, &h2, 2);
            std::memcpy(yh + oy + 256, &h3, 2);
        }
    }
}

size_t hybrid_table_bytes(int N) { return tab_bytes(hyb_npad(N)); }

bool hybrid_supported(const bfm_design_s* d, int dtype, int n_hist, double h_frac, const void* Y, int64_t m) {
    const size_t elt = dtype == BFM_F32 ? 4 : 2;
    if (!d->d_hyb || m < 1 || (uintptr_t)Y % 16 != 0 || ((size_t)m * elt) % 16 != 0) return false;
    return hyb_layout(n_hist, hyb_npad(d->N), hyb_hmax(n_hist, h_frac)).total <= kSmemCap;
}

namespace {

// Parameters and tensor map of one tile (false, with a message, when the
// hybrid form does not take it).
bool hyb_fill(const bfm_design_s* d, int dtype, const void* Y, const uint32_t* mask, int64_t m, int n_hist,
              double h_frac, double lambda, int32_t* brk, float* mean, float* sigma, float* beta, uint8_t* status,
              float* maxmo, HybridParams* Pout, CUtensorMap* tm) {
    if (!hybrid_supported(d, dtype, n_hist, h_frac, Y, m)) {
        set_error("the hybrid form needs Y with a 16-byte aligned base and rows of a multiple of 16 bytes, and "
                  "basis tables, stages and a residual ring of floor(h_frac * n_hist) slots for 512 pixels within "
                  "the shared memory of one SM");
        return false;
    }
    auto enc = encode_tiled();
    if (!enc) {
        set_error("hybrid form: cuTensorMapEncodeTiled is not available");
        return false;
    }
    const size_t elt = dtype == BFM_F32 ? 4 : 2;
    HybridParams P{};
    P.wait_ns = stage_wait_ns();
    P.mask = mask;
    P.m = m;
    P.mask_words = (m + 31) / 32;
    P.N = d->N;
    P.n = n_hist;
    P.hmax = hyb_hmax(n_hist, h_frac);
    P.npad = hyb_npad(d->N);
    P.h_frac = h_frac;
    P.tabs = static_cast<const unsigned char*>(d->d_hyb);
    P.lam2 = (float)(lambda * lambda);
    P.c_over_s = (float)(d->c / d->s);
    P.inv_s = (float)(1.0 / d->s);
    P.brk = brk;
    P.mean = mean;
    P.sigma = sigma;
    P.beta = beta;
    P.status = status;
    P.maxmo = maxmo;
    std::memset(tm, 0, sizeof *tm);
    const int G = dtype == BFM_F32 ? Dt<float>::G : Dt<int16_t>::G;
    const cuuint64_t gdim[2] = {(cuuint64_t)m, (cuuint64_t)d->N};
    const cuuint64_t gstride[1] = {(cuuint64_t)m * elt};
    const cuuint32_t box[2] = {(cuuint32_t)kBoxPx, (cuuint32_t)G};
    const cuuint32_t es[2] = {1u, 1u};
    if (enc(tm, elt == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16, 2,
            const_cast<void*>(Y), gdim, gstride, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
        set_error("hybrid form: cuTensorMapEncodeTiled failed for Y");
        return false;
    }
    *Pout = P;
    return true;
}

int sm_count_cur() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
    return sms;
}

}  // namespace

bfm_status launch_hybrid(const bfm_design_s* d, int dtype, const void* Y, const uint32_t* mask, int64_t m,
                         int n_hist, double h_frac, double lambda, int32_t* brk, float* mean, float* sigma,
                         float* beta, uint8_t* status, cudaStream_t stream, float* maxmo) {
    HybridParams P;
    CUtensorMap tm;
    if (!hyb_fill(d, dtype, Y, mask, m, n_hist, h_frac, lambda, brk, mean, sigma, beta, status, maxmo, &P, &tm))
        return BFM_EUNSUPPORTED;
    const int sms = sm_count_cur();
    const size_t smem = hyb_layout(n_hist, P.npad, P.hmax).total;
    const int64_t nblocks = (m + kGrpPx - 1) / kGrpPx;
    const int grid = (int)(nblocks < (int64_t)sms ? nblocks : (int64_t)sms);
    if (d->k == 1) return launch_kh<1>(tm, P, dtype, grid, smem, stream);
    if (d->k == 2) return launch_kh<2>(tm, P, dtype, grid, smem, stream);
    return launch_kh<3>(tm, P, dtype, grid, smem, stream);
}

// ---- batched launch (bfm_batch) --------------------------------------------------------------

struct HybGroup {
    int k, dtype;
    bool mask;
    int nmax = 0, npadmax = 0, hmaxmax = 0;  // the layout holds the largest of each
    int64_t blocks = 0;
    std::vector<HybBatchTile> tiles;
    HybBatchTile* d_tiles = nullptr;
    bool dirty = true;
};

HybGroup* hyb_group_create(int k, int dtype, bool has_mask) {
    auto* g = new HybGroup;
    g->k = k;
    g->dtype = dtype;
    g->mask = has_mask;
    return g;
}

void hyb_group_destroy(HybGroup* g) {
    if (!g) return;
    if (g->d_tiles) cudaFree(g->d_tiles);
    delete g;
}

bool hyb_group_variant(const HybGroup* g, int k, int dtype, bool has_mask) {
    return g->k == k && g->dtype == dtype && g->mask == has_mask;
}

int hyb_group_add(HybGroup* g, const bfm_design_s* d, const void* Y, const uint32_t* mask, int64_t m, int n_hist,
                  double h_frac, double lambda, int32_t* brk, float* mean, float* sigma, float* beta,
                  uint8_t* status) {
    HybBatchTile t;
    if (!hyb_fill(d, g->dtype, Y, mask, m, n_hist, h_frac, lambda, brk, mean, sigma, beta, status, nullptr, &t.P,
                  &t.tm))
        return -1;
    const int nmax = std::max(g->nmax, n_hist), npadmax = std::max(g->npadmax, t.P.npad),
              hmaxmax = std::max(g->hmaxmax, t.P.hmax);
    if (hyb_layout(nmax, npadmax, hmaxmax).total > kSmemCap) return 0;
    g->nmax = nmax;
    g->npadmax = npadmax;
    g->hmaxmax = hmaxmax;
    t.block0 = g->blocks;
    g->blocks += (m + kPx - 1) / kPx;
    g->tiles.push_back(t);
    g->dirty = true;
    return 1;
}

bfm_status hyb_group_upload(HybGroup* g) {
    if (!g->dirty) return BFM_OK;
    if (g->d_tiles) cudaFree(g->d_tiles);
    g->d_tiles = nullptr;
    cudaError_t e = cudaMalloc(&g->d_tiles, sizeof(HybBatchTile) * g->tiles.size());
    if (e == cudaSuccess)
        e = cudaMemcpy(g->d_tiles, g->tiles.data(), sizeof(HybBatchTile) * g->tiles.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(e, "bfm_batch: uploading hybrid tile descriptors");
    g->dirty = false;
    return BFM_OK;
}

namespace {
template <int KH, typename T, bool kMask>
void* hyb_batch_fn() {
    return (void*)hybrid_kernel<KH, T, kMask, true>;
}
}  // namespace

bfm_status hyb_group_node(HybGroup* g, cudaGraph_t graph, const cudaGraphNode_t* dep, cudaGraphNode_t* node) {
    void* fn = nullptr;
    const bool f32 = g->dtype == BFM_F32;
    switch (g->k) {
        case 1:
            fn = f32 ? (g->mask ? hyb_batch_fn<1, float, true>() : hyb_batch_fn<1, float, false>())
                     : (g->mask ? hyb_batch_fn<1, int16_t, true>() : hyb_batch_fn<1, int16_t, false>());
            break;
        case 2:
            fn = f32 ? (g->mask ? hyb_batch_fn<2, float, true>() : hyb_batch_fn<2, float, false>())
                     : (g->mask ? hyb_batch_fn<2, int16_t, true>() : hyb_batch_fn<2, int16_t, false>());
            break;
        default:
            fn = f32 ? (g->mask ? hyb_batch_fn<3, float, true>() : hyb_batch_fn<3, float, false>())
                     : (g->mask ? hyb_batch_fn<3, int16_t, true>() : hyb_batch_fn<3, int16_t, false>());
            break;
    }
    HybBatch bt{};
    bt.tiles = g->d_tiles;
    bt.ntiles = (int)g->tiles.size();
    bt.blocks = g->blocks;
    bt.lo = hyb_layout(g->nmax, g->npadmax, g->hmaxmax);
    const size_t smem = bt.lo.total;
    // the opt-in maximum: other groups of the same variant may need more than this one
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemCap);
    if (e != cudaSuccess) return cuda_fail(e, "bfm_batch: hybrid kernel shared memory attribute");
    // the single-tile parameters are unused but for the stage-wait bound
    static CUtensorMap tm_unused;  // zero; never read by the batched kernel
    HybridParams P{};
    P.wait_ns = g->tiles.empty() ? stage_wait_ns() : g->tiles[0].P.wait_ns;
    void* args[3] = {&tm_unused, &P, &bt};
    const int sms = sm_count_cur();
    cudaKernelNodeParams kp{};
    kp.func = fn;
    kp.gridDim = dim3((unsigned)std::min<int64_t>(g->blocks, sms));
    kp.blockDim = dim3(kThreads);
    kp.sharedMemBytes = (unsigned)smem;
    kp.kernelParams = args;
    e = cudaGraphAddKernelNode(node, graph, dep, dep ? 1 : 0, &kp);
    if (e != cudaSuccess) return cuda_fail(e, "bfm_batch: hybrid kernel node");
    return BFM_OK;
}

int64_t hyb_group_blocks(const HybGroup* g) { return g->blocks; }

}  // namespace bfm
