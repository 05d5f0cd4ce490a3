// Residuals and MOSUM process of selected pixels (bfm_trace).
//
// The many-core path returns the breaks and per-pixel summaries only; the
// residuals or the MOSUM process of an individual series can be examined
// afterwards, once the breaks say which series are of interest (Section 3.2,
// the remarks after Algorithm 2).  This file does that examination on the
// device for a list of pixels, one warp per pixel:
//   1. compaction of the pixel's valid observations (ballot + popcount over
//      32-date groups), n_p = valid history observations, N_p = all;
//   2. the least-squares fit of Eq. 5-6 on the valid history observations,
//      redone in FP64 from the design's table of Eq. 2 regressors (trend
//      centred and scaled) by Cholesky on the normal equations;
//   3. residuals y - x'beta (the sign of Eq. 3) of every valid observation,
//      sigma-hat with n_p - K degrees of freedom (Algorithm 1 step 5);
//   4. MO_j of Eq. 3 for every valid monitoring observation: the sum of the
//      h_p residuals ending at position j over sigma-hat * sqrt(n_p), from
//      FP64 prefix sums (the difference of two FP64 prefix sums is exact to
//      well below the float output).
// The pixel statuses written by bfm_monitor for the same data decide which
// pixels have a fit (OK, DEGENERATE, NO_MONITOR) so that the two calls agree
// on them; DEGENERATE pixels get MO = 0 at their monitoring dates.
//
// What bounds it: FP64 issue, 1/64 of the 32-bit rate, so FP64 instructions per
// pixel are what counts.  Evaluating the regressors in the kernel (six sincospi per
// date and pixel), summing the normal equations by butterflies over whole lanes and
// solving in every lane alike took about 2400 per warp and pixel: 709 us for 4096
// pixels of 414 dates.  Now the regressors are read from the design's table, the
// sums are folded (each exchange halves the values a lane carries) and the
// factorisation is spread over the lanes: about 400, 178 us; with runs of the prefix sums per lane and no division per
// date, 160 us.
#include <cmath>

#include "bfm_internal.cuh"

namespace bfm {
namespace {

struct TraceParams {
    const void* Y;
    const uint32_t* mask;
    int64_t m, mask_words;
    int N, n_hist, dtype;
    double h_frac;
    const double* x;  // regressors [N][K] of the design (Eq. 2, centred and scaled trend)
    const int64_t* pixels;
    int64_t count;
    const uint8_t* status;
    float* mo;
    float* resid;
};

// Shared memory of one warp: compacted values (double), their date indices
// and the compacted position of every date (-1 when missing).
constexpr int kBytesPerDate = 16;
constexpr int kMaxWarps = 4;
constexpr size_t kSmemTarget = 46 * 1024;  // beside the normal equations, within the default 48 KB

// Regressors of date t from the design's table (rows of K doubles, 16-byte aligned).
template <int K>
__device__ __forceinline__ void regressors(const double* tab, int t, double (&x)[K]) {
    const double2* r = reinterpret_cast<const double2*>(tab + (size_t)t * K);
#pragma unroll
    for (int a = 0; a < K / 2; ++a) {
        const double2 v = __ldg(r + a);
        x[2 * a] = v.x;
        x[2 * a + 1] = v.y;
    }
}

// Sums of n values over the warp's lanes, folded: at each exchange (lane
// distance kOff) a lane passes on the half of its values that its partner
// keeps, so n + n/2 + ... additions in place of n at every distance.  Ends with
// the sums of values first .. first + count - 1 in the lane, written to out.
template <int n, int kOff>
__device__ __forceinline__ void fold_sums(double (&v)[n], int lane, int first, int count, double* out) {
    if constexpr (kOff == 0) {
#pragma unroll
        for (int i = 0; i < n; ++i)
            if (i < count) out[first + i] = v[i];
    } else {
        constexpr int h = (n + 1) / 2;
        const bool up = (lane & kOff) != 0;
        double w[h];
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double lo = v[i], hi = i + h < n ? v[i + h < n ? i + h : 0] : 0.0;
            w[i] = (up ? hi : lo) + __shfl_xor_sync(~0u, up ? lo : hi, kOff);
        }
        fold_sums<h, kOff / 2>(w, lane, up ? first + h : first, up ? count - h : min(count, h), out);
    }
}

template <int KH>
__global__ void __launch_bounds__(32 * kMaxWarps) trace_kernel(const TraceParams P) {
    constexpr int K = 2 + 2 * KH;
    constexpr int NG = K * (K + 1) / 2;  // packed lower triangle, row a at a(a+1)/2
    constexpr int NE = NG + K;           // and the right-hand side as row K
    __shared__ double s_el[kMaxWarps][NE];
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + wib;
    if (i >= P.count) return;
    const int N = P.N;
    double* val = reinterpret_cast<double*>(smem + (size_t)wib * kBytesPerDate * N);
    int* tix = reinterpret_cast<int*>(val + N);
    int* pos = tix + N;
    float* mo_row = P.mo ? P.mo + i * N : nullptr;
    float* rs_row = P.resid ? P.resid + i * N : nullptr;
    const float qnan = __int_as_float(0x7fc00000);

    const int64_t p = P.pixels ? P.pixels[i] : i;
    int st = -1;
    if (p >= 0 && p < P.m) st = P.status[p];
    bool fit = st == BFM_PX_OK || st == BFM_PX_DEGENERATE || st == BFM_PX_NO_MONITOR;

    // 1. compaction
    int nv = 0, np = 0;
    if (fit) {
        constexpr int U = 4;  // groups of 32 dates whose loads are in flight together
        for (int tb = 0; tb < N; tb += 32 * U) {
            double y[U];
            bool v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int t = tb + 32 * u + lane;
                v[u] = false;
                y[u] = 0.0;
                if (t < N) {
                    const size_t o = (size_t)t * (size_t)P.m + (size_t)p;
                    if (P.dtype == BFM_F32) {
                        const float yf = __ldg(static_cast<const float*>(P.Y) + o);
                        v[u] = !isnan(yf);
                        y[u] = (double)yf;
                    } else {
                        const int16_t yq = __ldg(static_cast<const int16_t*>(P.Y) + o);
                        v[u] = yq != (int16_t)-32768;
                        y[u] = (double)yq;
                    }
                    if (P.mask)
                        v[u] = v[u] && ((__ldg(P.mask + (size_t)t * (size_t)P.mask_words + (size_t)(p >> 5)) >> (p & 31)) & 1u);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int t0 = tb + 32 * u, t = t0 + lane;
                const unsigned b = __ballot_sync(~0u, v[u]);
                const int q = nv + __popc(b & ((1u << lane) - 1u));
                if (t < N) pos[t] = v[u] ? q : -1;
                if (v[u]) {
                    val[q] = y[u];
                    tix[q] = t;
                }
                nv += __popc(b);
                const int hl = P.n_hist - t0;  // history dates in this group
                const unsigned hm = hl >= 32 ? ~0u : (hl > 0 ? (1u << hl) - 1u : 0u);
                np += __popc(b & hm);
            }
        }
        __syncwarp();
        fit = np > K;
    }

    // 2. normal equations of the history, right-hand side as a further row
    double beta[K];
    if (fit) {
        double* A = s_el[wib];
        {
            double g[NE];
#pragma unroll
            for (int a = 0; a < NE; ++a) g[a] = 0.0;
            for (int j = lane; j < np; j += 32) {
                double x[K];
                regressors<K>(P.x, tix[j], x);
                const double y = val[j];
#pragma unroll
                for (int a = 0; a < K; ++a) {
#pragma unroll
                    for (int b = 0; b <= a; ++b) g[a * (a + 1) / 2 + b] = fma(x[a], x[b], g[a * (a + 1) / 2 + b]);
                    g[NG + a] = fma(x[a], y, g[NG + a]);
                }
            }
            fold_sums<NE, 16>(g, lane, 0, NE, A);
        }
        __syncwarp();
        // Cholesky G = L L', column by column, the trailing elements (row i, column
        // c) spread over the lanes; row K becomes L^-1 rhs.  The diagonal keeps 1 / L_jj.
        constexpr int E = (NE + 31) / 32;
        int row[E], col[E];
        double own[E];
#pragma unroll
        for (int u = 0; u < E; ++u) {
            const int e = lane + 32 * u;
            int i = 0;
            while (i < K && (i + 1) * (i + 2) / 2 <= e) ++i;  // row i holds elements i(i+1)/2 ..
            row[u] = e < NE ? i : 0;
            col[u] = e < NE ? e - i * (i + 1) / 2 : -1;  // -1: no element
            own[u] = e < NE ? A[e] : 0.0;
        }
        auto at = [&](int i, int c) -> double& { return A[i * (i + 1) / 2 + c]; };
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const double d = at(j, j);
            fit = fit && d > 0.0;
            const double inv = rsqrt(d > 0.0 ? d : 1.0);
            double li[E], lc[E];
#pragma unroll
            for (int u = 0; u < E; ++u) {
                const bool upd = col[u] > j;
                li[u] = upd ? at(row[u], j) * inv : 0.0;
                lc[u] = upd ? (col[u] == row[u] ? li[u] : at(col[u], j) * inv) : 0.0;
            }
            __syncwarp();
#pragma unroll
            for (int u = 0; u < E; ++u) {
                own[u] = fma(-li[u], lc[u], own[u]);
                if (col[u] == j) own[u] = row[u] == j ? inv : own[u] * inv;
                if (col[u] >= j) A[lane + 32 * u] = own[u];
            }
            __syncwarp();
        }
#pragma unroll
        for (int a = K - 1; a >= 0; --a) {
            double v = at(K, a);
#pragma unroll
            for (int c = a + 1; c < K; ++c) v = fma(-at(c, a), beta[c], v);
            beta[a] = v * at(a, a);
        }
    }

    if (!fit) {
        for (int t = lane; t < N; t += 32) {
            if (mo_row) mo_row[t] = qnan;
            if (rs_row) rs_row[t] = qnan;
        }
        return;
    }

    // 3. residuals of every valid observation, sigma-hat from the history part
    double ss = 0.0;
    for (int j = lane; j < nv; j += 32) {
        double x[K];
        regressors<K>(P.x, tix[j], x);
        double yhat = 0.0;
#pragma unroll
        for (int a = 0; a < K; ++a) yhat = fma(x[a], beta[a], yhat);
        const double r = val[j] - yhat;
        val[j] = r;
        if (j < np) ss = fma(r, r, ss);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(~0u, ss, off);
    __syncwarp();
    if (rs_row)
        for (int t = lane; t < N; t += 32) {
            const int q = pos[t];
            rs_row[t] = q >= 0 ? (float)val[q] : qnan;
        }
    if (!mo_row) return;
    __syncwarp();

    // 4. prefix sums of the residuals in place (a run of consecutive ones per lane, then the
    // lanes' totals), then the windows of h_p terms
    {
        const int c = (nv + 31) / 32, j0 = lane * c, j1 = min(j0 + c, nv);
        double run = 0.0;
        for (int j = j0; j < j1; ++j) {
            run += val[j];
            val[j] = run;
        }
        double before = run;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const double u = __shfl_up_sync(~0u, before, off);
            if (lane >= off) before += u;
        }
        before = __shfl_up_sync(~0u, before, 1);
        if (lane > 0)
            for (int j = j0; j < j1; ++j) val[j] += before;
    }
    __syncwarp();
    int hp = (int)floor(P.h_frac * (double)np);
    hp = hp < 1 ? 1 : (hp > np ? np : hp);
    const double inv_scale = 1.0 / (sqrt(ss / (double)(np - K)) * sqrt((double)np));
    const bool degenerate = st == BFM_PX_DEGENERATE;
    for (int t = lane; t < N; t += 32) {
        float out = qnan;
        if (t >= P.n_hist) {
            const int q = pos[t];  // 0-based position: the window holds positions q-hp+1..q
            if (q >= np) out = degenerate ? 0.0f : (float)((val[q] - val[q - hp]) * inv_scale);
        }
        mo_row[t] = out;
    }
}

}  // namespace
}  // namespace bfm

using namespace bfm;

extern "C" bfm_status bfm_trace(bfm_design_t d, const void* Y, int dtype, const uint32_t* mask_bits, int64_t m,
                                int n_hist, double h_frac, const int64_t* pixels, int64_t count,
                                const uint8_t* status, float* mo, float* resid, void* stream) {
    if (!d) {
        set_error("bfm_trace: design handle is NULL");
        return BFM_EINVAL;
    }
    if (dtype != BFM_F32 && dtype != BFM_I16) {
        set_error("bfm_trace: dtype is not BFM_F32 or BFM_I16");
        return BFM_EINVAL;
    }
    if (m < 1 || count < 0) {
        set_error("bfm_trace: needs m >= 1 and count >= 0");
        return BFM_EINVAL;
    }
    if (!(n_hist >= 1 && n_hist < d->N)) {
        set_error("bfm_trace: n_hist outside 1 <= n_hist < N");
        return BFM_EINVAL;
    }
    if (!(h_frac > 0.0 && h_frac <= 1.0)) {
        set_error("bfm_trace: h_frac outside (0, 1]");
        return BFM_EINVAL;
    }
    if (count == 0) return BFM_OK;
    if (!Y || !status || (!mo && !resid)) {
        set_error("bfm_trace: Y, status and at least one of mo, resid must be non-NULL device pointers");
        return BFM_EINVAL;
    }
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != d->device) {
        set_error("bfm_trace: the design belongs to another device");
        return BFM_EINVAL;
    }
    TraceParams P{};
    P.Y = Y;
    P.mask = mask_bits;
    P.m = m;
    P.mask_words = (m + 31) / 32;
    P.N = d->N;
    P.n_hist = n_hist;
    P.dtype = dtype;
    P.h_frac = h_frac;
    P.x = d->d_xd;
    P.pixels = pixels;
    P.count = count;
    P.status = status;
    P.mo = mo;
    P.resid = resid;
    const size_t per_warp = (size_t)kBytesPerDate * (size_t)d->N;
    int warps = (int)(kSmemTarget / per_warp);
    warps = warps < 1 ? 1 : (warps > kMaxWarps ? kMaxWarps : warps);
    const int64_t grid = (count + warps - 1) / warps;
    if (grid > 0x7fffffffLL) {
        set_error("bfm_trace: count too large for one call");
        return BFM_EUNSUPPORTED;
    }
    const size_t smem = per_warp * (size_t)warps;
    cudaStream_t st = (cudaStream_t)stream;
    if (d->k == 1)
        trace_kernel<1><<<(unsigned)grid, 32 * warps, smem, st>>>(P);
    else if (d->k == 2)
        trace_kernel<2><<<(unsigned)grid, 32 * warps, smem, st>>>(P);
    else
        trace_kernel<3><<<(unsigned)grid, 32 * warps, smem, st>>>(P);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "bfm_trace: launch");
    return BFM_OK;
}
