// Single-pulse (boxcar matched-filter) search of dedispersed series: the
// step after dedispersion in the paper's pipeline (single_pulse_search.py,
// Sect. 2 step 7; long-period pulsars are found this way, Sect. 5.3).
//
// Per trial: mu = S1/N and sigma = sqrt((S2 - S1*S1/N)/N) from the exact
// integer moments S1 = sum s, S2 = sum s^2; for each boxcar width w,
// B_w[t] = sum_{k<w} s[t+k] (exact, t <= N - w) is a detection when
// B_w[t] >= w*mu + thr*sigma*sqrt(w) and it is a local maximum over its
// own width (strictly above the w - 1 values before it, not below the
// w - 1 after it).  The FP64 arithmetic is written with round-to-nearest
// intrinsics in the stated order so that no multiply-add is contracted and
// the threshold is the same number the host computes.
//
// k_sp_moments: one pass over the series, 64-bit integer sums.
// k_sp_thresholds: the integer threshold of every (trial, width), FP64.
// k_sp_detect: a CTA owns TS samples of one trial; it stages the samples
// [t0 - wmax + 1, t0 + TS + 2 wmax - 2] in shared memory as a prefix sum, so
// every B_w that the tile and its local-maximum windows need is one
// subtraction.  The sums are 32-bit modulo 2^32 when every window sum is below
// 2^31 (a difference is then exact), else 64-bit.  A thread keeps the prefix
// sums of its PT starts (256 apart: consecutive lanes, distinct banks) in
// registers and, per width, reads one more per start and compares the largest
// window sum with the threshold; the windows themselves are looked at only
// where it is reached.  Detections are appended with an atomic counter; past
// `cap` they are only counted.
//
// Bound: issue and shared-memory reads, about 3 instructions per start and
// width.  1001 trials x 257 689 samples, 13 widths: 2.64 ms with one branch
// per start and width and segment-wise (uncoalesced) staging, 1.03 ms
// here; tiles of 4096 keep the 450 staged neighbours at 11 %.
#include <limits.h>

#include "pss_internal.h"

namespace pss {

namespace {

constexpr int NT = 256;
constexpr int SP_CTAS = 4;  // CTAs per SM
// Samples per CTA (TS): tiles of 4096 stage few neighbours; a launch that then has fewer CTAs than fit the device at
// once takes tiles of 1024, which have a quarter of the serial work per CTA.  2^18 samples, 13
// widths, whole call: one trial 259 us with tiles of 4096 and 240 us with 1024, 8 trials 356 and 339 us.
constexpr int TS_LARGE = 4096, TS_SMALL = 1024;

__global__ void __launch_bounds__(NT) k_sp_moments(const int32_t* __restrict__ series, int64_t stride, int64_t n,
                                                   unsigned long long* s1, unsigned long long* s2) {
    const int b = blockIdx.y;
    const int32_t* s = series + (int64_t)b * stride;
    unsigned long long a1 = 0ull, a2 = 0ull;
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < n; i += (int64_t)gridDim.x * NT) {
        const unsigned long long v = (unsigned long long)(uint32_t)s[i];
        a1 += v;
        a2 += v * v;
    }
    for (int off = 16; off > 0; off >>= 1) {
        a1 += __shfl_xor_sync(0xffffffffu, a1, off);
        a2 += __shfl_xor_sync(0xffffffffu, a2, off);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(s1 + b, a1);
        atomicAdd(s2 + b, a2);
    }
}

// One thread per (trial, width): the integer threshold ceil(w*mu +
// thr*sigma*sqrt(w)) (B is an integer below 2^53, exact as a double, so
// (double)B >= thr exactly when B >= ceil(thr)); LLONG_MAX when sigma is 0.
__global__ void k_sp_thresholds(const __grid_constant__ SpArgs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.nb * a.nw) return;
    const int b = i / a.nw, wi = i - b * a.nw;
    const double fS1 = (double)a.s1[b], fS2 = (double)a.s2[b], fN = (double)a.n;
    const double mu = __ddiv_rn(fS1, fN);
    double var = __ddiv_rn(__dsub_rn(fS2, __ddiv_rn(__dmul_rn(fS1, fS1), fN)), fN);
    if (!(var > 0.0)) var = 0.0;
    const double sigma = __dsqrt_rn(var);
    long long t = LLONG_MAX;
    if (sigma > 0.0) {
        const double w = (double)a.w[wi];
        const double thr = __dadd_rn(__dmul_rn(w, mu), __dmul_rn(__dmul_rn(a.thr, sigma), __dsqrt_rn(w)));
        const double c = ceil(thr);
        t = c > 9.0e18 ? LLONG_MAX : (c < -9.0e18 ? LLONG_MIN : (long long)c);
    }
    a.thr_tab[i] = t;
}

// The windows of width w starting at t = t0 + tid + 256 i with sum B >= thr: kept when they are the local maximum
// (called by whole warps).  A lane looks at its NEAR neighbours on either side, nearest first (on the flank of a pulse
// the next window decides); what is left is looked at by the warp together, 32 distances at a time.  One trial of 2^18
// samples with a burst, widths 1 and 1000, whole call: 299 us with a lane walking all 1998 neighbours, 217 us here.
constexpr int NEAR = 8;
template <typename T, typename S>
__device__ __noinline__ void sp_hits(const SpArgs& a, const T* R, int64_t base, int b, int w, S thr, int64_t t0,
                                     int64_t tend, int64_t tmax) {
    const int lane = threadIdx.x & 31;
    auto sum = [&](int64_t u) { return (S)(R[u + w - base] - R[u - base]); };
    for (int64_t tb = t0; tb <= tend; tb += NT) {
        const int64_t t = tb + threadIdx.x;
        S B = 0;
        bool ok = t <= tend;
        if (ok) {
            B = sum(t);
            ok = B >= thr;
        }
        const int near = min(NEAR, w - 1);
        for (int k = 1; k <= near && ok; ++k) ok = t - k < 0 || B > sum(t - k);
        for (int k = 1; k <= near && ok; ++k) ok = t + k > tmax || B >= sum(t + k);
        if (w - 1 > NEAR)
            for (uint32_t m = __ballot_sync(0xffffffffu, ok); m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                const int64_t tt = __shfl_sync(0xffffffffu, (long long)t, src);
                const S BB = __shfl_sync(0xffffffffu, B, src);
                bool bad = false;
                for (int k0 = NEAR + 1; k0 < w && !bad; k0 += 32) {
                    const int k = k0 + lane;
                    if (k < w) bad = (tt - k >= 0 && BB <= sum(tt - k)) || (tt + k <= tmax && BB < sum(tt + k));
                    bad = __any_sync(0xffffffffu, bad);
                }
                if (bad && lane == src) ok = false;
            }
        if (!ok) continue;
        const unsigned long long slot = atomicAdd(a.count, 1ull);
        if ((int64_t)slot < a.cap) {
            SpRaw e;
            e.dm_idx = a.dm0 + b;
            e.w = w;
            e.t = t;
            e.B = (int64_t)B;
            a.out[slot] = e;
        }
    }
}

// T: the prefix sums' type (modulo its range), S: the window sums' (signed).
template <typename T, typename S, int TS>
__global__ void __launch_bounds__(NT, SP_CTAS) k_sp_detect(const __grid_constant__ SpArgs a) {
    constexpr int PT = TS / NT;  // boxcar starts per thread
    extern __shared__ __align__(16) unsigned char sp_raw[];
    T* R = reinterpret_cast<T*>(sp_raw);  // R[k]: sum of the k samples from `base` on
    __shared__ T s_tot[NT / 32];
    const int b = blockIdx.y;
    const int64_t n = a.n;
    const int64_t t0 = (int64_t)blockIdx.x * TS;
    const int32_t* s = a.series + (int64_t)b * a.stride;
    const long long* thr_b = a.thr_tab + (int64_t)b * a.nw;
    if (thr_b[0] == LLONG_MAX) return;  // sigma 0: no detections (uniform over the CTA)
    const int64_t base = max((int64_t)0, t0 - a.wmax + 1);
    const int64_t last = min(n, t0 + TS + 2 * (int64_t)a.wmax - 2);  // largest prefix index needed
    const int L = (int)(last - base);                                // samples staged
    const int C = TS + 3 * a.wmax;                                   // prefix sums kept (the last value past the samples)
#pragma unroll 8
    for (int k = threadIdx.x; k < C; k += NT) R[k + 1] = k < L ? (T)(uint32_t)__ldg(s + base + k) : (T)0;
    if (threadIdx.x == 0) R[0] = 0;
    __syncthreads();
    // per-thread segment sums (an odd stride: distinct banks), a block scan of them, and the sums in place
    const int seg = ((C + NT - 1) / NT) | 1;
    const int k0 = threadIdx.x * seg, k1 = min(C, k0 + seg);
    T tot = 0;
    for (int k = k0; k < k1; ++k) tot += R[k + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T incl = tot;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const T u = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += u;
    }
    if (lane == 31) s_tot[warp] = incl;
    __syncthreads();
    T run = incl - tot;
    for (int w = 0; w < warp; ++w) run += s_tot[w];
    for (int k = k0; k < k1; ++k) {
        run += R[k + 1];
        R[k + 1] = run;
    }
    __syncthreads();
    const T* Rt = R + (t0 - base) + threadIdx.x;
    T r0[PT];
#pragma unroll
    for (int i = 0; i < PT; ++i) r0[i] = Rt[i * NT];
    for (int i = 0; i < a.nw; ++i) {
        const int w = a.w[i];
        const int64_t tmax = n - w;  // last valid boxcar start
        if (tmax < t0) continue;
        // a threshold beyond S's range can never be met by a window sum that fits S
        const long long thr64 = thr_b[i];
        constexpr long long SMAX = sizeof(S) == 4 ? (long long)INT_MAX : LLONG_MAX;
        constexpr long long SMIN = sizeof(S) == 4 ? (long long)INT_MIN : LLONG_MIN;
        if (thr64 > SMAX) continue;
        const S thr = (S)(thr64 < SMIN ? SMIN : thr64);
        const T* Rw = Rt + w;
        S mx = (S)(Rw[0] - r0[0]);
#pragma unroll
        for (int q = 1; q < PT; ++q) mx = max(mx, (S)(Rw[q * NT] - r0[q]));
        // (starts past tmax are in mx too: their windows are cut off, and sp_hits leaves them out)
        if (__any_sync(0xffffffffu, mx >= thr)) sp_hits<T, S>(a, R, base, b, w, thr, t0, min(t0 + TS - 1, tmax), tmax);
    }
}

}  // namespace

// 32-bit prefix sums (modulo 2^32) suffice when every window sum is below 2^31
bool sp_narrow(const SpArgs& a) {
    return a.max_value >= 0 && (long long)a.wmax * a.max_value < (1ll << 31) - 1;
}

template <typename T, typename S, int TS>
cudaError_t launch_detect_t(const SpArgs& a, cudaStream_t s) {
    const size_t shm = (size_t)(TS + 3 * a.wmax + 1) * sizeof(T);
    cudaError_t e = allow_smem((const void*)k_sp_detect<T, S, TS>, shm);
    if (e != cudaSuccess) return e;
    dim3 gd((unsigned)((a.n + TS - 1) / TS), (unsigned)a.nb);
    k_sp_detect<T, S, TS><<<gd, NT, shm, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_detect(const SpArgs& a, cudaStream_t s) {
    const bool large = (a.n + TS_LARGE - 1) / TS_LARGE * a.nb >= (int64_t)(a.num_sms > 0 ? a.num_sms : 152) * SP_CTAS;
    if (sp_narrow(a))
        return large ? launch_detect_t<uint32_t, int32_t, TS_LARGE>(a, s) : launch_detect_t<uint32_t, int32_t, TS_SMALL>(a, s);
    return large ? launch_detect_t<unsigned long long, long long, TS_LARGE>(a, s)
                 : launch_detect_t<unsigned long long, long long, TS_SMALL>(a, s);
}

cudaError_t launch_single_pulse(const SpArgs& a, unsigned long long* s1, unsigned long long* s2, bool have_moments,
                                cudaStream_t s) {
    if (a.nb <= 0 || a.n <= 0) return cudaSuccess;
    if (a.nw < 1 || a.nw > SP_MAXW || a.wmax < 1 || a.wmax > SP_MAXWIDTH) return cudaErrorInvalidValue;
    cudaError_t e = have_moments ? cudaSuccess : launch_sp_moments(a.series, a.stride, a.n, a.nb, s1, s2, s);
    if (e != cudaSuccess) return e;
    k_sp_thresholds<<<(unsigned)((a.nb * a.nw + 127) / 128), 128, 0, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_detect(a, s);
}

cudaError_t launch_sp_moments(const int32_t* series, int64_t stride, int64_t n, int32_t nb, unsigned long long* s1,
                              unsigned long long* s2, cudaStream_t s) {
    if (nb <= 0 || n <= 0) return cudaSuccess;
    dim3 gm((unsigned)std::min<int64_t>((n + NT - 1) / NT, 64), (unsigned)nb);
    k_sp_moments<<<gm, NT, 0, s>>>(series, stride, n, s1, s2);
    return cudaGetLastError();
}

cudaError_t launch_sp_detect_only(const SpArgs& a, cudaStream_t s) {
    if (a.nb <= 0 || a.n <= 0) return cudaSuccess;
    return launch_detect(a, s);
}

}  // namespace pss
