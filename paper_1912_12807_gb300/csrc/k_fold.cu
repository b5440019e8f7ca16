// Folding of candidates' dedispersed series on a grid of trial frequencies
// (the prepfold step, paper Sect. 2 step 6).
//
// One CTA folds one (candidate, trial frequency): sample j has phase
// j x + j^2 g cycles (x = f dt, g = (fdot/2) dt^2) carried in 64-bit fixed
// point (X, G: rint(x 2^64), rint(g 2^64) modulo 2^64, rounded to nearest
// even from the exact binary values of the FP64 x and g formed with
// round-to-nearest intrinsics in the host's order; a negative g wraps),
// phase_j = j X + j^2 G modulo 2^64, and bin floor(phase_j nbin / 2^64) (the
// high word of the 128-bit product): integer arithmetic, so every sample
// lands in the bin the host reading assigns it, with no FP64 per sample.  The
// phase advances by d_j = X + (2 j + 1) G and d_j by 2 G, and
// (phase nbin) >> 64 is two 32-bit products (nbin < 2^32).
//
// A warp copies 32 RUN consecutive samples to shared memory (coalesced), then
// each lane walks RUN consecutive ones (an odd stride: distinct banks) and adds
// them with shared-memory atomics: a run of equal bins at once where a bin
// holds more than two samples, else every sample.  The bins are 32-bit
// (64-bit shared-memory atomics are loops) and are added to the 64-bit profile
// before they can overflow: every `rounds` tiles of all warps.  The profile
// and counts are exact integers.  The threads form the bins' chi-square terms
// against a flat profile and thread 0 sums them in order.
//
// Bound: issue and the atomics' bank conflicts.  64 candidates x 9 frequencies
// x 257 689 samples: 0.95 ms with each thread reading its own 4 KB run from
// global memory (32 cache lines per load) and 64-bit products and atomics per
// sample, 0.56 ms with coalesced tiles, 0.22 ms with 32-bit bins; RUN 47
// keeps four CTAs per SM.
#include "pss_internal.h"

namespace pss {

namespace {

constexpr int NT = 256;
constexpr int RUN = 47;                // consecutive samples of a lane (odd)
constexpr int TILE = 32 * RUN;         // samples of a warp's tile

// rint(v 2^64) modulo 2^64, round half to even: v - trunc(v) is exact in FP64
// and lies in (-1, 1), its scaling by 2^64 is exact, and a negative fraction
// wraps (2^64 - rint(|r| 2^64))
__device__ __forceinline__ unsigned long long fixed_point(double v) {
    const double r = __dsub_rn(v, trunc(v));
    if (r >= 0.0) return __double2ull_rn(ldexp(r, 64));
    return 0ull - __double2ull_rn(ldexp(-r, 64));
}

__global__ void __launch_bounds__(NT) k_fold(const __grid_constant__ FoldArgs a, int rounds) {
    // P [nbin], n [nbin] (u32), 32-bit sums [nbin] (u32, rounds > 0), staged samples [NT / 32][TILE] (then the
    // chi-square terms)
    extern __shared__ __align__(16) unsigned long long sm[];
    unsigned long long* P = sm;
    unsigned int* cnt = reinterpret_cast<unsigned int*>(sm + a.nbin);
    unsigned int* part = cnt + a.nbin;
    int32_t* stage = reinterpret_cast<int32_t*>(sm + 2 * a.nbin);
    const int r = blockIdx.x / a.nfreq, k = blockIdx.x - r * a.nfreq;
    const FoldItem it = a.items[r];
    __shared__ unsigned long long s_xg[2];
    __shared__ double s_f, s_mu, s_var;
    for (int b = threadIdx.x; b < a.nbin; b += NT) {
        P[b] = 0ull;
        cnt[b] = 0u;
        part[b] = 0u;
    }
    // FP64 is slow: one thread each forms the phase step and the moments
    if (threadIdx.x == 0) {
        const double f = __dadd_rn(it.f, __dmul_rn(__dsub_rn((double)k, __ddiv_rn((double)(a.nfreq - 1), 2.0)),
                                                   __ddiv_rn(a.step_bins, it.T)));
        // per-sample phase step x = f dt and drift g = (fdot / 2) dt^2 in 64-bit
        // fixed point (2^-64 cycle, modulo one cycle), rounded to nearest even
        s_xg[0] = fixed_point(__dmul_rn(f, it.dt));
        s_xg[1] = fixed_point(__dmul_rn(__dmul_rn(0.5, it.fdot), __dmul_rn(it.dt, it.dt)));
        s_f = f;
    } else if (threadIdx.x == 32) {
        const double fS1 = (double)it.s1, fS2 = (double)it.s2, fN = (double)it.n;
        s_mu = __ddiv_rn(fS1, fN);
        s_var = __ddiv_rn(__dsub_rn(fS2, __ddiv_rn(__dmul_rn(fS1, fS1), fN)), fN);
    }
    __syncthreads();
    const unsigned long long X = s_xg[0], G = s_xg[1], G2 = 2 * G;
    const uint32_t nb = (uint32_t)a.nbin;
    const int32_t* s = a.series + (int64_t)it.row * a.stride;
    const int64_t n = it.n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t* st = stage + warp * TILE;
    // bins per sample >= 1/2: most runs are one sample long
    const bool single = rounds > 0 && __umul64hi(X, 2ull * nb) >= 1;
    int round = 0;
    for (int64_t c0 = 0; c0 < n; c0 += (int64_t)(NT / 32) * TILE) {
        const int64_t j0 = c0 + (int64_t)warp * TILE;
        const int len = (int)max((int64_t)0, min((int64_t)TILE, n - j0));
#pragma unroll 16
        for (int q = lane; q < TILE; q += 32)
            if (q < len) st[q] = s[j0 + q];
        __syncwarp();
        const unsigned long long ju = (unsigned long long)(j0 + lane * RUN);
        unsigned long long ph = ju * X + (ju * ju) * G;  // wraps modulo 2^64: one cycle
        unsigned long long d = X + (2 * ju + 1) * G;
        const int mine = max(0, min(RUN, len - lane * RUN));
        const int32_t* my = st + lane * RUN;
        auto next_bin = [&]() -> uint32_t {
            const uint32_t hi = (uint32_t)(ph >> 32), lo = (uint32_t)ph;
            ph += d;
            d += G2;
            return (uint32_t)(((unsigned long long)hi * nb + __umulhi(lo, nb)) >> 32);
        };
        if (single) {
#pragma unroll 4
            for (int q = 0; q < mine; ++q) {
                const uint32_t bin = next_bin();
                atomicAdd(part + bin, (uint32_t)my[q]);
                atomicAdd(cnt + bin, 1u);
            }
        } else {
            uint32_t cur = 0, c = 0;
            unsigned long long acc = 0ull;
            auto flush = [&]() {
                if (rounds > 0) atomicAdd(part + cur, (uint32_t)acc);
                else atomicAdd(P + cur, acc);
                atomicAdd(cnt + cur, c);
            };
            for (int q = 0; q < mine; ++q) {
                const uint32_t v = (uint32_t)my[q], bin = next_bin();
                if (bin != cur) {
                    if (c) flush();
                    cur = bin;
                    acc = 0ull;
                    c = 0u;
                }
                acc += v;
                ++c;
            }
            if (c) flush();
        }
        __syncwarp();  // the tile is read: the next one overwrites it
        if (rounds > 0 && ++round == rounds) {
            round = 0;
            __syncthreads();
            for (int b = threadIdx.x; b < a.nbin; b += NT) {
                P[b] += part[b];
                part[b] = 0u;
            }
            __syncthreads();
        }
    }
    __syncthreads();
    if (rounds > 0)
        for (int b = threadIdx.x; b < a.nbin; b += NT) P[b] += part[b];
    __syncthreads();
    const int64_t o = (int64_t)blockIdx.x * a.nbin;
    for (int b = threadIdx.x; b < a.nbin; b += NT) {
        a.prof[o + b] = (long long)P[b];
        a.counts[o + b] = (long long)cnt[b];
    }
    const double mu = s_mu, var = s_var;
    double* term = reinterpret_cast<double*>(stage);
    if (var > 0.0)
        for (int b = threadIdx.x; b < a.nbin; b += NT) {
            if (cnt[b] == 0u) continue;
            const double nbv = (double)cnt[b];
            const double d = __dsub_rn((double)(long long)P[b], __dmul_rn(nbv, mu));
            term[b] = __ddiv_rn(__dmul_rn(d, d), __dmul_rn(nbv, var));
        }
    __syncthreads();
    if (threadIdx.x == 0) {
        double chi = 0.0;
        if (var > 0.0) {
            double sum = 0.0;
            int used = 0;
            for (int b = 0; b < a.nbin; ++b) {
                if (cnt[b] == 0u) continue;
                sum = __dadd_rn(sum, term[b]);
                ++used;
            }
            chi = used > 1 ? __ddiv_rn(sum, (double)(used - 1)) : 0.0;
        }
        a.chi2[blockIdx.x] = chi;
        a.freq[blockIdx.x] = s_f;
    }
}

}  // namespace

cudaError_t launch_fold(const FoldArgs& a, int64_t nitems, cudaStream_t s) {
    if (nitems <= 0) return cudaSuccess;
    if (a.nbin < 2 || a.nbin > 1024 || a.nfreq < 1 || a.nfreq > 64) return cudaErrorInvalidValue;
    static_assert((NT / 32) * TILE * sizeof(int32_t) >= 1024 * sizeof(double), "the terms fit over the staged samples");
    const size_t shm = 2 * (size_t)a.nbin * sizeof(unsigned long long) + (size_t)(NT / 32) * TILE * sizeof(int32_t);
    // tiles of all warps whose samples cannot overflow a 32-bit bin (0: 64-bit atomics)
    int rounds = 0;
    if (a.max_value > 0) rounds = (int)std::min<long long>(0xFFFFFFFFll / ((long long)(NT / 32) * TILE * a.max_value), 1 << 20);
    cudaError_t e = allow_smem((const void*)k_fold, shm);
    if (e != cudaSuccess) return e;
    k_fold<<<(unsigned)(nitems * a.nfreq), NT, shm, s>>>(a, rounds);
    return cudaGetLastError();
}

}  // namespace pss
