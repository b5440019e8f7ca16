// Harmonic summing, thresholding and candidate compaction (the paper's
// accelsearch, Sect. 2 step 4).
//
// For stage n = 2^s (1, 2, 4, .., numharm) the plane point (h, j) is taken
// as the n-th harmonic; its k-th harmonic is at half-bin
// h_k = floor((2kh + n)/(2n)) = (2kh + n) >> (s+1) and row
// j_k = Z + sgn(j-Z) ((2k|j-Z| + n) >> (s+1)), so
//   S_n(h, j) = sum_{k=1..n} P[j_k][h_k].
// Because h_{2m} at stage n equals h_m at stage n/2 (and likewise for rows),
// S_n = S_{n/2} + sum over odd k of P[j_k][h_k]: each stage adds only its odd
// harmonics to the previous stage's sums, kept in shared memory.
//
// A CTA owns a tile of TR rows x TH half-bins and keeps S for the tile plus
// a one-point halo, so the 3x3 local-maximum test (strictly larger than
// every in-plane neighbour, exact ties to the lower linear index j*nfft+h)
// needs no second pass.  Points that pass the stage threshold and the
// f >= f_lo cut are compacted with a warp ballot and one atomic per warp;
// the global counter always counts, so an overflow of `cap` is detected.
#include <math.h>
#include <stdlib.h>

#include "pss_internal.h"

namespace pss {

namespace {

constexpr int NT = 256;

struct Tile {
    int h0, j0, jlo, r0, halo_n, nfft, lane, b;
    const float* P;
};

// Stage SI (n = 2^SI): add the odd harmonics to the sums held in S, then
// test and compact the tile's points.  TR x TH is the tile; ONE_ROW is the
// zmax = 0 case (a single plane row, no row arithmetic).
template <int SI, int TR, int TH, bool ONE_ROW>
__device__ __forceinline__ void harm_stage(const HarmArgs& a, const Tile& t, float* S, const float* s_thr,
                                           const int* s_hmin) {
    constexpr int n = 1 << SI;
    constexpr int sh = SI + 1;
    constexpr int SW = TH + 2;
    for (int x = threadIdx.x; x < t.halo_n; x += NT) {
        const int rr = ONE_ROW ? 0 : x / SW;
        const int hc = ONE_ROW ? x : x - rr * SW;
        const int j = t.jlo + rr;
        const int h = t.h0 - 1 + hc;
        float* dst = S + (t.r0 + rr) * SW + hc;
        if (h < 0 || h >= t.nfft) {
            *dst = -INFINITY;
            continue;
        }
        float acc;
        if constexpr (SI == 0) {
            acc = __ldg(t.P + (ONE_ROW ? 0 : j * t.nfft) + h);
        } else {
            // the n/2 odd harmonics: independent loads, issued together
            float v[n / 2];
            const int h2 = 2 * h;
            if constexpr (ONE_ROW) {
#pragma unroll
                for (int q = 0; q < n / 2; ++q) v[q] = __ldg(t.P + (((2 * q + 1) * h2 + n) >> sh));
            } else {
                const int d = j - a.Z;
                const int ad2 = 2 * (d < 0 ? -d : d);
#pragma unroll
                for (int q = 0; q < n / 2; ++q) {
                    const int k = 2 * q + 1;
                    const int dk = (k * ad2 + n) >> sh;
                    const int jk = d < 0 ? a.Z - dk : a.Z + dk;
                    v[q] = __ldg(t.P + jk * t.nfft + ((k * h2 + n) >> sh));
                }
            }
            acc = *dst;
#pragma unroll
            for (int q = 0; q < n / 2; ++q) acc += v[q];
        }
        *dst = acc;
    }
    __syncthreads();
    const float thr = s_thr[SI];
    const int hmin = s_hmin[SI];
    constexpr int npts = TR * TH;
#pragma unroll 1
    for (int base = 0; base < npts; base += NT) {
        const int p = base + threadIdx.x;
        bool hit = false;
        int j = 0, h = 0;
        float s = 0.f;
        if (p < npts) {
            const int jr = p / TH, hc = p - jr * TH;
            j = t.j0 + jr;
            h = t.h0 + hc;
            if (j < a.nz && h < t.nfft && h >= hmin) {
                const int x = (jr + 1) * SW + hc + 1;
                s = S[x];
                if (s >= thr) {
                    hit = true;
#pragma unroll
                    for (int dj = -1; dj <= 1; ++dj) {
                        if (ONE_ROW && dj != 0) continue;
                        if (j + dj < 0 || j + dj >= a.nz) continue;
#pragma unroll
                        for (int dh = -1; dh <= 1; ++dh) {
                            if (dj == 0 && dh == 0) continue;
                            const float nb = S[x + dj * SW + dh];
                            // the neighbour's linear index is larger iff (dj, dh) > (0, 0)
                            const bool nb_later = (dj > 0) || (dj == 0 && dh > 0);
                            if (!(s > nb || (s == nb && nb_later))) hit = false;
                        }
                    }
                }
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (m) {
            unsigned long long slot0 = 0ull;
            if (t.lane == 0) slot0 = atomicAdd(a.counter, (unsigned long long)__popc(m));
            slot0 = __shfl_sync(0xffffffffu, slot0, 0);
            if (hit) {
                const unsigned long long slot = slot0 + __popc(m & ((1u << t.lane) - 1u));
                if ((int64_t)slot < a.cap) {
                    pss_raw_cand c;
                    c.dm_idx = a.row_dm ? a.row_dm[t.b] : a.dm0 + t.b;
                    c.numharm = n;
                    c.h = h;
                    c.j = j;
                    c.power = s;
                    c.reserved = a.row_file ? a.row_file[t.b] : 0;
                    a.out[slot] = c;
                }
            }
        }
    }
    __syncthreads();
}

template <int SI, int NSTAGES, int TR, int TH, bool ONE_ROW>
__device__ __forceinline__ void harm_stages(const HarmArgs& a, const Tile& t, float* S, const float* s_thr,
                                            const int* s_hmin) {
    if constexpr (SI < NSTAGES) {
        harm_stage<SI, TR, TH, ONE_ROW>(a, t, S, s_thr, s_hmin);
        harm_stages<SI + 1, NSTAGES, TR, TH, ONE_ROW>(a, t, S, s_thr, s_hmin);
    }
}

template <int NSTAGES, int TR, int TH, bool ONE_ROW>
__global__ void __launch_bounds__(NT) k_harm(const __grid_constant__ HarmArgs a) {
    __shared__ float S[(TR + 2) * (TH + 2)];  // row r <-> j = j0 - 1 + r
    __shared__ float s_thr[8];
    __shared__ int s_hmin[8];
#pragma unroll
    for (int q = 0; q < 6; ++q)
        if (threadIdx.x == q) {  // constant indices keep the parameter block out of local memory
            s_thr[q] = a.thr[q];
            s_hmin[q] = a.row_hmin ? a.row_hmin[8 * blockIdx.z + q] : a.hmin[q];
        }
    Tile t;
    t.b = blockIdx.z;
    t.h0 = blockIdx.x * TH;
    t.j0 = blockIdx.y * TR;
    t.nfft = (int)a.nfft;
    t.P = a.plane + (int64_t)t.b * a.plane_stride;
    // rows of the plane present in tile + halo
    t.jlo = ONE_ROW ? 0 : max(t.j0 - 1, 0);
    const int jhi = ONE_ROW ? 1 : min(t.j0 + TR + 1, a.nz);
    t.r0 = t.jlo - (t.j0 - 1);
    t.halo_n = (jhi - t.jlo) * (TH + 2);
    t.lane = threadIdx.x & 31;
    __syncthreads();
    harm_stages<0, NSTAGES, TR, TH, ONE_ROW>(a, t, S, s_thr, s_hmin);
}

template <int TR, int TH, bool ONE_ROW>
cudaError_t launch_variant(const HarmArgs& a, cudaStream_t s) {
    dim3 grid((unsigned)((a.nfft + TH - 1) / TH), (unsigned)((a.nz + TR - 1) / TR), (unsigned)a.nb);
    switch (a.nstages) {
        case 1: k_harm<1, TR, TH, ONE_ROW><<<grid, NT, 0, s>>>(a); break;
        case 2: k_harm<2, TR, TH, ONE_ROW><<<grid, NT, 0, s>>>(a); break;
        case 3: k_harm<3, TR, TH, ONE_ROW><<<grid, NT, 0, s>>>(a); break;
        case 4: k_harm<4, TR, TH, ONE_ROW><<<grid, NT, 0, s>>>(a); break;
        case 5: k_harm<5, TR, TH, ONE_ROW><<<grid, NT, 0, s>>>(a); break;
        case 6: k_harm<6, TR, TH, ONE_ROW><<<grid, NT, 0, s>>>(a); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// ---- register-blocked variant ------------------------------------------------
//
// A warp owns WR = 32 R consecutive half-bins of one plane row j; lane l
// holds the sums of the points h = hw + l + 32 i (i < R) in registers.  For
// stage n and odd harmonic k, point (h, j) reads row j_k (the same for the
// whole warp) at half-bin (2kh + n) >> (s+1); stepping h by 32 steps that
// index by exactly 32k/n (an integer for n <= 32), so one index computation
// per harmonic serves all R points and the loads use compile-time offsets,
// each coalesced across the warp.  Additions happen in the order of k_harm
// (stage by stage, odd k increasing), so the sums are bit-identical.
// Threshold tests run on the lane's maximum; a warp with a point above
// threshold takes same-row neighbours from adjacent lanes and recomputes any
// other neighbour (warp edges, rows j +- 1) from the plane.

// S_n at (h, j) from the plane (the same additions in the same order).
template <int SI>
__device__ float harm_sum_at(const float* P, int h, int j, int nfft, int nz, int Z) {
    if (h < 0 || h >= nfft || j < 0 || j >= nz) return -INFINITY;
    float acc = __ldg(P + j * nfft + h);
    const int d = j - Z, ad2 = 2 * (d < 0 ? -d : d);
#pragma unroll
    for (int s = 1; s <= SI; ++s) {
        const int n = 1 << s;
        for (int q = 0; q < n / 2; ++q) {
            const int k = 2 * q + 1;
            const int dk = (k * ad2 + n) >> (s + 1);
            const int jk = d < 0 ? Z - dk : Z + dk;
            acc += __ldg(P + jk * nfft + ((2 * k * h + n) >> (s + 1)));
        }
    }
    return acc;
}

// The same sum for the tiles' rare path, whose few warps hide no latency: every load issued before the first addition.
template <int SI>
__device__ __forceinline__ float harm_sum_ahead(const float* P, int h, int j, int nfft, int nz, int Z) {
    if (h < 0 || h >= nfft || j < 0 || j >= nz) return -INFINITY;
    const int d = j - Z, ad2 = 2 * (d < 0 ? -d : d);
    float v[1 << SI];
    v[0] = __ldg(P + j * nfft + h);
#pragma unroll
    for (int s = 1; s <= SI; ++s) {
        const int n = 1 << s;
#pragma unroll
        for (int q = 0; q < n / 2; ++q) {
            const int k = 2 * q + 1;
            const int dk = (k * ad2 + n) >> (s + 1);
            const int jk = d < 0 ? Z - dk : Z + dk;
            v[n / 2 + q] = __ldg(P + jk * nfft + ((2 * k * h + n) >> (s + 1)));
        }
    }
    float acc = v[0];
#pragma unroll
    for (int t = 1; t < 1 << SI; ++t) acc += v[t];
    return acc;
}

template <int SI, int R>
__device__ __forceinline__ void reg_test(const HarmArgs& a, const float* P, const float (&acc)[R], int hw, int j,
                                         int lane, int b) {
    const float thr = a.thr[SI];
    float mx = acc[0];
#pragma unroll
    for (int i = 1; i < R; ++i) mx = fmaxf(mx, acc[i]);
    if (!__any_sync(0xffffffffu, mx >= thr)) return;
    const int nfft = (int)a.nfft, hmin = a.row_hmin ? a.row_hmin[8 * b + SI] : a.hmin[SI], nz = a.nz, Z = a.Z;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        float left = __shfl_up_sync(0xffffffffu, acc[i], 1);
        float right = __shfl_down_sync(0xffffffffu, acc[i], 1);
        const float l31 = __shfl_sync(0xffffffffu, acc[i > 0 ? i - 1 : 0], 31);
        const float r0 = __shfl_sync(0xffffffffu, acc[i < R - 1 ? i + 1 : R - 1], 0);
        const float s = acc[i];
        const int h = hw + lane + 32 * i;
        if (s >= thr && h >= hmin) {
            if (lane == 0) left = i > 0 ? l31 : harm_sum_at<SI>(P, hw - 1, j, nfft, nz, Z);
            if (lane == 31) right = i < R - 1 ? r0 : harm_sum_at<SI>(P, hw + 32 * R, j, nfft, nz, Z);
            // strictly above every earlier neighbour, ties to the lower index against later ones
            bool hit = s > left && s >= right;
            if (nz > 1) {
#pragma unroll
                for (int dh = -1; dh <= 1; ++dh) {
                    if (!hit) break;
                    hit = s > harm_sum_at<SI>(P, h + dh, j - 1, nfft, nz, Z) &&
                          s >= harm_sum_at<SI>(P, h + dh, j + 1, nfft, nz, Z);
                }
            }
            if (hit) {
                const unsigned long long slot = atomicAdd(a.counter, 1ull);
                if ((int64_t)slot < a.cap) {
                    pss_raw_cand c;
                    c.dm_idx = a.row_dm ? a.row_dm[b] : a.dm0 + b;
                    c.numharm = 1 << SI;
                    c.h = h;
                    c.j = j;
                    c.power = s;
                    c.reserved = a.row_file ? a.row_file[b] : 0;
                    a.out[slot] = c;
                }
            }
        }
    }
}

template <int SI, int NSTAGES, int R>
__device__ __forceinline__ void reg_stages(const HarmArgs& a, const float* P, float (&acc)[R], int hw, int j,
                                           int lane, int b) {
    if constexpr (SI < NSTAGES) {
        if constexpr (SI > 0) {
            constexpr int n = 1 << SI;
            const int d = j - a.Z, ad2 = 2 * (d < 0 ? -d : d);
#pragma unroll
            for (int q = 0; q < n / 2; ++q) {
                const int k = 2 * q + 1;
                const int dk = (k * ad2 + n) >> (SI + 1);
                const int jk = d < 0 ? a.Z - dk : a.Z + dk;
                const float* p = P + jk * (int)a.nfft + ((2 * k * (hw + lane) + n) >> (SI + 1));
#pragma unroll
                for (int i = 0; i < R; ++i) acc[i] += __ldg(p + (32 / n) * k * i);
            }
        }
        reg_test<SI, R>(a, P, acc, hw, j, lane, b);
        reg_stages<SI + 1, NSTAGES, R>(a, P, acc, hw, j, lane, b);
    }
}

constexpr int REG_NT = 128;

template <int NSTAGES, int R, bool ROWS>
__global__ void __launch_bounds__(REG_NT) k_harm_reg(const __grid_constant__ HarmArgs a) {
    // blocks of consecutive launch order take the same h range of successive
    // rows, so the harmonic rows they read overlap while they are in L2; with
    // ROWS the warps of a block take consecutive rows of one h range, so the
    // harmonic rows they share are read through the same L1
    const int lane = threadIdx.x & 31;
    const int j = ROWS ? blockIdx.x * (REG_NT / 32) + (threadIdx.x >> 5) : blockIdx.x;
    if (ROWS && j >= a.nz) return;  // no barriers in this kernel
    const int b = blockIdx.z;
    const int hw = ROWS ? blockIdx.y * 32 * R : (blockIdx.y * (REG_NT / 32) + (threadIdx.x >> 5)) * 32 * R;
    const float* P = a.plane + (int64_t)b * a.plane_stride;
    float acc[R];
    const float* row = P + j * (int)a.nfft;
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] = __ldg(row + hw + lane + 32 * i);
    reg_stages<0, NSTAGES, R>(a, P, acc, hw, j, lane, b);
}

// ---- 2-D planes: tiles of rows ------------------------------------------------
//
// A thread owns RT rows at HP half-bins (lanes consecutive in h, 32 apart per
// point).  The rows of a tile are |j - Z| = RT a + r, r < RT, on one side of
// the centre row, and n divides RT, so harmonic k of stage n reads row
//   |j_k - Z| = (RT / n) k a + floor((2 k r + n) / (2 n)):
// which of the RT points share a row is known when the kernel is compiled, and
// each distinct row is loaded once (8 harmonics, 8 rows: 40 loads per half-bin
// instead of 64).  The additions are those of the kernels above in the same
// order, so the sums are bit-identical.
// Bound: the latency of plane reads that miss L2 (a plane of 201 rows is larger
// than L2; 1.5 planes come from HBM, 3.3 from L2).  301 trials, 201 rows of
// 2^18, 8 harmonics: 27.6 ms with one row per warp, 22.0 ms here; 1, 2 and 4
// half-bins per thread 31.2, 23.1 and 22.0 ms (longer contiguous reads and more
// of them in flight), 256 threads per block 22.3 ms.
// The rare path: a warp with points of row j at or above the threshold (v: the lane's sums; vi, vo: those of the rows
// one nearer to the centre row and one further, where the tile has them: bits 0 and 1 of `has`).  With interference it
// is not rare and most points it sees are on a ridge over many rows, so what the tile's own sums rule out comes first,
// and the loads of the sums it does not have are in flight together.  Uncleaned files, rows / tiles with a chain of
// loads per neighbour / here: 32 trials x 101 rows of 2^18, 342 k detections, 2.80 / 3.35 / 2.56 ms; 128 trials x 201
// rows 28.9 / 32.5 / 23.8 ms; a cleaned one 23.4 / 18.9 / 19.3 ms (held to 80 registers: 24.1 and 20.5 ms).
template <int SI, int HP>
__device__ __noinline__ void tile_hit(const HarmArgs& a, float4 v, float4 vi, float4 vo, int has, int sgn, int d, int hw,
                                      int b) {
    static_assert(HP == 4, "points by value");
    const float* P = a.plane + (int64_t)b * a.plane_stride;
    const int lane = threadIdx.x & 31, j = a.Z + sgn * d;
    const float4 vb = sgn > 0 ? vi : vo, va = sgn > 0 ? vo : vi;  // rows j - 1 and j + 1
    const bool kb = has & (sgn > 0 ? 1 : 2), ka = has & (sgn > 0 ? 2 : 1);
    const float thr = a.thr[SI], x[HP] = {v.x, v.y, v.z, v.w}, xb[HP] = {vb.x, vb.y, vb.z, vb.w}, xa[HP] = {va.x, va.y, va.z, va.w};
    const int nfft = (int)a.nfft, hmin = a.row_hmin ? a.row_hmin[8 * b + SI] : a.hmin[SI], nz = a.nz, Z = a.Z;
#pragma unroll
    for (int i = 0; i < HP; ++i) {
        // the points beside the lane's, in a row of sums; the warp's own first and last have none
        auto beside = [&](const float (&r)[HP], float& l, float& u) {
            l = __shfl_up_sync(0xffffffffu, r[i], 1);
            u = __shfl_down_sync(0xffffffffu, r[i], 1);
            const float l31 = __shfl_sync(0xffffffffu, r[i > 0 ? i - 1 : 0], 31);
            const float u0 = __shfl_sync(0xffffffffu, r[i < HP - 1 ? i + 1 : HP - 1], 0);
            if (lane == 0) l = l31;
            if (lane == 31) u = u0;
        };
        float left, right, bl, br, al, ar;
        beside(x, left, right);
        beside(xb, bl, br);
        beside(xa, al, ar);
        const bool first = i == 0 && lane == 0, end = i == HP - 1 && lane == 31;
        const float s = x[i];
        const int h = hw + lane + 32 * i;
        if (!(s >= thr && h >= hmin)) continue;
        if (first) left = harm_sum_ahead<SI>(P, h - 1, j, nfft, nz, Z);
        if (end) right = harm_sum_ahead<SI>(P, h + 1, j, nfft, nz, Z);
        // strictly above every earlier neighbour, ties to the lower index against later ones
        bool hit = s > left && s >= right;
        if (kb) hit = hit && s > xb[i] && (first || s > bl) && (end || s > br);
        if (ka) hit = hit && s >= xa[i] && (first || s >= al) && (end || s >= ar);
        if (!(kb && ka && !first && !end)) {
#pragma unroll 1
            for (int q = 0; q < 3 && hit; ++q) {
                const int dh = q == 0 ? 0 : 2 * q - 3;
                const bool out = (first && dh < 0) || (end && dh > 0);
                const float below = !kb || out ? harm_sum_ahead<SI>(P, h + dh, j - 1, nfft, nz, Z) : -INFINITY;
                const float above = !ka || out ? harm_sum_ahead<SI>(P, h + dh, j + 1, nfft, nz, Z) : -INFINITY;
                hit = s > below && s >= above;
            }
        }
        if (hit) {
            const unsigned long long slot = atomicAdd(a.counter, 1ull);
            if ((int64_t)slot < a.cap) {
                pss_raw_cand c;
                c.dm_idx = a.row_dm ? a.row_dm[b] : a.dm0 + b;
                c.numharm = 1 << SI;
                c.h = h;
                c.j = j;
                c.power = s;
                c.reserved = a.row_file ? a.row_file[b] : 0;
                a.out[slot] = c;
            }
        }
    }
}

template <int SI, int NSTAGES, int RT, int HP>
__device__ __forceinline__ void tile_stages(const HarmArgs& a, const char* Pz, int rstep, int ta, float (&acc)[RT][HP],
                                            int hw, int nrow, int sgn, int d0, int lane, int b) {
    if constexpr (SI < NSTAGES) {
        constexpr int n = 1 << SI;
        if constexpr (SI > 0) {
#pragma unroll
            for (int q = 0; q < n / 2; ++q) {
                const int k = 2 * q + 1;
                // (rows of the last tile past the plane's edge are loaded from the edge row and not tested)
                const int row0 = (RT / n) * k * ta;
                const int hb = 4 * ((2 * k * (hw + lane) + n) >> (SI + 1));
                float v[HP];
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    const int c = (2 * k * r + n) / (2 * n);
                    if (r == 0 || c != (2 * k * (r - 1) + n) / (2 * n)) {
                        const char* p = Pz + (int64_t)(min(row0 + c, a.Z) * rstep) + hb;
#pragma unroll
                        for (int i = 0; i < HP; ++i) v[i] = __ldg(reinterpret_cast<const float*>(p) + (32 / n) * k * i);
                    }
#pragma unroll
                    for (int i = 0; i < HP; ++i) acc[r][i] += v[i];
                }
            }
        }
        float mx = acc[0][0];
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int i = 0; i < HP; ++i) mx = fmaxf(mx, acc[r][i]);
        if (__any_sync(0xffffffffu, mx >= a.thr[SI])) {
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                float m = acc[r][0];
#pragma unroll
                for (int i = 1; i < HP; ++i) m = fmaxf(m, acc[r][i]);
                // (the centre row belongs to the side d >= 0)
                if (r < nrow && (r > 0 || d0 > 0 || sgn > 0) && __any_sync(0xffffffffu, m >= a.thr[SI])) {
                    auto row = [&](int q) { return make_float4(acc[q][0], acc[q][1], acc[q][2], acc[q][3]); };
                    const int has = (r > 0 ? 1 : 0) | (r + 1 < RT && r + 1 < nrow ? 2 : 0);
                    tile_hit<SI, HP>(a, row(r), row(r > 0 ? r - 1 : 0), row(r + 1 < RT ? r + 1 : r), has, sgn, d0 + r, hw, b);
                }
            }
        }
        tile_stages<SI + 1, NSTAGES, RT, HP>(a, Pz, rstep, ta, acc, hw, nrow, sgn, d0, lane, b);
    }
}

constexpr int TILE_RT = 8;  // rows of a tile: a multiple of every stage's number of harmonics
constexpr int TILE_HP = 4;
constexpr int TILE_NT = 128;

template <int NSTAGES>
__global__ void __launch_bounds__(TILE_NT) k_harm_tile(const __grid_constant__ HarmArgs a) {
    constexpr int RT = TILE_RT, HP = TILE_HP;
    const int lane = threadIdx.x & 31;
    // row tiles fastest: the harmonic rows that successive blocks read overlap while they are in L2
    const int sgn = (blockIdx.x & 1) ? -1 : 1, ta = blockIdx.x >> 1, d0 = RT * ta;
    const int b = blockIdx.z;
    const int hw = (blockIdx.y * (TILE_NT / 32) + (threadIdx.x >> 5)) * 32 * HP;
    const int nrow = min(RT, a.Z + 1 - d0);  // rows of the tile inside the plane
    const int rstep = sgn * (int)a.nfft * 4;
    const char* Pz = reinterpret_cast<const char*>(a.plane + (int64_t)b * a.plane_stride + (int64_t)a.Z * a.nfft);
    float acc[RT][HP];
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        const char* p = Pz + (int64_t)(min(d0 + r, a.Z) * rstep) + 4 * (hw + lane);
#pragma unroll
        for (int i = 0; i < HP; ++i) acc[r][i] = __ldg(reinterpret_cast<const float*>(p) + 32 * i);
    }
    tile_stages<0, NSTAGES, RT, HP>(a, Pz, rstep, ta, acc, hw, nrow, sgn, d0, lane, b);
}

// Planes with rows on both sides of the centre row, offsets within 31 bits of bytes from it, whole warps, up to 8
// harmonics (16 would need tiles of 16 rows, 64 sums per thread).
bool tile_usable(const HarmArgs& a) {
    return a.nz > 1 && a.nz == 2 * a.Z + 1 && a.nstages <= 4 && (int64_t)(a.Z + 16) * a.nfft * 4 < (int64_t(1) << 31) &&
           a.nfft % (TILE_NT * TILE_HP) == 0 && a.nfft / (TILE_NT * TILE_HP) <= 65535 && a.nb <= 65535;
}

// Where tiles gain: many trials of large planes, whose rows come from L2 or HBM anew for every harmonic.  A launch of
// tiles starts and drains about 0.03 ms slower than one of rows (fewer, longer warps), and a trial of it is shorter by
// a time that grows faster than the plane (more of it is out of L2): break-even is at 30 to 60 trials of 50 MiB, 5 to
// 9 of 100 MiB and 1 to 3 of 200 MiB, and below 40 MiB it is not reached with the trials that a batch can hold.
// Kernel times, rows and tiles, 8 harmonics: 51 rows of 2^18 (51 MiB) 16 trials 0.348 and 0.373 ms, 128 trials 2.65
// and 2.49; 201 rows of 2^16 (50 MiB) 32 trials 0.741 and 0.821, 128 trials 2.73 and 2.49; 101 rows of 2^17 (50 MiB) 32
// trials 0.684 and 0.718, 64 trials 1.348 and 1.290; 101 rows of 2^18 (101 MiB) 4 trials 0.180 and 0.188, 16 trials
// 0.678 and 0.604; 101 rows of 2^19 (202 MiB) 2 trials 0.201 and 0.221, 4 trials 0.387 and 0.375; 201 rows of 2^18
// (201 MiB) 4 trials 0.381 and 0.328; 201 rows of 2^19 (402 MiB) 1 trial 0.229 and 0.195; 35 rows of 2^18 (35 MiB) 128
// trials 1.83 and 1.87.  Rows of the last tile past the edge are summed in vain: at most 0.3 times the plane's.
bool tile_gains(const HarmArgs& a) {
    const int64_t rows = 2 * TILE_RT * (int64_t)((a.Z + TILE_RT) / TILE_RT);
    const double mib = (double)a.nz * (double)a.nfft * 4.0 / 1048576.0;
    return 10 * rows <= 13 * (int64_t)a.nz && mib >= 32.0 && a.nb * (mib / 50.0) * (mib / 50.0) >= 64.0;
}

template <int NSTAGES>
cudaError_t launch_tile_t(const HarmArgs& a, cudaStream_t s) {
    dim3 grid((unsigned)(2 * ((a.Z + TILE_RT) / TILE_RT)), (unsigned)(a.nfft / (TILE_NT * TILE_HP)), (unsigned)a.nb);
    k_harm_tile<NSTAGES><<<grid, TILE_NT, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_tile(const HarmArgs& a, cudaStream_t s) {
    switch (a.nstages) {
        case 1: return launch_tile_t<1>(a, s);
        case 2: return launch_tile_t<2>(a, s);
        case 3: return launch_tile_t<3>(a, s);
        case 4: return launch_tile_t<4>(a, s);
        default: return cudaErrorInvalidValue;
    }
}

// 2-D planes: tiles of rows where they gain, else the warps of a block take consecutive plane rows (31.1 -> 28.9 ms on
// the zmax 200 accel file).  PSS_HARM_ROWS=0: one row per block; 1: tiles wherever they can run.
int harm_rows() {
    static const int v = [] {
        const char* e = getenv("PSS_HARM_ROWS");
        return e ? (e[0] == '1' ? 1 : 0) : 2;
    }();
    return v;
}

template <int R, bool ROWS>
cudaError_t launch_reg_t(const HarmArgs& a, cudaStream_t s) {
    constexpr int W = REG_NT / 32;
    dim3 grid(ROWS ? (unsigned)((a.nz + W - 1) / W) : (unsigned)a.nz,
              ROWS ? (unsigned)(a.nfft / (32 * R)) : (unsigned)(a.nfft / (REG_NT * R)), (unsigned)a.nb);
    if (grid.y > 65535) return cudaErrorInvalidValue;
    switch (a.nstages) {
        case 1: k_harm_reg<1, R, ROWS><<<grid, REG_NT, 0, s>>>(a); break;
        case 2: k_harm_reg<2, R, ROWS><<<grid, REG_NT, 0, s>>>(a); break;
        case 3: k_harm_reg<3, R, ROWS><<<grid, REG_NT, 0, s>>>(a); break;
        case 4: k_harm_reg<4, R, ROWS><<<grid, REG_NT, 0, s>>>(a); break;
        case 5: k_harm_reg<5, R, ROWS><<<grid, REG_NT, 0, s>>>(a); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int R>
cudaError_t launch_reg(const HarmArgs& a, cudaStream_t s) {
    if (a.nz > 1 && harm_rows() && a.nfft / (32 * R) <= 65535) return launch_reg_t<R, true>(a, s);
    return launch_reg_t<R, false>(a, s);
}

}  // namespace

bool harm_takes_tiles(const HarmArgs& a) {
    return harm_rows() && tile_usable(a) && (harm_rows() == 1 || tile_gains(a));
}

cudaError_t launch_harm(const HarmArgs& a, cudaStream_t s) {
    if (a.nfft > (int64_t(1) << 24) || a.nstages > 6) return cudaErrorInvalidValue;
    if ((int64_t)a.nz * a.nfft > (int64_t(1) << 31)) return cudaErrorInvalidValue;  // 32-bit plane offsets
    if (harm_takes_tiles(a)) return launch_tile(a, s);
    // register-blocked kernel: up to 16 harmonics, whole warps of 32 x 16 points
    if (a.run == 8 && a.nstages <= 5 && a.nfft % (REG_NT * 8) == 0 && a.nfft / (REG_NT * 8) <= 65535 &&
        a.nb <= 65535)
        return launch_reg<8>(a, s);
    if (a.nstages <= 5 && a.nfft % (REG_NT * 16) == 0 && a.nfft / (REG_NT * 16) <= 65535 && a.nb <= 65535)
        return launch_reg<16>(a, s);
    if (a.nz == 1) return launch_variant<1, 2048, true>(a, s);
    return launch_variant<4, 256, false>(a, s);
}

}  // namespace pss
