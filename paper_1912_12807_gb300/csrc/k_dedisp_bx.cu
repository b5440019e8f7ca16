// Dedispersion of downsampled plan rows through a per-channel boxcar table
// (paper Sect. 2 step 2 with the downsampling of Tables 2-3), exact in
// integers.  With W_c[t] = sum_{k<ds} x[c][t + k] the downsampled series is
//
//     s_ds[j] = sum_c sum_{k<ds} x[c][j ds + d_c + k] = sum_c W_c[j ds + d_c],
//
// one term per channel and output sample instead of ds.  The table is laid
// out by phase, Wt[c][p][m] = W_c[m ds + p], so that with d_c = q ds + p a
// trial reads, for channel c, the contiguous run Wt[c][p][q + j], j < N_v:
// consecutive lanes read consecutive 16-bit words.  W_c[t] <= 255 ds fits 16
// bits for ds <= 256; the channel sum is accumulated in 32 bits.
//
// k_bx_table: one CTA per (channel, run of MT table columns) stages the
// MT ds + ds input bytes it needs, forms their prefix sums in shared
// memory (stored with a skew of one word per 2 ds so that lanes two columns
// apart read distinct banks) and writes two columns of a phase row as one
// 32-bit word: three prefix sums, two differences.  200 channels x 2^18
// samples, ds 8 to 128 (157 MB read and written each): 74 us per table with
// one 16-bit column per thread, 66 us here.
//
// k_dedisp_bx: a CTA owns GW consecutive trials (one warp each) and a tile
// of TJ output samples; the lanes of a warp turn 32 channels' delays into
// table offsets at once (ds is a power of two: a shift and a mask each) and
// list them in shared memory, even element offsets first.  A lane reads 32-bit words, two outputs of a
// channel each; words at an even and at an odd element offset are summed
// apart (16-bit halves, widened before they can overflow) and combined, one
// output shifted, at the end.  Adjacent trials mostly share a channel's phase
// row and offset, so their warps read the same lines through L1.  Bound: the
// latency of table reads that miss L1 (long scoreboard; L1 at 31 %, DRAM at 23 %
// of their rates), so a warp has the loads of four channels in flight at once.  979 trials of the six-row plan:
// 1.35 ms with 16-bit loads, 1.22 ms with a branch per channel, 0.60 ms here.
#include "pss_internal.h"

namespace pss {

namespace {

constexpr int TB_NT = 256;     // table builder threads
constexpr int TB_SPAN = 8192;  // native samples per table-builder CTA, plus a tail of ds
constexpr int GW = 8;          // trials (warps) per dedispersion CTA
constexpr int KW = 4;          // 32-bit words (2 outputs) per lane
constexpr int TJ = 64 * KW;    // outputs per tile

__device__ __forceinline__ int skew(int k, int lds) { return k + (k >> (lds + 1)); }

// ds = 2^lds <= 256 (plan rows are powers of two), MT = 2^lmt columns, so a
// CTA covers MT ds = TB_SPAN bytes of its channel plus a tail of ds bytes.
__global__ void __launch_bounds__(TB_NT) k_bx_table(const __grid_constant__ BxTableArgs a) {
    extern __shared__ __align__(16) unsigned char tb_sm[];
    const int lds = a.lds, ds = 1 << lds, lmt = a.lmt, MT = 1 << lmt;
    const int span = MT << lds;  // TB_SPAN
    const int L = span + ds;     // columns [m0, m0 + MT) need x[t0 .. t0 + L)
    uint8_t* xb = tb_sm;                                               // [L] staged bytes
    int32_t* P = reinterpret_cast<int32_t*>(tb_sm + ((L + 15) & ~15));  // skewed prefix sums P[0..L]
    __shared__ int32_t s_warp[TB_NT / 32];
    const int c = blockIdx.y;
    const int64_t m0 = (int64_t)blockIdx.x * MT;
    const int64_t t0 = m0 << lds;
    const uint8_t* row = a.xcm + (int64_t)c * a.pitch;
    if (t0 + L <= a.nsamp) {
        // row starts and t0 are 16-byte aligned (pitch is a multiple of 64, t0 of TB_SPAN)
        const uint4* src = reinterpret_cast<const uint4*>(row + t0);
        for (int k = threadIdx.x; k < span / 16; k += TB_NT) reinterpret_cast<uint4*>(xb)[k] = __ldg(src + k);
        for (int k = span + threadIdx.x; k < L; k += TB_NT) xb[k] = row[t0 + k];
    } else {
        for (int k = threadIdx.x; k < L; k += TB_NT) xb[k] = (t0 + k < a.nsamp) ? row[t0 + k] : (uint8_t)0;
    }
    __syncthreads();
    // exclusive prefix sums of the first `span` bytes: 32 per thread, then a block scan
    constexpr int SEG = TB_SPAN / TB_NT;
    const int k0 = threadIdx.x * SEG;
    int32_t v[SEG];
    int32_t tot = 0;
#pragma unroll
    for (int q = 0; q < SEG / 16; ++q) {
        const uint4 w = reinterpret_cast<const uint4*>(xb + k0)[q];
        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            v[16 * q + e] = (int32_t)((ww[e >> 2] >> (8 * (e & 3))) & 0xFFu);
            tot += v[16 * q + e];
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t incl = tot;
    for (int off = 1; off < 32; off <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += u;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    int32_t run = incl - tot;
    for (int w = 0; w < warp; ++w) run += s_warp[w];
#pragma unroll
    for (int e = 0; e < SEG; ++e) {
        P[skew(k0 + e, lds)] = run;
        run += v[e];
    }
    if (warp == 0) {
        // the tail P[span .. L]: a warp scan of the last ds bytes (at most 8 per lane)
        int32_t base = 0;
        for (int w = 0; w < TB_NT / 32; ++w) base += s_warp[w];
        const int per = (ds + 31) >> 5;
        int32_t loc[BX_MAX_DS / 32];
        int32_t t = 0;
#pragma unroll
        for (int e = 0; e < BX_MAX_DS / 32; ++e) {
            const int i = lane * per + e;
            loc[e] = (e < per && i < ds) ? (int32_t)xb[span + i] : 0;
            t += loc[e];
        }
        int32_t in = t;
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, in, off);
            if (lane >= off) in += u;
        }
        int32_t r = base + in - t;
#pragma unroll
        for (int e = 0; e < BX_MAX_DS / 32; ++e) {
            const int i = lane * per + e;
            if (e < per && i < ds) P[skew(span + i, lds)] = r;
            r += loc[e];
        }
        if (lane == 31) P[skew(L, lds)] = base + in;
    }
    __syncthreads();
    // W_c[m ds + p] = P[(m - m0) ds + p + ds] - P[(m - m0) ds + p], two columns m of a phase row p per thread (rows
    // start on 16-byte boundaries and hold whole words; a column past the last is written into the padding)
    uint32_t* out = reinterpret_cast<uint32_t*>(a.table + (int64_t)c * ds * a.mstride);
    const int64_t ncol = min((int64_t)MT, a.mstride - m0);
#pragma unroll 4
    for (int idx = threadIdx.x; idx < span / 2; idx += TB_NT) {
        const int p = idx >> (lmt - 1), mm = 2 * (idx & (MT / 2 - 1));
        if (mm >= ncol) continue;
        const int k = (mm << lds) + p;
        const int32_t p0 = P[skew(k, lds)], p1 = P[skew(k + ds, lds)], p2 = P[skew(k + 2 * ds, lds)];
        out[((int64_t)p * a.mstride + m0 + mm) / 2] = (uint32_t)(p1 - p0) | (uint32_t)(p2 - p1) << 16;
    }
}

// OFF: table offsets in elements, 32-bit where the table has fewer than 2^32.
template <bool INT_OUT, typename OFF>
__global__ void __launch_bounds__(32 * GW) k_dedisp_bx(const __grid_constant__ BxArgs a) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int my = blockIdx.y * GW + warp;
    if (my >= a.nb) return;
    const int64_t j0 = (int64_t)blockIdx.x * TJ;
    const int32_t* dl = a.delays + (int64_t)my * a.ck;
    const uint32_t* __restrict__ tab = reinterpret_cast<const uint32_t*>(a.table);
    // words that a lane may read of a channel's run: the outputs up to N_v and, at an odd offset, one more
    const int nword = (int)min((int64_t)(TJ / 2), (a.nv - j0 + 1) / 2);
    const bool full = nword == TJ / 2;
    const int period = 65535 / (255 << a.lds);  // channels whose sums fit 16 bits (>= 1)
    uint32_t ev[KW], od[KW], ox = 0u;           // 16-bit sums at even offsets, at odd ones (one early), the word past them
    uint32_t we[2 * KW], wo[2 * KW], wx = 0u;   // the same, widened
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        ev[k] = od[k] = 0u;
        we[2 * k] = we[2 * k + 1] = wo[2 * k] = wo[2 * k + 1] = 0u;
    }
    auto widen = [&]() {
#pragma unroll
        for (int k = 0; k < KW; ++k) {
            we[2 * k] += ev[k] & 0xFFFFu;
            we[2 * k + 1] += ev[k] >> 16;
            wo[2 * k] += od[k] & 0xFFFFu;
            wo[2 * k + 1] += od[k] >> 16;
            ev[k] = od[k] = 0u;
        }
        wx += ox & 0xFFFFu;
        ox = 0u;
    };
    int since = 0;
    // U channels at a time: their U KW loads are in flight together
    constexpr int U = 4;
    __shared__ __align__(16) OFF s_list[GW][32];
    OFF* list = s_list[warp];
    auto add = [&](uint32_t (&sum)[KW], const uint32_t (&w)[KW]) {
#pragma unroll
        for (int k = 0; k < KW; ++k) sum[k] += w[k];
        if (++since == period) {
            since = 0;
            widen();
        }
    };
    auto load = [&](const uint32_t* src, uint32_t (&w)[KW]) {
#pragma unroll
        for (int k = 0; k < KW; ++k) w[k] = full || lane + 32 * k < nword ? __ldg(src + lane + 32 * k) : 0u;
    };
    for (int cb = 0; cb < a.ck; cb += 32) {
        // lane l: the table offset of channel cb + l for this trial at output j0; even offsets first in the list
        const int cn = min(32, a.ck - cb);
        OFF o = 0;
        if (lane < cn) {
            const int32_t d = __ldg(dl + cb + lane);
            const int32_t q = d >> a.lds, p = d & ((1 << a.lds) - 1);
            o = (OFF)((((int64_t)(cb + lane) << a.lds) + p) * a.mstride + q + j0);
        }
        const uint32_t valid = cn == 32 ? 0xffffffffu : (1u << cn) - 1u;
        const uint32_t odd = __ballot_sync(0xffffffffu, (o & 1) != 0) & valid;
        const int ne = __popc(valid & ~odd);
        const uint32_t below = (1u << lane) - 1u;
        __syncwarp();
        if (lane < cn) list[(odd >> lane & 1) ? ne + __popc(odd & below) : __popc(~odd & below)] = o >> 1;
        __syncwarp();
        int i = 0;
        for (; i + U <= ne; i += U) {
            uint32_t w[U][KW];
#pragma unroll
            for (int u = 0; u < U; ++u) load(tab + list[i + u], w[u]);
#pragma unroll
            for (int u = 0; u < U; ++u) add(ev, w[u]);
        }
        for (; i < ne; ++i) {
            uint32_t w[KW];
            load(tab + list[i], w);
            add(ev, w);
        }
        for (; i + U <= cn; i += U) {
            uint32_t w[U][KW], x[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t* src = tab + list[i + u];
                load(src, w[u]);
                x[u] = lane == 0 ? __ldg(src + nword) : 0u;  // the word past the run: its first half is the last element
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                ox += x[u];
                add(od, w[u]);
            }
        }
        for (; i < cn; ++i) {
            const uint32_t* src = tab + list[i];
            uint32_t w[KW];
            load(src, w);
            if (lane == 0) ox += __ldg(src + nword);
            add(od, w);
        }
    }
    widen();
    wx = __shfl_sync(0xffffffffu, wx, 0);
    unsigned long long part = 0ull;
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        // the odd sums' next first half: the next lane's, lane 0's of the next k, or the word past the run
        const uint32_t give = lane == 0 ? (k + 1 < KW ? wo[2 * (k + 1 < KW ? k + 1 : k)] : wx) : wo[2 * k];
        uint32_t nx = __shfl_sync(0xffffffffu, give, (lane + 1) & 31);
        if (lane + 32 * k == nword - 1) nx = wx;
        const uint32_t v[2] = {we[2 * k] + wo[2 * k + 1], we[2 * k + 1] + nx};
        const int64_t j = j0 + 2 * (lane + 32 * k);
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if (j + e < a.nv) {
                part += v[e];
                if (INT_OUT) a.out_i[(int64_t)my * a.out_stride + j + e] = (int32_t)v[e];
                else a.out_f[(int64_t)my * a.out_stride + j + e] = (float)v[e];
            }
    }
    if (a.sums) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
        if (lane == 0) atomicAdd(a.sums + my, part);
    }
}

}  // namespace

int bx_table_cols(int ds) { return TB_SPAN / std::max(ds, 1); }

cudaError_t launch_bx_table(const BxTableArgs& a, cudaStream_t s) {
    if (a.ck <= 0 || a.mlen <= 0) return cudaSuccess;
    const int ds = 1 << a.lds;
    // grid.y is the channel: at most 65535 rows
    if (a.lds < 1 || ds > BX_MAX_DS || (1 << a.lmt) != bx_table_cols(ds) || a.mstride < a.mlen || (a.pitch & 15) ||
        a.ck > 65535)
        return cudaErrorInvalidValue;
    const int L = TB_SPAN + ds;
    const size_t shm = (size_t)((L + 15) & ~15) + (size_t)(L + 1 + (L >> (a.lds + 1)) + 2) * sizeof(int32_t);
    cudaError_t e = allow_smem((const void*)k_bx_table, shm);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((a.mlen + (1 << a.lmt) - 1) >> a.lmt), (unsigned)a.ck);
    k_bx_table<<<grid, TB_NT, shm, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_dedisp_bx(const BxArgs& a, cudaStream_t s) {
    if (a.nb <= 0 || a.nv <= 0) return cudaSuccess;
    if (a.lds < 1 || (1 << a.lds) > BX_MAX_DS || a.ck <= 0) return cudaErrorInvalidValue;
    dim3 grid((unsigned)((a.nv + TJ - 1) / TJ), (unsigned)((a.nb + GW - 1) / GW));
    if (((int64_t)a.ck << a.lds) * a.mstride < (int64_t(1) << 32)) {
        if (a.out_i) k_dedisp_bx<true, uint32_t><<<grid, 32 * GW, 0, s>>>(a);
        else k_dedisp_bx<false, uint32_t><<<grid, 32 * GW, 0, s>>>(a);
    } else {
        if (a.out_i) k_dedisp_bx<true, unsigned long long><<<grid, 32 * GW, 0, s>>>(a);
        else k_dedisp_bx<false, unsigned long long><<<grid, 32 * GW, 0, s>>>(a);
    }
    return cudaGetLastError();
}

}  // namespace pss
