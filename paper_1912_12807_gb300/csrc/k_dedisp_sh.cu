// Dedispersion of 8-bit files with partial sums shared between trials (paper
// Sect. 2 step 2; the same exact integers as k_dedisp.cu, added in another
// order).
//
// A CTA owns a group of up to 32 consecutive trials (16 warps, two trials
// each) and a tile of TN = 512 native samples, and walks the chunks of its
// group's table (host_dedisp.cpp):
//   1. the chunk's channel rows (the bytes its trials reach) and its table
//      come in by bulk copies while the previous chunk is being added up;
//   2. every thread forms 20 consecutive partial sums of a row at a time: S
//      channels, each six aligned words and a funnel shift to the row's own
//      byte offset, added as pairs of 16-bit halves;
//   3. every warp adds the row of its trial's pattern, at the trial's offset,
//      for each unit of the chunk: a 32-bit read holds 2 samples of S
//      channels, and two units go into one three-input add.
// Reads are aligned words whatever the offset: units at an even and at an odd
// offset are summed apart and combined, one sample shifted, at the end; the
// table lists a trial's even units first, so the loops do not branch.
//
// A 16-bit sum holds 257 channels; with more the sums are written out as
// 32-bit integers every 257 channels and added to by the same thread the
// next time.
//
// Bound: shared-memory wavefronts (79 % of their rate on the drift-scan file, 256
// channels, 0.5 pc cm^-3 steps; integer pipe 61 %).  The direct kernel reads one byte per
// channel and trial and spends five instructions on four of them; here a
// trial reads half a byte per channel, and a row costs 35 wavefronts per 640
// sums.  32 trials x 512 samples leave two CTAs per SM (row forming of one
// beside the adding of the other); five columns at a time because an odd
// stride reads distinct banks and 27-31 runs fill a warp; 64 rows per chunk are
// whole rounds of the 16 warps.  1001 drift-scan trials of 2^18 samples: 3.91 ms
// direct, 2.45 ms here; 301 trials at 1 pc cm^-3 steps: 1.57 and 1.23 ms.
//
// Waits are bounded as in k_dedisp.cu.
#include "bulk.cuh"
#include "pss_internal.h"

namespace pss {

namespace {

constexpr int TN = DD_TN, GT = DD_GT;
constexpr int NW = GT / 2;     // warps, two trials each
constexpr int NT = 32 * NW;
constexpr int KW = TN / 64;    // 32-bit words (2 sums) of a tile per lane

constexpr int SM_RAW = 0;
constexpr int SM_U = SM_RAW + DD_RAWCAP;  // the rows
constexpr int SM_BLOB = SM_U + DD_UCAP;
constexpr int BLOBCAP = DD_BLOBHEAD + DD_MAXROWS * 16 + GT * 2 + GT * (DD_MAXUNITS / 2 + 1) * 4;
constexpr int SM_BAR = SM_BLOB + 2 * BLOBCAP;
constexpr int SM_TOTAL = SM_BAR + 16;
static_assert(BLOBCAP % 16 == 0 && SM_BLOB % 16 == 0 && SM_U % 16 == 0 && SM_BAR % 8 == 0, "alignment");
static_assert(NW * TN * 4 <= DD_UCAP, "the epilogue's slices fit over the rows");
static_assert(2 * (SM_TOTAL + 1024) <= 228 * 1024, "two CTAs per SM");

// A thread forms M = DD_M consecutive columns (4 sums each) of a row at a time.
// M is odd, so that lanes M words apart read distinct banks, and each channel
// takes M + 1 words for M columns.
template <int S>
__device__ __forceinline__ void make_rows(const uint8_t* raw, uint2* rows, const uint4* src, const DdChunk& k) {
    constexpr int M = DD_M;
    const int nrun = k.nrun, ish = k.ishift, total = k.nrow << ish;
#pragma unroll 1
    for (int idx = threadIdx.x; idx < total; idx += NT) {
        const int r = idx >> ish, j = idx & ((1 << ish) - 1);
        if (j >= nrun) continue;
        const uint8_t* col = raw + 4 * M * j;
        const uint4 m4 = src[r];  // the same for the whole warp
        const uint32_t m[4] = {m4.x, m4.y, m4.z, m4.w};
        uint32_t e[M], o[M];
#pragma unroll
        for (int q = 0; q < M; ++q) e[q] = o[q] = 0u;
#pragma unroll
        for (int c = 0; c < S; ++c) {
            const uint32_t* p = reinterpret_cast<const uint32_t*>(col + (m[c] >> 5));
            uint32_t w[M + 1];
#pragma unroll
            for (int q = 0; q <= M; ++q) w[q] = p[q];
#pragma unroll
            for (int q = 0; q < M; ++q) {
                const uint32_t v = __funnelshift_r(w[q], w[q + 1], m[c]);  // the shift is taken modulo 32
                e[q] += v & 0x00FF00FFu;
                o[q] += __byte_perm(v, 0u, 0x4341);
            }
        }
#pragma unroll
        for (int q = 0; q < M; ++q) rows[M * (r * nrun + j) + q] = make_uint2(__byte_perm(e[q], o[q], 0x5410), __byte_perm(e[q], o[q], 0x7632));
    }
}

// A trial's running sums: words lane + 32 k of the tile from units at even
// offsets (a) and at odd ones (b, one sample early), and b's word past the tile.
struct Acc {
    uint32_t a[KW], b[KW], ext;
    __device__ __forceinline__ void clear() {
        ext = 0u;
#pragma unroll
        for (int k = 0; k < KW; ++k) a[k] = b[k] = 0u;
    }
    // u: the rows, as words, from this lane on; cnt: units at even offsets, and at odd ones << 8
    __device__ __forceinline__ void add(const uint32_t* u, const uint32_t* list, uint32_t cnt, int lane) {
        const uint32_t ne = cnt & 0xFFu, no = cnt >> 8;
#pragma unroll 1
        for (uint32_t i = 0; i < ne / 2; ++i) {
            const uint32_t w = *list++;
            const uint32_t *p = u + (w & 0xFFFFu), *q = u + (w >> 16);
#pragma unroll
            for (int k = 0; k < KW; ++k) a[k] = a[k] + p[32 * k] + q[32 * k];
        }
        if (ne & 1) {
            const uint32_t* p = u + (*list++ & 0xFFFFu);
#pragma unroll
            for (int k = 0; k < KW; ++k) a[k] += p[32 * k];
        }
#pragma unroll 1
        for (uint32_t i = 0; i < no / 2; ++i) {
            const uint32_t w = *list++;
            const uint32_t *p = u + (w & 0xFFFFu), *q = u + (w >> 16);
#pragma unroll
            for (int k = 0; k < KW; ++k) b[k] = b[k] + p[32 * k] + q[32 * k];
            ext = ext + p[32 * KW - lane] + q[32 * KW - lane];
        }
        if (no & 1) {
            const uint32_t* p = u + (*list & 0xFFFFu);
#pragma unroll
            for (int k = 0; k < KW; ++k) b[k] += p[32 * k];
            ext += p[32 * KW - lane];
        }
    }
    // the tile's sums as 32-bit integers in `nat` [TN] (the warp's own slice)
    __device__ __forceinline__ void write(uint32_t* nat, int lane) const {
#pragma unroll
        for (int k = 0; k < KW; ++k) {
            // b's word after this one: the next lane's, or lane 0's of the next k
            const uint32_t give = lane == 0 ? (k + 1 < KW ? b[k + 1 < KW ? k + 1 : k] : ext) : b[k];
            const uint32_t nx = __shfl_sync(0xffffffffu, give, (lane + 1) & 31);
            // 257 channels of 255: no half carries
            const uint32_t s = a[k] + __funnelshift_r(b[k], nx, 16);
            reinterpret_cast<uint2*>(nat)[lane + 32 * k] = make_uint2(s & 0xFFFFu, s >> 16);
        }
    }
};

// One trial's tile out: ds native samples to an output, 32-bit integers added
// to what an earlier flush of this tile left (`prev`), converted on the last.
// Adds the outputs and their squares to m1 and m2 (integer rows with a.squares: the moments of the single-pulse search).
template <bool INT_OUT>
__device__ __forceinline__ void put(const DdArgs& a, const uint32_t* nat, int my, int64_t t0, int lane, bool prev, bool last,
                                    unsigned long long& m1, unsigned long long& m2) {
    const int64_t j0 = t0 >> a.lds;
    int32_t* o = (INT_OUT ? a.out_i : reinterpret_cast<int32_t*>(a.out_f)) + (int64_t)my * a.out_stride + j0;
    const int left = (int)min((int64_t)(TN >> a.lds), a.nv - j0);  // outputs of this tile
    if (a.lds == 0 && !prev && last && left == TN && (INT_OUT || a.vec4)) {
        if (INT_OUT) {
            uint32_t sum = 0;
#pragma unroll
            for (int i = 0; i < TN / 32; ++i) {
                const uint32_t v = nat[lane + 32 * i];
                o[lane + 32 * i] = (int32_t)v;
                if (a.squares) {
                    sum += v;  // 16 values of at most 65535
                    m2 += (unsigned long long)v * v;
                }
            }
            m1 += sum;
            return;
        }
        uint32_t sum = 0;
#pragma unroll
        for (int i = 0; i < TN / 128; ++i) {
            const uint4 v = reinterpret_cast<const uint4*>(nat)[lane + 32 * i];
            sum += v.x + v.y + v.z + v.w;
            reinterpret_cast<float4*>(o)[lane + 32 * i] = make_float4((float)v.x, (float)v.y, (float)v.z, (float)v.w);
        }
        m1 += sum;
        return;
    }
    const int ds = 1 << a.lds;
    for (int q = lane; q < left; q += 32) {
        uint32_t v = 0;
        for (int e = 0; e < ds; ++e) v += nat[(q << a.lds) + e];
        if (prev) v += (uint32_t)o[q];
        if (last) {
            m1 += v;
            if (INT_OUT && a.squares) m2 += (unsigned long long)v * v;
        }
        if (INT_OUT || !last) o[q] = (int32_t)v;
        else reinterpret_cast<float*>(o)[q] = (float)v;
    }
}

// The warp's moments of trial `my` added to the trial's.
__device__ __forceinline__ void add_moments(const DdArgs& a, int my, int lane, unsigned long long m1, unsigned long long m2) {
    if (!a.sums) return;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m1 += __shfl_xor_sync(0xffffffffu, m1, off);
    if (lane == 0) atomicAdd(a.sums + my, m1);
    if (!a.squares) return;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, off);
    if (lane == 0) atomicAdd(a.squares + my, m2);
}

template <bool INT_OUT>
__global__ void __launch_bounds__(NT, 2) k_dedisp_sh(const __grid_constant__ DdArgs a) {
    extern __shared__ __align__(128) uint8_t sm[];
    uint64_t* bar = reinterpret_cast<uint64_t*>(sm + SM_BAR);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * TN;
    const int g = blockIdx.y;
    const int gn = min(GT, a.nb - g * GT);
    const int4 gi = *reinterpret_cast<const int4*>(a.tab + (size_t)g * sizeof(int4));
    const DdChunk* chunks = reinterpret_cast<const DdChunk*>(a.tab + a.chunk_off) + gi.x;
    const int2* chans = reinterpret_cast<const int2*>(a.tab + a.chan_off) + (int64_t)g * a.ck;
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // chunk c's table and channel rows: record k and channel entries ch (one copy per channel, spread over the warps)
    auto issue = [&](int c, const DdChunk& k, const int2* ch) {
        if (lane < 8) {
            // order this CTA's earlier generic-proxy reads of the staging area before the copies overwrite it
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (threadIdx.x == 0) {
                mbar_expect_tx(bar, (uint32_t)k.tx_bytes);
                bulk_g2s(sm + SM_BLOB + (c & 1) * BLOBCAP, a.tab + k.blob_off, (uint32_t)k.blob_bytes, bar);
            }
            for (int i = warp + NW * lane; i < k.nch; i += NW * 8) {
                const int2 e = ch[i];
                bulk_g2s(sm + SM_RAW + (size_t)(e.y & 0xFFFF) * 16, a.xcm + (int64_t)(k.c0 + i) * a.pitch + t0 + e.x,
                         (uint32_t)(e.y >> 16) * 16u, bar);
            }
        }
        __syncwarp();
    };
    Acc A0, A1;
    A0.clear();
    A1.clear();
    const bool act0 = warp < gn, act1 = warp + NW < gn;
    __syncthreads();
    issue(0, chunks[0], chans);
    int failed_at = -1;
    bool prev = false;
    for (int c = 0; c < gi.y; ++c) {
        // one warp polls the mbarrier; the others wait at the block barrier, which passes the bytes on
        const bool ok = warp == 0 ? mbar_wait(bar, (uint32_t)(c & 1), a.wait_polls) : true;
        if (__syncthreads_or(!ok)) {
            failed_at = c;
            break;
        }
        const uint8_t* blob = sm + SM_BLOB + (c & 1) * BLOBCAP;
        const DdChunk& k = *reinterpret_cast<const DdChunk*>(blob);
        uint32_t* u = reinterpret_cast<uint32_t*>(sm + SM_U);
        uint2* rows = reinterpret_cast<uint2*>(u);
        const uint4* src = reinterpret_cast<const uint4*>(blob + k.src_off);
        if (k.S == 4) make_rows<4>(sm + SM_RAW, rows, src, k);
        else if (k.S == 2) make_rows<2>(sm + SM_RAW, rows, src, k);
        else make_rows<1>(sm + SM_RAW, rows, src, k);
        __syncthreads();
        if (c + 1 < gi.y)
            issue(c + 1, *reinterpret_cast<const DdChunk*>(blob + sizeof(DdChunk)),
                  reinterpret_cast<const int2*>(blob + 2 * sizeof(DdChunk)));
        const uint16_t* cnt = reinterpret_cast<const uint16_t*>(blob + k.cnt_off);
        const uint32_t* list = reinterpret_cast<const uint32_t*>(blob + k.list_off);
        const uint32_t* uw = u + lane;
        if (act0) A0.add(uw, list + warp * k.npair, cnt[warp], lane);
        if (act1) A1.add(uw, list + (warp + NW) * k.npair, cnt[warp + NW], lane);
        if (k.flush) {
            // the sums leave through the row area (every warp is done with the rows), each warp its own
            // slice; copies of the next chunk may be landing in the staging area beside it
            const bool last = c + 1 == gi.y;
            __syncthreads();
            uint32_t* nat = u + warp * TN;
            if (act0) {
                unsigned long long m1 = 0ull, m2 = 0ull;
                A0.write(nat, lane);
                __syncwarp();
                put<INT_OUT>(a, nat, g * GT + warp, t0, lane, prev, last, m1, m2);
                if (last) add_moments(a, g * GT + warp, lane, m1, m2);
                __syncwarp();
            }
            if (act1) {
                unsigned long long m1 = 0ull, m2 = 0ull;
                A1.write(nat, lane);
                __syncwarp();
                put<INT_OUT>(a, nat, g * GT + warp + NW, t0, lane, prev, last, m1, m2);
                if (last) add_moments(a, g * GT + warp + NW, lane, m1, m2);
            }
            A0.clear();
            A1.clear();
            prev = true;
            // the next chunk's first barrier (after its data wait) orders these reads before its rows
        }
    }
    if (failed_at >= 0) {
        if (threadIdx.x == 0 && a.err) atomicExch(a.err, 1);
        // let the copies still in flight land before the CTA's shared memory is released (the full bound)
        mbar_wait(bar, (uint32_t)(failed_at & 1));
    }
}

template <bool INT_OUT>
cudaError_t launch_t(const DdArgs& a, dim3 grid, cudaStream_t s) {
    cudaError_t e = allow_smem((const void*)k_dedisp_sh<INT_OUT>, SM_TOTAL);
    if (e != cudaSuccess) return e;
    k_dedisp_sh<INT_OUT><<<grid, NT, SM_TOTAL, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_dedisp_sh(const DdArgs& a, cudaStream_t s) {
    if (a.nb <= 0 || a.nv <= 0) return cudaSuccess;
    if (a.lds < 0 || (TN >> a.lds) == 0 || a.ck <= 0) return cudaErrorInvalidValue;
    const int64_t L = a.nv << a.lds;
    dim3 grid((unsigned)((L + TN - 1) / TN), (unsigned)((a.nb + GT - 1) / GT));
    return a.out_i ? launch_t<true>(a, grid, s) : launch_t<false>(a, grid, s);
}

}  // namespace pss
