// Dedispersion of 1-bit files, bit-sliced (paper Sect. 2 step 2; the same
// exact integers as k_dedisp.cu).
//
// k_prep_bits keeps a 1-bit file as bits: channel-major rows of 32-bit words,
// bit i of word w the sample 32 w + i.  A trial's series is then a count of
// set bits over the channels, each row shifted by its delay, and 32 samples
// are counted at once: one word per channel goes into a tree of carry-save
// adders (two three-input logic operations each) whose outputs are the bit
// planes of the counts.
//
// A CTA owns a group of consecutive trials and a tile of 1024 KW samples.  The
// bits that its trials reach of every channel come in by one bulk copy per
// channel; the delays become word offsets and shifts in shared memory; then
// each warp takes its trials without a further block barrier: lane l counts
// samples 32 (l + 32 k) .. + 31, k < KW, reading two neighbouring words per
// channel and word and a funnel shift.  Per 32 samples and channel that is
// two shared-memory reads, one shift and 2.4 logic operations, against about
// 60 instructions of the byte form (k_dedisp.cu).  The planes become bytes by
// three rounds of masked swaps (8 x 8 bit transposes), and leave through the
// warp's slice of shared memory.
//
// Bound: shared-memory reads and logic operations together (76 % and 71 % of
// their rates, 96 channels x 10^6 samples, 96 trials).  32 trials share a staged tile of 4096 samples, which leaves
// two CTAs per SM with 96 channels (2048 samples where four words per lane do
// not fit).  96 channels x 10^6 samples, 1081 trials of ds 1, 2 and 4: 7.29 ms
// with the byte form, 1.17 ms here (2.2 TB/s of series written).
//
// The wait on the copies is bounded as in k_dedisp.cu.
#include "bulk.cuh"
#include "pss_internal.h"

namespace pss {

namespace {

constexpr int NW = 16;
constexpr int NT = 32 * NW;
constexpr int CB = 16;          // channels per counting block (rows are padded with zeros to a multiple)
constexpr int SLICE = 1024;     // epilogue bytes per warp

// ---- 1-bit file -> rows of bits --------------------------------------------
// A CTA takes 32 words (1024 samples) of 32 kept channels: a warp holds 32
// samples (one per lane), the file bytes that the channels lie in are loaded
// together (8 at a time), and a ballot gives a channel's word.  96 channels x
// 10^6 samples: 76 us with a byte loaded per group of 8 channels in turn,
// 55 us here.
__global__ void __launch_bounds__(256) k_prep_bits(const PrepArgs a, uint32_t* xb, int64_t pitchw) {
    __shared__ uint32_t tile[32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t w0 = (int64_t)blockIdx.x * 32;
    const int r0 = blockIdx.y * 32, rn = min(32, a.ck - r0);
    const int nb = a.nchan >> 3;
    const int mine = lane < rn ? __ldg(a.keep + r0 + lane) : 0;  // lane r: the channel of row r0 + r
    uint32_t word[4] = {0u, 0u, 0u, 0u};                         // lane r: words 4 warp .. 4 warp + 3 of row r0 + r
    for (int r = 0; r < rn;) {
        const int c0 = __shfl_sync(0xffffffffu, mine, r) >> 3;   // first of 8 bytes
        unsigned long long v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t t = (w0 + warp * 4 + i) * 32 + lane;
            const uint8_t* src = a.src + t * nb + c0;
            v[i] = 0ull;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (t < a.nsamp && c0 + q < nb) v[i] |= (unsigned long long)__ldg(src + q) << (8 * q);
        }
        for (; r < rn; ++r) {
            const int c = __shfl_sync(0xffffffffu, mine, r);
            if ((c >> 3) >= c0 + 8) break;
            const int bit = 8 * ((c >> 3) - c0) + 7 - (c & 7);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t m = __ballot_sync(0xffffffffu, (uint32_t)(v[i] >> bit) & 1u);
                if (lane == r) word[i] = m;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) tile[lane][warp * 4 + i] = word[i];
    __syncthreads();
    for (int r = warp; r < rn; r += 8)
        if (w0 + lane < pitchw) xb[(int64_t)(r0 + r) * pitchw + w0 + lane] = tile[r][lane];
}

// ---- counting ----------------------------------------------------------------
__device__ __forceinline__ uint32_t xor3(uint32_t a, uint32_t b, uint32_t c) { return a ^ b ^ c; }
__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a ^ b)); }

// Count 8 words into the planes of weight 1, 2 and 4; the carries of weight 8.
__device__ __forceinline__ uint32_t count8(const uint32_t (&x)[8], uint32_t& p1, uint32_t& p2, uint32_t& p4) {
    const uint32_t ta = maj3(p1, x[0], x[1]);
    p1 = xor3(p1, x[0], x[1]);
    const uint32_t tb = maj3(p1, x[2], x[3]);
    p1 = xor3(p1, x[2], x[3]);
    const uint32_t fa = maj3(p2, ta, tb);
    p2 = xor3(p2, ta, tb);
    const uint32_t tc = maj3(p1, x[4], x[5]);
    p1 = xor3(p1, x[4], x[5]);
    const uint32_t td = maj3(p1, x[6], x[7]);
    p1 = xor3(p1, x[6], x[7]);
    const uint32_t fb = maj3(p2, tc, td);
    p2 = xor3(p2, tc, td);
    const uint32_t e = maj3(p4, fa, fb);
    p4 = xor3(p4, fa, fb);
    return e;
}

// Exchange the bits of a s places above m with the bits of b under m.
__device__ __forceinline__ void swap_bits(uint32_t& a, uint32_t& b, int s, uint32_t m) {
    const uint32_t t = ((a >> s) ^ b) & m;
    b ^= t;
    a ^= t << s;
}

// Planes p[b] (bit j: bit b of sample j's count) -> n[m] (byte e: sample 4 m + e).
__device__ __forceinline__ void planes_to_bytes(uint32_t (&p)[8], uint32_t (&n)[8]) {
    // 8 x 8 transposes within each byte lane: p[i] byte L becomes the count of sample 8 L + i
#pragma unroll
    for (int i = 0; i < 4; ++i) swap_bits(p[i], p[i + 4], 4, 0x0F0F0F0Fu);
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if ((i & 2) == 0) swap_bits(p[i], p[i + 2], 2, 0x33333333u);
#pragma unroll
    for (int i = 0; i < 8; i += 2) swap_bits(p[i], p[i + 1], 1, 0x55555555u);
    // 4 x 4 byte transposes: samples in order
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t a = p[4 * h], b = p[4 * h + 1], c = p[4 * h + 2], d = p[4 * h + 3];
        const uint32_t ab0 = __byte_perm(a, b, 0x5140), ab1 = __byte_perm(a, b, 0x7362);
        const uint32_t cd0 = __byte_perm(c, d, 0x5140), cd1 = __byte_perm(c, d, 0x7362);
        n[h] = __byte_perm(ab0, cd0, 0x5410);      // byte lane 0: samples 4 h .. 4 h + 3
        n[2 + h] = __byte_perm(ab0, cd0, 0x7632);  // lane 1: 8 + 4 h ..
        n[4 + h] = __byte_perm(ab1, cd1, 0x5410);
        n[6 + h] = __byte_perm(ab1, cd1, 0x7632);
    }
}

// Bytes of 1024 consecutive samples (sl) summed by ds and written from output j; their sum, and the squares added
// to m2 (integer rows with a.squares).
template <bool INT_OUT>
__device__ __forceinline__ uint32_t put_bytes(const B1Args& a, const uint32_t* sl, int my, int64_t j, int lane,
                                              unsigned long long& m2) {
    const int ds = 1 << a.lds;
    int32_t* o = (INT_OUT ? a.out_i : reinterpret_cast<int32_t*>(a.out_f)) + (int64_t)my * a.out_stride + j;
    const int left = (int)min((int64_t)(SLICE >> a.lds), a.nv - j);
    uint32_t part = 0;
    auto store = [&](int q, uint32_t v) {
        part += v;
        if (INT_OUT && a.squares) m2 += (unsigned long long)v * v;
        if (INT_OUT) o[q] = (int32_t)v;
        else reinterpret_cast<float*>(o)[q] = (float)v;
    };
    if (a.lds == 0) {
        const uint8_t* b = reinterpret_cast<const uint8_t*>(sl);
        if (left == SLICE) {
            if (!INT_OUT && a.vec4) {
#pragma unroll
                for (int i = 0; i < SLICE / 128; ++i) {
                    const uint32_t w = sl[lane + 32 * i];
                    part = __dp4a(w, 0x01010101u, part);
                    // byte to float through the mantissa of 2^23
                    float4 f;
                    f.x = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440)) - 8388608.f;
                    f.y = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7441)) - 8388608.f;
                    f.z = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7442)) - 8388608.f;
                    f.w = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7443)) - 8388608.f;
                    reinterpret_cast<float4*>(o)[lane + 32 * i] = f;
                }
            } else {
#pragma unroll 8
                for (int i = 0; i < SLICE / 32; ++i) store(lane + 32 * i, b[lane + 32 * i]);
            }
        } else {
            for (int q = lane; q < left; q += 32) store(q, b[q]);
        }
    } else if (a.lds == 1) {
        const uint16_t* h = reinterpret_cast<const uint16_t*>(sl);
#pragma unroll 4
        for (int q = lane; q < left; q += 32) store(q, __dp4a((uint32_t)h[q], 0x01010101u, 0u));
    } else {
#pragma unroll 4
        for (int q = lane; q < left; q += 32) {
            uint32_t v = 0;
            for (int e = 0; e < ds / 4; ++e) v = __dp4a(sl[q * (ds / 4) + e], 0x01010101u, v);
            store(q, v);
        }
    }
    return part;
}

template <bool INT_OUT, int KW>
__global__ void __launch_bounds__(NT, 2) k_dedisp_b1(const __grid_constant__ B1Args a) {
    extern __shared__ __align__(128) uint8_t sm[];
    // rows [ck][rowb], a row of zeros, offsets [G][ckp], slices, barrier
    const int zrow = a.ck * a.rowb;
    uint32_t* offs = reinterpret_cast<uint32_t*>(sm + zrow + KW * 128 + 16);
    uint8_t* slices = reinterpret_cast<uint8_t*>(offs + a.G * a.ckp);
    uint64_t* bar = reinterpret_cast<uint64_t*>(slices + NW * SLICE);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * (1024 * KW);
    const int g0 = blockIdx.y * a.G;
    const int gn = min(a.G, a.nb - g0);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_expect_tx(bar, (uint32_t)(a.ck * a.rowb));
    __syncthreads();
    // (a limit of one poll, which tests set to see the wait run out, takes it here: after the offsets below the copies
    // have mostly landed)
    const bool in_time = a.wait_polls != 1 || warp != 0 || mbar_wait(bar, 0, 1);
    // channel c: the earliest delay of the group's trials, from a 16-byte boundary (128 samples), on
    bool bad = false;
    for (int c = threadIdx.x; c < a.ckp; c += NT) {
        if (c >= a.ck) {  // padding: the row of zeros
            for (int g = 0; g < gn; ++g) offs[g * a.ckp + c] = (uint32_t)zrow << 5;
            continue;
        }
        const int32_t* d = a.delays + (int64_t)g0 * a.ck + c;
        int32_t dmin = d[0];
#pragma unroll 8
        for (int g = 1; g < gn; ++g) dmin = min(dmin, d[(int64_t)g * a.ck]);
        const int32_t rs = dmin & ~127;
        bulk_g2s(sm + c * a.rowb, a.xb + (int64_t)c * a.pitchb + (t0 + rs) / 8, (uint32_t)a.rowb, bar);
#pragma unroll 8
        for (int g = 0; g < gn; ++g) {
            const int32_t o = d[(int64_t)g * a.ck] - rs;
            // the words o / 32 .. o / 32 + 32 KW of the row must be there
            const bool out = 4 * ((o >> 5) + 32 * KW + 1) > a.rowb;
            bad |= out;
            offs[g * a.ckp + c] = out ? (uint32_t)zrow << 5 : (uint32_t)(c * a.rowb + (o >> 5) * 4) << 5 | (o & 31);
        }
    }
    for (int i = threadIdx.x; i < KW * 32 + 4; i += NT) reinterpret_cast<uint32_t*>(sm + zrow)[i] = 0u;
    const int any_bad = __syncthreads_or(bad);
    const bool ok = in_time && (warp != 0 || mbar_wait(bar, 0, a.wait_polls));
    if (__syncthreads_or(!ok) || any_bad) {
        // (any_bad: a spread larger than the launch was sized for)
        if (threadIdx.x == 0 && a.err) atomicExch(a.err, any_bad ? 2 : 1);
        mbar_wait(bar, 0);  // let the copies in flight land before the shared memory is released (the full bound)
        return;
    }
    uint32_t* sl = reinterpret_cast<uint32_t*>(slices + warp * SLICE);
    const uint8_t* base = sm + 4 * lane;
    for (int tr = warp; tr < gn; tr += NW) {
        uint32_t p[KW][8];
#pragma unroll
        for (int k = 0; k < KW; ++k)
#pragma unroll
            for (int b = 0; b < 8; ++b) p[k][b] = 0u;
        const uint4* of = reinterpret_cast<const uint4*>(offs + tr * a.ckp);
#pragma unroll 1
        for (int cb = 0; cb < a.ckp; cb += CB) {
            uint32_t e[2][KW];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint4 ma = of[cb / 4 + 2 * h], mb = of[cb / 4 + 2 * h + 1];
                const uint32_t m[8] = {ma.x, ma.y, ma.z, ma.w, mb.x, mb.y, mb.z, mb.w};
#pragma unroll
                for (int k = 0; k < KW; ++k) {
                    uint32_t x[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t* w = reinterpret_cast<const uint32_t*>(base + (m[i] >> 5)) + 32 * k;
                        x[i] = __funnelshift_r(w[0], w[1], m[i]);  // the shift is taken modulo 32
                    }
                    e[h][k] = count8(x, p[k][0], p[k][1], p[k][2]);
                }
            }
#pragma unroll
            for (int k = 0; k < KW; ++k) {
                uint32_t s = maj3(p[k][3], e[0][k], e[1][k]);
                p[k][3] = xor3(p[k][3], e[0][k], e[1][k]);
#pragma unroll
                for (int b = 4; b < 8; ++b) {
                    const uint32_t t = p[k][b] & s;
                    p[k][b] ^= s;
                    s = t;
                }
            }
        }
        unsigned long long part = 0ull, m2 = 0ull;
#pragma unroll
        for (int k = 0; k < KW; ++k) {
            const int64_t t = t0 + 1024 * k;
            const int64_t j = t >> a.lds;
            if (j >= a.nv) break;
            uint32_t n[8];
            planes_to_bytes(p[k], n);
            __syncwarp();
            // lane l: samples 32 l .. 32 l + 31 of the 1024
            reinterpret_cast<uint4*>(sl)[2 * lane] = make_uint4(n[0], n[1], n[2], n[3]);
            reinterpret_cast<uint4*>(sl)[2 * lane + 1] = make_uint4(n[4], n[5], n[6], n[7]);
            __syncwarp();
            part += put_bytes<INT_OUT>(a, sl, g0 + tr, j, lane, m2);
        }
        if (a.sums) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
            if (lane == 0) atomicAdd(a.sums + g0 + tr, part);
        }
        if (INT_OUT && a.squares) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, off);
            if (lane == 0) atomicAdd(a.squares + g0 + tr, m2);
        }
    }
}

size_t b1_smem(int ck, int ckp, int rowb, int G, int KW) {
    return (size_t)ck * rowb + KW * 128 + 16 + (size_t)G * ckp * 4 + NW * SLICE + 16;
}

template <bool I, int KW>
cudaError_t launch_t(const B1Args& a, dim3 grid, size_t shm, cudaStream_t s) {
    cudaError_t e = allow_smem((const void*)k_dedisp_b1<I, KW>, shm);
    if (e != cudaSuccess) return e;
    k_dedisp_b1<I, KW><<<grid, NT, shm, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

// Launch sizes: words per lane (4, or 2 where four do not leave room for two
// CTAs per SM), the row bytes and the shared memory.
bool b1_sizes(int32_t spread, int32_t ck, int G, int* KW, int* rowb, size_t* shm) {
    if (ck < 1 || ck > 255 || spread < 0 || spread > 1 << 20) return false;  // counts are bytes
    const int ckp = (ck + CB - 1) / CB * CB;
    for (int kw = 4; kw >= 2; kw -= 2) {
        const int64_t rb = (4 * ((int64_t)(spread + 127) / 32 + 32 * kw + 1) + 15) & ~int64_t(15);
        if (rb > B1_SLACK) continue;
        const size_t need = b1_smem(ck, ckp, (int)rb, G, kw);
        if (need > (kw == 4 ? (size_t)112 : (size_t)220) * 1024) continue;
        *KW = kw;
        *rowb = (int)rb;
        *shm = need;
        return true;
    }
    return false;
}

cudaError_t launch_prep_bits(const PrepArgs& a, uint8_t* xb, int64_t pitchb, cudaStream_t s) {
    const int64_t pw = pitchb / 4;
    dim3 grid((unsigned)((pw + 31) / 32), (unsigned)((a.ck + 31) / 32));
    k_prep_bits<<<grid, 256, 0, s>>>(a, reinterpret_cast<uint32_t*>(xb), pw);
    return cudaGetLastError();
}

cudaError_t launch_dedisp_b1(B1Args a, int32_t spread, cudaStream_t s) {
    if (a.nb <= 0 || a.nv <= 0) return cudaSuccess;
    int KW = 0;
    size_t shm = 0;
    if (a.lds < 0 || a.lds > 10 || !b1_sizes(spread, a.ck, a.G, &KW, &a.rowb, &shm)) return cudaErrorInvalidValue;
    a.ckp = (a.ck + CB - 1) / CB * CB;
    const int64_t L = a.nv << a.lds;
    dim3 grid((unsigned)((L + 1024 * KW - 1) / (1024 * KW)), (unsigned)((a.nb + a.G - 1) / a.G));
    if (a.out_i) return KW == 4 ? launch_t<true, 4>(a, grid, shm, s) : launch_t<true, 2>(a, grid, shm, s);
    return KW == 4 ? launch_t<false, 4>(a, grid, shm, s) : launch_t<false, 2>(a, grid, shm, s);
}

}  // namespace pss
