// Work tables of the shared-sum dedispersion kernel (k_dedisp_sh.cu).
//
// The trials of a launch are cut into groups of consecutive ones.  Within a
// group the delays of S neighbouring channels relative to the first of them
// take only a few values (each moves by a fraction of a sample per trial), so
// the partial sum over those S channels is the same for many trials up to a
// shift in time.  A unit is such a run of channels; each distinct set of
// relative delays e_c in a group is a pattern, and its partial sums are one row:
//   row[x] = sum_c x_c[t0 + wmin + e_c + x],  x < TN + (wmax - wmin),
// wmin / wmax the smallest / largest delay a_i of the unit's first channel over
// the trials of the pattern.  Trial i then adds row[a_i - wmin + t], t < TN, of
// its pattern: the same integers in another order.
//
// Units are packed into chunks that fit the kernel's shared memory; all units
// of a chunk have the same S and all its rows the same length.
#include <string.h>

#include "pss_internal.h"

namespace pss {

namespace {

constexpr int TN = DD_TN, GT = DD_GT;

// Patterns of the unit [c0, c0 + S) for the trials of one group.
struct Unit {
    int c0 = 0, S = 0, npat = 0, width = 0;  // width: largest wmax - wmin
    int16_t pat[GT];                         // pattern of each trial
    int32_t first[GT];                       // a trial of each pattern
    int32_t wmin[GT], wmax[GT];
};

void unit_patterns(const int32_t* d, int ck, int n, int c0, int S, Unit* u) {
    u->c0 = c0;
    u->S = S;
    u->npat = 0;
    u->width = 0;
    for (int i = 0; i < n; ++i) {
        const int32_t* di = d + (int64_t)i * ck + c0;
        int p = u->npat - 1;  // neighbouring trials mostly share a pattern: search backwards
        for (; p >= 0; --p) {
            const int32_t* df = d + (int64_t)u->first[p] * ck + c0;
            bool same = true;
            for (int c = 1; c < S; ++c) same &= (di[c] - di[0]) == (df[c] - df[0]);
            if (same) break;
        }
        if (p < 0) {
            p = u->npat++;
            u->first[p] = i;
            u->wmin[p] = u->wmax[p] = di[0];
        }
        u->wmin[p] = std::min(u->wmin[p], di[0]);
        u->wmax[p] = std::max(u->wmax[p], di[0]);
        u->pat[i] = (int16_t)p;
    }
    for (int p = 0; p < u->npat; ++p) u->width = std::max(u->width, u->wmax[p] - u->wmin[p]);
}

// 4-sample columns of a row: what the trials read and one word past it, in whole runs of DD_M columns
int cols_of(int width) { return ((TN + width + 2 + 3) / 4 + DD_M - 1) / DD_M * DD_M; }

// Shared-memory wavefronts per 128 samples of a tile that a unit costs (the kernel is bound by them): a row reads
// (DD_M + 1) / DD_M words per channel and writes 2 words of sums, a trial reads 2 words.
double unit_cost(const Unit& u, int n) {
    return (double)u.npat * cols_of(u.width) * 4.0 / TN * (u.S * (1.0 + 1.0 / DD_M) + 2.5) + (double)n * 2.2;
}

struct GroupTab {
    std::vector<DdChunk> chunks;
    std::vector<int2> chans;
    std::vector<uint8_t> blob;
    double cost = 0;
    bool ok = true;
};

void build_group(const int32_t* d, int ck, int n, GroupTab* T) {
    std::vector<int32_t> lo(ck), hi(ck);
    for (int c = 0; c < ck; ++c) lo[c] = hi[c] = d[c];
    for (int i = 1; i < n; ++i)
        for (int c = 0; c < ck; ++c) {
            lo[c] = std::min(lo[c], d[(int64_t)i * ck + c]);
            hi[c] = std::max(hi[c], d[(int64_t)i * ck + c]);
        }
    auto raw_len = [&](int c) { return (hi[c] - (lo[c] & ~15) + TN + 4 + 15) & ~15; };
    // runs of 4 channels where that is cheaper than two runs of 2
    std::vector<Unit> units;
    Unit u4, a, b;
    for (int c = 0; c < ck;) {
        const int left = ck - c;
        if (left >= 4) {
            unit_patterns(d, ck, n, c, 4, &u4);
            unit_patterns(d, ck, n, c, 2, &a);
            unit_patterns(d, ck, n, c + 2, 2, &b);
            if (unit_cost(u4, n) <= unit_cost(a, n) + unit_cost(b, n)) {
                units.push_back(u4);
            } else {
                units.push_back(a);
                units.push_back(b);
            }
            c += 4;
        } else {
            const int S = left >= 2 ? 2 : 1;
            unit_patterns(d, ck, n, c, S, &a);
            units.push_back(a);
            c += S;
        }
    }
    T->chans.resize(ck);
    int since_flush = 0;
    for (size_t i0 = 0; i0 < units.size();) {
        DdChunk k{};
        k.c0 = units[i0].c0;
        k.S = units[i0].S;
        int raw = 0, rows = 0, ncol = 0;
        size_t i1 = i0;
        while (i1 < units.size() && units[i1].S == k.S && (int)(i1 - i0) < DD_MAXUNITS) {
            const Unit& u = units[i1];
            int r2 = raw;
            for (int c = 0; c < u.S; ++c) r2 += raw_len(u.c0 + c);
            const int rows2 = rows + u.npat, ncol2 = std::max(ncol, cols_of(u.width));
            if (r2 > DD_RAWCAP || rows2 > DD_MAXROWS || (int64_t)rows2 * ncol2 * 8 > DD_UCAP) break;
            // 16-bit sums hold 257 channels of 8 bits: a chunk stays within one flush period
            if (since_flush + (int)(u.c0 + u.S - k.c0) > 257) break;
            raw = r2;
            rows = rows2;
            ncol = ncol2;
            ++i1;
        }
        if (i1 == i0) {
            if (since_flush > 0 && !T->chunks.empty()) {
                T->chunks.back().flush = 1;
                since_flush = 0;
                continue;
            }
            T->ok = false;  // one unit alone does not fit (a very large delay spread)
            return;
        }
        k.nunit = (int32_t)(i1 - i0);
        k.nrow = rows;
        k.nrun = ncol / DD_M;
        k.ishift = 5;
        while ((1 << k.ishift) < k.nrun) ++k.ishift;
        int dst = 0;
        for (size_t i = i0; i < i1; ++i)
            for (int c = units[i].c0; c < units[i].c0 + units[i].S; ++c) {
                T->chans[c] = make_int2(lo[c] & ~15, (raw_len(c) / 16) << 16 | dst / 16);
                dst += raw_len(c);
                k.nch++;
            }
        // this record, the next chunk's record and channels (filled in dd_tables), the rows' sources, the trials'
        // unit counts, the trials' lists
        k.src_off = DD_BLOBHEAD;
        k.cnt_off = k.src_off + rows * 16;
        k.list_off = k.cnt_off + GT * 2;
        k.npair = k.nunit / 2 + 1;
        k.blob_bytes = (k.list_off + GT * k.npair * 4 + 15) & ~15;
        k.tx_bytes = dst + k.blob_bytes;
        k.blob_off = (int64_t)T->blob.size();
        T->blob.resize(T->blob.size() + k.blob_bytes, 0);
        uint8_t* blob = T->blob.data() + k.blob_off;
        uint32_t* src = reinterpret_cast<uint32_t*>(blob + k.src_off);
        uint16_t* cnt = reinterpret_cast<uint16_t*>(blob + k.cnt_off);
        uint32_t* list = reinterpret_cast<uint32_t*>(blob + k.list_off);
        int r = 0;
        std::vector<int> row0;
        for (size_t i = i0; i < i1; ++i) {
            const Unit& u = units[i];
            row0.push_back(r);
            for (int p = 0; p < u.npat; ++p) {
                const int32_t* df = d + (int64_t)u.first[p] * ck;
                for (int c = 0; c < u.S; ++c) {
                    const int ch = u.c0 + c;
                    const int rel = u.wmin[p] + (df[ch] - df[u.c0]) - T->chans[ch].x;  // >= 0: lo <= that delay
                    const int so = (T->chans[ch].y & 0xFFFF) * 16 + rel;
                    src[4 * (r + p) + c] = (uint32_t)(so & ~3) << 5 | (uint32_t)(so & 3) * 8;
                }
            }
            r += u.npat;
            T->cost += unit_cost(u, n);
        }
        // each trial's word offsets: units at even offsets first, then the odd ones from the next pair on
        for (int t = 0; t < n; ++t) {
            uint32_t* L = list + t * k.npair;
            int cntp[2] = {0, 0}, pairs = 0;
            for (int par = 0; par < 2; ++par) {
                int m = 0;
                for (size_t i = i0; i < i1; ++i) {
                    const Unit& u = units[i];
                    const int off = (row0[i - i0] + u.pat[t]) * ncol * 4 + (d[(int64_t)t * ck + u.c0] - u.wmin[u.pat[t]]);
                    if ((off & 1) != par) continue;
                    const uint32_t w = (uint32_t)(off / 2);
                    L[pairs + m / 2] |= (m & 1) ? w << 16 : w;
                    ++m;
                }
                cntp[par] = m;
                pairs += (m + 1) / 2;
            }
            cnt[t] = (uint16_t)(cntp[0] | cntp[1] << 8);
        }
        T->chunks.push_back(k);
        since_flush += k.nch;
        i0 = i1;
    }
    if (!T->chunks.empty()) T->chunks.back().flush = 1;
}

}  // namespace

bool dd_tables(const int32_t* delays, int64_t nb, int32_t ck, DdTables* out) {
    const int ng = (int)((nb + GT - 1) / GT);
    out->ngroups = ng;
    if (ng == 0 || ck <= 0) return false;
    std::vector<GroupTab> tabs(ng);
    parallel_for(ng, 1, [&](int64_t g) {
        build_group(delays + (size_t)g * GT * ck, ck, (int)std::min<int64_t>(GT, nb - g * GT), &tabs[g]);
    });
    size_t nchunk = 0, nblob = 0;
    double cost = 0;
    for (const auto& t : tabs) {
        if (!t.ok) return false;
        nchunk += t.chunks.size();
        nblob += t.blob.size();
        cost += t.cost;
    }
    // [groups int4][chunks][channels int2][blobs]; every part on a 16-byte boundary
    out->chunk_off = (size_t)ng * sizeof(int4);
    out->chan_off = out->chunk_off + nchunk * sizeof(DdChunk);
    const size_t blob0 = (out->chan_off + (size_t)ng * ck * sizeof(int2) + 15) & ~size_t(15);
    out->bytes.assign(blob0 + nblob, 0);
    uint8_t* B = out->bytes.data();
    size_t ci = 0, bo = blob0;
    for (int g = 0; g < ng; ++g) {
        GroupTab& t = tabs[g];
        const int4 gi = make_int4((int)ci, (int)t.chunks.size(), 0, 0);
        memcpy(B + (size_t)g * sizeof(int4), &gi, sizeof gi);
        for (auto& k : t.chunks) k.blob_off += (int64_t)bo;
        for (size_t i = 0; i < t.chunks.size(); ++i) {
            uint8_t* head = t.blob.data() + (t.chunks[i].blob_off - (int64_t)bo);
            memcpy(head, &t.chunks[i], sizeof(DdChunk));
            if (i + 1 == t.chunks.size()) continue;
            const DdChunk& nx = t.chunks[i + 1];
            memcpy(head + sizeof(DdChunk), &nx, sizeof(DdChunk));
            memcpy(head + 2 * sizeof(DdChunk), t.chans.data() + nx.c0, nx.nch * sizeof(int2));
        }
        memcpy(B + out->chunk_off + ci * sizeof(DdChunk), t.chunks.data(), t.chunks.size() * sizeof(DdChunk));
        memcpy(B + out->chan_off + (size_t)g * ck * sizeof(int2), t.chans.data(), (size_t)ck * sizeof(int2));
        memcpy(B + bo, t.blob.data(), t.blob.size());
        ci += t.chunks.size();
        bo += t.blob.size();
    }
    out->cost = cost;
    return true;
}

size_t dd_tables_bound(int64_t n, int64_t ck, int64_t nb) {
    const int64_t batches = (n + nb - 1) / nb, groups = n / GT + batches;
    // per channel at most one unit and one chunk: a row and a pair per trial, a chunk record, a channel entry
    return (size_t)groups * (sizeof(int4) + (size_t)ck * (GT * 28 + 16 + sizeof(DdChunk) + sizeof(int2))) + (size_t)batches * 512;
}

}  // namespace pss
