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
//
// A call on new trials or a new mask pays for this, so files that do not gain
// are left early, patterns are told apart by one key per trial, segments of
// channels and chunks are spread over the worker pool and written where they
// are uploaded from.  Calls with another DM range each time (16 Arm cores),
// without the kernel / with each group built and copied by one task / here:
// 8 trials x 1024 channels 256, 336, 239 us; 33 trials 445, 614, 412 us; a
// search of 101 trials x 64 channels (which does not take the tables) 584, 675,
// 570 us.
#include <string.h>

#include "pss_internal.h"

namespace pss {

namespace {

constexpr int TN = DD_TN, GT = DD_GT;

// Patterns of the unit [c0, c0 + S) for the trials of one group.
struct Unit {
    int c0 = 0, S = 0, npat = 0, width = 0;  // width: largest wmax - wmin
    uint8_t pat[GT];                         // pattern of each trial
    uint8_t first[GT];                       // a trial of each pattern
    int32_t wmin[GT], wmax[GT];
};
static_assert(GT <= 256, "trials of a group in bytes");

// A unit under construction: trial after trial by its key, which names the delays relative to the first channel's.
template <typename K>
struct Builder {
    K key[GT];
    void begin(Unit* u, int c0, int S) {
        u->c0 = c0;
        u->S = S;
        u->npat = 0;
        u->width = 0;
    }
    void add(Unit* u, int i, K k, int32_t a) {
        int p = u->npat - 1;  // neighbouring trials mostly share a pattern: search backwards
        while (p >= 0 && key[p] != k) --p;
        if (p < 0) {
            p = u->npat++;
            key[p] = k;
            u->first[p] = (uint8_t)i;
            u->wmin[p] = u->wmax[p] = a;
        }
        u->wmin[p] = std::min(u->wmin[p], a);
        u->wmax[p] = std::max(u->wmax[p], a);
        u->pat[i] = (uint8_t)p;
    }
    void end(Unit* u) {
        for (int p = 0; p < u->npat; ++p) u->width = std::max(u->width, u->wmax[p] - u->wmin[p]);
    }
};

// 4-sample columns of a row: what the trials read and one word past it, in whole runs of DD_M columns
int cols_of(int width) { return ((TN + width + 2 + 3) / 4 + DD_M - 1) / DD_M * DD_M; }

// Shared-memory wavefronts per 128 samples of a tile that a unit costs (the kernel is bound by them): a row reads
// (DD_M + 1) / DD_M words per channel and writes 2 words of sums, a trial reads 2 words.
double unit_cost(const Unit& u, int n) {
    return (double)u.npat * cols_of(u.width) * 4.0 / TN * (u.S * (1.0 + 1.0 / DD_M) + 2.5) + (double)n * 2.2;
}

constexpr int SEG = 128;  // channels whose patterns are found by one task (a multiple of 4)

struct Segment {
    std::vector<Unit> units;
    double cost = 0;
    bool ok = true;
};

struct Group {
    const int32_t* d = nullptr;   // delays [n][ck] of its trials
    int n = 0;
    std::vector<int32_t> lo, hi;  // smallest and largest delay of each channel
    std::vector<Segment> segs;
    std::vector<const Unit*> units;  // of all segments
    std::vector<DdChunk> chunks;
    std::vector<int> first;          // of each chunk: its first unit
    std::vector<int2> chans;
    size_t bytes = 0;                // of its chunks' tables
    int raw_len(int c) const { return (hi[c] - (lo[c] & ~15) + TN + 4 + 15) & ~15; }
};

// A run of 4 channels at once and as two runs of 2; true where the first is the cheaper.
struct Quad {
    Unit u4, a, b;
    Builder<uint64_t> k4;
    Builder<uint32_t> ka, kb;
    bool find(const Group& G, int ck, int c) {
        const int32_t* di = G.d + c;
        k4.begin(&u4, c, 4);
        ka.begin(&a, c, 2);
        kb.begin(&b, c + 2, 2);
        for (int i = 0; i < G.n; ++i, di += ck) {
            const uint32_t d0 = di[0], e1 = di[1] - d0, e2 = di[2] - d0, e3 = di[3] - d0;
            const uint64_t m = (1u << 21) - 1;
            k4.add(&u4, i, (e1 & m) | (e2 & m) << 21 | (e3 & m) << 42, di[0]);
            ka.add(&a, i, e1, di[0]);
            kb.add(&b, i, e3 - e2, di[2]);
        }
        k4.end(&u4);
        ka.end(&a);
        kb.end(&b);
        return unit_cost(u4, G.n) <= unit_cost(a, G.n) + unit_cost(b, G.n);
    }
};

// The units of channels [c0, c1), runs of 4 channels where that is cheaper than two runs of 2, and their cost.
void segment_units(Group& G, int ck, int c0, int c1, Segment* T) {
    const int n = G.n;
    for (int i = 0; i < n; ++i) {
        const int32_t* di = G.d + (int64_t)i * ck;
        for (int c = c0; c < c1; ++c) {
            G.lo[c] = i ? std::min(G.lo[c], di[c]) : di[c];
            G.hi[c] = i ? std::max(G.hi[c], di[c]) : di[c];
        }
    }
    // (a delay spread larger than the staging area; within it a channel's delay less the first one's differs by less
    // than 2^20 from trial to trial, so 21 bits of it tell the patterns apart)
    static_assert(DD_RAWCAP < 1 << 19, "21-bit keys");
    for (int c = c0; c < c1; ++c)
        if ((int64_t)G.hi[c] - G.lo[c] > DD_RAWCAP) {
            T->ok = false;
            return;
        }
    T->units.reserve((c1 - c0) / 2 + 2);
    Quad q;
    auto take = [&](const Unit& u) {
        T->cost += unit_cost(u, n);
        T->units.push_back(u);
    };
    int c = c0;
    for (; c + 4 <= c1; c += 4) {
        if (q.find(G, ck, c)) {
            take(q.u4);
        } else {
            take(q.a);
            take(q.b);
        }
    }
    while (c < c1) {
        const int32_t* di = G.d + c;
        q.ka.begin(&q.a, c, c1 - c >= 2 ? 2 : 1);
        for (int i = 0; i < n; ++i, di += ck) q.ka.add(&q.a, i, q.a.S == 2 ? (uint32_t)di[1] - (uint32_t)di[0] : 0u, di[0]);
        q.ka.end(&q.a);
        take(q.a);
        c += q.a.S;
    }
}

// Pack a group's units into chunks: their records (blob_off from the group's first) and channel entries.  False where
// one unit alone does not fit.
bool group_chunks(Group* G, int ck) {
    for (const Segment& sg : G->segs)
        for (const Unit& u : sg.units) G->units.push_back(&u);
    const std::vector<const Unit*>& units = G->units;
    G->chans.resize(ck);
    int since_flush = 0;
    for (size_t i0 = 0; i0 < units.size();) {
        DdChunk k{};
        k.c0 = units[i0]->c0;
        k.S = units[i0]->S;
        int raw = 0, rows = 0, ncol = 0;
        size_t i1 = i0;
        while (i1 < units.size() && units[i1]->S == k.S && (int)(i1 - i0) < DD_MAXUNITS) {
            const Unit& u = *units[i1];
            int r2 = raw;
            for (int c = 0; c < u.S; ++c) r2 += G->raw_len(u.c0 + c);
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
            if (since_flush > 0 && !G->chunks.empty()) {
                G->chunks.back().flush = 1;
                since_flush = 0;
                continue;
            }
            return false;  // one unit alone does not fit (a very large delay spread)
        }
        k.nunit = (int32_t)(i1 - i0);
        k.nrow = rows;
        k.nrun = ncol / DD_M;
        k.ishift = 5;
        while ((1 << k.ishift) < k.nrun) ++k.ishift;
        int dst = 0;
        for (size_t i = i0; i < i1; ++i)
            for (int c = units[i]->c0; c < units[i]->c0 + units[i]->S; ++c) {
                G->chans[c] = make_int2(G->lo[c] & ~15, (G->raw_len(c) / 16) << 16 | dst / 16);
                dst += G->raw_len(c);
                k.nch++;
            }
        // this record, the next chunk's record and channels, the rows' sources, the trials' unit counts, their lists
        k.src_off = DD_BLOBHEAD;
        k.cnt_off = k.src_off + rows * 16;
        k.list_off = k.cnt_off + GT * 2;
        k.npair = k.nunit / 2 + 1;
        k.blob_bytes = (k.list_off + GT * k.npair * 4 + 15) & ~15;
        k.tx_bytes = dst + k.blob_bytes;
        k.blob_off = (int64_t)G->bytes;
        G->bytes += k.blob_bytes;
        G->chunks.push_back(k);
        G->first.push_back((int)i0);
        since_flush += k.nch;
        i0 = i1;
    }
    if (!G->chunks.empty()) G->chunks.back().flush = 1;
    return true;
}

// Fill chunk ci's table (zeroed before).
void fill_chunk(const Group& G, int ck, int ci, uint8_t* blob) {
    const DdChunk& k = G.chunks[ci];
    memcpy(blob, &k, sizeof(DdChunk));
    if (ci + 1 < (int)G.chunks.size()) {
        const DdChunk& nx = G.chunks[ci + 1];
        memcpy(blob + sizeof(DdChunk), &nx, sizeof(DdChunk));
        memcpy(blob + 2 * sizeof(DdChunk), G.chans.data() + nx.c0, nx.nch * sizeof(int2));
    }
    const Unit* const* units = G.units.data() + G.first[ci];
    uint32_t* src = reinterpret_cast<uint32_t*>(blob + k.src_off);
    uint16_t* cnt = reinterpret_cast<uint16_t*>(blob + k.cnt_off);
    uint32_t* list = reinterpret_cast<uint32_t*>(blob + k.list_off);
    const int ncol = k.nrun * DD_M;
    int row0[DD_MAXUNITS], r = 0;
    for (int i = 0; i < k.nunit; ++i) {
        const Unit& u = *units[i];
        row0[i] = r;
        for (int p = 0; p < u.npat; ++p) {
            const int32_t* df = G.d + (int64_t)u.first[p] * ck;
            for (int c = 0; c < u.S; ++c) {
                const int ch = u.c0 + c;
                const int rel = u.wmin[p] + (df[ch] - df[u.c0]) - G.chans[ch].x;  // >= 0: lo <= that delay
                const int so = (G.chans[ch].y & 0xFFFF) * 16 + rel;
                src[4 * (r + p) + c] = (uint32_t)(so & ~3) << 5 | (uint32_t)(so & 3) * 8;
            }
        }
        r += u.npat;
    }
    // each trial's word offsets: units at even offsets first, then the odd ones from the next pair on
    for (int t = 0; t < G.n; ++t) {
        uint32_t* L = list + t * k.npair;
        const int32_t* dt = G.d + (int64_t)t * ck;
        uint16_t w[2][DD_MAXUNITS + 1];
        int m[2] = {0, 0};
        for (int i = 0; i < k.nunit; ++i) {
            const Unit& u = *units[i];
            const int off = (row0[i] + u.pat[t]) * ncol * 4 + (dt[u.c0] - u.wmin[u.pat[t]]);
            w[off & 1][m[off & 1]++] = (uint16_t)(off / 2);
        }
        for (int par = 0; par < 2; ++par) {
            w[par][m[par]] = 0;
            for (int q = 0; q < m[par]; q += 2) *L++ = (uint32_t)w[par][q] | (uint32_t)w[par][q + 1] << 16;
        }
        cnt[t] = (uint16_t)(m[0] | m[1] << 8);
    }
}

}  // namespace

bool dd_tables(const int32_t* delays, int64_t nb, int32_t ck, double max_cost, std::vector<uint8_t>* host, DdTables* out) {
    const int ng = (int)((nb + GT - 1) / GT);
    out->ngroups = ng;
    if (ng == 0 || ck <= 0) return false;
    // Groups of one stage cost nearly the same per trial (their delays move by the same steps), and neighbouring runs of
    // channels too: every fourth run of the first group tells what costs far too much
    {
        Group g;
        g.d = delays;
        g.n = (int)std::min<int64_t>(GT, nb);
        Quad q;
        double est = 0;
        int nq = 0;
        for (int c = 0; c + 4 <= ck; c += 16, ++nq)
            est += q.find(g, ck, c) ? unit_cost(q.u4, g.n) : unit_cost(q.a, g.n) + unit_cost(q.b, g.n);
        if (est > 1.02 * max_cost * 4 * nq * g.n) return false;
    }
    const int nseg = (ck + SEG - 1) / SEG;
    std::vector<Group> G(ng);
    for (int g = 0; g < ng; ++g) {
        G[g].d = delays + (size_t)g * GT * ck;
        G[g].n = (int)std::min<int64_t>(GT, nb - (int64_t)g * GT);
        G[g].lo.resize(ck);
        G[g].hi.resize(ck);
        G[g].segs.resize(nseg);
    }
    double cost = 0;
    // tasks of 10 us and more: handing less to the workers takes longer than doing it
    const int64_t grain = std::max<int64_t>(1, 4096 / ((int64_t)G[0].n * std::min<int32_t>(ck, SEG)));
    parallel_for((int64_t)ng * nseg, grain, [&](int64_t t) {
        const int g = (int)(t / nseg), sg = (int)(t % nseg);
        segment_units(G[g], ck, sg * SEG, std::min(ck, (sg + 1) * SEG), &G[g].segs[sg]);
    });
    for (const Group& g : G)
        for (const Segment& sg : g.segs) {
            if (!sg.ok) return false;
            cost += sg.cost;
        }
    out->cost = cost;
    if (cost > max_cost * (double)nb * ck) return false;
    size_t nchunk = 0, nblob = 0;
    std::vector<int2> at;  // (group, chunk) of every chunk
    for (int g = 0; g < ng; ++g) {
        if (!group_chunks(&G[g], ck)) return false;
        for (size_t i = 0; i < G[g].chunks.size(); ++i) at.push_back(make_int2(g, (int)i));
        nchunk += G[g].chunks.size();
        nblob += G[g].bytes;
    }
    // [groups int4][chunks][channels int2][blobs]; every part on a 16-byte boundary
    out->off = (host->size() + 255) & ~size_t(255);
    out->chunk_off = (size_t)ng * sizeof(int4);
    out->chan_off = out->chunk_off + nchunk * sizeof(DdChunk);
    const size_t blob0 = (out->chan_off + (size_t)ng * ck * sizeof(int2) + 15) & ~size_t(15);
    if (blob0 + nblob > dd_tables_bound(nb, ck)) return false;
    host->resize(out->off + blob0 + nblob);
    uint8_t* B = host->data() + out->off;
    size_t ci = 0, bo = blob0;
    for (int g = 0; g < ng; ++g) {
        Group& t = G[g];
        const int4 gi = make_int4((int)ci, (int)t.chunks.size(), 0, 0);
        memcpy(B + (size_t)g * sizeof(int4), &gi, sizeof gi);
        for (auto& k : t.chunks) k.blob_off += (int64_t)bo;
        memcpy(B + out->chunk_off + ci * sizeof(DdChunk), t.chunks.data(), t.chunks.size() * sizeof(DdChunk));
        memcpy(B + out->chan_off + (size_t)g * ck * sizeof(int2), t.chans.data(), (size_t)ck * sizeof(int2));
        ci += t.chunks.size();
        bo += t.bytes;
    }
    parallel_for((int64_t)at.size(), std::max(8, 256 / G[0].n), [&](int64_t i) {
        const Group& t = G[at[i].x];
        fill_chunk(t, ck, at[i].y, B + t.chunks[at[i].y].blob_off);
    });
    return true;
}

// (tables that gain take 2.2 to 6.5 bytes per trial and channel)
size_t dd_tables_bound(int64_t nb, int64_t ck) { return (size_t)(8 * nb * ck) + 16384; }

}  // namespace pss
