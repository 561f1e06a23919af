// Tables of the band rows (see aa_bands.h).  Host only.
#include <algorithm>
#include <climits>
#include <cstring>
#include <new>
#include <utility>

#include "aa_internal.h"

namespace aa {

namespace {

constexpr size_t kRowSmem = 36 * 1024;   // six CTAs of the row kernel per SM
constexpr size_t kSumSmem = 220 * 1024;  // one CTA of the summing kernel per SM

// Distinct keys of one band in first-seen order (open addressing; cleared by
// stamping).
class KeySet {
  public:
    KeySet() : keys_(kSize), ids_(kSize), stamp_(kSize, 0) {}
    void clear() { ++now_; n_ = 0; }
    // index of `key`; `fresh` set when it is new
    int add(uint64_t key, bool& fresh) {
        size_t h = (size_t)((key * 0x9e3779b97f4a7c15ull) >> 48) & (kSize - 1);
        while (stamp_[h] == now_) {
            if (keys_[h] == key) { fresh = false; return ids_[h]; }
            h = (h + 1) & (kSize - 1);
        }
        stamp_[h] = now_;
        keys_[h] = key;
        ids_[h] = n_;
        fresh = true;
        return n_++;
    }

  private:
    static constexpr size_t kSize = 4096;  // a segment has at most kBandSegment keys
    std::vector<uint64_t> keys_;
    std::vector<int> ids_;
    std::vector<uint32_t> stamp_;
    uint32_t now_ = 0;
    int n_ = 0;
};

// Tables for bands of k channels; false where a row's delays, a block's rows
// or a slot do not fit.
bool build(const RangePlan& r, int C, int k, BandPlan& bp) {
    bp = BandPlan{};
    bp.k = k;
    bp.nbands = (C + k - 1) / k;
    const int dec = r.desc.dec, ndm = r.desc.ndm;
    if (2 * k * 255 * dec > 65535) return false;  // the sum of two rows stays in a 16-bit lane
    const int npad = (bp.nbands + 1) & ~1;
    const int nblk_all = (ndm + kBandTrials - 1) / kBandTrials;
    bp.heads.resize((size_t)nblk_all * npad);
    bp.offs.resize((size_t)nblk_all * npad * kBandTrials);
    KeySet row_keys, quad_keys;
    std::vector<int> id(kBandSegment);
    std::vector<int32_t> sp(kBandSegment);
    std::vector<uint64_t> key;
    std::vector<int32_t> lo, hi, blo, bhi, bdst;
    std::vector<int> border, pair_dst((size_t)nblk_all, 0);
    int blk_base = 0;
    int max_quads = 0, max_e = 0, max_rq = 0;
    double cost = 0;
    for (int d0 = 0; d0 < ndm; d0 += kBandSegment) {
        BandSegment seg;
        seg.trial0 = d0;
        seg.ntrials = std::min(kBandSegment, ndm - d0);
        seg.nblk = (seg.ntrials + kBandTrials - 1) / kBandTrials;
        seg.blk0 = blk_base;
        const size_t first_copy = bp.copies.size();
        seg.row0 = (uint32_t)bp.rows.size();
        for (int b = 0; b < bp.nbands; ++b) {
            const int c0 = b * k, nch = std::min(k, C - c0);
            const int na = std::min(nch, 4), nb = nch - na;
            row_keys.clear();
            key.clear();
            lo.clear();
            hi.clear();
            for (int i = 0; i < seg.ntrials; ++i) {
                const int32_t* s = &r.shifts[(size_t)(d0 + i) * C + c0];
                int32_t mn = s[0];
                for (int j = 1; j < nch; ++j) mn = std::min(mn, s[j]);
                uint64_t kk = 0;
                for (int j = 0; j < nch; ++j) {
                    const int32_t e = s[j] - mn;
                    if (e > 255) return false;
                    kk |= (uint64_t)e << (8 * j);
                }
                bool fresh;
                const int q = row_keys.add(kk, fresh);
                if (fresh) {
                    key.push_back(kk);
                    lo.push_back(mn);
                    hi.push_back(mn);
                } else {
                    lo[q] = std::min(lo[q], mn);
                    hi[q] = std::max(hi[q], mn);
                }
                id[i] = q;
                sp[i] = mn;
            }
            const int n = (int)key.size();
            BandInfo info{};
            info.row0 = (uint32_t)bp.rows.size();
            info.quad0 = (uint32_t)bp.quads.size();
            info.nrows = (uint16_t)n;
            info.c0 = (uint16_t)c0;
            info.nch = (uint16_t)nch;
            const size_t first_row = bp.rows.size();
            int32_t umin = INT32_MAX, umax = 0;
            // quads of the two halves: their delays with the half's smallest removed
            auto half = [&](uint64_t kk, int j0, int cnt, uint16_t& e) {
                uint16_t rr[4];
                int mn = 255;
                for (int j = 0; j < cnt; ++j) mn = std::min(mn, (int)(kk >> (8 * (j0 + j)) & 255));
                uint64_t qk = 0;
                for (int j = 0; j < 4; ++j) {
                    rr[j] = j < cnt ? (uint16_t)((kk >> (8 * (j0 + j)) & 255) - mn) : 0xffff;
                    qk |= (uint64_t)(j < cnt ? rr[j] : 0) << (8 * j);
                }
                e = (uint16_t)mn;
                bool fresh;
                const int q = quad_keys.add(qk, fresh);
                if (fresh) {
                    BandQuad quad;
                    quad.blk0 = 0xffff;
                    quad.blk1 = 0;
                    std::memcpy(quad.r, rr, sizeof rr);
                    for (int j = 0; j < cnt; ++j) max_rq = std::max(max_rq, (int)rr[j]);
                    bp.quads.push_back(quad);
                }
                return (uint16_t)q;
            };
            for (int q = 0; q < n; ++q) {
                BandRow row{};
                row.qa = row.qb = 0xffff;
                row.smin = lo[q];
                row.span = hi[q] - lo[q];
                row.blk0 = 0xffff;
                umin = std::min(umin, lo[q]);
                umax = std::max(umax, hi[q]);
                bp.rows.push_back(row);
            }
            quad_keys.clear();
            for (int q = 0; q < n; ++q) bp.rows[first_row + q].qa = half(key[q], 0, na, bp.rows[first_row + q].ea);
            info.nqa = (uint16_t)(bp.quads.size() - info.quad0);
            if (nb > 0) {
                quad_keys.clear();
                for (int q = 0; q < n; ++q)
                    bp.rows[first_row + q].qb = (uint16_t)(half(key[q], 4, nb, bp.rows[first_row + q].eb) + info.nqa);
            }
            info.nqb = (uint16_t)(bp.quads.size() - info.quad0 - info.nqa);
            for (int q = 0; q < n; ++q)
                max_e = std::max({max_e, (int)bp.rows[first_row + q].ea, (int)bp.rows[first_row + q].eb});
            info.umin = umin;
            info.ulen = umax - umin;
            max_quads = std::max(max_quads, (int)info.nqa + info.nqb);
            bp.max_ulen = std::max(bp.max_ulen, info.ulen);
            bp.max_rows = std::max(bp.max_rows, n);
            // the blocks: which rows each uses, at which delays
            for (int g = 0; g < seg.nblk; ++g) {
                const int i0 = g * kBandTrials, i1 = std::min(seg.ntrials, i0 + kBandTrials);
                blo.assign((size_t)n, INT32_MAX);
                bhi.assign((size_t)n, -1);
                bdst.assign((size_t)n, 0);
                border.clear();
                for (int i = i0; i < i1; ++i) {
                    const int q = id[i];
                    if (bhi[q] < 0) border.push_back(q);
                    blo[q] = std::min(blo[q], sp[i]);
                    bhi[q] = std::max(bhi[q], sp[i]);
                }
                if ((int)border.size() > kBandMaxRows) return false;
                const size_t bb = (size_t)(blk_base + g) * npad + b;
                BandHead& h = bp.heads[bb];
                h.first = (uint32_t)bp.copies.size();
                h.n = (uint16_t)border.size();
                // the second band of a pair goes behind the first
                const int dst0 = b & 1 ? pair_dst[blk_base + g] : 0;
                int dst = dst0;
                for (int q : border) {
                    BandRow& row = bp.rows[first_row + q];
                    row.blk0 = std::min<uint16_t>(row.blk0, (uint16_t)g);
                    row.blk1 = std::max<uint16_t>(row.blk1, (uint16_t)g);
                    const int32_t at = blo[q] - row.smin;
                    BandCopy c;
                    c.row = (uint32_t)(first_row + q) - seg.row0;  // its place follows
                    c.rel = (uint32_t)(at & ~3);
                    c.dst = (uint32_t)dst;
                    c.n = (uint32_t)round_up(kBandWords + (bhi[q] - blo[q]) + (at & 3), 4);
                    bdst[q] = dst + (at & 3) - blo[q];  // slot word of delay s: bdst + s
                    dst += (int)c.n;
                    bp.copies.push_back(c);
                }
                if (dst > 65535) return false;
                pair_dst[blk_base + g] = dst;
                h.words = (uint16_t)(dst - dst0);
                uint16_t* of = &bp.offs[bb * kBandTrials];
                for (int t = 0; t < kBandTrials; ++t) {
                    const int i = std::min(i0 + t, i1 - 1);
                    of[t] = (uint16_t)(bdst[id[i]] + sp[i]);
                }
                // summing kernel: 8 words a lane for each trial, plus the ring's fill
                cost += 8.0 * kBandTrials + (dst - dst0) / 32.0;
            }
            // row kernel: 256 words of a row take 90 cycles (written at 2.8 TB/s,
            // measured, 152 SMs), read back once by the way
            cost += 90.0 * n;
            bp.infos.push_back(info);
        }
        seg.nrows = (int64_t)bp.rows.size() - seg.row0;
        BandRow* rows = bp.rows.data() + seg.row0;
        for (int b = 0; b < bp.nbands; ++b) {
            const BandInfo& info = bp.infos[bp.infos.size() - bp.nbands + b];
            for (int q = 0; q < info.nrows; ++q) {
                const BandRow& row = bp.rows[info.row0 + q];
                for (const uint16_t at : {row.qa, row.qb}) {
                    if (at == 0xffff) continue;
                    BandQuad& quad = bp.quads[info.quad0 + at];
                    quad.blk0 = std::min(quad.blk0, row.blk0);
                    quad.blk1 = std::max(quad.blk1, row.blk1);
                }
            }
        }
        // places by first block, counting sort
        std::vector<uint32_t> at((size_t)seg.nblk + 1, 0), order((size_t)seg.nrows);
        for (int64_t i = 0; i < seg.nrows; ++i) ++at[rows[i].blk0 + 1];
        for (int g = 0; g < seg.nblk; ++g) at[g + 1] += at[g];
        for (int64_t i = 0; i < seg.nrows; ++i) order[at[rows[i].blk0]++] = (uint32_t)i;
        uint64_t pre = 0;
        seg.first.assign((size_t)seg.nblk, BandSegment::Mark{-1, 0});
        seg.end.assign((size_t)seg.nblk, BandSegment::Mark{0, 0});
        int reached = 0;  // blocks whose first place is known
        for (int64_t i = 0; i < seg.nrows; ++i) {
            BandRow& row = rows[order[(size_t)i]];
            row.id = (uint32_t)i;
            row.pre = (uint32_t)pre;
            for (; reached <= row.blk1; ++reached) seg.first[(size_t)reached] = {i, (int64_t)pre};
            // a window may start up to 3 words early and end up to 3 late
            pre += (uint64_t)round_up(row.span + 8, 4);
            if (pre > UINT32_MAX / 4) return false;
            seg.end[row.blk0] = {i + 1, (int64_t)pre};
        }
        for (int g = 1; g < seg.nblk; ++g)
            if (seg.end[(size_t)g].id < seg.end[(size_t)g - 1].id) seg.end[(size_t)g] = seg.end[(size_t)g - 1];
        for (size_t i = first_copy; i < bp.copies.size(); ++i) {
            const BandRow& row = rows[bp.copies[i].row];
            bp.copies[i].row = row.id;
            bp.copies[i].rel += row.pre;
        }
        seg.pre = (int64_t)pre;
        bp.segs.push_back(seg);
        blk_base += seg.nblk;
    }
    // the ring: places one after the other, from the start again where the end
    // has no room; a place is free once every pair before it whose place it
    // overlaps is consumed (pairs are consumed in order)
    bp.ring_words = (int)(kSumSmem / 4);
    bp.smem_sum = kSumSmem;
    bp.by_two_pairs = 4 * k * 255 * dec <= 65535;
    for (int g = 0; g < nblk_all; ++g) {
        BandHead* h = &bp.heads[(size_t)g * npad];
        std::vector<std::pair<int, int>> place;
        int pos = 0, after = -1;
        for (int pr = 0; pr < npad / 2; ++pr) {
            const int w = kBandTrials + h[2 * pr].words + h[2 * pr + 1].words;
            if (w > bp.ring_words / (kBandLag + 2)) return false;  // the pair added, the lag behind it, one ahead
            if (pos + w > bp.ring_words) pos = 0;
            after = std::max(after, pr - kBandBars);
            for (int q = after + 1; q < pr; ++q)
                if (place[q].first < pos + w && pos < place[q].second) after = q;
            if (after >= 0 && after + kBandLag > pr) return false;
            if (after >= 0 && after + kBandLag > (pr & ~1)) bp.by_two_pairs = false;
            place.push_back({pos, pos + w});
            for (int u = 0; u < 2; ++u) {
                h[2 * pr + u].place = (uint32_t)pos;
                h[2 * pr + u].after = (int16_t)after;
                h[2 * pr + u].at = (int16_t)(after < 0 ? 0 : after + kBandLag);
            }
            pos += w;
        }
    }
    bp.max_quads = max_quads;
    for (bp.tile = 1024; bp.tile >= 128; bp.tile /= 2) {
        bp.quad_words = (int)round_up(bp.tile + max_e, 4);
        bp.raw_words = (int)round_up(bp.quad_words + max_rq, 4);
        bp.smem_rows = ((size_t)k * bp.raw_words + (size_t)max_quads * bp.quad_words) * 4 + (size_t)bp.max_rows * sizeof(BandRow) +
                       (size_t)max_quads * sizeof(BandQuad);
        if (bp.smem_rows <= kRowSmem) break;
    }
    if (bp.tile < 128) {  // a band of many quads: two CTAs per SM
        bp.tile = 128;
        if (bp.smem_rows > 2 * kRowSmem) return false;
    }
    bp.cost = cost;
    bp.ok = true;
    return true;
}

}  // namespace

bool band_shifts(const BandPlan& bp, int C, int ndm, int32_t* out) {
    for (size_t q = 0; q < bp.segs.size(); ++q) {
        const BandSegment& seg = bp.segs[q];
        std::vector<uint32_t> of((size_t)seg.nrows);  // row of each place
        for (int64_t i = 0; i < seg.nrows; ++i) {
            if (bp.rows[seg.row0 + i].id >= seg.nrows) return false;
            of[bp.rows[seg.row0 + i].id] = seg.row0 + (uint32_t)i;
        }
        for (int i = 0; i < seg.ntrials; ++i)
            for (int b = 0; b < bp.nbands; ++b) {
                const int npad = (bp.nbands + 1) & ~1;
                const size_t bb = (size_t)(seg.blk0 + i / kBandTrials) * npad + b;
                const BandHead& h = bp.heads[bb];
                const uint32_t off = bp.offs[bb * kBandTrials + i % kBandTrials];
                const BandCopy* c = nullptr;
                for (uint32_t j = 0; j < h.n; ++j) {
                    const BandCopy& x = bp.copies[h.first + j];
                    if (off >= x.dst && off < x.dst + x.n) c = &x;
                }
                if (!c || off + kBandWords > c->dst + c->n || c->dst + c->n > (uint32_t)h.words + (b & 1 ? bp.heads[bb - 1].words : 0) ||
                    h.place + kBandTrials + c->dst + c->n > (uint32_t)bp.ring_words || c->row >= seg.nrows) return false;
                const BandInfo& info = bp.infos[q * bp.nbands + b];
                const BandRow& row = bp.rows[of[c->row]];
                if (row.id != c->row || of[c->row] < info.row0 || of[c->row] >= info.row0 + info.nrows) return false;
                const int32_t at = (int32_t)(c->rel - row.pre + off - c->dst);  // row delay - row.smin
                const uint32_t next = c->row + 1 < seg.nrows ? bp.rows[of[c->row + 1]].pre : (uint32_t)seg.pre;
                if (at < 0 || at > row.span || c->rel + c->n > next + kBandWords) return false;
                const int g = i / kBandTrials;
                if (g < row.blk0 || g > row.blk1 || c->row < seg.first[(size_t)g].id || c->row >= seg.end[(size_t)g].id) return false;
                for (int j = 0; j < info.nch; ++j) {
                    const BandQuad& quad = bp.quads[info.quad0 + (j < 4 ? row.qa : row.qb)];
                    if (g < quad.blk0 || g > quad.blk1) return false;
                    out[(size_t)(seg.trial0 + i) * C + info.c0 + j] = row.smin + at + (j < 4 ? row.ea : row.eb) + quad.r[j & 3];
                }
            }
    }
    return true;
}

static void choose_bands(RangePlan& r, int C) {
    if (C > 65535 || r.desc.ndm < kBandTrials / 2) return;
    // Which ranges get tables at all (a launch looks at its length again, see
    // bands_pay): SM cycles per 512 output samples against the direct kernel's,
    // of which 64 trials of one channel take 991 (10.4e12 adds/s on 152 SMs at
    // 2.07 GHz, measured).  Bands of 8 channels cost about a seventh of that under
    // fine DM steps; at DM step 1 over 256 channels, bands of 2 to 8 cost about
    // half and run in 143 us against 180 (few CTAs: 1.5 waves).  Under half a
    // block of trials the row kernel's launch is not repaid.
    const double direct = 991.0 / 64 * (double)r.desc.ndm * C;
    BandPlan best;
    for (int k = 8; k >= 2; k /= 2) {
        BandPlan bp;
        if (!build(r, C, k, bp)) continue;
        // rows that many trials share: smaller bands would only add sums
        const bool shared = (double)bp.rows.size() < 64.0 * bp.nbands * (double)bp.segs.size();
        if (!best.ok || bp.cost < best.cost) best = std::move(bp);
        if (shared) break;
    }
    if (best.ok && best.cost < 0.6 * direct) r.bands = std::move(best);
}

void build_bands(RangePlan& r, int C) {
    r.bands = BandPlan{};
    try {
        choose_bands(r, C);
    } catch (const std::bad_alloc&) {  // the plan works without them
        r.bands = BandPlan{};
    }
}

void band_window(const BandSegment& s, int g0, int g1, int64_t& id, int64_t& pre, int64_t& nrows, int64_t& words) {
    id = s.first[(size_t)g0].id;
    pre = s.first[(size_t)g0].pre;
    nrows = s.end[(size_t)g1].id - id;
    words = s.end[(size_t)g1].pre - pre;
}

// bytes for ntiles tiles of the rows that any nblk blocks of a segment use
static int64_t bytes_for(const BandPlan& bp, int64_t ntiles, int nblk, int64_t limit = kBandBytesMax) {
    int64_t most = 0;
    for (const BandSegment& s : bp.segs)
        for (int g = 0; g < s.nblk; ++g) {
            int64_t id, pre, nrows, words;
            band_window(s, g, std::min(s.nblk, g + nblk) - 1, id, pre, nrows, words);
            most = std::max(most, nrows * ntiles * kBandWords + words);
        }
    return round_up(std::min(most * 4, limit), 256);
}

// blocks of a stripe: one that does not begin with a block touches one more
static int stripe_blocks(int32_t trials) { return std::max(1, trials / kBandTrials) + (trials % kBandTrials != 0); }

int64_t band_bytes(const BandPlan& bp, int64_t length) {
    if (!bp.ok || length <= 0) return 0;
    return bytes_for(bp, (length + 2 * kBandWords - 1) / (2 * kBandWords), kBandSegment / kBandTrials);
}

int64_t band_bytes_busy(const BandPlan& bp, int64_t length, int32_t trials) {
    if (!bp.ok || length <= 0) return 0;
    const int64_t nblk = std::max(1, trials / kBandTrials);
    const int64_t tiles = (length + 2 * kBandWords - 1) / (2 * kBandWords);
    return bytes_for(bp, std::min<int64_t>(tiles, std::max<int64_t>(kBandLeastTiles, (2 * kBandSms + nblk - 1) / nblk)), stripe_blocks(trials));
}

int64_t band_bytes_least(const BandPlan& bp, int64_t length, int32_t trials) {
    if (!bp.ok || length <= 0) return 0;
    const int64_t tiles = (length + 2 * kBandWords - 1) / (2 * kBandWords);
    return bytes_for(bp, std::min<int64_t>(tiles, kBandLeastTiles), stripe_blocks(trials), INT64_MAX);
}

namespace {

int64_t div_up(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Which side a launch takes.  Short outputs leave band rows the worse: a row is
// as long as the delays it is used at lie apart, whatever the output, so that at
// 300 samples of 1600 trials (1024 channels, DM step 1) rows and sums took 540 us
// where the direct kernel takes 160; at 16000 samples it is the other way round.
// Both times are estimated, in us, from what was measured on 6325 shapes (32 to
// 4096 channels, DM steps 0.05 to 1, 32 to 1600 trials, 200 to 64000 samples,
// decimations 1, 2 and 8), each with a row buffer and without: nine tenths of the
// estimates are within 10 %.  Where they decide, 28 of the shapes are more than
// 5 % slower than the other side (1.25x at most), 81 more than 5 % slower than
// band rows would be (1.23x); with band rows wherever they fit it was 1699, up to
// 3.4x.
double bands_us(const BandPlan& bp, int trial0, int ndm, int64_t length, int64_t bytes) {
    const int64_t all = div_up(length, 2 * kBandWords);
    double us = 0;
    for (const BandSegment& s : bp.segs) {
        const int d0 = std::max(trial0, s.trial0), d1 = std::min(trial0 + ndm, s.trial0 + s.ntrials);
        if (d0 >= d1) continue;
        const int g0 = (d0 - s.trial0) / kBandTrials, g1 = (d1 - 1 - s.trial0) / kBandTrials;
        int64_t id, pre, nrows, words;
        band_window(s, g0, g1, id, pre, nrows, words);
        const int64_t nt = std::max<int64_t>(1, std::min(all, (bytes / 4 - words) / (nrows * kBandWords)));
        const double slabs = (double)div_up(all, nt);
        // row kernel: six CTAs an SM, each a tile of one band's rows; its channels' loads where the rows are few
        const double ctas = std::max(1.0, (double)(div_up(nt * kBandWords + bp.max_ulen + 15, bp.tile) * bp.nbands) / (6 * kBandSms));
        const double row_us = std::max(1.02 * ctas * (1.0 + 0.1 * (double)nrows / bp.nbands * bp.tile / kBandWords) +
                                           0.042 * (double)(nrows * nt * kBandWords + words) / (kBandWords * kBandSms),
                                       5.0 * ctas * bp.k * bp.tile / 4096);
        // sums: one CTA an SM, whole tiles or halves as launch_bands takes them
        const int64_t n = nt * (g1 - g0 + 1), whole = div_up(n, kBandSms), half = div_up(2 * n, kBandSms);
        const double waves = half <= whole ? 0.74 * half : (double)whole;
        us += slabs * (5.2 + row_us + waves * (4.9 + 0.3 * bp.nbands));
    }
    return us;
}

// The strategy's own kernel: 16 trials x 512 samples a CTA, two an SM.
double strategy_us(int nchans, int ndm, int64_t length, bool grouped, double gwork, int elem) {
    const double c = nchans, wide = elem == 2 ? 1.0 : 0.0;
    const int64_t small = div_up(length, kSmallDirectTau) * ndm;
    if (!grouped && small <= kSmallDirect * kBandSms)
        return 5.6 + c * (0.009 + 0.015 * wide + 0.0585 * (double)small / (kSmallDirect * kBandSms));
    const int64_t n = div_up(ndm, kDmPerBlock) * div_up(length, kTau), full = n / (2 * kBandSms), rest = n % (2 * kBandSms);
    const double one = rest > 0 && rest <= kBandSms, two = rest > kBandSms;  // CTAs of an SM in the last wave
    if (!grouped) return 6.0 + c * ((0.222 + 0.018 * wide) * (double)full + (0.137 + 0.013 * wide) * one + (0.228 + 0.018 * wide) * two);
    return 10.0 + 2.0 * (1 - wide) + c * ((0.017 + 0.023 * wide + 0.24 * gwork) * (double)full +
                                          (0.0165 + 0.01 * wide + (0.157 + 0.03 * wide) * gwork) * one +
                                          (0.0154 + 0.021 * wide + (0.2575 + 0.02 * wide) * gwork) * two);
}

}  // namespace

int g_bands_always = 0;

bool bands_pay(const DedispArgs& a) {
    if (g_bands_always) return true;
    return bands_us(*a.bands, a.trial0, a.ndm, a.length, a.band_bytes) <=
           strategy_us(a.nchans, a.ndm, a.length, a.grouped != 0, a.gwork, a.elem);
}

bool bands_pay(const RangePlan& r, int nchans, int64_t length, int32_t trials, int64_t bytes) {
    if (!r.bands.ok || length <= 0 || bytes < band_bytes_least(r.bands, length, std::min(trials, r.desc.ndm))) return false;
    DedispArgs a{};
    a.nchans = nchans;
    a.ndm = std::min(trials, r.desc.ndm);
    a.length = length;
    a.elem = r.elem;
    a.grouped = r.strategy == 1;
    a.gwork = r.gwork;
    a.bands = &r.bands;
    a.band_bytes = bytes;
    return bands_pay(a);
}

}  // namespace aa
