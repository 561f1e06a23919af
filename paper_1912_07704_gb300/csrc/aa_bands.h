// Band rows: how a range of the grouped strategy runs when scratch for it is
// there (aa_band_plan.cpp builds the tables, aa_bands.cu holds the kernels).
//
// A band is k consecutive channels (k = 8, 4 or 2).  At trial i its channels
// have delays s'(i) + r_j(i), s' the smallest of them, r_j >= 0.  Over many
// trials the k-tuples r repeat (they are digital lines of nearly one slope),
// so each distinct tuple, a band row z[u] = sum_j x[c_j][u + r_j], is summed
// once and every trial adds one row per band: y_i[t] = sum_b z_{p(b,i)}[t +
// s'_b(i)], nchans / k adds per output sample.  Integer sums regrouped: the
// result is bit-identical.
//
// A range is cut into segments of kBandSegment trials (rows are shared inside
// one), a segment into blocks of kBandTrials trials (one CTA each per time
// tile), and the series into slabs of 2 hw samples: word u of a row holds the
// samples u and u + hw of the slab as two 16-bit lanes, so that any delay is
// a whole number of words.
#pragma once

#include <cstdint>
#include <vector>

namespace aa {

constexpr int kBandTrials = 64;    // trials per CTA: 16 warps x 4
constexpr int kBandSegment = 1536;  // trials that share rows
constexpr int kBandWords = 256;    // words (pairs of samples) per CTA
constexpr int kBandMaxRows = 32;   // rows of one band used by one block (one lane each)
constexpr int kBandBars = 32;      // pairs in the summing kernel's ring at most
constexpr int kBandLeastTiles = 16;  // fewer tiles in the row buffer are left to the other kernels
constexpr int kBandSms = 152;      // SMs that sizes and estimates assume, whatever plan is bound where
constexpr int kBandLag = 3;        // a place is refilled while the third pair behind its own is added

struct BandQuad {  // sum of up to four channels of one half of a band
    uint16_t r[4];  // delays inside the quad, 0xffff: no such channel
    uint16_t blk0, blk1;  // first and last block of the segment with a row of it
};
struct BandRow {
    uint16_t qa, qb;  // quads of the band's halves (index in the band's list, 0xffff: none)
    uint16_t ea, eb;  // their delays inside the row
    int32_t smin;     // smallest row delay s' over the segment's trials using it
    int32_t span;     // largest - smallest
    uint32_t pre;     // words before this row in the buffer beyond hw per earlier row
    uint16_t blk0, blk1;  // first and last block of the segment using it
    uint32_t id;      // its place among the segment's rows in the buffer: by first block
};
struct BandInfo {  // one band of one segment
    uint32_t row0, quad0;     // first row / quad (in the range's lists)
    uint16_t nrows, nqa, nqb;
    uint16_t c0, nch;         // its channels
    uint16_t pad;
    int32_t umin, ulen;       // smallest s', and largest - smallest s' over its rows
};
struct BandCopy {  // one row's window as a block uses it
    uint32_t row;  // place of the row (BandRow::id)
    uint32_t rel;  // words from the row's first to the window's (plus the tile's), multiple of 4
    uint32_t dst;  // words into the rows of its pair's place
    uint32_t n;    // words, multiple of 4
};
// Two consecutive bands of a block share a place in the summing kernel's ring:
// the trials' offsets of both (kBandTrials words of 16-bit pairs), then their
// row windows.  Places follow one another around the ring; where each lies and
// which pair must be consumed before it may be filled is laid down here.
struct BandHead {  // one (block, band)
    uint32_t first;   // first BandCopy
    uint16_t n;       // copies
    uint16_t words;   // words of all of them
    uint32_t place;   // words from the ring's start to the pair's place
    int16_t after;    // the pair whose consumption frees the place (-1: free from the start)
    int16_t at;       // the pair being added when it is filled
};
struct BandSegment {
    int32_t trial0 = 0, ntrials = 0, nblk = 0, blk0 = 0;
    int64_t nrows = 0, pre = 0;  // rows, and words of the buffer beyond hw per row
    uint32_t row0 = 0;
    // Rows that blocks g0 .. g1 use lie in places from first[g0] to end[g1]: a
    // launch over some of the blocks keeps only those in its buffer.
    struct Mark { int64_t id, pre; };
    std::vector<Mark> first, end;
};

struct BandPlan {
    bool ok = false;
    int k = 0, nbands = 0;
    int ring_words = 0;  // ring of the summing kernel
    bool by_two_pairs = false;  // two pairs' rows fit 16 bits, and their places fill in time to be added together
    int tile = 0;                    // words per CTA of the row kernel
    int raw_words = 0, quad_words = 0, max_quads = 0, max_rows = 0;
    size_t smem_rows = 0, smem_sum = 0;
    int32_t max_ulen = 0;
    double cost = 0;  // estimated SM cycles per 512 output samples of all trials
    std::vector<BandSegment> segs;
    std::vector<BandRow> rows;
    std::vector<BandQuad> quads;
    std::vector<BandInfo> infos;   // [segment][band]
    std::vector<BandCopy> copies;
    std::vector<BandHead> heads;   // [block][band (an even number)]
    std::vector<uint16_t> offs;    // [block][band (an even number)][kBandTrials]: each trial's word among its pair's rows
    const BandRow* d_rows = nullptr;
    const BandQuad* d_quads = nullptr;
    const BandInfo* d_infos = nullptr;
    const BandCopy* d_copies = nullptr;
    const BandHead* d_heads = nullptr;
    const uint16_t* d_offs = nullptr;
};

// Places that the rows of blocks g0 .. g1 of a segment take: from id (with pre
// words beyond hw per row before it), nrows of them with `words` beyond hw each.
void band_window(const BandSegment& s, int g0, int g1, int64_t& id, int64_t& pre, int64_t& nrows, int64_t& words);

}  // namespace aa
