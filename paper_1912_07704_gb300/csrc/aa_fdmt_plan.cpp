// Groups of depths of the tree form, built once per range.  A launch of
// aa_fdmt.cu merges several depths: each of its blocks owns some consecutive
// rows of the group's shallowest depth, loads the rows (or channels) they come
// from and merges depth after depth in shared memory.  This file lays the
// blocks out - which rows, which windows of them, in which slot - and chooses
// the groups by their modelled time.
#include <algorithm>
#include <cstdint>
#include <limits>

#include "aa_internal.h"

namespace aa {
namespace {

// One block before its tile is chosen: slots instead of word offsets.
struct Need {
    int32_t row;     // row of its depth, or reference of a load
    int64_t lo, hi;  // offsets of the window's first sample over its readers
    int32_t slot = -1;
    int32_t level = 0;  // loads: depth that reads it
};
struct Block {
    std::vector<Need> level[kFdmtMaxLevels];  // rows of depth top + i
    std::vector<Need> loads;
    int32_t slots = 0;
    int64_t spread = 0;  // most samples of a window beyond the tile
    int64_t adds = 0;
};

struct Builder {
    const FdmtPlan& fd;
    int32_t nchans;
    int elem;
    const std::vector<std::vector<int32_t>>& nodes;     // first row of each node, per depth
    std::vector<std::vector<int32_t>> at;               // [depth][row]: its index in the block under way
    std::vector<int32_t> at_chan;

    Builder(const FdmtPlan& f, int32_t c, int e, const std::vector<std::vector<int32_t>>& n)
        : fd(f), nchans(c), elem(e), nodes(n), at((size_t)f.depths), at_chan((size_t)c, -1) {
        for (int d = 0; d < fd.depths; ++d) at[(size_t)d].assign((size_t)rows(d), -1);
    }
    int64_t rows(int d) const { return fd.first[(size_t)(fd.depths - d)] - fd.first[(size_t)(fd.depths - 1 - d)]; }
    const FdmtRow& row(int d, int32_t i) const { return fd.rows[(size_t)(fd.first[(size_t)(fd.depths - 1 - d)] + i)]; }

    // rows [r0, r1) of the blocks: whole nodes together up to R rows, larger
    // nodes in equal parts of at most R
    std::vector<int32_t> cuts(int top, int32_t R) const {
        std::vector<int32_t> c{0};
        const int32_t n = (int32_t)rows(top);
        const auto& starts = nodes[(size_t)top];
        for (size_t j = 0; j < starts.size(); ++j) {
            const int32_t b = starts[j], e = j + 1 < starts.size() ? starts[j + 1] : n;
            if (e - c.back() <= R) continue;       // joins the block under way
            if (b > c.back()) c.push_back(b);      // close it before this node
            const int32_t parts = (e - b + R - 1) / R;
            for (int32_t k = 1; k < parts; ++k) c.push_back(b + (int32_t)((int64_t)(e - b) * k / parts));
        }
        if (c.back() < n) c.push_back(n);
        return c;
    }

    Need& want(std::vector<Need>& list, int32_t& index, int32_t ref, int64_t lo, int64_t hi, int level) {
        if (index < 0) {
            index = (int32_t)list.size();
            list.push_back(Need{ref, lo, hi, -1, level});
        } else {
            list[(size_t)index].lo = std::min(list[(size_t)index].lo, lo);
            list[(size_t)index].hi = std::max(list[(size_t)index].hi, hi);
        }
        return list[(size_t)index];
    }
    int32_t& load_index(int bottom, int32_t ref) {
        return ref < 0 ? at_chan[(size_t)(-(ref + 1))] : at[(size_t)bottom + 1][(size_t)ref];
    }

    // windows start and end at multiples of four samples
    static void whole(Need& n) {
        n.lo = n.lo & ~int64_t(3);
        n.hi = n.lo + round_up(n.hi - n.lo, 4);
    }
    void build(int top, int bottom, int32_t r0, int32_t r1, Block& b) {
        const int k = bottom - top + 1;
        b.loads.clear();
        b.adds = 0;
        for (auto& l : b.level) l.clear();
        for (int32_t r = r0; r < r1; ++r) b.level[0].push_back(Need{r, 0, 0, -1, 0});
        for (int i = 0; i < k; ++i) {
            const int d = top + i;
            b.adds += (int64_t)b.level[i].size();
            for (Need& n : b.level[i]) whole(n);
            for (size_t e = 0; e < b.level[i].size(); ++e) {
                const Need n = b.level[i][e];
                const FdmtRow& x = row(d, n.row);
                for (int half = 0; half < 2; ++half) {
                    const int32_t ref = half ? x.l : x.u;
                    const int64_t off = half ? x.gap : 0;
                    if (ref >= 0 && d < bottom) want(b.level[i + 1], at[(size_t)d + 1][(size_t)ref], ref, n.lo + off, n.hi + off, i);
                    else want(b.loads, load_index(bottom, ref), ref, n.lo + off, n.hi + off, i);
                }
            }
        }
        for (Need& n : b.loads) {
            whole(n);
            b.spread = std::max(b.spread, n.hi - n.lo);
        }
        for (int i = 1; i < k; ++i)
            for (const Need& n : b.level[i]) b.spread = std::max(b.spread, n.hi - n.lo);
        // slots: a depth's rows are placed before those it reads are given up
        std::vector<int32_t> free_slots;
        int32_t used = 0;
        auto take = [&]() {
            if (free_slots.empty()) return used++;
            const int32_t s = free_slots.back();
            free_slots.pop_back();
            return s;
        };
        for (Need& n : b.loads) n.slot = take();
        for (int i = k - 1; i >= 1; --i) {
            for (Need& n : b.level[i]) n.slot = take();
            for (const Need& n : b.loads)
                if (n.level == i) free_slots.push_back(n.slot);
            if (i + 1 < k)
                for (const Need& n : b.level[i + 1]) free_slots.push_back(n.slot);
        }
        b.slots = used;
    }
    void forget(int top, int bottom, const Block& b) {  // after a block: its rows' indices
        for (int i = 1; i <= bottom - top; ++i)
            for (const Need& n : b.level[i]) at[(size_t)(top + i)][(size_t)n.row] = -1;
        for (const Need& n : b.loads) load_index(bottom, n.row) = -1;
    }
};

// Windows of W words, the widest (a multiple of 32) whose slots leave room for
// two CTAs of an SM; the tile is what the spread leaves of it.
int width_of(int32_t slots, int64_t spread) {
    for (int w = 512; w >= 128; w -= 32)
        if ((int64_t)slots * w <= kFdmtSlotWords) return w - spread >= 64 ? w : 0;
    return 0;
}
int tile_of(int width, int64_t spread) { return (int)(width - spread) & ~7; }

}  // namespace

bool build_fdmt_groups(FdmtPlan& fd, int32_t nchans, int elem, const std::vector<std::vector<int32_t>>& nodes) {
    fd.groups.clear();
    fd.blocks.clear();
    fd.loads.clear();
    fd.ops.clear();
    if (fd.depths < 1) return true;
    Builder bl(fd, nchans, elem, nodes);
    Block b;
    // Modelled clocks of an SM for a group, per sample of the series, from at most
    // 16 of its blocks: memory at 6.8 TB/s (21.5 bytes a clock and SM), sums and
    // loads by the shared-memory words they move and the instructions they take.
    auto cost = [&](int top, int bottom, int32_t R) {
        const std::vector<int32_t> c = bl.cuts(top, R);
        const size_t n = c.size() - 1, step = (n + 15) / 16;
        double sum = 0;
        size_t seen = 0;
        for (size_t j = 0; j < n; j += step, ++seen) {
            b.spread = 0;
            bl.build(top, bottom, c[j], c[j + 1], b);
            bl.forget(top, bottom, b);
            const int W = width_of(b.slots, b.spread);
            const int tile = W ? tile_of(W, b.spread) : 0;
            if (!W) return std::numeric_limits<double>::infinity();
            double bytes = 0;
            for (const Need& l : b.loads) bytes += (l.row < 0 ? elem : 4) * (double)W;
            bytes += 4.0 * tile * (c[j + 1] - c[j]);
            const double passes = (W + 127) / 128;
            const double clocks = (double)(b.adds + b.loads.size()) * (0.125 * W + 8 * passes + 8) + 200.0 * (bottom - top + 2);
            sum += (bytes / 21.5 + clocks) / tile;
        }
        return sum / (double)seen * (double)n;
    };
    struct Choice { double cost = std::numeric_limits<double>::infinity(); int bottom = 0; int32_t R = 1; };
    std::vector<Choice> best((size_t)fd.depths + 1);
    best[(size_t)fd.depths].cost = 0;
    for (int top = fd.depths - 1; top >= 0; --top)
        for (int bottom = top; bottom < std::min(fd.depths, top + kFdmtMaxLevels); ++bottom)
            for (int32_t R : {64, 32, 16, 1}) {
                if (R == 1 && bottom > top) continue;  // the form that always fits, one depth deep
                const double t = cost(top, bottom, R) + best[(size_t)bottom + 1].cost;
                if (t < best[(size_t)top].cost) best[(size_t)top] = Choice{t, bottom, R};
            }
    for (int top = 0; top < fd.depths;) {
        const int bottom = best[(size_t)top].bottom;
        int32_t R = best[(size_t)top].R;
        std::vector<int32_t> c;
        int32_t slots = 0;
        int64_t spread = 0;
        int W = 0;
        for (;; R /= 2) {  // the sampled blocks need not be the largest
            if (R < 1) return false;
            c = bl.cuts(top, R);
            slots = 0;
            spread = 0;
            for (size_t j = 0; j + 1 < c.size(); ++j) {
                b.spread = 0;
                bl.build(top, bottom, c[j], c[j + 1], b);
                bl.forget(top, bottom, b);
                slots = std::max(slots, b.slots);
                spread = std::max(spread, b.spread);
            }
            W = width_of(slots, spread);
            if (W) break;
        }
        const int tile = tile_of(W, spread);
        FdmtGroup g;
        g.top = top;
        g.bottom = bottom;
        g.tile = tile;
        g.width = W;
        g.words = (int32_t)(slots * W);
        g.block0 = (int64_t)fd.blocks.size();
        for (size_t j = 0; j + 1 < c.size(); ++j) {
            b.spread = 0;
            bl.build(top, bottom, c[j], c[j + 1], b);
            FdmtBlock o{};
            o.load0 = (int32_t)fd.loads.size();
            o.nload = (int32_t)b.loads.size();
            o.op0 = (int32_t)fd.ops.size();
            for (const Need& n : b.loads) {
                g.leaves = g.leaves || n.row < 0;
                fd.loads.push_back(FdmtLoad{n.row, (int32_t)n.lo, (int32_t)(n.slot * W), (int32_t)(n.hi - n.lo) + tile});
            }
            const int k = bottom - top + 1;
            for (int i = k - 1, q = 0; i >= 0; --i, ++q) {
                const int d = top + i;
                for (const Need& n : b.level[i]) {
                    const FdmtRow& x = bl.row(d, n.row);
                    uint32_t off[2];
                    for (int half = 0; half < 2; ++half) {
                        const int32_t ref = half ? x.l : x.u;
                        const Need& s = ref >= 0 && d < bottom ? b.level[i + 1][(size_t)bl.at[(size_t)d + 1][(size_t)ref]]
                                                               : b.loads[(size_t)bl.load_index(bottom, ref)];
                        off[half] = (uint32_t)(s.slot * W + n.lo + (half ? x.gap : 0) - s.lo);
                    }
                    fd.ops.push_back(FdmtOp{off[0] | off[1] << 16, i ? (int32_t)(n.slot * W) : n.row, (int32_t)(n.hi - n.lo + tile), x.delta});
                }
                o.end[q] = (int32_t)((int64_t)fd.ops.size() - o.op0);
            }
            bl.forget(top, bottom, b);
            g.max_ops = std::max(g.max_ops, o.end[k - 1]);
            g.max_loads = std::max(g.max_loads, o.nload);
            fd.blocks.push_back(o);
        }
        g.nblocks = (int32_t)((int64_t)fd.blocks.size() - g.block0);
        fd.groups.push_back(g);
        top = bottom + 1;
    }
    return true;
}

// Channel delays of each trial read back from the blocks: their ops run on
// (source, offset) lists instead of samples, and every window is checked.
bool fdmt_shifts(const FdmtPlan& fd, int32_t nchans, int32_t ndm, int32_t* out) {
    struct Term { int32_t ref, off; };
    struct Slot { int32_t base = -1, n = 0; std::vector<Term> terms; };  // window [base, base + n) of the buffer, offsets from its start
    std::vector<std::vector<std::vector<Term>>> of(fd.groups.size());   // [group][row of its top depth]
    for (size_t q = 0; q < fd.groups.size(); ++q) {
        const FdmtGroup& g = fd.groups[q];
        of[q].resize((size_t)(fd.first[(size_t)(fd.depths - g.top)] - fd.first[(size_t)(fd.depths - 1 - g.top)]));
        const int64_t below = g.bottom + 1 < fd.depths
            ? fd.first[(size_t)(fd.depths - 1 - g.bottom)] - fd.first[(size_t)(fd.depths - 2 - g.bottom)] : 0;
        std::vector<Slot> slot((size_t)(g.words / g.width));
        for (int32_t bi = 0; bi < g.nblocks; ++bi) {
            const FdmtBlock& b = fd.blocks[(size_t)(g.block0 + bi)];
            for (auto& s : slot) s.n = 0;
            for (int32_t i = 0; i < b.nload; ++i) {
                const FdmtLoad& l = fd.loads[(size_t)(b.load0 + i)];
                if (l.dst % g.width || l.dst < 0 || l.dst / g.width >= (int32_t)slot.size() || l.n > g.width || l.n % 4 || l.n < 4 || l.lo < 0 || l.lo % 4 ||
                    l.ref >= below || -(l.ref + 1) >= nchans)
                    return false;
                slot[(size_t)(l.dst / g.width)] = Slot{l.dst, l.n, {Term{l.ref, l.lo}}};
            }
            int32_t o = 0;
            for (int i = 0; i <= g.bottom - g.top; ++i) {
                std::vector<Slot> made;
                for (; o < b.end[i]; ++o) {
                    const FdmtOp& op = fd.ops[(size_t)(b.op0 + o)];
                    Slot r;
                    if (op.n % 4 || (op.src & 3)) return false;
                    for (const int32_t src : {(int32_t)(op.src & 0xffff), (int32_t)(op.src >> 16)}) {
                        if (src / g.width >= (int32_t)slot.size()) return false;
                        const Slot& s = slot[(size_t)(src / g.width)];
                        if (src < s.base || src + op.n > s.base + s.n) return false;
                        for (const Term& t : s.terms) r.terms.push_back(Term{t.ref, t.off + src - s.base});
                    }
                    r.base = op.dst;
                    r.n = op.n;
                    if (i < g.bottom - g.top) {
                        if (op.dst % g.width || op.dst < 0 || op.dst / g.width >= (int32_t)slot.size() || op.n > g.width) return false;
                        made.push_back(std::move(r));
                    } else {
                        if (op.dst < 0 || (size_t)op.dst >= of[q].size() || op.n != g.tile || !of[q][(size_t)op.dst].empty()) return false;
                        of[q][(size_t)op.dst] = std::move(r.terms);
                    }
                }
                // a depth's rows must not lie where it still reads
                for (const Slot& r : made)
                    for (int32_t x = i ? b.end[i - 1] : 0; x < b.end[i]; ++x) {
                        const FdmtOp& op = fd.ops[(size_t)(b.op0 + x)];
                        if ((int32_t)(op.src & 0xffff) / g.width == r.base / g.width || (int32_t)(op.src >> 16) / g.width == r.base / g.width) return false;
                    }
                for (Slot& r : made) slot[(size_t)(r.base / g.width)] = std::move(r);
            }
            if (b.end[g.bottom - g.top] > g.max_ops || b.nload > g.max_loads) return false;
        }
        for (const auto& t : of[q])
            if (t.empty()) return false;
    }
    std::fill(out, out + (int64_t)ndm * nchans, -1);
    bool ok = true;
    auto walk = [&](auto&& self, size_t q, int32_t r, int64_t base, int32_t* e) -> void {
        for (const Term& t : of[q][(size_t)r]) {
            if (t.ref >= 0) { self(self, q + 1, t.ref, base + t.off, e); continue; }
            int32_t& s = e[-(t.ref + 1)];
            ok = ok && s == -1;
            s = (int32_t)(base + t.off);
        }
    };
    for (int32_t i = 0; i < ndm; ++i) walk(walk, 0, i, 0, out + (int64_t)i * nchans);
    for (int64_t i = 0; i < (int64_t)ndm * nchans; ++i) ok = ok && out[i] >= 0;
    return ok;
}

}  // namespace aa
