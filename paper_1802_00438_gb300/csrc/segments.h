// Segments of the contracted passes: which planes (2D: rows) of which tile columns each block
// streams.  Host code only.
//
// A segment costs w[col] per plane plus `fill` planes of pipeline fill, plus `edge` at the first
// and the last plane of the grid (boundary handling), and the slowest block sets the pass time.
// The tile columns overlap, so neighbouring columns should be at nearby planes at the same time:
// then the halo cells a tile reads again (and the partial sectors of its rows) are still in L2.
// So, level by level: with at least as many blocks as columns left, every column gets one block,
// all from the same first plane, for as many planes as the budget allows, and what is left of the
// columns goes to the blocks without work; with fewer blocks than columns, each block takes one
// whole rest of a column, the costliest first, and goes on with the budget that leaves it.  The
// budget is the smallest for which everything is dealt out (bisection).
// Measured on GB300 against contiguous ranges of (column, plane) units balanced the same way,
// where neighbours run at unrelated planes: see prepare3 and segments_2d in api.cu.
//
// One deal takes time proportional to the columns (times a logarithm for the rests that are cut):
// the whole columns are sorted once, and the rests go to a heap.  With more than kManyCols columns
// per block a bisection would buy nothing - a block's share is many columns, and the last of them
// are cut to fit - so the budget is the mean share with all its fills, raised by 0.25 % until it
// suffices.  One CPU core, 16384 x 16384 x 4 (82,919 columns, 152 blocks): 15 ms; with all rests
// sorted anew at every level and the budget bisected, 18.6 s.  10^8 x 10 (416,667 columns, 1216
// blocks): 93 ms, 81 s.  Up to kManyCols columns per block the segments are the same as those.
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

namespace stn {

struct Segment { int col, z0, z1, block; };

class SegmentDealer {
public:
    // w: cost per plane of each tile column; speed: each block's share of the budget (empty: all
    // alike)
    SegmentDealer(int nz, int slots, double fill, double edge, const std::vector<double> &w,
                  const std::vector<double> &speed = {})
        : nz_(nz), slots_(slots), fill_(fill), edge_(edge), w_(w), speed_(speed)
    {
        for (double x : w_) total_ += x * nz_;
    }

    // The smallest budget for which everything is dealt out, within tol (with very many columns
    // an estimate); with out != nullptr the segments, in the order in which they were dealt.
    double best(double tol, std::vector<Segment> *out)
    {
        if (w_.size() > (size_t)kManyCols * slots_) {
            double b = (total_ + (double)w_.size() * (fill_ + 2.0 * edge_)) / slots_;
            if (out)
                while (!deal(b, out)) b *= 1.0025;
            return b;
        }
        // (the upper end of the bracket is dealt only if nothing below it suffices)
        const double first = std::max(total_ / slots_, fill_ + 4.0);
        std::vector<Segment> list;
        for (double end = first + 3.0 * fill_ + edge_;; end *= 1.5) {
            double lo = first, hi = end;
            bool done = false;
            for (int i = 0; i < 40 && hi - lo > tol; i++) {
                const double mid = 0.5 * (lo + hi);
                if (deal(mid, out ? &list : nullptr)) {
                    hi = mid;
                    done = true;
                    if (out) out->swap(list);
                } else {
                    lo = mid;
                }
            }
            if (done || deal(hi, out)) return hi;
        }
    }

private:
    static constexpr int kManyCols = 8;

    struct Rest { int col, z0; };
    struct Block { double left; int id; };

    bool costlier(const Rest &a, const Rest &b) const
    {
        const double ca = (nz_ - a.z0) * w_[a.col], cb = (nz_ - b.z0) * w_[b.col];
        return ca != cb ? ca > cb : a.col < b.col;
    }

    // Block b takes what it can of q; true: q is now the rest, false: nothing is left of it.
    bool cut(Block &b, Rest &q, std::vector<Block> &spare, std::vector<Segment> *out) const
    {
        const int h = nz_ - q.z0;
        const double wc = w_[q.col], fixed = fill_ + (q.z0 == 0 ? edge_ : 0.0), room = b.left - fixed;
        const double fit = wc == 1.0 ? room : room / wc;   // (most columns weigh 1: no division)
        int take = fit >= h ? h : std::max(1, (int)fit);
        // a segment that reaches the end pays `edge` too; one that cannot, leaves a rest
        if (take == h && take > 1 && fixed + edge_ + h * wc > b.left)
            take = std::max(1, std::min(h - 1, (int)((room - edge_) / wc)));
        if (out) out->push_back(Segment{q.col, q.z0, q.z0 + take, b.id});
        if (take < h) {
            q.z0 += take;
            return true;
        }
        b.left -= fixed + edge_ + take * wc;
        if (b.left >= fill_ + 4) spare.push_back(b);
        return false;
    }

    bool deal(double budget, std::vector<Segment> *out)
    {
        // blocks with work to take, the largest budget first, from `head` on; `spare`: those that
        // have a segment and budget left, taken up when the others have run out
        std::vector<Block> &blocks = blocks_, &spare = spare_;
        blocks.resize(slots_);
        spare.clear();
        for (int b = 0; b < slots_; b++) blocks[b] = Block{speed_.empty() ? budget : budget * speed_[b], b};
        size_t head = 0;
        if (out) out->clear();
        auto more_blocks = [&]() {
            if (head < blocks.size()) return true;
            if (spare.empty()) return false;
            std::sort(spare.begin(), spare.end(), [](const Block &a, const Block &b) {
                return a.left != b.left ? a.left > b.left : a.id < b.id;
            });
            blocks.swap(spare);
            spare.clear();
            head = 0;
            return true;
        };
        const auto by_cost = [this](const Rest &a, const Rest &b) { return costlier(a, b); };
        const auto by_col = [](const Rest &a, const Rest &b) { return a.col < b.col; };
        const auto heap_less = [this](const Rest &a, const Rest &b) { return costlier(b, a); };
        std::vector<Rest> &rest = rest_, &next = next_;
        rest.clear();

        // more columns than blocks: whole columns in the order of their cost, and the rests of
        // those that were cut (a heap), whichever is costlier
        if (w_.size() > (size_t)slots_) {
            if (whole_.empty()) {
                whole_.resize(w_.size());
                for (size_t c = 0; c < w_.size(); c++) whole_[c] = Rest{(int)c, 0};
                std::sort(whole_.begin(), whole_.end(), by_cost);
            }
            size_t pos = 0;
            while (true) {
                if (!more_blocks()) return false;
                const size_t avail = blocks.size() - head;
                if (whole_.size() - pos + rest.size() <= avail) break;
                next.clear();
                for (size_t i = 0; i < avail; i++) {
                    Rest q;
                    if (rest.empty() || (pos < whole_.size() && costlier(whole_[pos], rest.front()))) {
                        q = whole_[pos++];
                    } else {
                        std::pop_heap(rest.begin(), rest.end(), heap_less);
                        q = rest.back();
                        rest.pop_back();
                    }
                    if (cut(blocks[head + i], q, spare, out)) next.push_back(q);
                }
                head += avail;
                for (const Rest &q : next) {
                    rest.push_back(q);
                    std::push_heap(rest.begin(), rest.end(), heap_less);
                }
            }
            rest.insert(rest.end(), whole_.begin() + pos, whole_.end());
            std::sort(rest.begin(), rest.end(), by_col);
        } else {
            rest.resize(w_.size());
            for (size_t c = 0; c < w_.size(); c++) rest[c] = Rest{(int)c, 0};
        }
        // no more rests than blocks were left at some point: few enough to sort them at each level
        while (!rest.empty()) {
            if (!more_blocks()) return false;
            const size_t avail = blocks.size() - head, n = std::min(avail, rest.size());
            const bool whole = rest.size() > avail;
            if (whole) std::sort(rest.begin(), rest.end(), by_cost);
            next.clear();
            for (size_t i = 0; i < rest.size(); i++)
                if (i >= avail || cut(blocks[head + i], rest[i], spare, out)) next.push_back(rest[i]);
            head += n;
            if (whole) std::sort(next.begin(), next.end(), by_col);
            rest.swap(next);
        }
        return true;
    }

    const int nz_, slots_;
    const double fill_, edge_;
    const std::vector<double> w_, speed_;
    double total_ = 0.0;
    std::vector<Block> blocks_, spare_;   // a deal's, kept for the next one
    std::vector<Rest> rest_, next_;
    std::vector<Rest> whole_;   // whole columns, the costliest first (only with more columns than blocks)
};

}  // namespace stn
