// lpb_resident.h -- the layout of a matrix for the resident interval kernel
// (lpb_resident.cu): which thread takes a row, and the order in which a
// row's entries are summed.  Plain host code, checked without a GPU by
// tests/native/resident_layout_test.cu.  Rows sorted by length and taken in
// slices of as many rows as lanes, each padded to its longest, are the
// SELL-C-sigma format of Kreutzer, Hager, Wellein, Fehske and Bishop (SIAM J.
// Sci. Comput. 36(5), 2014), here with one window over all rows; cutting the
// long rows in the step kernels' pieces is this kernel's own.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

namespace lpb {

// A lane's word: a row (or, for a piece, the place of its partial sum), and
// whether it has no entries.
constexpr uint32_t kResIdle = 0xffffu;   // an idle lane's row
constexpr uint32_t kResEmpty = 0x10000u;
constexpr int kResMaxRow = 0xfffe;       // most rows, places and columns

// One product.  Rows are taken 32 at a time, a slice, one row per lane of a
// warp, longest first, so that the lanes run about the same number of
// entries.  A long row is cut into pieces that lanes of piece slices sum; a
// lane of a long slice adds the partial sums.
struct ResLayout {
    struct Head {
        int off, pairs;  // entries of a slice: pairs [off, off + pairs) of each lane
    };
    struct Long {
        int pieces, slot0, flag0;  // of a long slice: the most pieces of a row, its first slot (32 to a piece) and flag
    };
    int shorts = 0, longs = 0, pieces = 0;  // slices
    std::vector<Head> head;                 // piece slices, then short slices
    std::vector<uint32_t> word;             // 32 per slice: short slices, long slices, piece slices
    std::vector<int> beg, len;              // first entry and entries of each lane of the short, then the piece slices
    std::vector<Long> lhead;
    std::vector<int> np;                    // pieces of each lane of the long slices
    std::vector<uint32_t> flag;             // per slot of a long slice: the lanes in which a segment begins
    std::vector<int> pos;                   // row -> place among the lanes of the short and long slices
    int slots = 0;                          // partial sums (32 to a slot)
    int total_pairs = 0;
    int places() const { return 32 * (shorts + longs); }
};

// Lays the rows (pointers rp) out.  A row longer than long_thr is cut as the
// step kernels cut it: ceil(len / seg) segments of equal length, each split
// into contiguous pieces over `groups` row groups; the partial sums are added
// in that order (pieces of a segment, then segments).  false: too many rows,
// or more than max_pairs pairs of entries to a lane in all.
inline bool res_layout(int rows, const int* rp, int long_thr, int seg, int groups, long long max_pairs, ResLayout& o) {
    o = ResLayout{};
    if (rows > kResMaxRow - 64) return false;
    int top = 0;
    for (int i = 0; i < rows; ++i) top = std::max(top, rp[i + 1] - rp[i]);
    // rows by length, longest first (counting sort)
    std::vector<int> start((size_t)top + 2, 0), order(rows);
    for (int i = 0; i < rows; ++i) ++start[top - (rp[i + 1] - rp[i]) + 1];
    for (int k = 0; k <= top; ++k) start[k + 1] += start[k];
    for (int i = 0; i < rows; ++i) order[start[top - (rp[i + 1] - rp[i])]++] = i;
    int n_long = 0;
    while (n_long < rows && rp[order[n_long] + 1] - rp[order[n_long]] > long_thr) ++n_long;
    o.shorts = (rows - n_long + 31) / 32;
    o.longs = (n_long + 31) / 32;
    o.pos.assign(rows, 0);
    o.word.assign((size_t)o.places(), kResIdle);
    o.beg.assign(32 * (size_t)o.shorts, 0);
    o.len.assign(32 * (size_t)o.shorts, 0);
    o.np.assign(32 * (size_t)o.longs, 0);
    for (int k = n_long; k < rows; ++k) {
        const int row = order[k], at = k - n_long;
        o.pos[row] = at;
        o.beg[at] = rp[row];
        o.len[at] = rp[row + 1] - rp[row];
        o.word[at] = (uint32_t)row | (o.len[at] == 0 ? kResEmpty : 0u);
    }
    // the pieces of the long rows, and the slots of their partial sums
    struct Piece {
        int beg, len;
        uint32_t slot;
    };
    std::vector<Piece> pieces;
    for (int s = 0; s < o.longs; ++s) {
        ResLayout::Long lh{0, o.slots, (int)o.flag.size()};
        for (int lane = 0; lane < 32 && 32 * s + lane < n_long; ++lane) {
            const int row = order[32 * s + lane], rb0 = rp[row], re0 = rp[row + 1], len = re0 - rb0;
            const int at = 32 * (o.shorts + s) + lane;
            o.pos[row] = at;
            o.word[at] = (uint32_t)row;
            const int ns = std::max(1, (len + seg - 1) / seg), sl = (len + ns - 1) / ns;
            int np = 0;
            for (int q = 0; q < ns; ++q) {
                const int rb = std::min(re0, rb0 + q * sl), re = std::min(re0, rb + sl);
                const int piece = (re - rb + groups - 1) / groups;
                for (int g = 0; g < groups; ++g) {
                    const int beg = std::min(re, rb + g * piece), end = std::min(re, beg + piece);
                    if (beg == end) continue;
                    if (np == lh.pieces) {
                        ++lh.pieces;
                        o.flag.push_back(0u);
                    }
                    if (g == 0) o.flag[(size_t)lh.flag0 + np] |= 1u << lane;
                    const long long slot = 32LL * (o.slots + np) + lane;
                    if (slot > kResMaxRow) return false;
                    pieces.push_back({beg, end - beg, (uint32_t)slot});
                    ++np;
                }
            }
            o.np[32 * (size_t)s + lane] = np;
        }
        o.slots += lh.pieces;
        o.lhead.push_back(lh);
    }
    std::stable_sort(pieces.begin(), pieces.end(), [](const Piece& x, const Piece& y) { return x.len > y.len; });
    o.pieces = (int)(pieces.size() + 31) / 32;
    const size_t p0 = o.beg.size();
    o.beg.resize(p0 + 32 * (size_t)o.pieces, 0);
    o.len.resize(p0 + 32 * (size_t)o.pieces, 0);
    o.word.resize(o.word.size() + 32 * (size_t)o.pieces, kResIdle);
    for (size_t k = 0; k < pieces.size(); ++k) {
        o.beg[p0 + k] = pieces[k].beg;
        o.len[p0 + k] = pieces[k].len;
        o.word[32 * (size_t)(o.shorts + o.longs) + k] = pieces[k].slot;
    }
    // a slice takes as many pairs as its longest lane, and one at least
    long long at = 0;
    for (int s = 0; s < o.pieces + o.shorts; ++s) {
        const size_t lane0 = s < o.pieces ? p0 + 32 * (size_t)s : 32 * (size_t)(s - o.pieces);
        int most = 1;
        for (int q = 0; q < 32; ++q) most = std::max(most, o.len[lane0 + q]);
        o.head.push_back({(int)at, (most + 1) / 2});
        at += (most + 1) / 2;
        if (at > max_pairs) return false;
    }
    o.total_pairs = (int)at;
    return true;
}

}  // namespace lpb
