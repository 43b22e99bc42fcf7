// Host-side check of the resident kernel's layout (lpb_resident.h): over
// seeded random matrices and cuts, every entry of every row is summed once,
// in the step kernels' order (the pieces of a segment, then the segments), by
// lanes that fit in their slices.  Compiled by nvcc for the host; makes no
// CUDA call.  Prints "ok" or the first failure.
#include <cstdio>
#include <map>
#include <random>

#include "lpb_resident.h"

using namespace lpb;

static int fail_at(const char* what, int row) {
    std::printf("%s (row %d)\n", what, row);
    return 1;
}

int main() {
    std::mt19937 rng(7);
    for (int trial = 0; trial < 400; ++trial) {
        const int rows = 1 + rng() % 200, thr = 1 + rng() % 40, seg = 16 << rng() % 5, groups = 4 << rng() % 6;
        std::vector<int> rp(1, 0);
        for (int i = 0; i < rows; ++i) rp.push_back(rp.back() + (int)(rng() % 4 ? rng() % 12 : rng() % 700));
        ResLayout l;
        if (!res_layout(rows, rp.data(), thr, seg, groups, 1 << 20, l)) return fail_at("no layout", -1);
        // slot -> piece
        std::map<uint32_t, std::pair<int, int>> piece;
        const size_t p0 = 32 * (size_t)l.shorts, w0 = 32 * (size_t)(l.shorts + l.longs);
        for (int k = 0; k < 32 * l.pieces; ++k) {
            const uint32_t slot = l.word[w0 + k];
            if (slot == kResIdle) continue;
            if (!piece.insert({slot, {l.beg[p0 + k], l.len[p0 + k]}}).second) return fail_at("slot used twice", -1);
            if ((l.len[p0 + k] + 1) / 2 > l.head[k / 32].pairs) return fail_at("piece exceeds its slice", -1);
            if ((int)slot >= 32 * l.slots) return fail_at("slot out of range", -1);
        }
        std::vector<int> seen(rows, 0);
        for (int at = 0; at < l.places(); ++at) {
            const uint32_t w = l.word[at];
            if ((w & 0xffffu) == kResIdle) continue;
            const int row = (int)(w & 0xffffu), len = rp[row + 1] - rp[row];
            if (row >= rows || seen[row]++ || l.pos[row] != at) return fail_at("place", row);
            if (at < 32 * l.shorts) {
                if (len > thr || l.beg[at] != rp[row] || l.len[at] != len || ((w & kResEmpty) != 0) != (len == 0))
                    return fail_at("short row", row);
                if ((len + 1) / 2 > l.head[l.pieces + at / 32].pairs) return fail_at("row exceeds its slice", row);
                continue;
            }
            if (len <= thr) return fail_at("short row among the long ones", row);
            // the pieces that the step kernels make, in order
            const int s = (at - 32 * l.shorts) / 32, lane = at % 32;
            const ResLayout::Long& h = l.lhead[s];
            int t = 0;
            const int ns = (len + seg - 1) / seg, sl = (len + ns - 1) / ns;
            for (int q = 0; q < ns; ++q) {
                const int rb = std::min(rp[row + 1], rp[row] + q * sl), re = std::min(rp[row + 1], rb + sl);
                const int per = (re - rb + groups - 1) / groups;
                bool first = true;
                for (int e = rb; e < re; e += per, ++t, first = false) {
                    const auto it = piece.find((uint32_t)(32 * (h.slot0 + t) + lane));
                    if (t >= h.pieces || it == piece.end() || it->second.first != e ||
                        it->second.second != std::min(per, re - e))
                        return fail_at("piece", row);
                    if ((l.flag[(size_t)h.flag0 + t] >> lane & 1u) != (first ? 1u : 0u)) return fail_at("segment flag", row);
                    piece.erase(it);
                }
            }
            if (t != l.np[32 * (size_t)s + lane]) return fail_at("pieces of a row", row);
        }
        for (int i = 0; i < rows; ++i)
            if (!seen[i]) return fail_at("row without a place", i);
        if (!piece.empty()) return fail_at("a piece of no row", -1);
        int at = 0;
        for (const auto& h : l.head) {
            if (h.off != at || h.pairs < 1) return fail_at("slice offsets", -1);
            at += h.pairs;
        }
        if (at != l.total_pairs) return fail_at("pairs", -1);
    }
    // more rows than a word holds, or more pairs than asked for
    ResLayout l;
    std::vector<int> many(kResMaxRow + 2, 0);
    if (res_layout(kResMaxRow + 1, many.data(), 32, 256, 8, 1 << 20, l)) return fail_at("too many rows", -1);
    const int two[] = {0, 40, 80};
    if (res_layout(2, two, 64, 256, 8, 10, l)) return fail_at("too many pairs", -1);
    std::printf("ok\n");
    return 0;
}
