// Host-side check of the short rows' order (lpb_row_order.h): over row counts
// that are and are not whole windows, and thresholds up to the largest, the
// records written are the rows of at most thr entries, once each, as many as
// are counted, and none past the last row.  Restates the counting and the
// sorted writing of the set-up kernels around the shared key; compiled by nvcc
// for the host, makes no CUDA call.  Prints "ok" or the first failure.
#include <algorithm>
#include <climits>
#include <cstdio>
#include <random>
#include <vector>

#include "lpb_row_order.h"

using namespace lpb;

static int fail_at(const char* what, int rows, int window, int thr) {
    std::printf("%s (%d rows, windows of %d, threshold %d)\n", what, rows, window, thr);
    return 1;
}

int main() {
    std::mt19937 rng(3);
    for (int rows : {1, 2, 127, 128, 129, 300, 2047, 2048, 2049, 5000})
        for (int window : {128, 2048})
            for (int thr : {1, 32, 300, INT_MAX - 1, INT_MAX}) {
                std::vector<int> len(rows);
                for (int& v : len) v = rng() % 3 ? rng() % 40 : rng() % 500;
                std::vector<int> out;  // rows in the order of their records
                for (int base = 0; base < rows; base += window) {
                    int counted = 0;
                    std::vector<unsigned long long> key(window);
                    for (int q = 0; q < window; ++q) {
                        const int i = base + q;
                        if (i < rows && len[i] <= thr) ++counted;
                        key[q] = short_key(i < rows, i < rows ? len[i] : 0, thr, q);
                    }
                    std::sort(key.begin(), key.end());
                    const int first = (int)out.size();
                    for (int q = 0; q < window; ++q) {
                        if (!is_short(key[q])) continue;
                        if (first + q != (int)out.size()) return fail_at("short rows do not come first", rows, window, thr);
                        out.push_back(base + (int)(key[q] & 0xffffffffull));
                    }
                    if ((int)out.size() - first != counted) return fail_at("records and count differ", rows, window, thr);
                    for (size_t k = first; k + 1 < out.size(); ++k) {
                        const int a = out[k], b = out[k + 1];
                        if (len[a] < len[b] || (len[a] == len[b] && a >= b)) return fail_at("order", rows, window, thr);
                    }
                }
                std::vector<char> seen(rows, 0);
                for (int i : out) {
                    if (i >= rows) return fail_at("a record past the last row", rows, window, thr);
                    if (len[i] > thr || seen[i]++) return fail_at("a long row, or a row twice", rows, window, thr);
                }
                for (int i = 0; i < rows; ++i)
                    if (len[i] <= thr && !seen[i]) return fail_at("a row is left out", rows, window, thr);
            }
    std::printf("ok\n");
    return 0;
}
