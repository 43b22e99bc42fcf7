// lpb_row_order.h -- the order in which the step kernels take the short rows
// (lpb_setup.cu): the sort key of a row within its window.  Host and device
// code, checked without a GPU by tests/native/row_order_test.cu.
#pragma once

#ifdef __CUDACC__
#define LPB_RO_HD __host__ __device__
#else
#define LPB_RO_HD
#endif

namespace lpb {

// Upper half of the key of a place that is no short row: a row of more than
// thr entries, or a place past the last row, whatever thr is (the largest
// threshold, 2^31 - 1, makes every row short).
constexpr unsigned kNotShort = 0xffffffffu;

// Key of place q of a window, which is a row of len entries when in_matrix:
// rows of at most thr entries, longest first, equal lengths in their order,
// and then the places that are no short row.
LPB_RO_HD inline unsigned long long short_key(bool in_matrix, int len, int thr, int q) {
    const unsigned upper = in_matrix && len <= thr ? (unsigned)(thr - len) : kNotShort;
    return (unsigned long long)upper << 32 | (unsigned)q;
}
LPB_RO_HD inline bool is_short(unsigned long long key) { return (unsigned)(key >> 32) != kNotShort; }

}  // namespace lpb
