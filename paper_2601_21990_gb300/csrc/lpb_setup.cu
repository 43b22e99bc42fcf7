// lpb_setup.cu -- once-per-matrix device work of lpb_create:
//   transpose of A (A and A^T are both stored, Sec. 6 "Implementation details"),
//   Ruiz + Pock-Chambolle equilibration, scaled values and vectors,
//   power iteration for ||A~||_2 (eta = 0.998 / ||A~||_2, Sec. 4 "Step-size"),
//   lists of long rows for the SpMM kernels.
// Every kernel is deterministic: sums run in a fixed order, the transpose is
// sorted by the original entry index inside each row of A^T.
#include <algorithm>
#include <climits>
#include <cstdio>
#include <vector>

#include "lpb_internal.h"
#include "lpb_row_order.h"

namespace lpb {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// scratch of one call, from the stream's pool; goes with the scope, also where
// a later step fails
struct StreamMem {
    void* p = nullptr;
    cudaStream_t s;
    explicit StreamMem(cudaStream_t stream) : s(stream) {}
    StreamMem(const StreamMem&) = delete;
    StreamMem& operator=(const StreamMem&) = delete;
    cudaError_t take(size_t bytes) { return cudaMallocAsync(&p, bytes, s); }
    ~StreamMem() {
        if (p) cudaFreeAsync(p, s);
    }
};

// ---------------------------------------------------------------------------
// exclusive scan of int32 (block = 1024 threads, 2 elements per thread)
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 1024;
constexpr int kScanTile = 2 * kScanThreads;

__global__ void k_scan_tile(const int* __restrict__ in, int* __restrict__ out, int count,
                            int* __restrict__ tile_sums) {
    __shared__ int warp_tot[kScanThreads / 32];
    const int base = blockIdx.x * kScanTile + 2 * threadIdx.x;
    int a0 = base < count ? in[base] : 0;
    int a1 = base + 1 < count ? in[base + 1] : 0;
    int local = a0 + a1;
    // inclusive warp scan of `local`
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = local;
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int w = warp_tot[lane];
        int wi = w;
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(kFull, wi, o);
            if (lane >= o) wi += t;
        }
        warp_tot[lane] = wi - w;  // exclusive prefix of warp totals
    }
    __syncthreads();
    int excl = inc - local + warp_tot[warp];
    if (base < count) out[base] = excl;
    if (base + 1 < count) out[base + 1] = excl + a0;
    if (threadIdx.x == kScanThreads - 1 && tile_sums) tile_sums[blockIdx.x] = excl + local;
}

__global__ void k_scan_add(int* __restrict__ out, int count, const int* __restrict__ tile_offs) {
    const int base = blockIdx.x * kScanTile + 2 * threadIdx.x;
    const int add = tile_offs[blockIdx.x];
    if (base < count) out[base] += add;
    if (base + 1 < count) out[base + 1] += add;
}

__global__ void k_copy_total(const int* in_last, const int* out_last, int* total) {
    *total = *in_last + *out_last;
}

// ---------------------------------------------------------------------------
// transpose
// ---------------------------------------------------------------------------
__global__ void k_count_cols(const int* __restrict__ ci, int nnz, int* __restrict__ cnt) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += gridDim.x * blockDim.x)
        atomicAdd(&cnt[ci[e]], 1);
}

// one warp per row of A: every entry takes a slot in its column's segment
__global__ void k_fill_slots(const int* __restrict__ rp, const int* __restrict__ ci, int rows,
                             const int* __restrict__ rp_t, int* __restrict__ cursor, int* __restrict__ key) {
    const int warps = gridDim.x * blockDim.x / 32;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) / 32; i < rows; i += warps) {
        for (int e = rp[i] + (threadIdx.x & 31); e < rp[i + 1]; e += 32) {
            int j = ci[e];
            int pos = rp_t[j] + atomicAdd(&cursor[j], 1);
            key[pos] = e;
        }
    }
}

// segments of <= 32 keys: one warp, bitonic network in registers
__global__ void k_segsort_warp(const int* __restrict__ seg, int nseg, int* __restrict__ key) {
    const int warps = gridDim.x * blockDim.x / 32;
    const int lane = threadIdx.x & 31;
    for (int s = (blockIdx.x * blockDim.x + threadIdx.x) / 32; s < nseg; s += warps) {
        const int beg = seg[s], len = seg[s + 1] - beg;
        if (len <= 1 || len > 32) continue;
        int v = lane < len ? key[beg + lane] : INT_MAX;
        for (int k = 2; k <= 32; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                int o = __shfl_xor_sync(kFull, v, j);
                bool asc = (lane & k) == 0, lower = (lane & j) == 0;
                v = (asc == lower) ? min(v, o) : max(v, o);
            }
        if (lane < len) key[beg + lane] = v;
    }
}

// segments of 33..2048 keys: one block, bitonic network in shared memory
constexpr int kSegBlock = 2048;
__global__ void k_segsort_block(const int* __restrict__ seg, int nseg, int* __restrict__ key) {
    __shared__ int buf[kSegBlock];
    for (int s = blockIdx.x; s < nseg; s += gridDim.x) {
        const int beg = seg[s], len = seg[s + 1] - beg;
        if (len <= 32 || len > kSegBlock) continue;
        int p = 64;
        while (p < len) p <<= 1;
        for (int i = threadIdx.x; i < p; i += blockDim.x) buf[i] = i < len ? key[beg + i] : INT_MAX;
        __syncthreads();
        for (int k = 2; k <= p; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int i = threadIdx.x; i < p; i += blockDim.x) {
                    int q = i ^ j;
                    if (q > i) {
                        bool asc = (i & k) == 0;
                        int a = buf[i], b = buf[q];
                        if ((a > b) == asc) { buf[i] = b; buf[q] = a; }
                    }
                }
                __syncthreads();
            }
        for (int i = threadIdx.x; i < len; i += blockDim.x) key[beg + i] = buf[i];
        __syncthreads();
    }
}

__device__ int lower_bound_i(const int* a, int n, int v) {
    int lo = 0, hi = n;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// segments of > 2048 keys: one block, bottom-up merge sort through `tmp`
// (keys are distinct entry indices, so a key's rank in the other run fixes
// its output position)
__global__ void k_segsort_big(const int* __restrict__ seg, int nseg, int* __restrict__ key, int* __restrict__ tmp) {
    for (int s = blockIdx.x; s < nseg; s += gridDim.x) {
        const int beg = seg[s], len = seg[s + 1] - beg;
        if (len <= kSegBlock) continue;
        int* src = key + beg;
        int* dst = tmp + beg;
        for (int w = 1; w < len; w <<= 1) {
            for (int p = threadIdx.x; p < len; p += blockDim.x) {
                int lo = (p / (2 * w)) * (2 * w);
                int mid = min(lo + w, len), hi = min(lo + 2 * w, len);
                int v = src[p];
                int pos = p < mid ? (p - lo) + lower_bound_i(src + mid, hi - mid, v)
                                  : (p - mid) + lower_bound_i(src + lo, mid - lo, v);
                dst[lo + pos] = v;
            }
            __syncthreads();
            int* t = src; src = dst; dst = t;
        }
        if (src != key + beg)
            for (int p = threadIdx.x; p < len; p += blockDim.x) key[beg + p] = src[p];
        __syncthreads();
    }
}

// A^T entry at `pos` comes from A entry key[pos]: its column in A^T is the
// row of that entry in A (binary search in row_ptr), its value is A's value.
__global__ void k_finish_transpose(const int* __restrict__ rp, int rows, const int* __restrict__ key, int nnz,
                                   const double* __restrict__ vals, int* __restrict__ ci_t,
                                   double* __restrict__ vals_t) {
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += gridDim.x * blockDim.x) {
        int e = key[p];
        int lo = 0, hi = rows;  // last row with rp[row] <= e
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (rp[mid] <= e) lo = mid; else hi = mid;
        }
        ci_t[p] = lo;
        vals_t[p] = vals[e];
    }
}

// ---------------------------------------------------------------------------
// long-row lists
// ---------------------------------------------------------------------------
__global__ void k_long_flags(const int* __restrict__ rp, int rows, int thr, int* __restrict__ flag) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows; i += gridDim.x * blockDim.x)
        flag[i] = (rp[i + 1] - rp[i]) > thr ? 1 : 0;
}

// each long row with its entries' range
__global__ void k_long_ranges(const int* __restrict__ rp, const int* __restrict__ rows, int count,
                              int4* __restrict__ out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        out[i] = make_int4(rows[i], rp[rows[i]], rp[rows[i] + 1], 0);
}

__global__ void k_long_scatter(const int* __restrict__ flag, const int* __restrict__ pos, int rows,
                               int* __restrict__ list) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows; i += gridDim.x * blockDim.x)
        if (flag[i]) list[pos[i]] = i;
}

// ---------------------------------------------------------------------------
// short rows in the order of the step kernels
// ---------------------------------------------------------------------------
// Two lists (Csr::srec, Csr::nrec; step_args says which step takes which).
// The first: windows of kWindow rows, each sorted by length, longest first (the
// windows of the SELL-C-sigma format of Kreutzer, Hager, Wellein, Fehske and
// Bishop, SIAM J. Sci. Comput. 36(5), 2014): the row groups of a warp then take
// rows of about the same length, and rows that lie near one another stay near
// (a window's rows share what they gather in L2).  The second: the rows as they
// stand, so that a warp's narrow row groups read and write their points, 16 to
// 128 bytes a row, in whole lines.
constexpr int kWindow = 2048;

// per window: its rows of at most thr entries
__global__ void __launch_bounds__(256) k_short_count(const int* __restrict__ rp, int rows, int thr,
                                                     int* __restrict__ cnt) {
    __shared__ int sum;
    if (threadIdx.x == 0) sum = 0;
    __syncthreads();
    int mine = 0;
    for (int q = threadIdx.x; q < kWindow; q += blockDim.x) {
        const int i = blockIdx.x * kWindow + q;
        if (i < rows && rp[i + 1] - rp[i] <= thr) ++mine;
    }
    if (mine) atomicAdd(&sum, mine);
    __syncthreads();
    if (threadIdx.x == 0) cnt[blockIdx.x] = sum;
}

// one block per window: bitonic sort of the places' keys (short_key), the
// rows of more than thr entries and the places past the last row at the end;
// equal lengths keep their order
__global__ void __launch_bounds__(1024) k_short_order(const int* __restrict__ rp, int rows, int thr,
                                                      const int* __restrict__ first, int4* __restrict__ out) {
    __shared__ unsigned long long key[kWindow];
    const int base = blockIdx.x * kWindow;
    for (int q = threadIdx.x; q < kWindow; q += blockDim.x) {
        const int i = base + q;
        key[q] = short_key(i < rows, i < rows ? rp[i + 1] - rp[i] : 0, thr, q);
    }
    __syncthreads();
    for (int k = 2; k <= kWindow; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int q = threadIdx.x; q < kWindow; q += blockDim.x) {
                const int p = q ^ j;
                if (p > q) {
                    const unsigned long long x = key[q], y = key[p];
                    if ((x > y) == ((q & k) == 0)) {
                        key[q] = y;
                        key[p] = x;
                    }
                }
            }
            __syncthreads();
        }
    for (int q = threadIdx.x; q < kWindow; q += blockDim.x) {
        if (!is_short(key[q])) continue;
        const int i = base + (int)(key[q] & 0xffffffffull);
        out[first[blockIdx.x] + q] = make_int4(i, 0, 0, rp[i + 1] - rp[i]);
    }
}

// fours of entries of each record
__global__ void k_short_fours(const int4* __restrict__ rec, int n, int* __restrict__ cnt) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        cnt[i] = (rec[i].w + 3) / 4;
}
__global__ void k_short_place(int4* __restrict__ rec, int n, const int* __restrict__ first) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        rec[i].y = first[i];
        rec[i].z = (rec[i].w + 1) / 2;
    }
}

// the record of each row, and from it the records in the rows' order (first:
// how many short rows stand before a row)
__global__ void k_short_where(const int4* __restrict__ rec, int n, int* __restrict__ place) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) place[rec[i].x] = i;
}
__global__ void k_short_flags(const int* __restrict__ rp, int rows, int thr, int* __restrict__ flag) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows; i += gridDim.x * blockDim.x)
        flag[i] = rp[i + 1] - rp[i] <= thr ? 1 : 0;
}
__global__ void k_short_narrow(const int4* __restrict__ rec, const int* __restrict__ place,
                               const int* __restrict__ rp, int rows, int thr, const int* __restrict__ first,
                               int4* __restrict__ out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows; i += gridDim.x * blockDim.x)
        if (rp[i + 1] - rp[i] <= thr) {
            const int p = place[i];
            const int4 r = rec[p];
            out[first[i]] = make_int4(i, r.y, r.z, p);
        }
}
// (last: the entries are counted by the word until then)
__global__ void k_short_self(int4* __restrict__ rec, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) rec[i].w = i;
}

// columns of the packed entries, and their values and the rows' vectors: a
// warp per record; an odd row's last pair is filled up with its last entry's
// column and the value 0
__global__ void k_short_cols(const int4* __restrict__ rec, int n, const int* __restrict__ rp,
                             const int* __restrict__ ci, int* __restrict__ out) {
    const int warps = gridDim.x * blockDim.x / 32, lane = threadIdx.x & 31;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) / 32; i < n; i += warps) {
        const int4 r = rec[i];
        const int b = rp[r.x];
        for (int e = lane; e < (r.w + 3) / 4 * 4; e += 32)
            out[(size_t)r.y * 4 + e] = ci[b + (e < r.w ? e : r.w - 1)];
    }
}
template <typename T>
__global__ void k_short_vals(const int4* __restrict__ rec, int n, const int* __restrict__ rp, RowVectors<T> v,
                             T* __restrict__ out, T* __restrict__ k) {
    const int warps = gridDim.x * blockDim.x / 32, lane = threadIdx.x & 31;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) / 32; i < n; i += warps) {
        const int4 r = rec[i];
        const int b = rp[r.x];
        for (int e = lane; e < (r.w + 3) / 4 * 4; e += 32)
            out[(size_t)r.y * 4 + e] = e < r.w ? v.vals[b + e] : T(0);
        if (lane == 0) {
            k[4 * (size_t)i] = v.c ? v.c[r.x] : T(0);
            k[4 * (size_t)i + 1] = v.lo[r.x];
            k[4 * (size_t)i + 2] = v.hi[r.x];
            k[4 * (size_t)i + 3] = T(0);
        }
    }
}

// ---------------------------------------------------------------------------
// equilibration
// ---------------------------------------------------------------------------
// One warp per CSR row: max or sum of |D_r[i] * a * D_c[j]| where, for the
// CSR of A^T, the row is a variable j and the column a constraint i (the
// product is always formed in the order D_r * a * D_c).
template <bool SUM>
__global__ void k_row_stat(const int* __restrict__ rp, const int* __restrict__ ci, const double* __restrict__ v,
                           int rows, const double* __restrict__ d_row, const double* __restrict__ d_col,
                           bool rows_are_constraints, double* __restrict__ out) {
    const int warps = gridDim.x * blockDim.x / 32;
    const int lane = threadIdx.x & 31;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) / 32; i < rows; i += warps) {
        double acc = 0.0;
        for (int e = rp[i] + lane; e < rp[i + 1]; e += 32) {
            int j = ci[e];
            double a = rows_are_constraints ? fabs(d_row[i] * v[e] * d_col[j]) : fabs(d_col[j] * v[e] * d_row[i]);
            acc = SUM ? acc + a : fmax(acc, a);
        }
        for (int o = 16; o > 0; o >>= 1) {
            double t = __shfl_down_sync(kFull, acc, o);
            acc = SUM ? acc + t : fmax(acc, t);
        }
        if (lane == 0) out[i] = acc;
    }
}

__global__ void k_apply_scale(double* __restrict__ d, const double* __restrict__ stat, int count) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        if (stat[i] > 0.0) d[i] /= sqrt(stat[i]);
}

__global__ void k_fill_d(double* d, int count, double v) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) d[i] = v;
}

// scaled values: warp per row, D_r[i] * a * D_c[j] with i the constraint
__global__ void k_scale_vals(const int* __restrict__ rp, const int* __restrict__ ci, const double* __restrict__ v,
                             int rows, const double* __restrict__ d_r, const double* __restrict__ d_c,
                             bool rows_are_constraints, double* __restrict__ o64, float* __restrict__ o32) {
    const int warps = gridDim.x * blockDim.x / 32;
    const int lane = threadIdx.x & 31;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) / 32; i < rows; i += warps) {
        for (int e = rp[i] + lane; e < rp[i + 1]; e += 32) {
            int j = ci[e];
            double s = rows_are_constraints ? d_r[i] * v[e] * d_c[j] : d_r[j] * v[e] * d_c[i];
            o64[e] = s;
            if (o32) o32[e] = (float)s;
        }
    }
}

__global__ void k_scale_vectors(int m, int n, const double* __restrict__ d_r, const double* __restrict__ d_c,
                                const double* __restrict__ c, const double* __restrict__ l,
                                const double* __restrict__ u, const double* __restrict__ xl,
                                const double* __restrict__ xu, double* cs, double* ls, double* us, double* xls,
                                double* xus) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < max(m, n); i += gridDim.x * blockDim.x) {
        if (i < n) {
            cs[i] = d_c[i] * c[i];
            xls[i] = xl[i] / d_c[i];
            xus[i] = xu[i] / d_c[i];
        }
        if (i < m) {
            ls[i] = d_r[i] * l[i];
            us[i] = d_r[i] * u[i];
        }
    }
}

__global__ void k_to_f32(const double* __restrict__ in, float* __restrict__ out, int count) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) out[i] = (float)in[i];
}

// ---------------------------------------------------------------------------
// deterministic two-stage sums
// ---------------------------------------------------------------------------
constexpr int kSumBlocks = 256;
constexpr int kSumThreads = 256;

__device__ __forceinline__ double block_sum(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (warp == 0) {
        t = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(kFull, t, o);
    }
    __syncthreads();
    return t;  // valid in thread 0
}

// mode 0: sum v^2; mode 1: sum over rows of b~_i^2 (finite bound of larger magnitude)
__global__ void k_sum_stage1(const double* __restrict__ a, const double* __restrict__ b, int count, int mode,
                             double* __restrict__ part) {
    __shared__ double sh[32];
    double acc = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        if (mode == 0) {
            acc += a[i] * a[i];
        } else {
            double l = a[i], u = b[i], r = 0.0;
            bool fl = isfinite(l), fu = isfinite(u);
            if (fl && fu) r = fabs(l) > fabs(u) ? l : u;
            else if (fl) r = l;
            else if (fu) r = u;
            acc += r * r;
        }
    }
    double t = block_sum(acc, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

__global__ void k_sum_stage2(const double* __restrict__ part, int count, double* __restrict__ out) {
    __shared__ double sh[32];
    double acc = 0.0;
    for (int i = threadIdx.x; i < count; i += blockDim.x) acc += part[i];
    double t = block_sum(acc, sh);
    if (threadIdx.x == 0) *out = t;
}

// ---------------------------------------------------------------------------
// power iteration
// ---------------------------------------------------------------------------
// SplitMix64 (Steele, Lea, Flood, OOPSLA 2014): the index-th output of the
// generator whose state starts at `seed`.
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t index) {
    uint64_t z = seed + (index + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void k_power_init(double* v, int n, uint64_t seed) {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
        v[j] = 2.0 * ((double)(splitmix64(seed, (uint64_t)j) >> 11) * 0x1.0p-53) - 1.0;
}

// One product of A~^T A~ takes two launches of k_power_spmv.  Each block
// leaves its share of the squared norm of the result as one partial, and the
// next launch adds the partials in block order: the forward launch in every
// block (it scales by the norm), the other in its first block (which only
// records it).  The first block decides whether the iteration has stopped;
// launches queued past that point return at once.  The grid is fixed, so the
// rows each block covers and the order of every sum are the same on every
// run.  The vector is kept near unit norm by a power of two, which rounds
// nothing: u = 2^-e A~ w with e the exponent of ||w||, and the estimate
// ||A~ w|| / ||w|| = ||u|| / (2^-e ||w||) is formed once.
//
// What bounds a launch on a matrix in L2 is the FP64 pipe (a warp's
// multiply-add takes it 16 cycles; a division by ||w|| per row took some 200)
// and the chain of round trips around it.  So a short row has few lanes, only
// the multiply-adds that some lane of a warp needs are issued, the blocks are
// few and large (one ticket per block, 512 to 3125 of them, took 28 to 48 us
// a launch), a row group has its next row's entries on their way while it
// gathers for this one, and the first row's are loaded ahead of the wait for
// the previous launch (programmatic dependent launch).
constexpr int kPowBlocks = 152;
constexpr int kPowThreads = 1024;
constexpr int kPowGroup = 4;      // lanes of a short row
constexpr int kPowLong = 1024;    // rows with more entries take a block, other long rows a warp

struct PowArgs {
    const int* rp;
    const int* ci;
    const double* v;
    int rows;
    const int* mid;         // rows of more than kLongRow entries
    int n_mid;
    const int* longs;       // rows of more than kPowLong entries
    int n_long;
    const double* x;
    double* y;
    const double* pin;      // partials of the operand's squared norm
    double* pout;
    double* xnorm;          // forward: the operand's scaled norm, read by the second launch
    double* est;            // estimate of each product
    int it;
    int* stop;
    double tol;
};

// 2^-e with e the exponent of v (1 for a v that has none)
__device__ __forceinline__ double pow2_below(double v) {
    const long long e = __double_as_longlong(v) >> 52 & 0x7ff;
    return e >= 1 && e <= 2045 ? __longlong_as_double((2046 - e) << 52) : 1.0;
}

// sum of part[0 .. count) in a fixed order; warp 0 calls it, the sum is in
// all its lanes
__device__ __forceinline__ double warp_sum(const double* part, int count, bool global) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < count; i += 32) acc += global ? __ldcg(part + i) : part[i];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
    return acc;
}

// y = 2^-e M x with e the exponent of ||x|| (FWD; 0 when the norm is 0), or
// y = M x, and the partials of its norm.
template <bool FWD>
__global__ void __launch_bounds__(kPowThreads, 1) k_power_spmv(const PowArgs a) {
    constexpr int U = 4, kGroups = kPowThreads / kPowGroup, kWarps = kPowThreads / 32;
    __shared__ double sh[kGroups];
    __shared__ double sh_nx;
    const int tid = threadIdx.x, lane = tid % kPowGroup, grp = tid / kPowGroup;
    const int stride = kPowBlocks * kGroups;
    int i = (int)blockIdx.x * kGroups + grp;
    // entries [b, e) of a short row; none of another
    auto bounds = [&](int r, int& b, int& e) {
        b = r < a.rows ? __ldg(a.rp + r) : 0;
        e = r < a.rows ? __ldg(a.rp + r + 1) : 0;
        if (e - b > kLongRow) e = b;
    };
    auto load = [&](int e0, int step, int end, int (&c)[U], double (&w)[U]) {
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int e = e0 + k * step;
            c[k] = e < end ? __ldg(a.ci + e) : -1;
            w[k] = e < end ? __ldg(a.v + e) : 0.0;
        }
    };
    // x was written by the previous launch: read through L2
    auto gather = [&](const int (&c)[U], double (&xs)[U]) {
#pragma unroll
        for (int k = 0; k < U; ++k) xs[k] = c[k] >= 0 ? __ldcg(a.x + c[k]) : 0.0;
    };
    int beg, end, nbeg, nend, c[U];
    double w[U];
    bounds(i, beg, end);
    load(beg + lane, kPowGroup, end, c, w);
    bounds(i + stride, nbeg, nend);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (*(volatile const int*)a.stop) return;
    if (tid < 32 && (FWD || blockIdx.x == 0)) {
        const double nx = sqrt(warp_sum(a.pin, kPowBlocks, true));
        if (tid == 0) sh_nx = nx;
        if (tid == 0 && blockIdx.x == 0) {
            if (FWD) {
                *a.xnorm = nx * pow2_below(nx);
                // product it - 1 is complete
                const int p = a.it - 1;
                const double now = p > 1 ? __ldcg(a.est + p) : 0.0, before = p > 1 ? __ldcg(a.est + p - 1) : 0.0;
                if (p >= 1 && (!(nx > 0.0) || (p > 1 && fabs(now - before) <= a.tol * now))) *a.stop = p;
            } else {
                const double xn = __ldcg(a.xnorm);
                a.est[a.it] = xn > 0.0 ? nx / xn : 0.0;
            }
        }
    }
    double sc = 1.0;
    if (FWD) {
        __syncthreads();
        sc = sh_nx > 0.0 ? pow2_below(sh_nx) : 0.0;
    }
    double sq = 0.0;  // this thread's rows' squares
    // the longest rows: a block each
    for (int q = blockIdx.x; q < a.n_long; q += kPowBlocks) {
        const int r = a.longs[q], b = __ldg(a.rp + r), e1 = __ldg(a.rp + r + 1);
        double acc = 0.0;
        for (int e = b + tid; e < e1; e += U * kPowThreads) {
            int cc[U];
            double ww[U], xs[U];
            load(e, kPowThreads, e1, cc, ww);
            gather(cc, xs);
#pragma unroll
            for (int k = 0; k < U; ++k) acc += ww[k] * xs[k];
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
        __syncthreads();
        if ((tid & 31) == 0) sh[tid >> 5] = acc;
        __syncthreads();
        if (tid < 32) {
            const double yi = warp_sum(sh, kWarps, false) * sc;
            if (tid == 0) {
                a.y[r] = yi;
                sq += yi * yi;
            }
        }
    }
    // the other long rows: a warp each
    for (int q = (int)blockIdx.x * kWarps + (tid >> 5); q < a.n_mid; q += kPowBlocks * kWarps) {
        const int r = a.mid[q], b = __ldg(a.rp + r), e1 = __ldg(a.rp + r + 1);
        if (e1 - b > kPowLong) continue;
        double acc = 0.0;
        for (int e = b + (tid & 31); e - (tid & 31) < e1; e += U * 32) {
            int cc[U];
            double ww[U], xs[U];
            load(e, 32, e1, cc, ww);
            gather(cc, xs);
#pragma unroll
            for (int k = 0; k < U; ++k)
                if (e - (tid & 31) + k * 32 < e1) acc += ww[k] * xs[k];
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
        if ((tid & 31) == 0) {
            const double yi = acc * sc;
            a.y[r] = yi;
            sq += yi * yi;
        }
    }
    // the short rows: kPowGroup lanes each (the trip count is the block's, so
    // that every lane reaches the shuffles)
    for (int base = (int)blockIdx.x * kGroups; base < a.rows; base += stride) {
        const int row = i, b = beg, e1 = end;
        double xs[U], ws[U];
        gather(c, xs);
#pragma unroll
        for (int k = 0; k < U; ++k) ws[k] = w[k];
        beg = nbeg;
        end = nend;
        load(beg + lane, kPowGroup, end, c, w);
        i += stride;
        bounds(i + stride, nbeg, nend);
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < U; ++k)
            if (__any_sync(kFull, b + lane + k * kPowGroup < e1)) acc += ws[k] * xs[k];
        for (int e = b + lane + U * kPowGroup; __any_sync(kFull, e < e1); e += U * kPowGroup) {
            int cc[U];
            load(e, kPowGroup, e1, cc, ws);
            gather(cc, xs);
#pragma unroll
            for (int k = 0; k < U; ++k)
                if (__any_sync(kFull, e + k * kPowGroup < e1)) acc += ws[k] * xs[k];
        }
        for (int o = kPowGroup / 2; o > 0; o >>= 1) acc += __shfl_down_sync(kFull, acc, o, kPowGroup);
        if (lane == 0 && row < a.rows && __ldg(a.rp + row + 1) - __ldg(a.rp + row) <= kLongRow) {
            const double yi = acc * sc;
            a.y[row] = yi;
            sq += yi * yi;
        }
    }
    // squares sit in the groups' first lanes (the block's and the warps' rows
    // in lanes that are among them)
    __syncthreads();
    if (lane == 0) sh[grp] = sq;
    __syncthreads();
    if (tid < 32) {
        const double t = warp_sum(sh, kGroups, false);
        if (tid == 0) a.pout[blockIdx.x] = t;
    }
}

// partials of the squared norm of x
__global__ void __launch_bounds__(256) k_power_norm(const double* __restrict__ x, int count, double* __restrict__ part) {
    __shared__ double sh[32];
    double acc = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) acc += x[i] * x[i];
    const double t = block_sum(acc, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

// Blocks of the Ruiz and Pock-Chambolle row statistics (a warp per row, so
// the grid changes no result): up to 16384, about 8 rows per warp on a
// 1M-row matrix
constexpr int kStatCap = 16384;

inline int grid_for(long long work, int threads, int cap = 4096) {
    long long g = (work + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

}  // namespace

// ---------------------------------------------------------------------------
// host wrappers
// ---------------------------------------------------------------------------
cudaError_t exclusive_scan_i32(const int* in, int* out, int count, int* total_dev, cudaStream_t s) {
    if (count <= 0) {
        if (total_dev) return cudaMemsetAsync(total_dev, 0, sizeof(int), s);
        return cudaSuccess;
    }
    const int tiles = (count + kScanTile - 1) / kScanTile;
    StreamMem mem(s);
    int* sums = nullptr;
    int* offs = nullptr;
    cudaError_t e = cudaSuccess;
    if (tiles > 1) {
        if ((e = mem.take(sizeof(int) * (size_t)tiles * 2)) != cudaSuccess) return e;
        sums = (int*)mem.p;
        offs = sums + tiles;
    }
    k_scan_tile<<<tiles, kScanThreads, 0, s>>>(in, out, count, sums);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (tiles > 1) {
        if ((e = exclusive_scan_i32(sums, offs, tiles, nullptr, s)) != cudaSuccess) return e;
        k_scan_add<<<tiles, kScanThreads, 0, s>>>(out, count, offs);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (total_dev) {
        k_copy_total<<<1, 1, 0, s>>>(in + count - 1, out + count - 1, total_dev);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return e;
}

cudaError_t transpose_csr(const Csr& a, const double* a_vals, Csr& at, int* perm_out, cudaStream_t s) {
    // at.rp (cols + 1), at.ci (nnz) and perm_out-sized scratch are allocated by the caller;
    // perm_out receives the A^T slot -> A entry map, vals_t is written into at.v64.
    cudaError_t e;
    const int nnz = a.nnz, cols = a.cols;
    int *cnt = nullptr, *cursor = nullptr, *tmp = nullptr;
    if ((e = cudaMallocAsync((void**)&cnt, sizeof(int) * (size_t)(cols + 1) * 2, s)) != cudaSuccess) return e;
    cursor = cnt + cols + 1;
    if ((e = cudaMemsetAsync(cnt, 0, sizeof(int) * (size_t)(cols + 1) * 2, s)) != cudaSuccess) return e;
    if (nnz > 0) {
        k_count_cols<<<grid_for(nnz, 256), 256, 0, s>>>(a.ci, nnz, cnt);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = exclusive_scan_i32(cnt, at.rp, cols + 1, nullptr, s)) != cudaSuccess) return e;
    if (nnz > 0) {
        k_fill_slots<<<grid_for((long long)a.rows * 32, 256), 256, 0, s>>>(a.rp, a.ci, a.rows, at.rp, cursor, perm_out);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_segsort_warp<<<grid_for((long long)cols * 32, 256), 256, 0, s>>>(at.rp, cols, perm_out);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_segsort_block<<<grid_for(cols, 1, 1024), 1024, 0, s>>>(at.rp, cols, perm_out);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = cudaMallocAsync((void**)&tmp, sizeof(int) * (size_t)nnz, s)) != cudaSuccess) return e;
        k_segsort_big<<<grid_for(cols, 1, 256), 1024, 0, s>>>(at.rp, cols, perm_out, tmp);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_finish_transpose<<<grid_for(nnz, 256), 256, 0, s>>>(a.rp, a.rows, perm_out, nnz, a_vals, at.ci, at.v64);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = cudaFreeAsync(tmp, s)) != cudaSuccess) return e;
    }
    return cudaFreeAsync(cnt, s);
}

// Segments of the long rows for the step kernels: a long row of len entries
// gets ceil(len / kStepSeg) segments of ceil(len / segments) entries, the
// last ones shorter; blocks are listed segment-major.
static cudaError_t build_long_segments(Csr& a, cudaStream_t s) {
    cudaError_t e;
    if (a.n_long == 0) return cudaSuccess;
    std::vector<int4> rows(a.n_long);
    StreamMem mem(s);
    if ((e = mem.take(sizeof(int4) * (size_t)a.n_long)) != cudaSuccess) return e;
    int4* dev = (int4*)mem.p;
    k_long_ranges<<<grid_for(a.n_long, 256), 256, 0, s>>>(a.rp, a.long_rows, a.n_long, dev);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(rows.data(), dev, sizeof(int4) * a.n_long, cudaMemcpyDeviceToHost, s)) != cudaSuccess)
        return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    std::vector<int> part0(a.n_long + 1, 0);
    int most = 0;
    for (int i = 0; i < a.n_long; ++i) {
        a.long_nnz += rows[i].z - rows[i].y;
        const int segs = std::max(1, (rows[i].z - rows[i].y + kStepSeg - 1) / kStepSeg);
        part0[i + 1] = part0[i] + segs;
        most = std::max(most, segs);
    }
    std::vector<LongSeg> lseg;
    lseg.reserve((size_t)part0[a.n_long]);
    for (int seg = most - 1; seg >= 0; --seg)
        for (int i = 0; i < a.n_long; ++i) {
            const int segs = part0[i + 1] - part0[i];
            if (seg >= segs) continue;
            const int each = (rows[i].z - rows[i].y + segs - 1) / segs;
            const int beg = std::min(rows[i].z, rows[i].y + seg * each), end = std::min(rows[i].z, beg + each);
            lseg.push_back(LongSeg{rows[i].x, beg, end, i, seg, segs, part0[i], 0});
        }
    a.n_lseg = part0[a.n_long];
    if ((e = cudaMalloc((void**)&a.lseg, sizeof(LongSeg) * lseg.size())) != cudaSuccess) return e;
    return cudaMemcpy(a.lseg, lseg.data(), sizeof(LongSeg) * lseg.size(), cudaMemcpyHostToDevice);
}

void free_long_rows(Csr& a) {
    if (a.long_rows) cudaFree(a.long_rows);
    if (a.lseg) cudaFree(a.lseg);
    a.long_rows = nullptr;
    a.lseg = nullptr;
    a.n_long = a.n_lseg = 0;
    a.long_nnz = 0;
}

cudaError_t build_long_rows(Csr& a, cudaStream_t s) {
    cudaError_t e;
    if (a.long_rows || a.lseg) {
        if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
        free_long_rows(a);
    }
    a.n_long = 0;
    a.long_nnz = 0;
    a.n_lseg = 0;
    if (a.rows == 0) return cudaSuccess;
    StreamMem mem(s);
    if ((e = mem.take(sizeof(int) * ((size_t)a.rows * 2 + 1))) != cudaSuccess) return e;
    int *flag = (int*)mem.p, *pos = flag + a.rows, *total = pos + a.rows;
    k_long_flags<<<grid_for(a.rows, 256), 256, 0, s>>>(a.rp, a.rows, a.long_thr, flag);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = exclusive_scan_i32(flag, pos, a.rows, total, s)) != cudaSuccess) return e;
    int h_total = 0;
    if ((e = cudaMemcpyAsync(&h_total, total, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    a.n_long = h_total;
    if (h_total > 0) {
        if ((e = cudaMalloc((void**)&a.long_rows, sizeof(int) * (size_t)h_total)) != cudaSuccess) return e;
        k_long_scatter<<<grid_for(a.rows, 256), 256, 0, s>>>(flag, pos, a.rows, a.long_rows);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return build_long_segments(a, s);
}

void free_short_rows(Csr& a) {
    if (a.srec) cudaFree(a.srec);  // with all that lies behind it
    a.srec = a.nrec = nullptr;
    a.pci = nullptr;
    a.pv32 = a.pk32 = nullptr;
    a.pv64 = a.pk64 = nullptr;
    a.pvdf = a.pkdf = nullptr;
    a.n_short = 0;
}

template <typename T>
static cudaError_t pack_vals(const Csr& a, int n, RowVectors<T> v, T* out, T* k, cudaStream_t s) {
    if (!v.vals) return cudaSuccess;
    k_short_vals<T><<<grid_for((long long)n * 32, 256, kStatCap), 256, 0, s>>>(a.srec, n, a.rp, v, out, k);
    return cudaGetLastError();
}

cudaError_t build_short_rows(Csr& a, RowVectors<float> v32, RowVectors<double> v64, RowVectors<dfloat> vdf,
                             cudaStream_t s) {
    cudaError_t e;
    if (a.srec && (e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    free_short_rows(a);
    const int n = a.rows - a.n_long;
    if (n <= 0) return cudaSuccess;
    // one allocation: the records, the rows' vectors, and the entries, at most
    // three a row more than the short rows have (their exact number would cost
    // a wait); the long rows' entries stay where they are
    const size_t entries = (size_t)(a.nnz - a.long_nnz) + 3 * (size_t)n;
    size_t bytes = 0;
    auto take = [&](bool wanted, size_t size) {
        const size_t at = bytes;
        if (wanted) bytes += (size + 255) / 256 * 256;
        return at;
    };
    const size_t at_rec = take(true, sizeof(int4) * n), at_nrec = take(true, sizeof(int4) * n), at_ci = take(true, 4 * entries);
    const size_t at_v32 = take(v32.vals, 4 * entries), at_k32 = take(v32.vals, 16 * (size_t)n);
    const size_t at_v64 = take(v64.vals, 8 * entries), at_k64 = take(v64.vals, 32 * (size_t)n);
    const size_t at_vdf = take(vdf.vals, 8 * entries), at_kdf = take(vdf.vals, 32 * (size_t)n);
    char* mem = nullptr;
    if ((e = cudaMalloc((void**)&mem, bytes)) != cudaSuccess) return e;
    a.srec = (int4*)(mem + at_rec);
    a.nrec = (int4*)(mem + at_nrec);
    a.pci = (int*)(mem + at_ci);
    if (v32.vals) {
        a.pv32 = (float*)(mem + at_v32);
        a.pk32 = (float*)(mem + at_k32);
    }
    if (v64.vals) {
        a.pv64 = (double*)(mem + at_v64);
        a.pk64 = (double*)(mem + at_k64);
    }
    if (vdf.vals) {
        a.pvdf = (dfloat*)(mem + at_vdf);
        a.pkdf = (dfloat*)(mem + at_kdf);
    }
    const int windows = (a.rows + kWindow - 1) / kWindow;
    const size_t most = std::max((size_t)a.rows, (size_t)n);
    StreamMem scratch(s);
    if ((e = scratch.take(sizeof(int) * most * 2)) != cudaSuccess) return e;
    int *cnt = (int*)scratch.p, *first = cnt + most;
    k_short_count<<<windows, 256, 0, s>>>(a.rp, a.rows, a.long_thr, cnt);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = exclusive_scan_i32(cnt, first, windows, nullptr, s)) != cudaSuccess) return e;
    k_short_order<<<windows, 1024, 0, s>>>(a.rp, a.rows, a.long_thr, first, a.srec);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_short_fours<<<grid_for(n, 256), 256, 0, s>>>(a.srec, n, cnt);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = exclusive_scan_i32(cnt, first, n, nullptr, s)) != cudaSuccess) return e;
    k_short_place<<<grid_for(n, 256), 256, 0, s>>>(a.srec, n, first);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_short_flags<<<grid_for(a.rows, 256), 256, 0, s>>>(a.rp, a.rows, a.long_thr, cnt);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = exclusive_scan_i32(cnt, first, a.rows, nullptr, s)) != cudaSuccess) return e;
    k_short_where<<<grid_for(n, 256), 256, 0, s>>>(a.srec, n, cnt);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_short_narrow<<<grid_for(a.rows, 256), 256, 0, s>>>(a.srec, cnt, a.rp, a.rows, a.long_thr, first, a.nrec);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_short_cols<<<grid_for((long long)n * 32, 256, kStatCap), 256, 0, s>>>(a.srec, n, a.rp, a.ci, a.pci);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = pack_vals<float>(a, n, v32, a.pv32, a.pk32, s)) != cudaSuccess) return e;
    if ((e = pack_vals<double>(a, n, v64, a.pv64, a.pk64, s)) != cudaSuccess) return e;
    if ((e = pack_vals<dfloat>(a, n, vdf, a.pvdf, a.pkdf, s)) != cudaSuccess) return e;
    k_short_self<<<grid_for(n, 256), 256, 0, s>>>(a.srec, n);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    a.n_short = n;
    return cudaSuccess;
}

cudaError_t ruiz_pock_chambolle(const Csr& a, const double* a_vals, const Csr& at, const double* at_vals,
                                int ruiz_iters, int pock_chambolle, double* d_r, double* d_c, double* tmp_r,
                                double* tmp_c, cudaStream_t s) {
    cudaError_t e;
    const int m = a.rows, n = a.cols;
    if (m > 0) k_fill_d<<<grid_for(m, 256), 256, 0, s>>>(d_r, m, 1.0);
    k_fill_d<<<grid_for(n, 256), 256, 0, s>>>(d_c, n, 1.0);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    for (int it = 0; it < ruiz_iters + (pock_chambolle ? 1 : 0); ++it) {
        const bool pc = it >= ruiz_iters;
        // both statistics from the same A~, then both factors updated
        if (m > 0) {
            if (pc) k_row_stat<true><<<grid_for((long long)m * 32, 256, kStatCap), 256, 0, s>>>(a.rp, a.ci, a_vals, m, d_r, d_c, true, tmp_r);
            else k_row_stat<false><<<grid_for((long long)m * 32, 256, kStatCap), 256, 0, s>>>(a.rp, a.ci, a_vals, m, d_r, d_c, true, tmp_r);
        }
        if (pc) k_row_stat<true><<<grid_for((long long)n * 32, 256, kStatCap), 256, 0, s>>>(at.rp, at.ci, at_vals, n, d_c, d_r, false, tmp_c);
        else k_row_stat<false><<<grid_for((long long)n * 32, 256, kStatCap), 256, 0, s>>>(at.rp, at.ci, at_vals, n, d_c, d_r, false, tmp_c);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (m > 0) k_apply_scale<<<grid_for(m, 256), 256, 0, s>>>(d_r, tmp_r, m);
        k_apply_scale<<<grid_for(n, 256), 256, 0, s>>>(d_c, tmp_c, n);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t scale_values(const Csr& a, const double* a_vals, const double* d_r, const double* d_c,
                         bool rows_are_constraints, double* out64, float* out32, cudaStream_t s) {
    if (a.rows == 0 || a.nnz == 0) return cudaSuccess;
    k_scale_vals<<<grid_for((long long)a.rows * 32, 256), 256, 0, s>>>(a.rp, a.ci, a_vals, a.rows, d_r, d_c,
                                                                         rows_are_constraints, out64, out32);
    return cudaGetLastError();
}

cudaError_t scale_vectors(int m, int n, const double* d_r, const double* d_c, const double* c, const double* l,
                          const double* u, const double* xl, const double* xu, double* cs, double* ls, double* us,
                          double* xls, double* xus, cudaStream_t s) {
    k_scale_vectors<<<grid_for(m > n ? m : n, 256), 256, 0, s>>>(m, n, d_r, d_c, c, l, u, xl, xu, cs, ls, us, xls, xus);
    return cudaGetLastError();
}

cudaError_t convert_f32(const double* in, float* out, int count, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    k_to_f32<<<grid_for(count, 256), 256, 0, s>>>(in, out, count);
    return cudaGetLastError();
}

namespace {
// hi = value rounded to FP32, lo = the rounding error rounded to FP32; an
// infinite value is {+-inf, 0}
__global__ void k_split_df(const double* __restrict__ in, df* __restrict__ out, int count, bool recip) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const double v = recip ? 1.0 / in[i] : in[i];
        const float hi = (float)v;
        out[i] = df{hi, isfinite(v) && isfinite(hi) ? (float)(v - (double)hi) : 0.0f};
    }
}
__global__ void k_split_lo(const double* __restrict__ v64, const float* __restrict__ v32, float* __restrict__ lo,
                           int count) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        lo[i] = (float)(v64[i] - (double)v32[i]);
}
}  // namespace

cudaError_t split_df(const double* in, df* out, int count, bool recip, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    k_split_df<<<grid_for(count, 256), 256, 0, s>>>(in, out, count, recip);
    return cudaGetLastError();
}

cudaError_t split_lo(const double* v64, const float* v32, float* lo, int count, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    k_split_lo<<<grid_for(count, 256), 256, 0, s>>>(v64, v32, lo, count);
    return cudaGetLastError();
}

static cudaError_t two_stage(const double* a, const double* b, int count, int mode, double* out_dev, double* part,
                             cudaStream_t s) {
    k_sum_stage1<<<kSumBlocks, kSumThreads, 0, s>>>(a, b, count, mode, part);
    k_sum_stage2<<<1, kSumThreads, 0, s>>>(part, kSumBlocks, out_dev);
    return cudaGetLastError();
}

cudaError_t sq_norm(const double* v, int count, double* out_dev, cudaStream_t s) {
    double* part = nullptr;
    cudaError_t e = cudaMallocAsync((void**)&part, sizeof(double) * kSumBlocks, s);
    if (e != cudaSuccess) return e;
    if ((e = two_stage(v, nullptr, count, 0, out_dev, part, s)) != cudaSuccess) return e;
    return cudaFreeAsync(part, s);
}

cudaError_t rhs_norm2(const double* ls, const double* us, int m, double* out_dev, cudaStream_t s) {
    double* part = nullptr;
    cudaError_t e = cudaMallocAsync((void**)&part, sizeof(double) * kSumBlocks, s);
    if (e != cudaSuccess) return e;
    if ((e = two_stage(ls, us, m, 1, out_dev, part, s)) != cudaSuccess) return e;
    return cudaFreeAsync(part, s);
}

size_t power_work_doubles(int m, int n, int max_iter) {
    return (size_t)n + (size_t)(m > 0 ? m : 1) + 2 * (size_t)kPowBlocks + 2 + ((size_t)max_iter + 1);
}

// a launch of the product as a programmatic dependent of the previous one
static cudaError_t launch_power(void (*f)(PowArgs), const PowArgs& a, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kPowBlocks);
    cfg.blockDim = dim3(kPowThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, f, a);
}

// The products of power_norm; va and vat list the rows of more than kPowLong
// entries of A~ and A~^T.  `work` as power_work_doubles lays it out: w (n), u
// (m), the partials of ||u||^2 and ||w||^2, the scaled ||w||, the stop flag,
// the estimates; w starts as the unnormalised start vector.
static cudaError_t power_iterate(const Csr& a, const Csr& at, const Csr& va, const Csr& vat, int max_iter,
                                 double tol, uint64_t seed, double* work, double* est_out, int* iters_out,
                                 cudaStream_t s) {
    const int m = a.rows, n = a.cols;
    double* w = work;
    double* u = w + n;
    double* part_u = u + (m > 0 ? m : 1);
    double* part_w = part_u + kPowBlocks;
    double* xnorm = part_w + kPowBlocks;
    int* stop = reinterpret_cast<int*>(xnorm + 1);
    double* est = xnorm + 2;
    cudaError_t e;
    if ((e = cudaMemsetAsync(stop, 0, sizeof(double), s)) != cudaSuccess) return e;
    k_power_init<<<grid_for(n, 256), 256, 0, s>>>(w, n, seed);
    k_power_norm<<<kPowBlocks, 256, 0, s>>>(w, n, part_w);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    PowArgs fwd{a.rp,  a.ci, a.v64, m, a.long_rows, a.n_long, va.long_rows, va.n_long, w,
                u, part_w, part_u, xnorm, est, 0, stop, tol};
    PowArgs back{at.rp, at.ci, at.v64, n, at.long_rows, at.n_long, vat.long_rows, vat.n_long, u,
                 w, part_u, part_w, xnorm, est, 0, stop, tol};
    // products queued between two looks at the stop flag (those past it return at once)
    constexpr int kChunk = 64;
    int last = 0;
    for (int base = 1; base <= max_iter; base += kChunk) {
        last = base + kChunk - 1 < max_iter ? base + kChunk - 1 : max_iter;
        for (int it = base; it <= last; ++it) {
            // u = 2^-e A~ w, then w = A~^T u and est[it] = ||A~ w|| / ||w||
            fwd.it = back.it = it;
            if ((e = launch_power(k_power_spmv<true>, fwd, s)) != cudaSuccess) return e;
            if ((e = launch_power(k_power_spmv<false>, back, s)) != cudaSuccess) return e;
        }
        int stopped = 0;
        if ((e = cudaMemcpyAsync(&stopped, stop, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
        if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
        if (stopped) {
            last = stopped;
            break;
        }
    }
    *iters_out = last;
    if ((e = cudaMemcpyAsync(est_out, est + last, sizeof(double), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    return cudaStreamSynchronize(s);
}

// Power iteration on A~^T A~: sigma_est = ||A~ v|| for unit v.  Stops at the
// first product where the estimate moves by <= tol relative, or when
// ||A~^T A~ v|| = 0, or after max_iter products.
cudaError_t power_norm(const Csr& a, const Csr& at, int max_iter, double tol, uint64_t seed, double* work,
                       double* est_out, int* iters_out, cudaStream_t s) {
    cudaError_t e;
    *est_out = 0.0;
    *iters_out = 0;
    if (a.rows == 0 || a.nnz == 0) return cudaSuccess;
    // the rows of more than kPowLong entries of A~ and A~^T, one block each
    Csr va = a, vat = at;
    for (Csr* c : {&va, &vat}) {
        const bool some = c->n_long > 0;  // rows of more than kLongRow entries
        c->long_rows = nullptr;
        c->lseg = nullptr;
        c->n_long = 0;
        c->long_thr = kPowLong;
        if (some && (e = build_long_rows(*c, s)) != cudaSuccess) {
            free_long_rows(va);
            free_long_rows(vat);
            return e;
        }
    }
    e = power_iterate(a, at, va, vat, max_iter, tol, seed, work, est_out, iters_out, s);
    if (e != cudaSuccess) cudaStreamSynchronize(s);
    free_long_rows(va);
    free_long_rows(vat);
    return e;
}

}  // namespace lpb
