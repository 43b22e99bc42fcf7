// lpb_resident.cu -- a whole interval of a small matrix in one launch.
//
// The columns of a batch do not touch one another between checks, so a tile
// of C columns can run its L iterations by itself: one block keeps the tile's
// reflected point (n x C), dual iterate (m x C), the two gathered blocks, and
// their anchors in shared memory and walks all rows of A~^T and A~ in every
// iteration, with block barriers in place of kernel boundaries.  The matrix
// and the row records are read through L1.  At the interval's last iteration
// the block writes the state and the check's operands to the same global
// blocks as the step kernels, so the checks, compaction and migration do not
// know which kernel ran.
//
// Every row is summed in the order in which the step kernel at this batch
// width sums it (pieces and segments of long rows among it) and the
// elementwise steps are the same code (primal_element, dual_element): while
// the points are finite, the iterates are bitwise those of the step kernels.
// (A lane that is shorter than its slice adds 0 times its first entry's point,
// a packed row of an odd length 0 times its last one's: an infinite point
// can make the one sum NaN and leave the other infinite.)
//
// Why one block and no cluster: splitting the rows over the blocks of a
// cluster needs each block's rows in every other block's shared memory twice
// an iteration; such stores move 18 bytes a cycle and SM here, an exchange
// takes 900 cycles at least, and the cluster barrier's acquire drops the
// matrix from L1.  Four to eight blocks a tile took 5 to 12 us an iteration on
// the 1k x 2k matrix, one block 4.6.  What bounds it then: the gathers' bank
// conflicts and issue (FP32), the FP64 pipe (FP64), and L1, which has to hold
// the matrix (res_us says where that ends and the step kernels are faster).
// A pass of 512 iterations and 8 checks, step kernels and this one: 37 LPs on
// 1k x 2k, FP32, 4.5 and 3.2 ms; 16 LPs on 200 x 400, FP64, 4.7 and 2.9 ms.
#include <atomic>
#include <climits>
#include <cstring>
#include <memory>
#include <new>
#include <utility>

#include "lpb_engine.h"
#include "lpb_resident.h"
#include "lpb_step.h"

namespace lpb {

namespace {

constexpr int kResThreads = 1024;  // most threads of a block
constexpr int kResStatic = 1024;   // shared memory left to the tile's parameters

// A row's bounds, cost (primal) and word.
template <typename T>
struct alignas(16) ResRec {
    T lo, hi, c;
    uint32_t word;
};
template <typename T>
struct alignas(2 * sizeof(T)) Pair {
    T a, b;
};

// One product's layout (ResLayout) on the device.
template <typename T>
struct ResDir {
    int shorts, longs, pieces;
    const int2* head;         // piece slices, then short slices: first pair, pairs
    const ResRec<T>* rec;     // lanes of the short slices, then of the long slices
    const uint32_t* pword;    // lanes of the piece slices
    const Pair<T>* va;        // [pair][32]
    const uint32_t* ci;       // the same: two 16-bit places
    const int4* lhead;        // long slices
    const int* np;            // their lanes' pieces
    const uint32_t* flag;
};

template <typename T>
struct ResPart {
    int ld, ncol, ce, uni;
    T *Xbar, *Y, *Xh, *DX, *Yh, *DY, *DYp;
    const T *X0, *Y0;
    const T* hal;
    ColParams<T> col;
    ResDir<T> p, d;  // rows of A~^T and of A~
};

template <typename T>
struct ResArgs {
    int nparts, L;
    int tile0[kMaxParts + 1];  // part p has blocks [tile0[p], tile0[p + 1]), a tile of columns each
    ResPart<T> part[kMaxParts];
};
static_assert(sizeof(ResArgs<double>) <= 4096, "resident kernel arguments exceed 4 KB");

template <typename T, int C>
struct alignas(sizeof(T) * C) Pk {
    T v[C];
};

__host__ __device__ inline int up16(int v) { return (v + 15) / 16 * 16; }

// acc += U pairs of one lane's entries, in order, against the resident block
// src
template <typename T, int C, int U>
__device__ __forceinline__ void res_pairs(const Pair<T>* __restrict__ va, const uint32_t* __restrict__ ci,
                                          const T* src, T (&acc)[C]) {
    Pair<T> b[U];
    Pk<T, C> x[U], y[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
        const uint32_t c = __ldg(ci + j * 32);
        b[j] = va[j * 32];
        x[j] = *reinterpret_cast<const Pk<T, C>*>(src + (c & 0xffffu) * C);
        y[j] = *reinterpret_cast<const Pk<T, C>*>(src + (c >> 16) * C);
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
#pragma unroll
        for (int v = 0; v < C; ++v) acc[v] = dot_acc(b[j].a, x[j].v[v], acc[v]);
#pragma unroll
        for (int v = 0; v < C; ++v) acc[v] = dot_acc(b[j].b, y[j].v[v], acc[v]);
    }
}
// the pairs of a slice: every lane runs as many; past its own entries it has
// a factor 0 and the place of its first entry
template <typename T, int C>
__device__ __forceinline__ void res_sum(const Pair<T>* __restrict__ va, const uint32_t* __restrict__ ci, int pairs,
                                        const T* src, T (&acc)[C]) {
#pragma unroll 1
    for (; pairs >= 4; pairs -= 4, va += 128, ci += 128) res_pairs<T, C, 4>(va, ci, src, acc);
    if (pairs >= 2) {
        res_pairs<T, C, 2>(va, ci, src, acc);
        pairs -= 2;
        va += 64;
        ci += 64;
    }
    if (pairs > 0) res_pairs<T, C, 1>(va, ci, src, acc);
}

// the sum of a long row from its pieces' partial sums (32 to a slot): the
// pieces of each segment in order, then the segments in order
template <typename T, int C>
__device__ __forceinline__ void res_long_sum(const T* part, const uint32_t* __restrict__ flag, int np, int lane,
                                             T (&acc)[C]) {
    Pk<T, C> s = *reinterpret_cast<const Pk<T, C>*>(part);
    bool first = true;
#pragma unroll 4
    for (int t = 1; t < np; ++t) {
        const Pk<T, C> p = *reinterpret_cast<const Pk<T, C>*>(part + t * 32 * C);
        if (__ldg(flag + t) >> lane & 1u) {
#pragma unroll
            for (int v = 0; v < C; ++v) {
                acc[v] = first ? s.v[v] : add(acc[v], s.v[v]);
                s.v[v] = p.v[v];
            }
            first = false;
        } else {
#pragma unroll
            for (int v = 0; v < C; ++v) s.v[v] += p.v[v];
        }
    }
#pragma unroll
    for (int v = 0; v < C; ++v) acc[v] = first ? s.v[v] : add(acc[v], s.v[v]);
}

// One product over all rows: begin(place) ahead of a row's sum, for what does
// not depend on it, then finish(record, place, sum).
template <typename T, int C, typename B, typename F>
__device__ __forceinline__ void res_rows(const ResDir<T>& d, const T* src, T* sP, B begin, F finish) {
    using Pack = Pk<T, C>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (d.pieces > 0) {
#pragma unroll 1
        for (int s = warp; s < d.pieces; s += nw) {
            const int2 h = __ldg(d.head + s);
            const uint32_t w = __ldg(d.pword + s * 32 + lane);
            T acc[C];
#pragma unroll
            for (int v = 0; v < C; ++v) acc[v] = T(0);
            res_sum<T, C>(d.va + (size_t)h.x * 32 + lane, d.ci + (size_t)h.x * 32 + lane, h.y, src, acc);
            fin<C>(acc);
            if (w != kResIdle) {
                Pack q;
#pragma unroll
                for (int v = 0; v < C; ++v) q.v[v] = acc[v];
                *reinterpret_cast<Pack*>(sP + w * C) = q;
            }
        }
        __syncthreads();
    }
#pragma unroll 1
    for (int s = warp; s < d.longs + d.shorts; s += nw) {
        const bool is_long = s < d.longs;
        const int place = 32 * (is_long ? d.shorts + s : s - d.longs) + lane;
        const ResRec<T> r = d.rec[place];
        T acc[C];
        const bool mine = (r.word & 0xffffu) != kResIdle;
        auto early = begin(place);
        if (is_long) {
            const int4 h = __ldg(d.lhead + s);
            if (mine) res_long_sum<T, C>(sP + (h.y * 32 + lane) * C, d.flag + h.z, __ldg(d.np + s * 32 + lane), lane, acc);
        } else {
            const int2 h = __ldg(d.head + d.pieces + s - d.longs);
#pragma unroll
            for (int v = 0; v < C; ++v) acc[v] = T(0);
            res_sum<T, C>(d.va + (size_t)h.x * 32 + lane, d.ci + (size_t)h.x * 32 + lane, h.y, src, acc);
            fin<C>(acc);
            if (r.word & kResEmpty)
#pragma unroll
                for (int v = 0; v < C; ++v) acc[v] = T(0);
        }
        if (mine) finish(r, place, early, acc);
    }
}

// The block's part and its columns' parameters, in shared memory: held in
// registers over the interval, their pointers would spill.
template <typename T, int C>
struct ResTile {
    ResPart<T> a;
    T tau[C], sigma[C], isigma[C], lo[C], hi[C], c[C];
    int kind[C], var[C], hal[C];  // hal: the column's row of the weight table, -1 past the last column
};
static_assert(sizeof(ResTile<dfloat, 2>) <= kResStatic && sizeof(ResTile<float, 4>) <= kResStatic, "tile parameters");

template <typename T, int C, bool CHECK>
__device__ __forceinline__ void res_primal(const ResTile<T, C>& P, T* sX, const T* sX0, const T* sY, T* sP, int col0,
                                           int t) {
    using Pack = Pk<T, C>;
    const ResDir<T> d = P.a.p;
    T pa[C], pb[C], tau[C];
    int var[C];
    bool obj[C];
#pragma unroll
    for (int v = 0; v < C; ++v) {
        const int h = P.hal[v];
        pa[v] = h >= 0 ? ldg1(P.a.hal + h + 2 * t) : T(0);
        pb[v] = h >= 0 ? ldg1(P.a.hal + h + 2 * t + 1) : T(0);
        tau[v] = P.tau[v];
        var[v] = P.var[v];
        obj[v] = P.kind[v] == 2;
    }
    res_rows<T, C>(
        d, sY, sP,
        [&](int place) {
            const Pack xb = *reinterpret_cast<const Pack*>(sX + place * C);
            const Pack x0 = *reinterpret_cast<const Pack*>(sX0 + place * C);
            Pack x;
#pragma unroll
            for (int v = 0; v < C; ++v) x.v[v] = primal_iterate(pa[v], pb[v], xb.v[v], x0.v[v]);
            return x;
        },
        [&](const ResRec<T>& r, int place, const Pack& x, const T(&acc)[C]) {
            const int row = (int)(r.word & 0xffffu);
            Pack xh, xb, dz;
#pragma unroll
            for (int v = 0; v < C; ++v) {
                T cj = obj[v] ? T(0) : r.c, lo = r.lo, hi = r.hi;
                if (var[v] == row) {
                    if (obj[v]) {
                        cj = P.c[v];
                    } else {
                        lo = P.lo[v];
                        hi = P.hi[v];
                    }
                }
                primal_element<T, CHECK>(x.v[v], acc[v], tau[v], cj, lo, hi, xh.v[v], xb.v[v], dz.v[v]);
            }
            *reinterpret_cast<Pack*>(sX + place * C) = xb;
            if (CHECK) {
                const size_t at = (size_t)row * P.a.ld + col0;
                *reinterpret_cast<Pack*>(P.a.Xbar + at) = xb;
                *reinterpret_cast<Pack*>(P.a.Xh + at) = xh;
                *reinterpret_cast<Pack*>(P.a.DX + at) = dz;
            }
        });
}

template <typename T, int C>
struct Dual {
    Pk<T, C> y, ys, y0;
};

template <typename T, int C, bool CHECK>
__device__ __forceinline__ void res_dual(const ResTile<T, C>& P, const T* sX, T* sY, const T* sY0, T* sP, int col0,
                                         int t) {
    using Pack = Pk<T, C>;
    const ResDir<T> d = P.a.d;
    T ca[C], cb[C], sg[C], isg[C];
#pragma unroll
    for (int v = 0; v < C; ++v) {
        const int h = P.hal[v];
        ca[v] = h >= 0 ? ldg1(P.a.hal + h + 2 * t + 2) : T(0);
        cb[v] = h >= 0 ? ldg1(P.a.hal + h + 2 * t + 3) : T(0);
        sg[v] = P.sigma[v];
        isg[v] = P.isigma[v];
    }
    res_rows<T, C>(
        d, sX, sP,
        [&](int place) {
            Dual<T, C> e;
            e.y = *reinterpret_cast<const Pack*>(sY + place * C);
            e.y0 = *reinterpret_cast<const Pack*>(sY0 + place * C);
#pragma unroll
            for (int v = 0; v < C; ++v) e.ys.v[v] = over_sigma(e.y.v[v], sg[v], isg[v]);
            return e;
        },
        [&](const ResRec<T>& r, int place, const Dual<T, C>& e, const T(&acc)[C]) {
            Pack yh, yn, dz;
#pragma unroll
            for (int v = 0; v < C; ++v)
                dual_element(ca[v], cb[v], e.y.v[v], e.ys.v[v], e.y0.v[v], acc[v], sg[v], r.lo, r.hi, yh.v[v],
                             yn.v[v], dz.v[v]);
            if (!CHECK) {
                *reinterpret_cast<Pack*>(sY + place * C) = yn;
            } else {
                const size_t at = (size_t)(r.word & 0xffffu) * P.a.ld + col0;
                Pack dzp;
#pragma unroll
                for (int v = 0; v < C; ++v) dzp.v[v] = barrier(dz.v[v], r.lo, r.hi);
                *reinterpret_cast<Pack*>(P.a.Y + at) = yn;
                *reinterpret_cast<Pack*>(P.a.Yh + at) = yh;
                *reinterpret_cast<Pack*>(P.a.DY + at) = dz;
                *reinterpret_cast<Pack*>(P.a.DYp + at) = dzp;
            }
        });
}

template <typename T, int C>
__global__ void __launch_bounds__(kResThreads, 1) k_resident(const __grid_constant__ ResArgs<T> g) {
    extern __shared__ __align__(16) char res_smem[];
    __shared__ ResTile<T, C> P;
    using Pack = Pk<T, C>;
    int pi = 0;
    while (pi + 1 < g.nparts && (int)blockIdx.x >= g.tile0[pi + 1]) ++pi;
    const int col0 = ((int)blockIdx.x - g.tile0[pi]) * C, tid = threadIdx.x, nt = blockDim.x;
    const ResPart<T>& a = g.part[pi];
    if (tid == 0) P.a = a;
    if (tid < C) {
        const int j = col0 + tid;
        const bool in = j < a.ncol;
        P.kind[tid] = in ? a.col.kind[j] : 0;
        P.var[tid] = P.kind[tid] != 0 ? a.col.var[j] : -1;
        P.tau[tid] = in ? a.col.tau[j] : T(0);
        P.lo[tid] = in ? a.col.lo[j] : T(0);
        P.hi[tid] = in ? a.col.hi[j] : T(0);
        P.c[tid] = in ? a.col.c[j] : T(0);
        P.sigma[tid] = in ? a.col.sigma[j] : T(1);
        P.isigma[tid] = std::is_same<T, dfloat>::value ? T(1) / P.sigma[tid] : T(0);
        P.hal[tid] = in ? 2 * ((a.uni >= 0 ? a.uni : a.col.grp[j]) * (a.ce + 1)) : -1;
    }
    // shared memory: the two gathered blocks and their anchors, by place, and
    // the long rows' partial sums
    const int np = 32 * (a.p.shorts + a.p.longs), nd = 32 * (a.d.shorts + a.d.longs);
    T* sX = reinterpret_cast<T*>(res_smem);
    T* sX0 = sX + np * C;
    T* sY = sX0 + np * C;
    T* sY0 = sY + nd * C;
    T* sP = sY0 + nd * C;
    for (int i = tid; i < np + nd; i += nt) {
        const bool dual = i >= np;
        const int place = dual ? i - np : i;
        const uint32_t row = (dual ? a.d.rec : a.p.rec)[place].word & 0xffffu;
        if (row == kResIdle) continue;
        const size_t at = (size_t)row * a.ld + col0;
        *reinterpret_cast<Pack*>((dual ? sY : sX) + place * C) = *reinterpret_cast<const Pack*>((dual ? a.Y : a.Xbar) + at);
        *reinterpret_cast<Pack*>((dual ? sY0 : sX0) + place * C) = *reinterpret_cast<const Pack*>((dual ? a.Y0 : a.X0) + at);
    }
    __syncthreads();
#pragma unroll 1
    for (int t = 0; t + 1 < g.L; ++t) {
        res_primal<T, C, false>(P, sX, sX0, sY, sP, col0, t);
        __syncthreads();
        res_dual<T, C, false>(P, sX, sY, sY0, sP, col0, t);
        __syncthreads();
    }
    res_primal<T, C, true>(P, sX, sX0, sY, sP, col0, g.L - 1);
    __syncthreads();
    res_dual<T, C, true>(P, sX, sY, sY0, sP, col0, g.L - 1);
}

// The records and entries of a layout, from the CSR matrix and the vectors by
// row; pos gives a column's place.  Thread i takes a lane of the short slices,
// then of the piece slices, then of the long slices.
template <typename T>
__global__ void k_res_fill(ResDir<T> d, ResRec<T>* rec, Pair<T>* ova, uint32_t* oci, const uint32_t* __restrict__ word,
                           const int* __restrict__ beg, const int* __restrict__ len, const int* __restrict__ pos,
                           const int* __restrict__ ci, const T* __restrict__ va, const T* __restrict__ rlo,
                           const T* __restrict__ rhi, const T* __restrict__ rc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, ns = 32 * d.shorts, np = 32 * d.pieces, nl = 32 * d.longs;
    if (i >= ns + np + nl) return;
    if (i < ns || i >= ns + np) {
        const int place = i < ns ? i : i - np;
        const uint32_t w = word[place], row = w & 0xffffu;
        ResRec<T> r;
        r.lo = row != kResIdle ? rlo[row] : T(0);
        r.hi = row != kResIdle ? rhi[row] : T(0);
        r.c = row != kResIdle && rc ? rc[row] : T(0);
        r.word = w;
        rec[place] = r;
        if (i >= ns) return;
    }
    const int2 h = d.head[i < ns ? d.pieces + i / 32 : (i - ns) / 32];
    const int b = beg[i], n = len[i];
    for (int k = 0; k < h.y; ++k) {
        const size_t at = ((size_t)h.x + k) * 32 + i % 32;
        const uint32_t first = n > 0 ? (uint32_t)pos[ci[b]] : 0u;
        const uint32_t c0 = 2 * k < n ? (uint32_t)pos[ci[b + 2 * k]] : first;
        const uint32_t c1 = 2 * k + 1 < n ? (uint32_t)pos[ci[b + 2 * k + 1]] : first;
        oci[at] = c0 | c1 << 16;
        ova[at] = Pair<T>{2 * k < n ? va[b + 2 * k] : T(0), 2 * k + 1 < n ? va[b + 2 * k + 1] : T(0)};
    }
}

}  // namespace

// A matrix's two layouts for one iterate type and set of row-group widths and
// thresholds.  Measured on the host first (measure); on the device only once
// an interval is to run from them (res_build).
struct ResPlan {
    int prec = -1, lanes_p = 0, lanes_d = 0, thr_p = 0, thr_d = 0;
    bool fits = false;   // the matrix has the layouts, and no allocation for them has failed
    int places = 0;      // rows of both products, idle lanes among them
    int slots = 0;       // partial sums (32 to a slot) of the product with more
    int slices = 0;      // slices of the longest phase
    long long pairs = 0; // of a lane, both products
    std::unique_ptr<ResLayout[]> lay;  // until they are on the device
    void* mem = nullptr;               // both layouts and what they were filled from, one allocation
    int64_t charged = 0;               // bytes of it on a server's account
    ResDir<double> dir[2];             // pointers; the value type follows prec
    // (rp: the row pointers of A~^T, then of A~); false: no such layouts
    bool measure(const std::vector<int>* rp, long long max_pairs) {
        const int thr[2] = {thr_p, thr_d}, lanes[2] = {lanes_p, lanes_d};
        lay.reset(new ResLayout[2]);
        places = slots = slices = 0;
        pairs = 0;
        for (int q = 0; q < 2; ++q) {
            ResLayout& l = lay[q];
            if (!res_layout((int)rp[q].size() - 1, rp[q].data(), thr[q], kStepSeg, kBlock / lanes[q], max_pairs, l)) {
                lay.reset();
                return false;
            }
            places += l.places();
            slots = std::max(slots, l.slots);
            slices = std::max(slices, std::max(l.pieces, l.shorts + l.longs));
            pairs += l.total_pairs;
        }
        return true;
    }
};

namespace {

// the pieces of one allocation, each from a multiple of 256 bytes on
struct Carve {
    size_t bytes = 0;
    size_t take(size_t size) {
        const size_t at = bytes;
        bytes += (size + 255) / 256 * 256;
        return at;
    }
};

// where the arrays of a plan's two layouts lie in its allocation: those that
// the host fills, then those that k_res_fill does
struct ResPlaces {
    struct {
        size_t head, pword, lhead, np, flag, word, beg, len, pos, rec, va, ci;
    } at[2];
    size_t upload = 0, bytes = 0;
};
template <typename T>
ResPlaces res_places(const ResPlan* plan) {
    ResPlaces p;
    Carve c;
    for (int q = 0; q < 2; ++q) {
        const ResLayout& l = plan->lay[q];
        p.at[q].head = c.take(l.head.size() * sizeof(int2));
        p.at[q].lhead = c.take(l.lhead.size() * sizeof(int4));
        p.at[q].np = c.take(l.np.size() * 4);
        p.at[q].flag = c.take(l.flag.size() * 4);
        p.at[q].word = c.take(l.word.size() * 4);
        p.at[q].pword = p.at[q].word + 4 * (size_t)l.places();  // the words of the piece slices are the last
        p.at[q].beg = c.take(l.beg.size() * 4);
        p.at[q].len = c.take(l.len.size() * 4);
        p.at[q].pos = c.take(l.pos.size() * 4);
    }
    p.upload = c.bytes;
    for (int q = 0; q < 2; ++q) {
        const ResLayout& l = plan->lay[q];
        p.at[q].rec = c.take((size_t)l.places() * sizeof(ResRec<T>));
        p.at[q].va = c.take(32 * (size_t)l.total_pairs * sizeof(Pair<T>));
        p.at[q].ci = c.take(32 * (size_t)l.total_pairs * 4);
    }
    p.bytes = c.bytes;
    return p;
}

// The measured layouts on the device.  The allocation is stream-ordered and
// the only wait is for the handle's own stream: cudaMalloc and cudaFree wait
// for the whole device, and a server runs other matrices' intervals meanwhile.
template <typename T>
cudaError_t res_build(lpb_ctx* h, ResPlan* plan, const ResPlaces& places) {
    cudaStream_t s = h->stream;
    const IterData<T> it = lane_iter_data<T>(h, h->lane[0]);  // matrix and vectors only
    const Csr* csr[2] = {&h->At, &h->A};
    const auto& at = places.at;
    std::vector<char> host(places.upload);
    auto put = [&](size_t to, const void* from, size_t bytes) {
        if (bytes) std::memcpy(host.data() + to, from, bytes);
    };
    for (int q = 0; q < 2; ++q) {
        const ResLayout& l = plan->lay[q];
        std::vector<int4> lh;
        for (const auto& x : l.lhead) lh.push_back(make_int4(x.pieces, x.slot0, x.flag0, 0));
        put(at[q].head, l.head.data(), l.head.size() * sizeof(int2));
        put(at[q].lhead, lh.data(), lh.size() * sizeof(int4));
        put(at[q].np, l.np.data(), l.np.size() * 4);
        put(at[q].flag, l.flag.data(), l.flag.size() * 4);
        put(at[q].word, l.word.data(), l.word.size() * 4);
        put(at[q].beg, l.beg.data(), l.beg.size() * 4);
        put(at[q].len, l.len.data(), l.len.size() * 4);
        put(at[q].pos, l.pos.data(), l.pos.size() * 4);
    }
    cudaError_t e;
    if ((e = cudaMallocAsync(&plan->mem, places.bytes, s)) != cudaSuccess) return e;
    char* mem = (char*)plan->mem;
    if ((e = cudaMemcpyAsync(mem, host.data(), places.upload, cudaMemcpyHostToDevice, s)) != cudaSuccess) return e;
    for (int q = 0; q < 2; ++q) {
        const ResLayout& l = plan->lay[q];
        const auto& p = at[q];
        ResDir<T> d{};
        d.shorts = l.shorts;
        d.longs = l.longs;
        d.pieces = l.pieces;
        d.head = (const int2*)(mem + p.head);
        d.rec = (const ResRec<T>*)(mem + p.rec);
        d.pword = (const uint32_t*)(mem + p.pword);
        d.va = (const Pair<T>*)(mem + p.va);
        d.ci = (const uint32_t*)(mem + p.ci);
        d.lhead = (const int4*)(mem + p.lhead);
        d.np = (const int*)(mem + p.np);
        d.flag = (const uint32_t*)(mem + p.flag);
        const int all = 32 * (l.shorts + l.longs + l.pieces);
        k_res_fill<T><<<(all + 127) / 128, 128, 0, s>>>(
            d, (ResRec<T>*)d.rec, (Pair<T>*)d.va, (uint32_t*)d.ci, (const uint32_t*)(mem + p.word),
            (const int*)(mem + p.beg), (const int*)(mem + p.len), (const int*)(mem + at[1 - q].pos), csr[q]->ci,
            q == 0 ? it.at_vals : it.a_vals, q == 0 ? it.xl : it.l, q == 0 ? it.xu : it.u, q == 0 ? it.c : nullptr);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        std::memcpy((void*)&plan->dir[q], (const void*)&d, sizeof(d));
    }
    // the host's copy goes, and other streams run from the layouts
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    plan->lay.reset();
    return cudaSuccess;
}
static_assert(sizeof(ResDir<float>) == sizeof(ResDir<double>) && sizeof(ResDir<dfloat>) == sizeof(ResDir<double>),
              "pointers and counts only");

template <typename T>
ResDir<T> typed(const ResDir<double>& d) {
    ResDir<T> r;
    std::memcpy((void*)&r, (const void*)&d, sizeof(r));
    return r;
}

// SM count and the most dynamic shared memory of a block on the device
cudaError_t res_limits(int* sms, int* smem) {
    static std::atomic<int> cache[kShapeDevices][2];  // static storage: starts at 0
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool in = dev >= 0 && dev < kShapeDevices;
    *sms = in ? cache[dev][0].load(std::memory_order_acquire) : 0;
    *smem = in ? cache[dev][1].load(std::memory_order_acquire) : 0;
    if (*sms > 0 && *smem > 0) return cudaSuccess;
    if ((e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
    if (in) {
        cache[dev][0].store(*sms, std::memory_order_release);
        cache[dev][1].store(*smem, std::memory_order_release);
    }
    return cudaSuccess;
}

template <typename T, int C>
cudaError_t res_launch(const ResArgs<T>& g, int threads, size_t smem, cudaStream_t s) {
    static std::atomic<int> set[kShapeDevices];
    int dev = 0, sms = 0, most = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kShapeDevices || !set[dev].load(std::memory_order_acquire)) {
        if ((e = res_limits(&sms, &most)) != cudaSuccess) return e;
        e = cudaFuncSetAttribute(k_resident<T, C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 most - kResStatic);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < kShapeDevices) set[dev].store(1, std::memory_order_release);
    }
    k_resident<T, C><<<g.tile0[g.nparts], threads, smem, s>>>(g);
    return cudaGetLastError();
}

}  // namespace

void set_res_account(lpb_ctx* h, std::function<bool(int64_t)> account) {
    h->res_charge = std::move(account);
    for (ResPlan* p : h->res_plans) p->charged = 0;
}

void free_res_plans(lpb_ctx* h, bool keep_stream) {
    if (!h->res_plans.empty()) h->ws_epoch += 1;  // captured intervals hold them
    for (ResPlan* p : h->res_plans) {
        if (p->mem) keep_stream ? cudaFreeAsync(p->mem, h->stream) : cudaFree(p->mem);
        if (p->charged > 0 && h->res_charge) h->res_charge(-p->charged);
        delete p;
    }
    h->res_plans.clear();
}

namespace {

// Estimated microseconds of an iteration: of the resident kernel for a layout
// of `pairs` (of a lane, both products) and C columns a block, and of the step
// kernels for the same matrix at ncol columns.  Fitted on GB300 at 2070 MHz
// over matrices of 200 to 2750 rows and 1 to 900 LPs; the constants are where
// each bound lies:
//   resident, FP32: a pair of entries per lane takes the block 7 ns (issue,
//   bank conflicts of the gathers), 14 ns once the entries exceed what L1
//   holds beside the resident blocks (550 pairs, 210 KB); FP64 and
//   double-float wait on their pipe.  Long rows in batches of one or two
//   lanes are many short pieces, added one after another.
//   steps: about 2 us a launch and its chain of round trips, 1 us more each
//   where rows are cut into segments, then L2 traffic.
// 16 FP64 LPs on 200 x 400 (pairs 75): 4.1 us against 7.4; 37 LPs on a 1k x
// 2k power-law matrix (pairs 500): 4.6 against 7.2; 24 LPs on 2k x 2k with 10
// entries a row (pairs 720): 5.7 against 4.6, the step kernels'.
template <typename T>
double res_us(long long pairs, bool longs, int lanes, int C) {
    const bool f32 = std::is_same<T, float>::value, f64 = std::is_same<T, double>::value;
    const double in = (double)std::min<long long>(pairs, 550), out = (double)pairs - in;
    double us = 0.6 + (f64 ? 0.045 * pairs : f32 ? 0.0068 * in + 0.0145 * out : 0.02 * pairs);
    if (longs && lanes < 4) us += 0.0105 * pairs;
    return us * (C == 1 ? 1.0 : C == 2 ? 1.4 : 2.3);
}
template <typename T>
double step_us(long long pairs, bool longs, int ncol) {
    const bool f64 = std::is_same<T, double>::value;
    return (f64 ? 6.3 : 4.3 + (longs ? 2.0 : 0.0)) + (f64 ? 2.5e-4 : 5.2e-5) * (double)pairs * ncol;
}

// The handle's layouts for iterate type T (of lane precision prec) at a batch
// width, measured when they are not yet; null when the matrix has none of at
// most max_pairs, or no memory was left for them.
template <typename T>
lpb_err res_plan(lpb_ctx* h, int prec, int ncol, long long max_pairs, ResPlan** out) {
    *out = nullptr;
    // the width decides how long rows are cut; without long rows it does not matter
    const int lp = h->At.n_long > 0 ? row_group_lanes<T>(ncol, h->At.g_shift) : 32;
    const int ld = h->A.n_long > 0 ? row_group_lanes<T>(ncol, h->A.g_shift) : 32;
    for (ResPlan* q : h->res_plans)
        if (q->prec == prec && q->lanes_p == lp && q->lanes_d == ld && q->thr_p == h->At.long_thr &&
            q->thr_d == h->A.long_thr) {
            if (q->fits) *out = q;
            return LPB_OK;
        }
    const Csr* csr[2] = {&h->At, &h->A};
    for (int q = 0; q < 2; ++q)
        if (h->rp_host[q].empty()) {
            std::vector<int> rp((size_t)csr[q]->rows + 1);
            LPB_CU(cudaMemcpyAsync(rp.data(), csr[q]->rp, sizeof(int) * rp.size(), cudaMemcpyDeviceToHost, h->stream));
            LPB_CU(cudaStreamSynchronize(h->stream));
            h->rp_host[q].swap(rp);
        }
    std::unique_ptr<ResPlan> p(new ResPlan());
    p->prec = prec;
    p->lanes_p = lp;
    p->lanes_d = ld;
    p->thr_p = h->At.long_thr;
    p->thr_d = h->A.long_thr;
    p->fits = p->measure(h->rp_host, max_pairs);
    h->res_plans.reserve(h->res_plans.size() + 1);
    if (p->fits) *out = p.get();
    h->res_plans.push_back(p.release());
    return LPB_OK;
}

// A measured plan's layouts on the device, if they are not there yet; *ok =
// false when no memory is left for them, or a server has none to give just
// now.  The step kernels need none and give the same results, so that is no
// error of the solve.
template <typename T>
lpb_err res_ready(lpb_ctx* h, ResPlan* p, long long max_pairs, bool* ok) {
    *ok = true;
    if (p->mem) return LPB_OK;
    cudaError_t e = cudaErrorMemoryAllocation;
    try {
        if (p->lay || p->measure(h->rp_host, max_pairs)) {
            const ResPlaces places = res_places<T>(p);
            if (h->res_charge) {
                if (!h->res_charge((int64_t)places.bytes)) {
                    *ok = false;
                    return LPB_OK;
                }
                p->charged = (int64_t)places.bytes;
            }
            e = res_build<T>(h, p, places);
        }
    } catch (const std::bad_alloc&) {
    }
    if (e == cudaSuccess) return LPB_OK;
    if (p->charged > 0) h->res_charge(-p->charged);
    p->charged = 0;
    *ok = false;
    cudaStreamSynchronize(h->stream);
    if (p->mem) cudaFreeAsync(p->mem, h->stream);
    p->mem = nullptr;
    if (e != cudaErrorMemoryAllocation) return cuda_fail(e, "layout of the resident kernel");
    p->fits = false;
    p->lay.reset();
    cudaGetLastError();  // the next launch's error is its own
    return LPB_OK;
}

}  // namespace

template <typename T>
lpb_err res_choose(lpb_ctx* const* hs, Lane* const* lns, int count, ResShape* shape, ResPlan** plans) {
    *shape = ResShape{};
    if (count > kMaxParts) return LPB_OK;
    int sms = 0, most = 0;
    LPB_CU(res_limits(&sms, &most));
    const int ts = (int)sizeof(T);
    // the fewest columns a block with which the tiles are one wave
    int C = 0;
    long long tiles = 0;
    for (int c = 1; c * ts <= 16 && C == 0; c *= 2) {
        tiles = 0;
        for (int i = 0; i < count; ++i) tiles += (lns[i]->ncol + c - 1) / c;
        if (tiles <= sms) C = c;
    }
    if (C == 0) return LPB_OK;
    // more pairs than the slowest step would be worth are not laid out
    constexpr long long kMostPairs = 1000;
    const long long limit = most - kResStatic;
    for (int i = 0; i < count; ++i) {
        const lpb_ctx* h = hs[i];
        if (h->m == 0 || h->nnz == 0 || lns[i]->ncol == 0) return LPB_OK;
        if (2 * ((long long)h->m + h->n) * ts * C > limit || h->nnz > 32 * kMostPairs) return LPB_OK;
    }
    int slices = 1;
    long long smem = 0;
    double us_res = 0.0, us_step = 0.0, fixed_us = 0.0;
    for (int i = 0; i < count; ++i) {
        lpb_ctx* h = hs[i];
        ResPlan* p = nullptr;
        lpb_err rc = LPB_OK;
        try {
            rc = res_plan<T>(h, lns[i]->prec, lns[i]->ncol, kMostPairs, &p);
        } catch (const std::bad_alloc&) {
        }
        if (rc != LPB_OK) return rc;
        if (!p) return LPB_OK;
        plans[i] = p;
        const bool longs = h->A.n_long > 0 || h->At.n_long > 0;
        slices = std::max(slices, p->slices);
        smem = std::max(smem, (2LL * p->places + 32LL * p->slots) * ts * C);
        us_res = std::max(us_res, res_us<T>(p->pairs, longs, std::min(p->lanes_p, p->lanes_d), C));
        // (a joint step's launches overlap their parts' chains, not their traffic)
        const double fixed = step_us<T>(0, longs, 0);
        us_step += step_us<T>(p->pairs, longs, lns[i]->ncol) - fixed;
        fixed_us = std::max(fixed_us, fixed);
    }
    if (smem > limit || us_res > 0.92 * (us_step + fixed_us)) {
        for (int i = 0; i < count; ++i) plans[i]->lay.reset();  // (measured again should another width want it)
        return LPB_OK;
    }
    for (int i = 0; i < count; ++i) {
        bool ok = false;
        const lpb_err rc = res_ready<T>(hs[i], plans[i], kMostPairs, &ok);
        if (rc != LPB_OK || !ok) return rc;
    }
    shape->C = C;
    shape->threads = std::min(kResThreads, std::max(64, slices * 32));
    shape->smem = (size_t)smem;
    return LPB_OK;
}

template <typename T>
cudaError_t launch_resident(const IterPart<T>* parts, ResPlan* const* plans, int count, int L, const ResShape& shape,
                            cudaStream_t s) {
    ResArgs<T> g{};
    g.nparts = count;
    g.L = L;
    int tiles = 0;
    for (int i = 0; i < count; ++i) {
        const IterPart<T>& q = parts[i];
        g.tile0[i] = tiles;
        tiles += (q.ncol + shape.C - 1) / shape.C;
        ResPart<T>& a = g.part[i];
        a.ld = q.ld;
        a.ncol = q.ncol;
        a.ce = q.ce;
        a.uni = q.uni;
        a.Xbar = q.b.Xbar;
        a.Y = q.b.Y;
        a.Xh = q.b.Xh;
        a.DX = q.b.DX;
        a.Yh = q.b.Yh;
        a.DY = q.b.DY;
        a.DYp = q.b.DYp;
        a.X0 = q.b.X0;
        a.Y0 = q.b.Y0;
        a.hal = q.hal;
        a.col = q.d.col;
        a.p = typed<T>(plans[i]->dir[0]);
        a.d = typed<T>(plans[i]->dir[1]);
    }
    g.tile0[count] = tiles;
    if constexpr (std::is_same<T, float>::value) {
        if (shape.C == 4) return res_launch<T, 4>(g, shape.threads, shape.smem, s);
    }
    if (shape.C == 2) return res_launch<T, 2>(g, shape.threads, shape.smem, s);
    return res_launch<T, 1>(g, shape.threads, shape.smem, s);
}

#define LPB_RES_INSTANTIATE(T)                                                                                \
    template lpb_err res_choose<T>(lpb_ctx* const*, Lane* const*, int, ResShape*, ResPlan**);                 \
    template cudaError_t launch_resident<T>(const IterPart<T>*, ResPlan* const*, int, int, const ResShape&, \
                                            cudaStream_t);
LPB_RES_INSTANTIATE(float)
LPB_RES_INSTANTIATE(double)
LPB_RES_INSTANTIATE(dfloat)

}  // namespace lpb
