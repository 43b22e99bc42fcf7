// lpb_step.h -- device code of the step kernels (the fused CSR SpMM with
// its primal or dual epilogue, described in lpb_iter.cu) and the host
// helpers that shape their launches, shared by the launches of one matrix
// (lpb_iter.cu) and the joint launches over several matrices (lpb_multi.cu).
#pragma once

#include <atomic>
#include <climits>
#include <type_traits>

#include "lpb_internal.h"

// Resident blocks per SM the step kernels are compiled for (register caps
// without spills; a spilled byte goes through the same L1 as the gathers, and
// a few of them per row cost more than a block less).  FP32: the row groups
// of 32 lanes wait on HBM and gain from every block (10 at 48 registers; on
// the 1M-row matrix 8 blocks took 140 ms a pass, 10 took 138 ms); the
// narrower ones run from L2 (8).  Double-float and FP64 hold wider sums.
#ifndef LPB_STEP_MIN_BLOCKS_WIDE
#define LPB_STEP_MIN_BLOCKS_WIDE 10
#endif
#ifndef LPB_STEP_MIN_BLOCKS
#define LPB_STEP_MIN_BLOCKS 8
#endif
#ifndef LPB_STEP_MIN_BLOCKS_F64
#define LPB_STEP_MIN_BLOCKS_F64 5
#endif
#ifndef LPB_STEP_MIN_BLOCKS_DF
#define LPB_STEP_MIN_BLOCKS_DF 7
#endif
// the same for the deep kernels (kDeep), whose grids are less than a wave
#ifndef LPB_STEP_MIN_BLOCKS_DEEP
#define LPB_STEP_MIN_BLOCKS_DEEP 4
#endif

namespace lpb {

namespace {

template <typename T> struct Vec;
template <> struct Vec<float> { static constexpr int V = 4; };
template <> struct Vec<double> { static constexpr int V = 2; };
template <> struct Vec<dfloat> { static constexpr int V = 2; };

// Gathers a lane issues before it consumes them.  Four keep the registers low
// enough for the resident warps that fill the memory pipeline.  A step of
// fewer blocks than one wave has nothing but its rows' chains of round trips:
// its kernels are the deep ones, eight at a time (sixteen need so many
// registers that the next step's blocks find no room to start early: 4 LPs on
// 100k x 100k 6.6 ms a pass of 256 iterations, with eight 6.1).  Row groups of
// 32 lanes have no deep kernel: a step that wide and that small runs alone
// only for a few hundred rows.
template <int G> constexpr int kDeep = G >= 32 ? 0 : 8;
constexpr int kFlat = 4;

template <typename T, int G, int B> struct MinBlocks {
    static constexpr int v = B > kFlat                       ? LPB_STEP_MIN_BLOCKS_DEEP
                             : std::is_same<T, double>::value ? LPB_STEP_MIN_BLOCKS_F64
                             : std::is_same<T, dfloat>::value ? LPB_STEP_MIN_BLOCKS_DF
                             : G >= 32                        ? LPB_STEP_MIN_BLOCKS_WIDE
                                                              : LPB_STEP_MIN_BLOCKS;
};

__device__ __forceinline__ void ldv(const float* p, float (&r)[4]) {
    float4 u = *reinterpret_cast<const float4*>(p);
    r[0] = u.x; r[1] = u.y; r[2] = u.z; r[3] = u.w;
}
__device__ __forceinline__ void ldv(const double* p, double (&r)[2]) {
    double2 u = *reinterpret_cast<const double2*>(p);
    r[0] = u.x; r[1] = u.y;
}
__device__ __forceinline__ void ldg_v(const float* p, float (&r)[4]) {
    float4 u = __ldg(reinterpret_cast<const float4*>(p));
    r[0] = u.x; r[1] = u.y; r[2] = u.z; r[3] = u.w;
}
__device__ __forceinline__ void ldg_v(const double* p, double (&r)[2]) {
    double2 u = __ldg(reinterpret_cast<const double2*>(p));
    r[0] = u.x; r[1] = u.y;
}
__device__ __forceinline__ void stv(float* p, const float (&r)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(r[0], r[1], r[2], r[3]);
}
__device__ __forceinline__ void stv(double* p, const double (&r)[2]) {
    *reinterpret_cast<double2*>(p) = make_double2(r[0], r[1]);
}
__device__ __forceinline__ void ldv(const dfloat* p, dfloat (&r)[2]) {
    float4 u = *reinterpret_cast<const float4*>(p);
    r[0] = dfloat(u.x, u.y); r[1] = dfloat(u.z, u.w);
}
__device__ __forceinline__ void ldg_v(const dfloat* p, dfloat (&r)[2]) {
    float4 u = __ldg(reinterpret_cast<const float4*>(p));
    r[0] = dfloat(u.x, u.y); r[1] = dfloat(u.z, u.w);
}
__device__ __forceinline__ void stv(dfloat* p, const dfloat (&r)[2]) {
    *reinterpret_cast<float4*>(p) = make_float4(r[0].hi, r[0].lo, r[1].hi, r[1].lo);
}

// scalar read-only load, multiply-add and infinity test for each iterate type
__device__ __forceinline__ float ldg1(const float* p) { return __ldg(p); }
__device__ __forceinline__ double ldg1(const double* p) { return __ldg(p); }
__device__ __forceinline__ dfloat ldg1(const dfloat* p) {
    const float2 u = __ldg(reinterpret_cast<const float2*>(p));
    return dfloat(u.x, u.y);
}
__device__ __forceinline__ float mad(float a, float x, float acc) { return fmaf(a, x, acc); }
__device__ __forceinline__ double mad(double a, double x, double acc) { return fma(a, x, acc); }
// the SpMM's running sums: for dfloat the low part stays unnormalised until
// fin() (dfl_dot_acc), which shortens the dependent chain per nonzero
__device__ __forceinline__ dfloat mad(dfloat a, dfloat x, dfloat acc) { return dfl_fma(a, x, acc); }
__device__ __forceinline__ float dot_acc(float a, float x, float acc) { return fmaf(a, x, acc); }
__device__ __forceinline__ double dot_acc(double a, double x, double acc) { return fma(a, x, acc); }
__device__ __forceinline__ dfloat dot_acc(dfloat a, dfloat x, dfloat acc) { return dfl_dot_acc(a, x, acc); }
// a product and a difference, each rounded by itself (never joined into one
// multiply-add by the compiler)
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ dfloat mul(dfloat a, dfloat b) { return a * b; }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ dfloat sub(dfloat a, dfloat b) { return a - b; }
// x - tau q with one rounding in FP32 and FP64
__device__ __forceinline__ float step_from(float x, float tau, float q) { return fmaf(-tau, q, x); }
__device__ __forceinline__ double step_from(double x, double tau, double q) { return fma(-tau, q, x); }
__device__ __forceinline__ dfloat step_from(dfloat x, dfloat tau, dfloat q) { return x - tau * q; }
// ca v + cb w: the second product rounded, then one multiply-add
template <typename T>
__device__ __forceinline__ T blend(T ca, T v, T cb, T w) {
    return mad(ca, v, mul(cb, w));
}
__device__ __forceinline__ dfloat blend(dfloat ca, dfloat v, dfloat cb, dfloat w) { return ca * v + cb * w; }
// 2 v, exact in every iterate type (for dfloat both parts scale)
__device__ __forceinline__ float twice(float v) { return 2.0f * v; }
__device__ __forceinline__ double twice(double v) { return 2.0 * v; }
__device__ __forceinline__ dfloat twice(dfloat v) { return dfloat(2.0f * v.hi, 2.0f * v.lo); }
// y / sigma: FP32 and FP64 divide; dfloat multiplies by the column's
// reciprocal 1/sigma (staged once per block), which a double-float division
// would recompute per element at several times the cost
__device__ __forceinline__ float over_sigma(float y, float sg, float) { return y / sg; }
__device__ __forceinline__ double over_sigma(double y, double sg, double) { return y / sg; }
__device__ __forceinline__ dfloat over_sigma(dfloat y, dfloat, dfloat isg) { return y * isg; }
template <int V> __device__ __forceinline__ void fin(float (&)[V]) {}
template <int V> __device__ __forceinline__ void fin(double (&)[V]) {}
template <int V> __device__ __forceinline__ void fin(dfloat (&acc)[V]) {
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = dfl_norm(acc[v]);
}
__device__ __forceinline__ bool is_inf(float v) { return isinf(v); }
__device__ __forceinline__ bool is_inf(double v) { return isinf(v); }
__device__ __forceinline__ bool is_inf(dfloat v) { return isinf(v.hi); }

// A vector of the gathered block, row c.  The previous kernel of the interval
// writes that block, and may still be writing it when this one starts: plain
// loads, which no compiler moves ahead of the wait for that kernel (pdl_wait)
// and which see what it wrote.  Read-only loads (ld.global.nc) are neither held
// back by the wait nor defined for such data; the matrix, the records and the
// bounds, which no step writes, take those.  Plain loads cost nothing: with
// read-only ones and with these, a pass of 64 LPs on the 20k x 50k power-law
// matrix 6.25 and 6.21 ms, 1024 LPs on 100k x 100k 59.7 and 59.9, 128 LPs on
// 1M x 2M 125.1 and 124.9.
template <typename T, int V>
__device__ __forceinline__ void ld_iterate(const char* src, unsigned c, unsigned pitch, T (&r)[V]) {
    ldv(reinterpret_cast<const T*>(src + (size_t)c * pitch), r);
}

// Entries are summed in rounds of kRound<G>; a row's last batch is filled up
// with a factor 0 and the column of its round's first entry (no branch
// between the gathers, and an infinite operand gives what it gives at every
// batch size).
template <int G> constexpr int kRound = G >= 8 ? G : 8;

// acc += entries [beg, end) of a long row, in order, from shared memory; every
// lane of the row group is at the same ones, and the gathers of B entries are
// issued together
template <typename T, int V, int G, int B>
__device__ __forceinline__ void gather_held(const int* ci, const T* va, const char* src, unsigned pitch, int beg,
                                            int end, T (&acc)[V]) {
#pragma unroll 1
    for (int e = beg; e < end; e += B) {
        T w[B], xs[B][V];
        const int first = beg + (e - beg) / kRound<G> * kRound<G>;
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const bool in = e + j < end;
            const unsigned c = (unsigned)ci[in ? e + j : first];
            w[j] = in ? va[e + j] : T(0);
            ld_iterate(src, c, pitch, xs[j]);
        }
#pragma unroll
        for (int j = 0; j < B; ++j)
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v] = dot_acc(w[j], xs[j][v], acc[v]);
    }
}

// four or two values from an address that they fill
__device__ __forceinline__ void ldg4(const int* p, unsigned (&r)[4]) {
    const int4 u = __ldg(reinterpret_cast<const int4*>(p));
    r[0] = u.x; r[1] = u.y; r[2] = u.z; r[3] = u.w;
}
__device__ __forceinline__ void ldg4(const float* p, float (&r)[4]) { ldg_v(p, r); }
template <typename T>
__device__ __forceinline__ void ldg4(const T* p, T (&r)[4]) {
    T u[2], v[2];
    ldg_v(p, u);
    ldg_v(p + 2, v);
    r[0] = u[0]; r[1] = u[1]; r[2] = v[0]; r[3] = v[1];
}
__device__ __forceinline__ void ldg2(const int* p, unsigned (&r)[2]) {
    const int2 u = __ldg(reinterpret_cast<const int2*>(p));
    r[0] = u.x; r[1] = u.y;
}
__device__ __forceinline__ void ldg2(const float* p, float (&r)[2]) {
    const float2 u = __ldg(reinterpret_cast<const float2*>(p));
    r[0] = u.x; r[1] = u.y;
}
template <typename T>
__device__ __forceinline__ void ldg2(const T* p, T (&r)[2]) { ldg_v(p, r); }

template <typename T, int V, int B>
__device__ __forceinline__ void gather_batch(const unsigned (&c)[B], const T (&w)[B], const char* src, unsigned pitch,
                                             T (&acc)[V]) {
    T xs[B][V];
#pragma unroll
    for (int j = 0; j < B; ++j) ld_iterate(src, c[j], pitch, xs[j]);
#pragma unroll
    for (int j = 0; j < B; ++j)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = dot_acc(w[j], xs[j][v], acc[v]);
}

// acc += the packed entries of a short row, in order: B at a time (their
// columns and values are one broadcast load per four), then by fours, then the
// last two
template <typename T, int V, int B>
__device__ __forceinline__ void gather_packed(const int* __restrict__ ci, const T* __restrict__ va, int pairs,
                                              const char* src, unsigned pitch, T (&acc)[V]) {
    if (B > 4) {
#pragma unroll 1
        for (; pairs >= B / 2; pairs -= B / 2, ci += B, va += B) {
            unsigned c[B];
            T w[B];
#pragma unroll
            for (int j = 0; j < B; j += 4) {
                ldg4(ci + j, *reinterpret_cast<unsigned(*)[4]>(c + j));
                ldg4(va + j, *reinterpret_cast<T(*)[4]>(w + j));
            }
            gather_batch<T, V, B>(c, w, src, pitch, acc);
        }
    }
#pragma unroll 1
    for (; pairs >= 2; pairs -= 2, ci += 4, va += 4) {
        unsigned c[4];
        T w[4];
        ldg4(ci, c);
        ldg4(va, w);
        gather_batch<T, V, 4>(c, w, src, pitch, acc);
    }
    if (pairs > 0) {
        unsigned c[2];
        T w[2];
        ldg2(ci, c);
        ldg2(va, w);
        gather_batch<T, V, 2>(c, w, src, pitch, acc);
    }
}

template <typename T>
struct StepArgs {
    // sparse operator (rows of A~^T for the primal step, of A~ for the dual step)
    int rows;
    const int* ci;
    const T* va;
    // the other rows in the order in which they are taken, their entries in
    // fours, their cost and bounds (Csr::srec ..)
    const int4* srec;
    const int* pci;
    const T* pva;
    const T* pk;
    int n_short;
    const LongSeg* lseg;  // long-row blocks
    int n_lseg, per;      // segments, and how many a block takes
    T* part;          // partial sums of multi-segment rows, [segment][ld]
    unsigned* ticket; // completion count per (long row, column tile), tile stride ntix
    int ntix;
    const T* src;     // gathered block: Y^k (primal) or Xbar (dual)
    // row-side state
    T* Z;             // dual: Y^k -> Y^{k+1}, in place (unused by the primal step)
    const T* Z0;      // anchor
    T* Zbar;          // primal: Xbar of the previous iteration in, the new Xbar out (in place)
    T* Zh;            // check: x^ / y^
    T* DZ;            // check: x^ - X^k / y^ - Y^k
    T* Aux;           // check, dual: Pi_B(y^ - Y^k)
    const T* rc;      // primal: scaled c (n)
    const T* rlo;     // scaled lower bounds of the rows (xlo or l)
    const T* rhi;
    ColParams<T> col;
    int ld, ncol;
    const T* hal;     // per group g, entry e = 0 .. ce: (k+1)/(k+2), 1/(k+2) of Eq. mainiter
                      // for k = k_start - 1 + e at [2 (g (ce + 1) + e)]; iteration t of the
                      // interval uses entry t + 1, and entry t rebuilds its X^k
    int t, ce;
    int uni;          // the group of every active column, or -1 if they belong to several
    int pdl;          // launched as a programmatic dependent of the previous step kernel
    int hold;         // the next step kernel's blocks start when this grid has ended
    int hbm;          // the gathered block exceeds half of L2: the iterates come from HBM
};

// Reduce the row groups' partial sums of a long row through shared memory;
// on return only row group 0 holds the sum.  Every thread of the block calls it.
template <typename T, int V, int G>
__device__ __forceinline__ bool long_row_reduce(T (&acc)[V], T* red) {
    constexpr int GPB = kBlock / G;
    const int lane = threadIdx.x % G, grp = threadIdx.x / G;
#pragma unroll
    for (int v = 0; v < V; ++v) red[threadIdx.x * V + v] = acc[v];
    __syncthreads();
    if (grp != 0) return false;
    for (int g = 1; g < GPB; ++g)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] += red[(g * G + lane) * V + v];
    return true;
}

// Segments of long rows that a block takes at one or two lanes a row, where
// they are so many that a block each would be more than a wave of mostly
// prologue (long_per): 4 for one lane, 2 for two.  Measured with a block a
// segment and with these: 2 LPs on the 20k x 50k power-law matrix (1500
// segments) 5.0 and 4.4 ms a pass of 256 iterations (3.5 with the short rows
// in their own order), 8 LPs 4.1 and 3.7; on 100k x 200k with 50 long rows (200
// segments), 2 LPs, 6.05 and 6.4.
// Not in FP64, whose blocks are bound by their SM's FP64 pipe: few large ones,
// started as the previous step's blocks leave room (programmatic dependent
// launch), pile up on some SMs (1 and 2 LPs on the 20k x 50k matrix, 84 us an
// iteration with four segments a block, 58 with one).
template <typename T, int G>
constexpr int kSegPer = std::is_same<T, double>::value || G > 2 ? 1 : 4 / G;
template <typename T, int G>
int long_per(int segments, int sms) {
    return kSegPer<T, G> > 1 && segments > 4 * sms ? kSegPer<T, G> : 1;
}
// Dynamic shared memory of a long-row block: its partial sums, a vector per
// lane, before them (a block of one segment) its entries.  None where the matrix has no long row: L1 keeps what is not taken.
template <typename T, int G>
int long_smem(int segments, int per) {
    if (segments == 0) return 0;
    const int sums = per * kBlock * 16, entries = per == 1 ? kStepSeg * (int)(sizeof(int) + sizeof(T)) : 0;
    return sums > entries ? sums : entries;
}

template <typename T>
__device__ __forceinline__ T barrier(T v, T lo, T hi) {
    const bool li = is_inf(lo), hi_ = is_inf(hi);
    if (li && hi_) return T(0);
    if (li) return v > T(0) ? v : T(0);
    if (hi_) return v < T(0) ? v : T(0);
    return v;
}

// per-column parameters of the block's column tile, staged in shared memory;
// ca, cb are the Halpern weights of the column's restart group
template <typename T, int TN>
struct TileParams {
    T tau[TN], lo[TN], hi[TN], c[TN], sigma[TN], isigma[TN], ca[TN], cb[TN], pa[TN], pb[TN];
    int key[TN];  // the override's row: var of a box, ~var of an objective, INT_MAX if none
};

// The elementwise steps state where a product is rounded before it is added
// (mul, step_from, blend), so that every kernel that runs them gives the same
// bits.
//
// The iterate of one element, rebuilt from the previous reflection:
// X^k = k/(k+1) Xb + X^0/(k+1), weights pa and pb.
template <typename T>
__device__ __forceinline__ T primal_iterate(T pa, T pb, T xbar, T x0) {
    return mad(pa, xbar, mul(pb, x0));
}

// The primal step of one element: box projection, reflection (the Halpern
// update of Eq. mainiter is applied when the next step rebuilds its
// iterate).  acc is the row's product.
template <typename T, bool CHECK>
__device__ __forceinline__ void primal_element(T x, T acc, T tau, T cj, T lo, T hi, T& xh, T& xb, T& dz) {
    const T q = cj + acc, step = mul(tau, q);
    T s = CHECK ? sub(x, step) : step_from(x, tau, q);
    const bool inside = s < hi && s > lo;
    s = s < hi ? s : hi;
    s = s > lo ? s : lo;
    xh = s;
    xb = twice(s) - x;
    // x^ - x: where the box is not active it is -tau (c + G) exactly,
    // which stays accurate when |x| is large (diverging iterates of an
    // infeasible LP); elsewhere the difference with the bound
    dz = inside ? -step : s - x;
}

// The dual step of one element: row projection and Halpern update.  ys is
// y / sigma (over_sigma).
template <typename T>
__device__ __forceinline__ void dual_element(T ca, T cb, T y, T ys, T y0, T acc, T sg, T lr, T ur, T& yh, T& yn,
                                             T& dz) {
    const T s = ys + acc;
    T p = s < ur ? s : ur;
    p = p > lr ? p : lr;
    yh = sg * (s - p);
    yn = blend(ca, twice(yh) - y, cb, y0);
    // y^ - y: y^ = 0 exactly where the row bound is not active; where it
    // is, y^ - y = sigma (A xb - Pi(v)) without the cancellation of y
    dz = p == s ? -y : sg * (acc - p);
}

// A row's own operands in the lane's columns: its stored point (primal: the
// reflection Xbar; dual: Y) and anchor; and its cost and bounds.
template <typename T, int V>
struct RowOwn {
    T z[V], z0[V];
};
template <typename T>
struct RowK {
    T c, lo, hi;
};

// the point and its anchor, by plain loads (previous kernels write them)
template <typename T, int V, bool PRIMAL>
__device__ __forceinline__ RowOwn<T, V> load_own(const StepArgs<T>& a, int row, int col0) {
    RowOwn<T, V> o;
    const size_t off = (size_t)row * a.ld + col0;
    ldv((PRIMAL ? a.Zbar : a.Z) + off, o.z);
    ldv(a.Z0 + off, o.z0);
    return o;
}

// primal epilogue for row `row`, lane columns col0 .. col0+V (q0 = their
// offset in the tile): the iterate rebuilt from the previous reflection,
// X^k = k/(k+1) Xb + X^0/(k+1), then the step
template <typename T, int V, int TN, bool CHECK>
__device__ __forceinline__ void primal_epilogue(const StepArgs<T>& a, const TileParams<T, TN>& P, int row, int col0,
                                                int q0, const T (&acc)[V], const RowOwn<T, V>& o, const RowK<T>& k,
                                                T upa, T upb) {
    const size_t off = (size_t)row * a.ld + col0;
    T xh[V], xb[V], dz[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int q = q0 + v;
        const T pa = a.uni >= 0 ? upa : P.pa[q], pb = a.uni >= 0 ? upb : P.pb[q];
        const T x = primal_iterate(pa, pb, o.z[v], o.z0[v]);
        const int key = P.key[q];
        T cj = key < 0 ? T(0) : k.c, lo = k.lo, hi = k.hi;
        if (key == row) {
            lo = P.lo[q];
            hi = P.hi[q];
        }
        if (key == ~row) cj = P.c[q];
        primal_element<T, CHECK>(x, acc[v], P.tau[q], cj, lo, hi, xh[v], xb[v], dz[v]);
    }
    stv(a.Zbar + off, xb);
    if (CHECK) {
        stv(a.Zh + off, xh);
        stv(a.DZ + off, dz);
    }
}

// dual epilogue
template <typename T, int V, int TN, bool CHECK>
__device__ __forceinline__ void dual_epilogue(const StepArgs<T>& a, const TileParams<T, TN>& P, int row, int col0,
                                              int q0, const T (&acc)[V], const RowOwn<T, V>& o, const RowK<T>& k, T uca,
                                              T ucb) {
    const size_t off = (size_t)row * a.ld + col0;
    T yh[V], yn[V], dz[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const T ca = a.uni >= 0 ? uca : P.ca[q0 + v], cb = a.uni >= 0 ? ucb : P.cb[q0 + v];
        const T sg = P.sigma[q0 + v], ys = over_sigma(o.z[v], sg, P.isigma[q0 + v]);
        dual_element(ca, cb, o.z[v], ys, o.z0[v], acc[v], sg, k.lo, k.hi, yh[v], yn[v], dz[v]);
    }
    stv(a.Z + off, yn);
    if (CHECK) {
        T dzp[V];
#pragma unroll
        for (int v = 0; v < V; ++v) dzp[v] = barrier(dz[v], k.lo, k.hi);
        stv(a.Zh + off, yh);
        stv(a.DZ + off, dz);
        stv(a.Aux + off, dzp);
    }
}

// Programmatic dependent launch: what a step kernel reads before this wait
// (the matrix, costs and bounds, per-column parameters, Halpern weights) the
// previous kernel does not write, so its round trips overlap
// the end of that kernel.  That holds because only step kernels after an
// interval's first are launched as programmatic dependents, and their
// predecessor is a step kernel; the first primal step of an interval follows
// the check, admission, extraction, compaction and migration kernels that do
// write those, and is launched without the attribute (launch_iteration).
// Then let the next step kernel start its own prologue on the SMs this grid
// frees.
// (hold: not before this grid ends, see early_release.)
__device__ __forceinline__ void pdl_wait(int pdl, int hold) {
    if (pdl) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (!hold) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
}

__device__ __forceinline__ void stv_cg(float* p, const float (&r)[4]) {
    __stcg(reinterpret_cast<float4*>(p), make_float4(r[0], r[1], r[2], r[3]));
}
__device__ __forceinline__ void stv_cg(double* p, const double (&r)[2]) {
    __stcg(reinterpret_cast<double2*>(p), make_double2(r[0], r[1]));
}
__device__ __forceinline__ void stv_cg(dfloat* p, const dfloat (&r)[2]) {
    __stcg(reinterpret_cast<float4*>(p), make_float4(r[0].hi, r[0].lo, r[1].hi, r[1].lo));
}
__device__ __forceinline__ void ldv_cg(const float* p, float (&r)[4]) {
    const float4 u = __ldcg(reinterpret_cast<const float4*>(p));
    r[0] = u.x; r[1] = u.y; r[2] = u.z; r[3] = u.w;
}
__device__ __forceinline__ void ldv_cg(const double* p, double (&r)[2]) {
    const double2 u = __ldcg(reinterpret_cast<const double2*>(p));
    r[0] = u.x; r[1] = u.y;
}
__device__ __forceinline__ void ldv_cg(const dfloat* p, dfloat (&r)[2]) {
    const float4 u = __ldcg(reinterpret_cast<const float4*>(p));
    r[0] = dfloat(u.x, u.y); r[1] = dfloat(u.z, u.w);
}
__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ dfloat add(dfloat a, dfloat b) { return a + b; }

// One step (primal or dual) of the iteration on one column tile.
//   The first blocks: one segment of a long row each (at most kStepSeg
//   entries), split into contiguous pieces over the block's G-lane row groups
//   and reduced in shared memory; at one or two lanes, several segments
//   (long_per).  A row of one segment is finished by its
//   block; for a row of several, each block stores its partial sums, and the
//   block that completes the row (the last to take the row's ticket; no block
//   waits) adds the partials in segment order and finishes the row, so the
//   result does not depend on which block ends last.
//   What bounds a long row is its block's chain of round trips, so the chain is
//   short: one record (LongSeg) where there were four dependent loads, and
//   the entries are in shared memory or registers before the wait (64 LPs on
//   the 20k x 50k power-law matrix, 256 iterations: 6.45 to 6.28 ms a pass; at
//   32 lanes, 100 LPs, microseconds an iteration: on 3k x 6k 17.5 to 16.8, on
//   200k x 400k 379 to 375, on 1M x 2M 1823 to 1807).
//   The other blocks: persistent over the short rows (srec), row group
//   g taking records g, g + stride, ...; a warp's row groups take rows of
//   about the same length (build_short_rows).
//   What bounds a short row: its gathers move 16 G bytes an entry from L2
//   (at most 64 bytes a cycle and SM), and everything else that goes through
//   L1 takes a turn from them.  So a lane reads four columns and four values
//   with one broadcast load each from the packed rows, where shuffled entries
//   took two shuffles an entry, and the row's cost and bounds come in one
//   load.  Measured with the shuffles and with the packed rows (a pass of the
//   benchmark's power-law batch, 256 iterations: 7.8 and 6.5 ms; 64 LPs on a
//   10k x 10k matrix, mostly double-float: 7.9 and 6.3 ms; 101 LPs on a 200k
//   x 400k matrix, 64 iterations: 30.5 and 26.2 ms; the bound-tightening
//   batch of 1024 LPs, 64 iterations: 65.4 and 61.1 ms; 128 LPs on the 1M x
//   2M matrix: 139.6 and 133.0 ms).  Evict-first hints on a row's own
//   operands cost 2-4% in this form; prefetching the next row's own operands
//   to L2 gains 1-2% where they come from HBM.
//   (bx, by) is the block's place in the step's own grid (bx over the
//   long-row and persistent blocks, gx of them; by over the column tiles).
template <typename T, int G, int B, bool CHECK, bool PRIMAL>
__device__ __forceinline__ void step_body(const StepArgs<T>& a, const int bx, const int by, const int gx) {
    constexpr int V = Vec<T>::V, GPB = kBlock / G, TN = G * V;
    extern __shared__ uint4 red[];  // a long-row block's entries, then its partial sums (long_smem)
    __shared__ TileParams<T, TN> P;
    const int tile0 = by * TN;
    for (int q = threadIdx.x; q < TN; q += kBlock) {
        const int j = tile0 + q;
        const bool in = j < a.ncol;
        if (a.uni < 0) {
            // entry t + 1 of the column's group: this iteration's weights;
            // entry t: the previous iteration's, which rebuild X^k
            const int h = in ? 2 * (a.col.grp[j] * (a.ce + 1) + a.t + 1) : 2;
            if (PRIMAL) {
                P.pa[q] = in ? a.hal[h - 2] : T(0);
                P.pb[q] = in ? a.hal[h - 1] : T(0);
            } else {
                P.ca[q] = in ? a.hal[h] : T(0);
                P.cb[q] = in ? a.hal[h + 1] : T(0);
            }
        }
        if (PRIMAL) {
            const int kind = in ? a.col.kind[j] : 0;
            P.key[q] = kind == 1 ? a.col.var[j] : kind == 2 ? ~a.col.var[j] : INT_MAX;
            P.tau[q] = in ? a.col.tau[j] : T(0);
            P.lo[q] = in ? a.col.lo[j] : T(0);
            P.hi[q] = in ? a.col.hi[j] : T(0);
            P.c[q] = in ? a.col.c[j] : T(0);
        } else {
            P.sigma[q] = in ? a.col.sigma[j] : T(1);
            if (std::is_same<T, dfloat>::value) P.isigma[q] = T(1) / P.sigma[q];
        }
    }
    // one restart group in the whole batch: its Halpern weights as scalars
    // (the primal step takes the previous iteration's, the dual step this one's)
    const int hu = a.uni >= 0 ? 2 * (a.uni * (a.ce + 1) + a.t + (PRIMAL ? 0 : 1)) : 0;
    const T uca = a.uni >= 0 ? a.hal[hu] : T(0), ucb = a.uni >= 0 ? a.hal[hu + 1] : T(0);
    const unsigned pitch = (unsigned)a.ld * (unsigned)sizeof(T);

    const int lane = threadIdx.x % G, grp = threadIdx.x / G;
    const int col0 = tile0 + lane * V;
    const bool active = col0 < a.ncol;
    const unsigned gmask = G == 32 ? 0xffffffffu : (((1u << G) - 1u) << ((threadIdx.x & 31) & ~(G - 1)));
    const char* const src = reinterpret_cast<const char*>(a.src + (active ? col0 : tile0));
    const int per = kSegPer<T, G> > 1 ? a.per : 1, nlb = (a.n_lseg + per - 1) / per;
    if (bx < nlb) {
        const int st = kBlock / per, sub = threadIdx.x / st, is = bx * per + sub;  // threads of a segment
        const bool some = is < a.n_lseg;
        const int4* const rec = reinterpret_cast<const int4*>(a.lseg + (some ? is : bx * per));
        const int4 r0 = __ldg(rec), r1 = __ldg(rec + 1);
        const int row = r0.x, rb = r0.y, re = r0.z, ns = r1.y, s0 = r1.z;
        const int piece = (re - rb + GPB - 1) / GPB;
        T acc[V];
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = T(0);
        if (kSegPer<T, G> > 1 && per > 1) {
            constexpr int SP = kSegPer<T, G>, ST = kBlock / SP;
            // a row group takes SP pieces, next to one another, of at most E
            // entries; their columns and values come before the wait
            constexpr int E = (kStepSeg + GPB - 1) / GPB, PC = B / E < 1 ? 1 : B / E < SP ? B / E : SP;
            const int first = (threadIdx.x % ST) / G * SP;
            T* const part = reinterpret_cast<T*>(red) + (size_t)sub * kBlock * V;
            unsigned c[SP][E];
            T w[SP][E];
#pragma unroll
            for (int p = 0; p < SP; ++p)
#pragma unroll
                for (int j = 0; j < E; ++j) {
                    const int beg = rb + (first + p) * piece, e = beg + j;
                    const bool in = j < piece && e < re;
                    c[p][j] = (unsigned)__ldg(a.ci + (in ? e : beg < re ? beg : rb));
                    w[p][j] = in ? ldg1(a.va + e) : T(0);
                }
            __syncthreads();
            pdl_wait(a.pdl, a.hold);
#pragma unroll
            for (int p0 = 0; p0 < SP; p0 += PC) {
                T xs[PC][E][V];
#pragma unroll
                for (int p = 0; p < PC; ++p)
#pragma unroll
                    for (int j = 0; j < E; ++j)
                        ld_iterate(src, c[p0 + p][j], pitch, xs[p][j]);
#pragma unroll
                for (int p = 0; p < PC; ++p) {
                    const int k = first + p0 + p, left = re - rb - k * piece;
                    T sum[V];
#pragma unroll
                    for (int v = 0; v < V; ++v) sum[v] = T(0);
                    if (left > 0) {
#pragma unroll
                        for (int j = 0; j < E; ++j)
#pragma unroll
                            for (int v = 0; v < V; ++v) sum[v] = dot_acc(w[p0 + p][j], xs[p][j][v], sum[v]);
                        if (E % 4 != 0) {  // (the last batch of four is filled up)
#pragma unroll
                            for (int v = 0; v < V; ++v) sum[v] = dot_acc(T(0), xs[p][0][v], sum[v]);
                        }
                    }
                    fin<V>(sum);
#pragma unroll
                    for (int v = 0; v < V; ++v) part[(k * G + lane) * V + v] = sum[v];
                }
            }
            __syncthreads();
            if (!some || threadIdx.x % ST >= G) return;
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v] = part[lane * V + v];
#pragma unroll 8
            for (int g = 1; g < GPB; ++g)
#pragma unroll
                for (int v = 0; v < V; ++v) acc[v] += part[(g * G + lane) * V + v];
        } else {
            const int beg = min(re, rb + grp * piece), end = min(re, beg + piece);
            // the segment's entries before the wait
            T* const va = reinterpret_cast<T*>(red);
            int* const ci = reinterpret_cast<int*>(va + kStepSeg);
            for (int q = threadIdx.x; q < re - rb; q += kBlock) {
                ci[q] = __ldg(a.ci + rb + q);
                va[q] = ldg1(a.va + rb + q);
            }
            __syncthreads();
            pdl_wait(a.pdl, a.hold);
            gather_held<T, V, G, B>(ci, va, src, pitch, beg - rb, end - rb, acc);
            __syncthreads();
            fin<V>(acc);
            if (!long_row_reduce<T, V, G>(acc, reinterpret_cast<T*>(red))) return;
        }
        // only the segment's first row group continues
        if (ns > 1) {
            if (active) stv_cg(a.part + (size_t)(s0 + r1.x) * a.ld + col0, acc);
            __threadfence();
            __syncwarp(gmask);
            unsigned last = 0;
            if (lane == 0) {
                unsigned* t = a.ticket + (size_t)r0.w * a.ntix + by;
                last = atomicAdd(t, 1u) == (unsigned)(ns - 1);
                if (last) *t = 0u;  // ready for the next launch
            }
            last = __shfl_sync(gmask, last, 0, G);
            if (!last) return;
            __threadfence();
            if (!active) return;
            T p[V];
            ldv_cg(a.part + (size_t)s0 * a.ld + col0, acc);
#pragma unroll 1
            for (int t = 1; t < ns; ++t) {
                ldv_cg(a.part + (size_t)(s0 + t) * a.ld + col0, p);
#pragma unroll
                for (int v = 0; v < V; ++v) acc[v] = add(acc[v], p[v]);
            }
        }
        if (!active) return;
        const RowOwn<T, V> o = load_own<T, V, PRIMAL>(a, row, col0);
        const RowK<T> k{PRIMAL ? a.rc[row] : T(0), a.rlo[row], a.rhi[row]};
        if (PRIMAL) primal_epilogue<T, V, TN, CHECK>(a, P, row, col0, lane * V, acc, o, k, uca, ucb);
        else dual_epilogue<T, V, TN, CHECK>(a, P, row, col0, lane * V, acc, o, k, uca, ucb);
        return;
    }

    const int stride = (gx - nlb) * GPB;
    int i = (bx - nlb) * GPB + grp;
    int4 rec = make_int4(0, 0, 0, 0);
    if (i < a.n_short) rec = __ldg(a.srec + i);
    __syncthreads();
    pdl_wait(a.pdl, a.hold);
#pragma unroll 1
    for (; i < a.n_short; i += stride) {
        const int row = rec.x, first = rec.y, pairs = rec.z, place = rec.w;
        if (i + stride < a.n_short) rec = __ldg(a.srec + i + stride);
        T acc[V];
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = T(0);
        gather_packed<T, V, B>(a.pci + 4 * (size_t)first, a.pva + 4 * (size_t)first, pairs, src, pitch, acc);
        fin<V>(acc);
        // the next row's own operands towards L2, when they come from HBM
        if (a.hbm && active && i + stride < a.n_short) {
            const size_t off = (size_t)rec.x * a.ld + col0;
            asm volatile("prefetch.global.L2 [%0];" ::"l"((PRIMAL ? a.Zbar : a.Z) + off));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.Z0 + off));
        }
        if (active) {
            const RowOwn<T, V> o = load_own<T, V, PRIMAL>(a, row, col0);
            T kk[4];
            ldg4(a.pk + 4 * (size_t)place, kk);
            const RowK<T> k{kk[0], kk[1], kk[2]};
            if (PRIMAL) primal_epilogue<T, V, TN, CHECK>(a, P, row, col0, lane * V, acc, o, k, uca, ucb);
            else dual_epilogue<T, V, TN, CHECK>(a, P, row, col0, lane * V, acc, o, k, uca, ucb);
        }
    }
}

// Launch shapes are cached per device: SM count and resident blocks per SM
// packed into one int (sms * 64 + per_sm, 0 = not yet looked up), published
// with release / acquire so that every thread (the server runs one worker per
// matrix) reads both values of one lookup or does the lookup itself.
constexpr int kShapeDevices = 64;
inline int pack_shape(int sms, int per_sm) {
    sms = sms > 0 ? sms : 1;
    per_sm = per_sm > 0 ? (per_sm < 63 ? per_sm : 63) : 1;
    return sms * 64 + per_sm;
}

// SM count and resident blocks per SM of kernel f (kBlock threads, at most
// smem bytes of dynamic shared memory) on the current device, through f's per-device cache `shape` (static storage)
template <typename F>
cudaError_t launch_shape(std::atomic<int>* shape, F f, int smem, int* sms, int* per_sm) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int packed = dev >= 0 && dev < kShapeDevices ? shape[dev].load(std::memory_order_acquire) : 0;
    if (packed == 0) {
        int b = 0, n = 0;
        if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, f, kBlock, smem)) != cudaSuccess) return e;
        packed = pack_shape(n, b);
        if (dev >= 0 && dev < kShapeDevices) shape[dev].store(packed, std::memory_order_release);
    }
    *sms = packed / 64;
    *per_sm = packed % 64;
    return cudaSuccess;
}

// f<<<grid, kBlock, smem, s>>>(a), as a programmatic dependent of the previous
// kernel in s when pdl is set
template <typename A>
cudaError_t launch_with(void (*f)(A), dim3 grid, int smem, const A& a, bool pdl, cudaStream_t s) {
    if (!pdl) {
        f<<<grid, kBlock, smem, s>>>(a);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kBlock);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, f, a);
}

// Lanes per row group for a batch of ncol columns (one vector of V columns
// per lane), halved g_shift times: narrower groups make more column tiles,
// each row's gathers split over more blocks.
template <typename T>
int row_group_lanes(int ncol, int g_shift) {
    constexpr int V = Vec<T>::V;
    int vecs = (ncol + V - 1) / V;
    for (int q = 0; q < g_shift && vecs > 1; ++q) vecs = (vecs + 1) / 2;
    return vecs <= 1 ? 1 : vecs <= 2 ? 2 : vecs <= 4 ? 4 : vecs <= 8 ? 8 : vecs <= 16 ? 16 : 32;
}

// L2 bytes of the current device, looked up once per device
inline cudaError_t l2_bytes(long long* out) {
    static std::atomic<long long> cache[kShapeDevices];  // static storage: starts at 0
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    long long v = dev >= 0 && dev < kShapeDevices ? cache[dev].load(std::memory_order_acquire) : 0;
    if (v == 0) {
        int b = 0;
        if ((e = cudaDeviceGetAttribute(&b, cudaDevAttrL2CacheSize, dev)) != cudaSuccess) return e;
        v = b > 0 ? b : 1;
        if (dev >= 0 && dev < kShapeDevices) cache[dev].store(v, std::memory_order_release);
    }
    *out = v;
    return cudaSuccess;
}

// Whether a step lets the next step's blocks start before its own have ended.
// They start wherever there is room, and where long-row blocks, the largest,
// do, the FP64 pipes of some SMs get most of them.  At one and two lanes what
// the early start saves still counts for more.  Microseconds an iteration, FP64,
// long rows, with the early start and without: 8 LPs on 5k x 10k 21.7 and 19.5,
// on 20k x 50k 50.1 and 45.2, 32 LPs on 3k x 6k 24.6 and 22.9; 4 LPs on 5k x 10k
// 18.2 and 21.4; without long rows, 8 LPs on 20k x 20k 24.2 and 24.7.
template <typename T>
bool early_release(int lanes, bool long_rows) {
    return !std::is_same<T, double>::value || lanes < 4 || !long_rows;
}

// Whether a step takes the short rows in their own order (Csr::nrec) and not
// by length (Csr::srec); own: the bytes of the rows' two own blocks.  By
// length, a warp's row groups run about as many entries each, but the rows'
// points lie apart.  Narrow row groups' points (16 bytes a lane) then come in
// parts of lines, the more so from HBM, where the primal step, of few entries a
// row, moves more of its own points than it gathers.  FP64, bound by its pipe,
// wants the equal lengths at every width; double-float lies between.
// Microseconds of a step kernel pair by length and in the rows' order: FP32,
// 4 LPs on 200k x 400k 63 and 60, 8 LPs on 1M x 2M 245 and 220, 16 LPs 474 and
// 390, 32 LPs 656 and 600 (with 32 LPs on 100k x 100k 40 and 44, and on 200k x
// 400k the dual step 78 and 90: by length); double-float, 2 LPs on 400k x 1M
// 134 and 120, 4 LPs 122 and 128, 8 LPs 206 and 195, on 1M x 2M 512 and 454, on
// 200k x 400k 110 and 114; FP64, 8 LPs on 200k x 400k 311 and 345.
template <typename T>
bool natural_order(int lanes, bool primal, long long own, long long l2) {
    if (std::is_same<T, double>::value) return false;
    const int any = std::is_same<T, float>::value ? 4 : 1, far = std::is_same<T, float>::value ? 8 : 4;
    return lanes <= any || (lanes <= far && primal && 2 * own > l2);
}

// The arguments of one matrix's primal step (rows of A~^T gathering Y) or
// dual step (rows of A~ gathering Xbar) at iteration t of its interval;
// pdl is left to the caller.  l2: the device's L2 bytes, which decide whether
// a row's own operands are prefetched.
template <typename T>
StepArgs<T> step_args(bool primal, const IterData<T>& d, const IterBufs<T>& b, int ld, int ncol, const T* hal,
                      int t, int ce, int uni, long long l2) {
    const Csr& c = primal ? d.At : d.A;
    StepArgs<T> a{};
    a.rows = c.rows;
    a.ci = c.ci;
    a.va = primal ? d.at_vals : d.a_vals;
    const int lanes = row_group_lanes<T>(ncol, c.g_shift);
    a.hold = !early_release<T>(lanes, d.A.n_long > 0 || d.At.n_long > 0);
    const long long own = 2LL * c.rows * ld * (long long)sizeof(T);
    a.srec = natural_order<T>(lanes, primal, own, l2) ? c.nrec : c.srec;
    a.pci = c.pci;
    a.pva = primal ? d.at_pv : d.a_pv;
    a.pk = primal ? d.at_pk : d.a_pk;
    a.n_short = c.n_short;
    a.lseg = c.lseg;
    a.n_lseg = c.n_lseg;
    a.part = (T*)c.part;
    a.ticket = c.ticket;
    a.ntix = c.ntix;
    // the gathered block: Y (m x ld) for the primal step, Xbar (n x ld) for the dual step
    const long long gbytes = (long long)(primal ? d.A.rows : d.A.cols) * ld * (long long)sizeof(T);
    a.hbm = 2 * gbytes > l2;
    if (primal) {
        a.src = b.Y;
        a.Z = nullptr;
        a.Z0 = b.X0;
        a.Zbar = b.Xbar;
        a.Zh = b.Xh;
        a.DZ = b.DX;
        a.Aux = nullptr;
        a.rc = d.c;
        a.rlo = d.xl;
        a.rhi = d.xu;
    } else {
        a.src = b.Xbar;
        a.Z = b.Y;
        a.Z0 = b.Y0;
        a.Zbar = nullptr;
        a.Zh = b.Yh;
        a.DZ = b.DY;
        a.Aux = b.DYp;
        a.rc = nullptr;
        a.rlo = d.l;
        a.rhi = d.u;
    }
    a.col = d.col;
    a.ld = ld;
    a.ncol = ncol;
    a.hal = hal;
    a.t = t;
    a.ce = ce;
    a.uni = uni;
    return a;
}

}  // namespace

}  // namespace lpb
