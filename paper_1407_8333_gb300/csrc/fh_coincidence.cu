// Candidate clustering and coincidences on the GPU (Sec. "Candidate clustering
// and coincidences", Eq. norm; App. "Theory of coincidences").
//
//   fh_cluster       single-linkage clusters of one candidate set: candidates
//                    whose distance (Eq. norm, in mean coarse-bin widths) is at
//                    most d_max are linked; every cluster is labelled by its
//                    smallest member
//   fh_coincidences  the coincident pairs of two sets: frequencies referred to a
//                    common time, every parameter within its window in bins
//
// Both put the candidates in a grid of cells over frequency and spin-down.  A
// cell is at least as wide as the largest difference a link (or a coincidence)
// allows, reach x the largest width (reach: d_max, or the window), so a
// candidate's partners lie in its own cell and the eight around it.  The cells
// are numbered with the spin-down index innermost, so the three cells of one
// frequency index are one contiguous range of the sorted candidates.  (The
// sky widths grow without bound towards the poles and the equator, where they
// cover the whole range, so the sky is left to the tests of each pair.)  The
// sorted order carries a 32-byte binary32 record per candidate (four parameters,
// four half widths): what the pair loop reads, coalesced or broadcast, with the
// binary64 records read only by the few pairs that the binary32 arithmetic
// cannot decide (sets whose records do not fit in memory form them at each use).
//
// Clustering links each candidate to those behind it in the sorted order through
// a lock-free union-find: a root is only ever hung below a smaller root (one
// compare-and-swap), so the root of every cluster is its smallest member and the
// labels do not depend on the order of the links.  Coincidences count each
// set-1 candidate's partners (keeping the first few of them), scan the counts
// into output offsets, then write the partners sorted by index, so the pairs
// come out in (i, j) order.
//
// Arithmetic: every k and the distance are the binary64 operations of the
// definition in the order written (|x2 - x1|, 2 pi - that above pi for
// longitudes, divided by (w1 + w2) * 0.5; ((k_l^2 + k_b^2) + k_f^2) + k_fd^2 and
// its square root), so every link and every coincidence is decided exactly as
// the definition decides it.
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <algorithm>

#include "fh_internal.h"

namespace fh {
namespace {

constexpr double kPi = 3.141592653589793;
constexpr double kTwoPi = 6.283185307179586;
constexpr int kMaxCells = 1 << 22;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kUnionLimit = 1 << 20;  // retries of one union (each follows another's progress)

__device__ __forceinline__ double bins_apart(double x1, double x2, double w1, double w2,
                                             bool wrap)
{
    double a = fabs(__dsub_rn(x2, x1));
    if (wrap && a > kPi) a = __dsub_rn(kTwoPi, a);
    return __ddiv_rn(a, __dmul_rn(__dadd_rn(w1, w2), 0.5));
}

__device__ __forceinline__ double norm_distance(const fh_cand_params &a, const fh_cand_params &b,
                                                double fa, double fb)
{
    const double kl = bins_apart(a.lam, b.lam, a.dlam, b.dlam, true);
    const double kb = bins_apart(a.beta, b.beta, a.dbeta, b.dbeta, false);
    const double kf = bins_apart(fa, fb, a.df, b.df, false);
    const double kd = bins_apart(a.fdot, b.fdot, a.dfdot, b.dfdot, false);
    return __dsqrt_rn(__dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(kl, kl), __dmul_rn(kb, kb)),
                                          __dmul_rn(kf, kf)),
                                __dmul_rn(kd, kd)));
}

// order-preserving map of doubles to unsigned 64-bit keys (for atomic max)
__device__ __forceinline__ unsigned long long okey(double x)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double from_okey(unsigned long long k)
{
    const unsigned long long u = (k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k;
    return __longlong_as_double((long long)u);
}

// Per candidate the checks, the rounding to binary32 and the limits of a cell are
// integer operations on the bits: a binary64 compare or conversion takes a slot of the
// binary64 pipe (1.68 results per SM and clock), which had bound the three kernels
// that build the cells (ranges, counts and scatter of two sets of 10^6: 79, 65 and
// 119 us with them, now 37, 42 and 73).
__device__ __forceinline__ bool finite(double x)
{
    return (__double2hiint(x) & 0x7FF00000) != 0x7FF00000;
}
__device__ __forceinline__ bool positive(double x)  // and finite
{
    return (unsigned long long)(__double_as_longlong(x) - 1) < 0x7FEFFFFFFFFFFFFFull;
}
__device__ __forceinline__ bool cand_ok(const fh_cand_params &c)
{
    return finite(c.lam) & finite(c.beta) & finite(c.f) & finite(c.fdot) & positive(c.dlam) &
           positive(c.dbeta) & positive(c.df) & positive(c.dfdot);
}
// x in binary32, to nearest (a tie away from zero)
__device__ __forceinline__ float to_float(double x)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const unsigned e = (unsigned)(u >> 52) & 0x7FFu;
    if (e - 897u > 252u) return (float)x;  // zero, or out of the normal range
    const unsigned m = (unsigned)((u + (1ull << 28)) >> 29) - (896u << 23);
    return __uint_as_float(m | ((unsigned)(u >> 63) << 31));
}

// ---------------------------------------------------------------- the grid of cells
// What one call keeps on the device beside its arrays; zeroed before the first
// kernel (the largest keys start at 0; a minimum is the largest complement).
enum { kMinF, kMaxF, kMinD, kMaxD, kWidF, kWidD, kAbsL, kAbsB, kStats };
struct Head {
    unsigned long long stat[kStats];
    unsigned blocks_done;
    int32_t err;
    int32_t n_roots;   // clustering: clusters
    int32_t pad;
    // the grid: cell (floor((f - f0) inv_wf), floor((fdot - d0) inv_wd))
    double f0, inv_wf, d0, inv_wd;
    int32_t nbf, nbd;
    float4 tol;        // bound of the error of a binary32 difference (lam, beta, f, fdot)
};

// The binary32 difference of two parameters x stored as float(x - origin) is off
// by at most 2^-24 (|xa| + |xb|) from the roundings and 2^-24 |xa - xb| from the
// subtraction: below 2.4e-7 times the largest |x| (5e-7 is taken, plus a term above the
// subnormals); values beyond 1e30 are left to binary64 (an infinite bound
// neither rejects nor accepts).
__device__ __forceinline__ float diff_bound(double largest)
{
    return largest < 1e30 ? (float)(5e-7 * largest + 5e-38) : INFINITY;
}

// Cell widths: at least reach x the largest width, 1e-6 wider so that two values
// that far apart never land two cells apart after rounding, and wide enough for
// at most max_cells cells (at most 32 spin-down cells then, unless the frequency
// needs few).  An infinite or undefined width puts everything in one cell.
__device__ void grid_setup(Head *h, double reach_f, double reach_d, int32_t max_cells)
{
    const double lo_f = from_okey(~h->stat[kMinF]), hi_f = from_okey(h->stat[kMaxF]);
    const double lo_d = from_okey(~h->stat[kMinD]), hi_d = from_okey(h->stat[kMaxD]);
    const double rf = hi_f - lo_f, rd = hi_d - lo_d;
    // (the sum of two widths may overflow: such sets take one cell)
    const double mf = from_okey(h->stat[kWidF]), md = from_okey(h->stat[kWidD]);
    double wf = mf < 8e307 ? reach_f * mf * (1.0 + 1e-6) : INFINITY;
    double wd = md < 8e307 ? reach_d * md * (1.0 + 1e-6) : INFINITY;
    auto ideal = [](double r, double w) {
        const double n = floor(r / w) + 1.0;
        return n >= 1.0 && n < 1e9 ? n : (n >= 1e9 ? 1e9 : 1.0);
    };
    const double nf = ideal(rf, wf), nd = ideal(rd, wd), cap = (double)max_cells;
    double bf = nf, bd = nd;
    if (nf * nd > cap) {
        bd = fmin(nd, 32.0);
        bf = fmin(nf, floor(cap / bd));
        bd = fmin(nd, floor(cap / bf));
    }
    wf = fmax(wf, rf / bf * (1.0 + 1e-6));
    wd = fmax(wd, rd / bd * (1.0 + 1e-6));
    h->f0 = lo_f;
    h->d0 = lo_d;
    // (0 puts every candidate in the first cell)
    const double vf = 1.0 / wf, vd = 1.0 / wd;
    h->inv_wf = (bf > 1.0 && wf > 0.0 && isfinite(vf)) ? vf : 0.0;
    h->inv_wd = (bd > 1.0 && wd > 0.0 && isfinite(vd)) ? vd : 0.0;
    h->nbf = (int32_t)bf;
    h->nbd = (int32_t)bd;
    // lam: + the binary32 2 pi; f, fdot: set 1 reaches up to a cell beyond the grid
    h->tol = make_float4(diff_bound(from_okey(h->stat[kAbsL])) + 1e-6f,
                         diff_bound(from_okey(h->stat[kAbsB])), diff_bound(rf + 2.0 * wf),
                         diff_bound(rd + 2.0 * wd));
}

// One candidate set of a call: its records and how its frequencies are shifted
// (f + fdot dt where shift is set, else f).
struct CandSet {
    const fh_cand_params *c;
    double dt;
    int32_t n, shift;
    __device__ __forceinline__ double freq(const fh_cand_params &x) const
    {
        return shift ? __dadd_rn(x.f, __dmul_rn(x.fdot, dt)) : x.f;
    }
};

// Ranges of frequency and spin-down (set b), largest widths and sky values (both
// sets), the checks of every candidate; the last block lays out the grid.
// One block-wide reduction per statistic and one atomic per block (with an atomic
// per warp the same-address atomics set the time: 69 us for three statistics of
// 10^6 candidates, 26 us for these eight).  label (clustering): label[i] = i.
constexpr int kRangeThreads = 256;
__global__ void __launch_bounds__(kRangeThreads)
range_kernel(CandSet a, CandSet b, double reach_f, double reach_d, int32_t max_cells, Head *h,
             int32_t *label)
{
    let_next_start();
    unsigned long long st[kStats];
#pragma unroll
    for (int q = 0; q < kStats; ++q) st[q] = 0ull;
    bool bad = false;
    const unsigned n = (unsigned)a.n + (unsigned)b.n;  // at most 2^31
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const bool in_b = k >= (unsigned)a.n;
        const fh_cand_params x = in_b ? b.c[k - a.n] : a.c[k];
        bad = bad || !cand_ok(x);
        if (in_b) {
            const unsigned long long f = okey(b.freq(x)), d = okey(x.fdot);
            st[kMinF] = max(st[kMinF], ~f);
            st[kMaxF] = max(st[kMaxF], f);
            st[kMinD] = max(st[kMinD], ~d);
            st[kMaxD] = max(st[kMaxD], d);
            if (label) label[k - a.n] = (int32_t)(k - a.n);
        }
        st[kWidF] = max(st[kWidF], okey(x.df));
        st[kWidD] = max(st[kWidD], okey(x.dfdot));
        st[kAbsL] = max(st[kAbsL], okey(fabs(x.lam)));
        st[kAbsB] = max(st[kAbsB], okey(fabs(x.beta)));
    }
    __shared__ unsigned long long red[kStats][kRangeThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < kStats; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) st[q] = max(st[q], __shfl_xor_sync(kFull, st[q], o));
        if (lane == 0) red[q][warp] = st[q];
    }
    if (__syncthreads_or(bad ? 1 : 0) && threadIdx.x == 0) atomicOr(&h->err, kErrInvalid);
    if (threadIdx.x < kStats) {
        unsigned long long m = 0ull;
#pragma unroll
        for (int w = 0; w < kRangeThreads / 32; ++w) m = max(m, red[threadIdx.x][w]);
        atomicMax(&h->stat[threadIdx.x], m);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&h->blocks_done, 1u) == gridDim.x - 1) {
        __threadfence();
        // (the other blocks' maxima came by atomics: read them past this SM's L1)
        for (int q = 0; q < kStats; ++q) h->stat[q] = atomicMax(&h->stat[q], 0ull);
        grid_setup(h, reach_f, reach_d, max_cells);
    }
}

// cell of a candidate, or -1: too far outside the grid to have a partner in it
__device__ __forceinline__ int32_t cell_of(const Head &h, double f, double fdot)
{
    const double x = h.inv_wf > 0.0 ? __dmul_rn(__dsub_rn(f, h.f0), h.inv_wf) : 0.0;
    const double y = h.inv_wd > 0.0 ? __dmul_rn(__dsub_rn(fdot, h.d0), h.inv_wd) : 0.0;
    // (the conversion saturates, and takes NaN to the lowest value)
    const int32_t i = __double2int_rd(x), j = __double2int_rd(y);
    if (i < -1 || i > h.nbf || j < -1 || j > h.nbd) return -1;
    return min(max(i, 0), h.nbf - 1) * h.nbd + min(max(j, 0), h.nbd - 1);
}

// every candidate's cell and its rank among those of the cell (the order within
// a cell decides nothing).  cnt: set a's cells at [0, max_cells), b's behind them
__global__ void __launch_bounds__(256)
cell_count_kernel(CandSet a, CandSet b, const Head *hp, int32_t max_cells, int32_t *cnt,
                  int2 *at)
{
    let_next_start();
    wait_for_previous();
    const Head h = *hp;
    const unsigned n = (unsigned)a.n + (unsigned)b.n;  // at most 2^31
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const bool in_b = k >= (unsigned)a.n;
        const fh_cand_params *p = in_b ? b.c + (k - a.n) : a.c + k;
        // (8 bytes at a time: a caller's records start on any multiple of 8)
        const double2 q = make_double2(p->f, p->fdot);
        const CandSet &s = in_b ? b : a;
        const double f = s.shift ? __dadd_rn(q.x, __dmul_rn(q.y, s.dt)) : q.x;
        const int32_t c = cell_of(h, f, q.y);
        int32_t r = 0;
        if (c >= 0) r = atomicAdd(cnt + (in_b ? max_cells : 0) + c, 1);
        at[k] = make_int2(c, r);
    }
}

// a candidate's binary32 record: (lam, beta, f, fdot), f and fdot from the grid's
// origin, and the half widths (never below 1e-37: the rejects take a product with the
// widths, and `ordinary` leaves such narrow ones to binary64)
__device__ __forceinline__ float4 record_x(const CandSet &s, const fh_cand_params &x, double f0,
                                           double d0)
{
    return make_float4(to_float(x.lam), to_float(x.beta), to_float(__dsub_rn(s.freq(x), f0)),
                       to_float(__dsub_rn(x.fdot, d0)));
}
__device__ __forceinline__ float4 record_h(const fh_cand_params &x)
{
    auto half = [](double width) { return fmaxf(0.5f * to_float(width), 1e-37f); };
    return make_float4(half(x.dlam), half(x.dbeta), half(x.df), half(x.dfdot));
}

// sorted candidates (set a's, then set b's): [position] -> index and cell, and the
// record, a sector of 32 bytes
struct Sorted {
    int2 *who;
    float4 *rec;
    __device__ __forceinline__ int32_t index(unsigned t) const { return who[t].x; }
    __device__ __forceinline__ int32_t cell(unsigned t) const { return who[t].y; }
    __device__ __forceinline__ float4 x(unsigned t) const { return rec[2 * (size_t)t]; }
    __device__ __forceinline__ float4 h(unsigned t) const { return rec[2 * (size_t)t + 1]; }
};
// the same without the records, formed anew at each use: for sets whose 32 bytes per
// candidate do not fit in memory
struct SortedLean {
    int2 *who;
    CandSet a, b;
    const int32_t *n_a;  // candidates of set a among the sorted ones
    const Head *head;
    __device__ __forceinline__ int32_t index(unsigned t) const { return who[t].x; }
    __device__ __forceinline__ int32_t cell(unsigned t) const { return who[t].y; }
    __device__ __forceinline__ const CandSet &set(unsigned t) const
    {
        return t < (unsigned)*n_a ? a : b;
    }
    __device__ __forceinline__ float4 x(unsigned t) const
    {
        const CandSet &s = set(t);
        return record_x(s, s.c[who[t].x], head->f0, head->d0);
    }
    __device__ __forceinline__ float4 h(unsigned t) const
    {
        return record_h(set(t).c[who[t].x]);
    }
};

__global__ void __launch_bounds__(256)
cell_scatter_kernel(CandSet a, CandSet b, const Head *hp, int32_t max_cells, const int32_t *start,
                    const int2 *at, Sorted o)
{
    let_next_start();
    wait_for_previous();
    const double f0 = hp->f0, d0 = hp->d0;
    const unsigned n = (unsigned)a.n + (unsigned)b.n;  // at most 2^31
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const bool in_b = k >= (unsigned)a.n;
        const int i = (int)(in_b ? k - a.n : k);
        const int2 w = at[k];
        if (w.x < 0) continue;
        const fh_cand_params x = in_b ? b.c[i] : a.c[i];
        const unsigned t = (unsigned)start[(in_b ? max_cells : 0) + w.x] + (unsigned)w.y;
        o.who[t] = make_int2(i, w.x);
        if (!o.rec) continue;
        o.rec[2 * (size_t)t] = record_x(in_b ? b : a, x, f0, d0);
        o.rec[2 * (size_t)t + 1] = record_h(x);
    }
}

// The cells around a candidate's cell with frequency index shifted by k, as one
// range [lo, hi) of sorted positions (empty where the index is off the grid).
__device__ __forceinline__ void cell_range(const int32_t *start, int32_t cell, int32_t nbf,
                                           int32_t nbd, int k, unsigned &lo, unsigned &hi)
{
    const int i = cell / nbd + k, j = cell % nbd;
    if (i < 0 || i >= nbf) {
        lo = hi = 0;
        return;
    }
    lo = start[i * nbd + max(j - 1, 0)];
    hi = start[i * nbd + min(j + 1, nbd - 1) + 1];
}

// Binary32 decisions of a pair.  apart(): |x2 - x1| (wrapped for lam) of two
// records, each within tol of the binary64 value; wid(): the mean widths, to a
// few 2^-24.  The bounds below carry 2e-5 against those relative errors.
struct Limits {
    float4 hi, lo;       // a little above and below the reach
    float d2_hi, d2_lo;  // clustering: d_max^2 likewise
    bool exact;          // the reach is out of the binary32 arithmetic's range
};
__device__ __forceinline__ float4 apart(const float4 &a, const float4 &b)
{
    const float l = fabsf(a.x - b.x);
    return make_float4(fminf(l, 6.28318531f - l), fabsf(a.y - b.y), fabsf(a.z - b.z),
                       fabsf(a.w - b.w));
}
__device__ __forceinline__ float4 wid(const float4 &a, const float4 &b)
{
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
// some parameter is more than its reach apart: such a pair neither links (its
// distance is at least each k) nor coincides.  NaN and infinities never reject.
__device__ __forceinline__ bool far_apart(const float4 &d, const float4 &w, const float4 &hi,
                                          const float4 &tol)
{
    return (d.x - tol.x > hi.x * w.x) | (d.y - tol.y > hi.y * w.y) |
           (d.z - tol.z > hi.z * w.z) | (d.w - tol.w > hi.w * w.w);
}
__device__ __forceinline__ bool ordinary(const float4 &d, const float4 &w)
{
    const float big = fmaxf(fmaxf(fmaxf(fabsf(d.x), d.y), fmaxf(d.z, d.w)),
                            fmaxf(fmaxf(w.x, w.y), fmaxf(w.z, w.w)));
    return big < 1e30f && fminf(fminf(w.x, w.y), fminf(w.z, w.w)) > 1e-30f;
}

// ---------------------------------------------------------------- clustering
__device__ __forceinline__ int32_t uf_find(int32_t *parent, int32_t x, int32_t *err)
{
    for (int it = 0; it < kUnionLimit; ++it) {
        const int32_t p = ((volatile int32_t *)parent)[x];
        if (p == x) return x;
        const int32_t gp = ((volatile int32_t *)parent)[p];
        if (gp != p) atomicCAS(parent + x, p, gp);  // path halving: point to an ancestor
        x = gp;
    }
    atomicOr(err, kErrRange);
    return x;
}

__device__ __forceinline__ void uf_union(int32_t *parent, int32_t a, int32_t b, int32_t *err)
{
    for (int it = 0; it < kUnionLimit; ++it) {
        const int32_t ra = uf_find(parent, a, err), rb = uf_find(parent, b, err);
        if (ra == rb) return;
        const int32_t lo = min(ra, rb), hi = max(ra, rb);
        // hang the larger root below the smaller one, unless it stopped being a root
        if (atomicCAS(parent + hi, hi, lo) == hi) return;
        a = lo;
        b = hi;
    }
    atomicOr(err, kErrRange);
}

// The scan of clustering and coincidences.  Four lanes share a candidate and step
// through its ranges of sorted positions (neighbouring lanes read neighbouring
// records); pairs that the rejects leave go to the warp's list, and 32 of them at a
// time are decided, a lane each.  (Decided where they are found, one lane in four was
// busy and the scan of 10^5 candidates took 144 us, link, and 98 us, coincidences,
// now 56 and 25; a thread per candidate also left three quarters of the warps empty.)
//   range(t, k, lo, hi): the k-th of `ranges` ranges of position t
//   decide(t, u): what to do with the pair of positions t and u
constexpr int kScanLanes = 4;
constexpr int kPairThreads = 256;
constexpr int kPairCands = kPairThreads / kScanLanes;  // candidates of a block
template <typename S, typename R, typename D>
__device__ __forceinline__ void scan_pairs(const S &o, unsigned n, int ranges,
                                           const float4 &hi_lim, const float4 &tol, R &&range, D &&decide)
{
    __shared__ uint2 list_s[kPairThreads / 32][96];
    uint2 *list = list_s[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31, sub = lane % kScanLanes;
    const unsigned lt = (1u << lane) - 1u;
    int listed = 0;
    const unsigned t = blockIdx.x * kPairCands + threadIdx.x / kScanLanes;
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 xa = t < n ? o.x(t) : none, ha = t < n ? o.h(t) : none;
    for (int k = 0; k < ranges; ++k) {
        unsigned lo = 0, hi = 0;
        if (t < n) range(t, k, lo, hi);
        // every lane takes the warp's longest share, two records at a time
        const unsigned longest =
            __reduce_max_sync(kFull, hi > lo ? (hi - lo + kScanLanes - 1) / kScanLanes : 0u);
        unsigned u = lo + sub;
        for (unsigned step = 0; step < longest; step += 2, u += 2 * kScanLanes) {
            float4 xu[2], hu[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const unsigned v = u + r * kScanLanes < hi ? u + r * kScanLanes : 0u;
                xu[r] = o.x(v);
                hu[r] = o.h(v);
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const unsigned v = u + r * kScanLanes;
                const bool near =
                    v < hi && !far_apart(apart(xa, xu[r]), wid(ha, hu[r]), hi_lim, tol);
                const unsigned m = __ballot_sync(kFull, near);
                if (near) list[listed + __popc(m & lt)] = make_uint2(t, v);
                listed += __popc(m);
            }
            while (listed >= 32) {
                __syncwarp();
                listed -= 32;
                const uint2 q = list[listed + lane];
                decide(q.x, q.y);
                __syncwarp();
            }
        }
    }
    __syncwarp();
    if (lane < listed) {
        const uint2 q = list[lane];
        decide(q.x, q.y);
    }
}

// Every pair is looked at once, from its first candidate in the sorted order: the rest
// of that one's own and the next spin-down cell, and the three cells of the next
// frequency index.  The distance is formed in binary32 with its error bound; only pairs
// whose distance lies within the bound of d_max take the binary64 divisions and
// square root (GB300's binary64 rate is a small fraction of its binary32 one).
// 10^5 candidates of one 1 Hz band: 4.0 ms with buckets of frequency alone and the
// binary64 records gathered per pair, 56 us now; 10^6 over 10 Hz: 25.4 -> 0.37 ms (0.41
// with the 64 registers that leave four blocks on an SM).
template <typename S>
__global__ void __launch_bounds__(kPairThreads, 5)
link_kernel(const fh_cand_params *c, int32_t max_cells, double d_max, Limits lim, const Head *hp,
            const int32_t *start, S o, int32_t *parent, int32_t *err)
{
    let_next_start();
    wait_for_previous();
    const int32_t nbf = hp->nbf, nbd = hp->nbd;
    const float4 tol = hp->tol;
    scan_pairs(
        o, (unsigned)start[max_cells], 2, lim.hi, tol,
        [&](unsigned t, int k, unsigned &lo, unsigned &hi) {
            cell_range(start, o.cell(t), nbf, nbd, k, lo, hi);
            if (k == 0) lo = t + 1;
        },
        [&](unsigned t, unsigned u) {
            const float4 d = apart(o.x(t), o.x(u)), w = wid(o.h(t), o.h(u));
            bool in = false, sure = false;
            if (!lim.exact && ordinary(d, w)) {
                const float ax = fabsf(d.x);
                const float p0 = (ax + tol.x) / w.x, p1 = (d.y + tol.y) / w.y,
                            p2 = (d.z + tol.z) / w.z, p3 = (d.w + tol.w) / w.w;
                const float m0 = fmaxf(ax - tol.x, 0.f) / w.x, m1 = fmaxf(d.y - tol.y, 0.f) / w.y,
                            m2 = fmaxf(d.z - tol.z, 0.f) / w.z, m3 = fmaxf(d.w - tol.w, 0.f) / w.w;
                in = p0 * p0 + p1 * p1 + p2 * p2 + p3 * p3 < lim.d2_lo;
                sure = in || m0 * m0 + m1 * m1 + m2 * m2 + m3 * m3 > lim.d2_hi;
            }
            if (sure && !in) return;
            const int32_t i = o.index(t), j = o.index(u);
            if (!sure) {
                const fh_cand_params a = c[i], b = c[j];
                in = norm_distance(a, b, a.f, b.f) <= d_max;
            }
            if (in) uf_union(parent, i, j, err);
        });
}

// every candidate's root, in place (roots only ever move to ancestors, so a
// concurrent find still ends at the same root), and the number of roots
__global__ void __launch_bounds__(256) finish_labels_kernel(int32_t *label, int32_t n, Head *h)
{
    let_next_start();
    wait_for_previous();
    int roots = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int32_t r = uf_find(label, i, &h->err);
        label[i] = r;
        roots += r == i;
    }
    roots = __reduce_add_sync(kFull, roots);
    __shared__ int sum;
    if (threadIdx.x == 0) sum = 0;
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && roots) atomicAdd(&sum, roots);
    __syncthreads();
    if (threadIdx.x == 0 && sum) atomicAdd(&h->n_roots, sum);
}

// ---------------------------------------------------------------- coincidences
constexpr int kKeep = 8;  // partners of a candidate kept from the count for the write
template <typename S>
struct CoinArgs {
    CandSet s1, s2;
    double w[4];          // windows: lam, beta, f, fdot
    Limits lim;
    const Head *h;
    const int32_t *start; // set 1's cells, then set 2's (max_cells each)
    int32_t max_cells;
    S o;                  // set 1's candidates, then set 2's
    int32_t *keep;        // [set-1 sorted position][kKeep], 16-byte aligned; null: the
                          // write looks for every candidate's partners again
};

// bins_apart(...) <= window, mostly without its division.  With a the distance, b the
// mean width and t = RN(a - window b), which has the sign of the exact difference:
// t <= 0 means a / b <= window, and so its rounding; t above 2^-50 a means a quotient
// more than two units above the window; the division decides in between, and for
// widths and windows next to the ends of binary64's range.  (b and the window are at
// least 2^-500 each, so their product lies far above the subnormals and a t that
// rounds to zero means a quotient that rounds to the window.)
__device__ __forceinline__ bool within(double x1, double x2, double w1, double w2, bool wrap,
                                       double window)
{
    double a = fabs(__dsub_rn(x2, x1));
    if (wrap && a > kPi) a = __dsub_rn(kTwoPi, a);
    const double b = __dmul_rn(__dadd_rn(w1, w2), 0.5);
    const double t = __fma_rn(-window, b, a);
    const int ea = __double2hiint(a) >> 20, eb = __double2hiint(b) >> 20,
              ew = __double2hiint(window) >> 20, et = __double2hiint(t) >> 20;
    // (signs would make these negative or 2048 and more)
    if (ea < 2047 && eb > 523 && eb < 2000 && ew > 523 && ew < 2000) {
        if (__double_as_longlong(t) <= 0) return true;
        if (et >= ea - 49) return false;
    }
    return __ddiv_rn(a, b) <= window;
}

// whether the records at sorted positions t (set 1) and u coincide, after the rejects:
// each parameter clearly inside its window in binary32, else the exact test of that
// one (values on the grid of a search are often whole windows apart)
template <typename S>
__device__ __forceinline__ bool inside(const CoinArgs<S> &a, unsigned t, unsigned u,
                                       const float4 &tol)
{
    const float4 d = apart(a.o.x(t), a.o.x(u)), w = wid(a.o.h(t), a.o.h(u));
    const bool ok = !a.lim.exact && ordinary(d, w);
    const bool il = ok && d.x + tol.x < a.lim.lo.x * w.x, ib = ok && d.y + tol.y < a.lim.lo.y * w.y,
               jf = ok && d.z + tol.z < a.lim.lo.z * w.z, id = ok && d.w + tol.w < a.lim.lo.w * w.w;
    if (il && ib && jf && id) return true;
    const fh_cand_params &x = a.s1.c[a.o.index(t)], &y = a.s2.c[a.o.index(u)];
    return (jf || within(a.s1.freq(x), a.s2.freq(y), x.df, y.df, false, a.w[2])) &&
           (id || within(x.fdot, y.fdot, x.dfdot, y.dfdot, false, a.w[3])) &&
           (ib || within(x.beta, y.beta, x.dbeta, y.dbeta, false, a.w[1])) &&
           (il || within(x.lam, y.lam, x.dlam, y.dlam, true, a.w[0]));
}

// Partners of every set-1 candidate, counted, the first kKeep found kept (in any
// order; the write sorts them).  10^5 x 10^5 candidates of one 1 Hz band: 1.20 ms -> 25 us
// for the count and 1.45 ms -> 30 us for the write; 10^6 x 10^6 over 10 Hz: 9.7 -> 0.18 ms
// and 11.4 ms -> 44 us.  (With the four divisions of every pair that binary32 left open,
// binary64 operations set the count's time, 55 us and 0.37 ms.)  cnt1 starts at zero.
template <typename S>
__global__ void __launch_bounds__(kPairThreads) coin_count_kernel(const CoinArgs<S> a,
                                                                  int32_t *cnt1, int32_t *cnt2)
{
    let_next_start();
    wait_for_previous();
    const int32_t nbf = a.h->nbf, nbd = a.h->nbd;
    const float4 tol = a.h->tol;
    scan_pairs(
        a.o, (unsigned)a.start[a.max_cells], 3, a.lim.hi, tol,
        [&](unsigned t, int k, unsigned &lo, unsigned &hi) {
            cell_range(a.start + a.max_cells, a.o.cell(t), nbf, nbd, k - 1, lo, hi);
        },
        [&](unsigned t, unsigned u) {
            if (!inside(a, t, u, tol)) return;
            const int32_t j = a.o.index(u);
            const int c = atomicAdd(cnt1 + a.o.index(t), 1);
            if (a.keep && c < kKeep) a.keep[(int64_t)t * kKeep + c] = j;
            if (cnt2) atomicAdd(cnt2 + j, 1);
        });
}

// the partners of set 1's candidate at sorted position t, one thread: f(index in set 2)
template <typename S, typename F>
__device__ __forceinline__ void for_partners(const CoinArgs<S> &a, unsigned t, F &&f)
{
    const float4 tol = a.h->tol;
    for (int k = -1; k <= 1; ++k) {
        unsigned lo, hi;
        cell_range(a.start + a.max_cells, a.o.cell(t), a.h->nbf, a.h->nbd, k, lo, hi);
        for (unsigned u = lo; u < hi; ++u)
            if (!far_apart(apart(a.o.x(t), a.o.x(u)), wid(a.o.h(t), a.o.h(u)), a.lim.hi, tol) &&
                inside(a, t, u, tol))
                f(a.o.index(u));
    }
}

template <typename S>
__global__ void __launch_bounds__(256)
coin_write_kernel(const CoinArgs<S> a, const int32_t *cnt1, const int64_t *off, int64_t capacity,
                  int32_t *pairs)
{
    let_next_start();
    wait_for_previous();
    const int n = a.start[a.max_cells];
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        const int32_t i = a.o.index(t);
        const int c = cnt1[i];
        if (c == 0) continue;
        const int64_t o0 = off[i];
        int64_t o = o0;
        auto put = [&](int32_t j) {
            if (o < capacity) {
                // insertion into the candidate's list, kept sorted by j
                int64_t q = o;
                while (q > o0 && pairs[2 * (q - 1) + 1] > j) {
                    pairs[2 * q + 1] = pairs[2 * (q - 1) + 1];
                    --q;
                }
                pairs[2 * o] = i;
                pairs[2 * q + 1] = j;
            }
            ++o;
        };
        if (!a.keep || c > kKeep) {
            for_partners(a, t, put);
            continue;
        }
        // the kept ones, sorted in registers (insertion in memory waits for each store)
        const int4 *kept = reinterpret_cast<const int4 *>(a.keep + (int64_t)t * kKeep);
        const int4 p0 = kept[0], p1 = kept[1];
        int32_t v[kKeep] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
        for (int k = 0; k < kKeep; ++k)
            if (k >= c) v[k] = INT_MAX;
#pragma unroll
        for (int r = 0; r < kKeep; ++r)
#pragma unroll
            for (int k = r & 1; k + 1 < kKeep; k += 2) {
                const int32_t lo = min(v[k], v[k + 1]);
                v[k + 1] = max(v[k], v[k + 1]);
                v[k] = lo;
            }
#pragma unroll
        for (int k = 0; k < kKeep; ++k)
            if (k < c && o0 + k < capacity) {
                pairs[2 * (o0 + k)] = i;
                pairs[2 * (o0 + k) + 1] = v[k];
            }
    }
}

// ---------------------------------------------------------------- cluster coincidences
// Each coincident pair of clusters keeps its nearest coincident pair.  A hash
// table (open addressing, 64-bit keys cluster1 << 32 | cluster2, twice as many
// slots as pairs) gives every pair of clusters a slot; the slot keeps the
// smallest distance (atomic minimum of the bits of a non-negative double, which
// order like the values) and then the smallest pair index at that distance.
// The pairs come in (i, j) order, so the representatives, compacted in pair
// order, come out in (i, j) order too.
constexpr unsigned long long kEmptyKey = ~0ull;

struct CCArgs {
    const fh_cand_params *c1, *c2;
    const int32_t *label1, *label2, *pairs;
    int32_t n1, n2;
    int64_t n_pairs;
    double dt1, dt2;  // t_c - t_ref of each set
    unsigned long long *keys, *dmin, *best;
    int64_t tmask;
    int32_t *slot, *flag;
    double *dist;
    int32_t *err;
};

__device__ __forceinline__ unsigned long long mix64(unsigned long long z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void cc_insert_kernel(const CCArgs a)
{
    let_next_start();
    wait_for_previous();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < a.n_pairs;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t i = a.pairs[2 * p], j = a.pairs[2 * p + 1];
        bool ok = i >= 0 && i < a.n1 && j >= 0 && j < a.n2;
        if (ok && p > 0) {
            const int32_t pi = a.pairs[2 * p - 2], pj = a.pairs[2 * p - 1];
            ok = pi < i || (pi == i && pj < j);  // strictly increasing (i, j)
        }
        const int32_t la = ok ? a.label1[i] : -1, lb = ok ? a.label2[j] : -1;
        ok = ok && la >= 0 && la < a.n1 && lb >= 0 && lb < a.n2;
        if (!ok) {
            atomicOr(a.err, kErrInvalid);
            a.slot[p] = -1;
            continue;
        }
        // (the distance before the probes: the lanes part there, and binary64
        // operations of half-empty warps had doubled the time)
        const fh_cand_params x = a.c1[i], y = a.c2[j];
        const double fx = __dadd_rn(x.f, __dmul_rn(x.fdot, a.dt1));
        const double fy = __dadd_rn(y.f, __dmul_rn(y.fdot, a.dt2));
        const double d = norm_distance(x, y, fx, fy);
        const unsigned long long key = ((unsigned long long)(uint32_t)la << 32) | (uint32_t)lb;
        int64_t h = (int64_t)(mix64(key) & (unsigned long long)a.tmask);
        int32_t at = -1;
        for (int64_t it = 0; it <= a.tmask; ++it) {  // the table is at most half full
            const unsigned long long old = atomicCAS(a.keys + h, kEmptyKey, key);
            if (old == kEmptyKey || old == key) {
                at = (int32_t)h;
                break;
            }
            h = (h + 1) & a.tmask;
        }
        if (at < 0) {
            atomicOr(a.err, kErrRange);
            a.slot[p] = -1;
            continue;
        }
        a.dist[p] = d;
        a.slot[p] = at;
        atomicMin(a.dmin + at, (unsigned long long)__double_as_longlong(d));
    }
}

__global__ void cc_best_kernel(const CCArgs a)
{
    let_next_start();
    wait_for_previous();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < a.n_pairs;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t h = a.slot[p];
        if (h >= 0 &&
            (unsigned long long)__double_as_longlong(a.dist[p]) == a.dmin[h])
            atomicMin(a.best + h, (unsigned long long)p);
    }
}

__global__ void cc_flag_kernel(const CCArgs a)
{
    let_next_start();
    wait_for_previous();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < a.n_pairs;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t h = a.slot[p];
        a.flag[p] = (h >= 0 && a.best[h] == (unsigned long long)p) ? 1 : 0;
    }
}

__global__ void cc_write_kernel(const CCArgs a, const int64_t *off, int64_t capacity,
                                int32_t *out, double *out_d)
{
    let_next_start();
    wait_for_previous();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < a.n_pairs;
         p += (int64_t)gridDim.x * blockDim.x) {
        if (!a.flag[p]) continue;
        const int64_t k = off[p];
        if (k >= capacity) continue;
        const int32_t i = a.pairs[2 * p], j = a.pairs[2 * p + 1];
        out[4 * k] = a.label1[i];
        out[4 * k + 1] = a.label2[j];
        out[4 * k + 2] = i;
        out[4 * k + 3] = j;
        if (out_d) out_d[k] = a.dist[p];
    }
}

int grid_for(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 4096)); }

unsigned pair_grid(int64_t n) { return (unsigned)((n + kPairCands - 1) / kPairCands); }

// reach per parameter -> binary32 bounds (see Limits); a positive reach below 1e-30 is
// rejected as if it were that, so that the bound is no subnormal
Limits make_limits(const double *reach, double d_max)
{
    Limits l{};
    l.exact = false;
    const double up = 1.0 + 2e-5, dn = 1.0 - 2e-5;
    float hi[4];
    for (int q = 0; q < 4; ++q) {
        if (!(reach[q] > 1e-6 && reach[q] < 1e9)) l.exact = true;
        hi[q] = reach[q] > 0.0 ? (float)(std::max(reach[q], 1e-30) * up) : 0.0f;
    }
    l.hi = make_float4(hi[0], hi[1], hi[2], hi[3]);
    l.lo = make_float4((float)(reach[0] * dn), (float)(reach[1] * dn), (float)(reach[2] * dn),
                       (float)(reach[3] * dn));
    l.d2_hi = (float)(d_max * d_max * (1.0 + 4e-5));
    l.d2_lo = (float)(d_max * d_max * (1.0 - 4e-5));
    return l;
}

// the candidates of a and b in cells: head, start (2 max_cells + 1) and the
// sorted arrays (set a's candidates first), on scratch memory.  52 bytes per candidate;
// where the records' 32 do not fit, without them (o.rec null: lean()).
struct Cells {
    Head *head = nullptr;
    int32_t *start = nullptr, max_cells = 0;
    Sorted o{};
    SortedLean lean(const CandSet &a, const CandSet &b) const
    {
        return SortedLean{o.who, a, b, start + max_cells, head};
    }
};
cudaError_t build_cells(const CandSet &a, const CandSet &b, double reach_f, double reach_d,
                        int32_t *label, Cells &g, Scratch &sc, cudaStream_t s)
{
    const size_t n = (size_t)a.n + (size_t)b.n;
    g.max_cells = (int32_t)std::min<size_t>(kMaxCells, std::max<size_t>(n, 256));
    const size_t cells = 2 * (size_t)g.max_cells;
    // one allocation: the head and the counts (zeroed together), starts, the
    // candidates' cells and ranks, the sorted arrays
    char *base = nullptr;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at += (bytes + 255) / 256 * 256;
        return o;
    };
    const size_t o_head = take(sizeof(Head)), o_cnt = take(4 * cells), zeroed = at;
    const size_t o_start = take(4 * (cells + 1)), o_at = take(8 * n), o_who = take(8 * n),
                 o_rec = take(32 * n);
    cudaError_t e = sc.get(&base, at);
    const bool lean = e == cudaErrorMemoryAllocation;
    if (lean) {
        cudaGetLastError();
        e = sc.get(&base, o_rec);
    }
    if (e != cudaSuccess) return e;
    g.head = reinterpret_cast<Head *>(base + o_head);
    int32_t *cnt = reinterpret_cast<int32_t *>(base + o_cnt);
    g.start = reinterpret_cast<int32_t *>(base + o_start);
    int2 *where = reinterpret_cast<int2 *>(base + o_at);
    g.o.who = reinterpret_cast<int2 *>(base + o_who);
    g.o.rec = lean ? nullptr : reinterpret_cast<float4 *>(base + o_rec);
    e = cudaMemsetAsync(base, 0, zeroed, s);
    if (e != cudaSuccess) return e;
    const int grid = grid_for((int64_t)n);
    range_kernel<<<std::min(grid, 608), kRangeThreads, 0, s>>>(a, b, reach_f, reach_d,
                                                               g.max_cells, g.head, label);
    launch_after(cell_count_kernel, grid, 256, 0, s, a, b, g.head, g.max_cells, cnt, where);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = scan_exclusive(cnt, (int64_t)cells, g.start, sc, s);
    if (e == cudaSuccess) {
        launch_after(cell_scatter_kernel, grid, 256, 0, s, a, b, g.head, g.max_cells, g.start,
                     where, g.o);
        e = cudaGetLastError();
    }
    return e;
}

int report(int32_t h_err)
{
    if (h_err & kErrInvalid)
        return set_error(FH_ERR_INVALID_ARG, "a candidate value is not finite or a width <= 0");
    if (h_err & kErrRange) return set_error(FH_ERR_TIMEOUT, "union-find retry limit reached");
    return FH_OK;
}

}  // namespace
}  // namespace fh

using namespace fh;

extern "C" {

int fh_cluster(const fh_cand_params *cands, int32_t n, double d_max, int32_t *label,
               int32_t *n_clusters, void *stream)
{
    if ((n > 0 && (!cands || !label)) || !n_clusters || n < 0 || n > (1 << 30) ||
        !(d_max >= 0.0) || !std::isfinite(d_max))
        return set_error(FH_ERR_INVALID_ARG, "need cands, label, n in [0, 2^30], finite d_max >= 0");
    *n_clusters = 0;
    if (n == 0) return FH_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    Scratch sc(s);
    const CandSet none{nullptr, 0.0, 0, 0}, set{cands, 0.0, n, 0};
    const double reach[4] = {d_max, d_max, d_max, d_max};
    Cells g;
    cudaError_t e = build_cells(none, set, d_max, d_max, label, g, sc, s);
    if (e == cudaSuccess) {
        // (with no set a the starts of the second half are the set's own)
        auto link = [&](auto o) {
            launch_after(link_kernel<decltype(o)>, pair_grid(n), kPairThreads, 0, s, cands,
                         g.max_cells, d_max, make_limits(reach, d_max), g.head,
                         g.start + g.max_cells, o, label, &g.head->err);
        };
        if (g.o.rec)
            link(g.o);
        else
            link(g.lean(none, set));
        launch_after(finish_labels_kernel, grid_for(n), 256, 0, s, label, n, g.head);
        e = cudaGetLastError();
    }
    Head h{};
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, g.head, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_error(e, "cluster");
    *n_clusters = h.n_roots;
    return report(h.err);
}

int fh_coincidences(const fh_cand_params *c1, int32_t n1, double t_ref1,
                    const fh_cand_params *c2, int32_t n2, double t_ref2, double t_c,
                    const double *win, int32_t *pairs, int64_t capacity, int64_t *n_pairs,
                    int32_t *n_match1, int32_t *n_match2, void *stream)
{
    if ((n1 > 0 && !c1) || (n2 > 0 && !c2) || !win || !n_pairs || (capacity > 0 && !pairs) ||
        n1 < 0 || n2 < 0 || n1 > (1 << 30) || n2 > (1 << 30) || capacity < 0)
        return set_error(FH_ERR_INVALID_ARG, "bad candidate sets or outputs");
    for (int q = 0; q < 4; ++q)
        if (!(win[q] >= 0.0) || !std::isfinite(win[q]))
            return set_error(FH_ERR_INVALID_ARG, "windows must be finite and >= 0");
    if (!std::isfinite(t_ref1) || !std::isfinite(t_ref2) || !std::isfinite(t_c))
        return set_error(FH_ERR_INVALID_ARG, "reference times must be finite");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    *n_pairs = 0;
    cudaError_t e = cudaSuccess;
    if (n_match2 && n2 > 0) e = cudaMemsetAsync(n_match2, 0, 4 * (size_t)n2, s);
    if (e == cudaSuccess && n_match1 && n1 > 0 && n2 == 0)
        e = cudaMemsetAsync(n_match1, 0, 4 * (size_t)n1, s);
    if (e != cudaSuccess) return cuda_error(e, "cudaMemsetAsync (coincidences)");
    if (n1 == 0 || n2 == 0) {
        e = cudaStreamSynchronize(s);
        return e == cudaSuccess ? FH_OK : cuda_error(e, "coincidences");
    }
    Scratch sc(s);
    // frequencies at the common time: f + fdot (t_c - t_ref)
    const CandSet s1{c1, t_c - t_ref1, n1, 1}, s2{c2, t_c - t_ref2, n2, 1};
    Cells g;
    int64_t *off = nullptr;
    int32_t *cnt1 = n_match1, *keep = nullptr;
    if (!cnt1) e = sc.get(&cnt1, (size_t)n1);
    if (e == cudaSuccess) e = sc.get(&off, (size_t)n1 + 1);
    if (e == cudaSuccess) e = build_cells(s1, s2, win[2], win[3], nullptr, g, sc, s);
    // (sets so large that these 32 bytes per candidate do not fit do without)
    if (e == cudaSuccess && sc.get(&keep, (size_t)n1 * kKeep) != cudaSuccess) {
        cudaGetLastError();
        keep = nullptr;
    }
    // (candidates of set 1 outside the grid have no partner and no sorted position)
    if (e == cudaSuccess) e = cudaMemsetAsync(cnt1, 0, 4 * (size_t)n1, s);
    if (e != cudaSuccess) return cuda_error(e, "coincidences set-up");
    auto run = [&](auto o) {
        CoinArgs<decltype(o)> a{};
        a.s1 = s1;
        a.s2 = s2;
        for (int q = 0; q < 4; ++q) a.w[q] = win[q];
        a.lim = make_limits(win, 0.0);
        a.keep = keep;
        a.h = g.head;
        a.start = g.start;
        a.max_cells = g.max_cells;
        a.o = o;
        launch_after(coin_count_kernel<decltype(o)>, pair_grid(n1), kPairThreads, 0, s, a, cnt1,
                     n_match2);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = scan_exclusive(cnt1, n1, off, sc, s);
        if (e == cudaSuccess && capacity > 0) {
            launch_after(coin_write_kernel<decltype(o)>, grid_for(n1), 256, 0, s, a, cnt1, off,
                         capacity, pairs);
            e = cudaGetLastError();
        }
    };
    if (g.o.rec)
        run(g.o);
    else
        run(g.lean(s1, s2));
    int64_t total = 0;
    int32_t h_err = 0;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&total, off + n1, sizeof(total), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&h_err, &g.head->err, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_error(e, "coincidences");
    const int rc = report(h_err);
    if (rc) return rc;
    *n_pairs = total;
    if (total > capacity)
        return set_error(FH_ERR_CAPACITY, "%lld coincident pairs, capacity %lld",
                         (long long)total, (long long)capacity);
    return FH_OK;
}

int fh_cluster_coincidences(const fh_cand_params *c1, int32_t n1, double t_ref1,
                            const int32_t *label1, const fh_cand_params *c2, int32_t n2,
                            double t_ref2, const int32_t *label2, double t_c,
                            const int32_t *pairs, int64_t n_pairs, int32_t *out, double *out_d,
                            int64_t capacity, int64_t *n_out, void *stream)
{
    if (!n_out || n_pairs < 0 || n_pairs > ((int64_t)1 << 30) || capacity < 0 || n1 < 0 ||
        n2 < 0 || (n_pairs > 0 && (!c1 || !c2 || !label1 || !label2 || !pairs)) ||
        (capacity > 0 && !out))
        return set_error(FH_ERR_INVALID_ARG, "bad candidate sets, labels, pairs or outputs");
    if (!std::isfinite(t_ref1) || !std::isfinite(t_ref2) || !std::isfinite(t_c))
        return set_error(FH_ERR_INVALID_ARG, "reference times must be finite");
    *n_out = 0;
    if (n_pairs == 0) return FH_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    Scratch sc(s);
    int64_t tsize = 2;
    while (tsize < 2 * n_pairs) tsize <<= 1;
    unsigned long long *keys = nullptr, *dmin = nullptr, *best = nullptr;
    int32_t *slot = nullptr, *flag = nullptr, *err = nullptr;
    double *dist = nullptr;
    int64_t *off = nullptr;
    cudaError_t e = sc.get(&keys, (size_t)tsize);
    if (e == cudaSuccess) e = sc.get(&dmin, (size_t)tsize);
    if (e == cudaSuccess) e = sc.get(&best, (size_t)tsize);
    if (e == cudaSuccess) e = sc.get(&slot, (size_t)n_pairs);
    if (e == cudaSuccess) e = sc.get(&flag, (size_t)n_pairs);
    if (e == cudaSuccess) e = sc.get(&dist, (size_t)n_pairs);
    if (e == cudaSuccess) e = sc.get(&off, (size_t)n_pairs + 1);
    if (e == cudaSuccess) e = sc.get(&err, 1);
    if (e != cudaSuccess) return cuda_error(e, "cudaMallocAsync (cluster coincidences)");
    e = cudaMemsetAsync(keys, 0xFF, 8 * (size_t)tsize, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(dmin, 0xFF, 8 * (size_t)tsize, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(best, 0xFF, 8 * (size_t)tsize, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, 4, s);
    CCArgs a{c1, c2, label1, label2, pairs, n1, n2, n_pairs, t_c - t_ref1, t_c - t_ref2,
             keys, dmin, best, tsize - 1, slot, flag, dist, err};
    const int grid = grid_for(n_pairs);
    if (e == cudaSuccess) {
        launch_after(cc_insert_kernel, grid, 256, 0, s, a);
        launch_after(cc_best_kernel, grid, 256, 0, s, a);
        launch_after(cc_flag_kernel, grid, 256, 0, s, a);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = scan_exclusive(flag, n_pairs, off, sc, s);
    if (e == cudaSuccess && capacity > 0) {
        launch_after(cc_write_kernel, grid, 256, 0, s, a, off, capacity, out, out_d);
        e = cudaGetLastError();
    }
    int64_t total = 0;
    int32_t h_err = 0;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&total, off + n_pairs, sizeof(total), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h_err, err, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_error(e, "cluster coincidences");
    if (h_err & kErrInvalid)
        return set_error(FH_ERR_INVALID_ARG, "pairs out of range or not in (i, j) order, or "
                                             "labels out of range");
    if (h_err) return set_error(FH_ERR_RANGE, "cluster-pair table full");
    *n_out = total;
    if (total > capacity)
        return set_error(FH_ERR_CAPACITY, "%lld cluster pairs, capacity %lld", (long long)total,
                         (long long)capacity);
    return FH_OK;
}

}  // extern "C"
