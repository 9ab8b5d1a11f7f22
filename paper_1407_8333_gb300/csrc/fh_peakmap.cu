// Peakmap construction and cleaning on the GPU (the step before the transform).
//
//   fh_peakmap_select            Sec. "Peakmap", Eq. pm: R = S_P / S_AR bin by bin
//                                (binary32), peaks = bins above theta that are strict
//                                local maxima of R in their FFT
//   fh_peakmap_gross_veto        Sec. "Removal of spectral wandering lines": the
//                                "gross histogram" of a Delta t_H x Delta f_H grid;
//                                peaks in cells above the threshold are removed
//   fh_peakmap_persistency_veto  Sec. "Removal of spectral lines of constant
//                                frequency" with App. "Robust statistic": per-bin
//                                FFT counts, m1 = median, m2 = median(|x - m1|) /
//                                0.6745; bins above m1 + k m2 lose their peaks
//
// Selection streams the two spectra once (8 bytes per bin, the HBM-bound part):
// a block takes 4096 bins of one FFT, keeps R in shared memory with one halo
// bin on each side, and writes one selection bit per bin (a warp ballot per 32
// bins) and the segment's count; a single-block scan turns the counts into the
// CSR offsets and per-segment bases; a second pass expands the bits into bin
// indices.  Cleaning works on the peak lists: histograms by global atomics, a
// block per FFT for the passes that need the FFT (ballot ranks keep the order), the
// same scan for the new offsets.  GB300's binary64 rate is a small fraction of its
// integer rate, so no per-peak step uses binary64 where integers say the same:
// gross columns come from integer column edges, the persistency threshold is
// compared as an integer, and a power-of-two T_FFT gives a frequency's bits by
// shifts.  The robust statistic needs only the histogram of
// the per-bin counts (values 0 .. n_fft), so its medians are order statistics
// found by one block scanning that histogram; every median is exact (integers
// and half-integers), and m2 and the threshold are single binary64 operations
// in the order written above.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <vector>

#include "fh_internal.h"

namespace fh {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kSegBins = 4096;    // bins of one FFT per selection block
constexpr int kSegThreads = 256;  // 16 bins per thread
constexpr int kSegWords = kSegBins / 32;
constexpr int kScanThreads = 1024;

// (k0 + b) / t_fft, the IEEE quotient.  When t_fft is a power of two the
// quotient of an integer x in [1, 2^53) is x itself with another exponent: its
// bits come from integer shifts (a dozen integer instructions; a conversion and
// a binary64 multiply cost several times that on GB300).
struct FreqOf {
    int64_t k0;
    double t_fft;
    int32_t ex;     // t_fft = 2^ex where pow2
    bool pow2;
    __device__ __forceinline__ double operator()(int32_t b) const
    {
        const int64_t x = k0 + b;
        if (pow2 && x > 0 && x < (int64_t(1) << 53)) {
            const int lz = __clzll(x);
            // the leading one at bit 52, then dropped (the hidden bit)
            const uint64_t m = ((uint64_t)x << (lz - 11)) & 0xFFFFFFFFFFFFFull;
            return __longlong_as_double(
                (long long)(((uint64_t)(1023 + 63 - lz - ex) << 52) | m));
        }
        return __ddiv_rn((double)x, t_fft);
    }
};

FreqOf make_freq_of(int64_t k0, double t_fft)
{
    int ex = 0;
    const double m = std::frexp(t_fft, &ex);
    FreqOf f;
    f.k0 = k0;
    f.t_fft = t_fft;
    f.ex = ex - 1;
    f.pow2 = m == 0.5 && ex > -900 && ex < 900;  // every quotient is a normal number
    return f;
}

// ---------------------------------------------------------------- selection
struct SelArgs {
    const float *s_p, *s_ar;
    int64_t pitch;
    int32_t n_fft, n_bins, n_seg, n_words;
    float theta;
    uint32_t *mask;     // [fft][word]
    int32_t *seg_count; // [fft][seg]
    int32_t *err;       // bulk-copy waits that ran out (Result)
};

__device__ __forceinline__ float ratio_at(const float *sp, const float *sa, int j, int n_bins)
{
    // bins outside the FFT are never compared (the flags of bins 0 and
    // n_bins - 1 are false), so any value serves there
    return (j >= 0 && j < n_bins) ? __fdiv_rn(__ldg(sp + j), __ldg(sa + j)) : 0.0f;
}

constexpr int kBulkPolls = 1 << 22;  // a bulk copy always completes; this only bounds the wait

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return ok != 0;
}

// The selection pass with the two spectrum rows of a tile brought into shared
// memory by bulk copies (cp.async.bulk, the 1-D form of the tensor memory
// accelerator) that complete on one mbarrier: 32 KB per block in flight at
// once, no registers held by loads.  Used when both spectra are 16-byte
// aligned, the pitch is a multiple of 4 floats and so is n_bins, so that every
// copy starts on a 16-byte boundary and moves a multiple of 16 bytes.  The
// ratios are formed in place; flags and counts as in select_mask_kernel.
__global__ void __launch_bounds__(kSegThreads) select_mask_bulk_kernel(const SelArgs a)
{
    let_next_start();
    __shared__ __align__(128) float p_s[kSegBins + 8];  // p_s[4 + k]: S_P, then R, of bin j0 + k
    __shared__ __align__(128) float q_s[kSegBins];
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int32_t warp_cnt[kSegThreads / 32];
    const int row = blockIdx.y, seg = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j0 = seg * kSegBins;
    const int nb = min(kSegBins, a.n_bins - j0);
    const float *sp = a.s_p + (int64_t)row * a.pitch;
    const float *sa = a.s_ar + (int64_t)row * a.pitch;
    const uint32_t bar_a = (uint32_t)__cvta_generic_to_shared(&bar);
    if (tid == 0) {
        const uint32_t bytes = 4u * (uint32_t)nb;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_a),
                     "r"(2u * bytes)
                     : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
            "[%3];" ::"r"((uint32_t)__cvta_generic_to_shared(p_s + 4)),
            "l"(sp + j0), "r"(bytes), "r"(bar_a)
            : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
            "[%3];" ::"r"((uint32_t)__cvta_generic_to_shared(q_s)),
            "l"(sa + j0), "r"(bytes), "r"(bar_a)
            : "memory");
    }
    // the halo bins (outside the copies)
    if (tid == 32) p_s[3] = ratio_at(sp, sa, j0 - 1, a.n_bins);
    if (tid == 64) p_s[4 + kSegBins] = ratio_at(sp, sa, j0 + kSegBins, a.n_bins);
    __syncthreads();  // the barrier is initialised before anyone waits on it
    bool done = false;
    for (int it = 0; it < kBulkPolls && !done; ++it) done = mbar_try_wait(bar_a, 0);
    if (!done) {
        // never expected: report, then still wait (bounded) for the block's own
        // copies before the shared memory is given up
        if (tid == 0) atomicOr(a.err, kErrRange);
        for (int it = 0; it < kBulkPolls && !done; ++it) done = mbar_try_wait(bar_a, 0);
    }
    for (int k = tid; k < nb; k += kSegThreads) p_s[4 + k] = __fdiv_rn(p_s[4 + k], q_s[k]);
    __syncthreads();
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < kSegWords / (kSegThreads / 32); ++k) {
        const int wl = k * (kSegThreads / 32) + warp;  // word of the segment
        const int loc = wl * 32 + lane;
        const int j = j0 + loc;
        const float r = p_s[4 + loc];
        const bool f = j >= 1 && j <= a.n_bins - 2 && r > a.theta && r > p_s[3 + loc] &&
                       r > p_s[5 + loc];
        const unsigned word = __ballot_sync(kFull, f);
        const int w = seg * kSegWords + wl;
        if (lane == 0 && w < a.n_words) a.mask[(int64_t)row * a.n_words + w] = word;
        cnt += __popc(word);
    }
    if (lane == 0) warp_cnt[warp] = cnt;
    __syncthreads();
    if (warp == 0) {
        int c = lane < kSegThreads / 32 ? warp_cnt[lane] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(kFull, c, o);
        if (lane == 0) a.seg_count[(int64_t)row * a.n_seg + seg] = c;
    }
}


// A block takes 4096 bins of one FFT.  Loads: 16 bins per thread, as four
// float4 per spectrum when the rows are 16-byte aligned (VEC), so that each
// SM keeps ~256 KB of loads in flight; the ratios go to shared memory with one
// halo bin on each side.  Flags: warp w takes words w, w + 8, ... (32 bins
// each), one ballot per word.
template <bool VEC>
__global__ void __launch_bounds__(kSegThreads) select_mask_kernel(const SelArgs a)
{
    let_next_start();
    __shared__ float r_s[kSegBins + 2];  // r_s[1 + k] = R(j0 + k); halos at 0 and kSegBins + 1
    __shared__ int32_t warp_cnt[kSegThreads / 32];
    const int row = blockIdx.y, seg = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j0 = seg * kSegBins;
    const float *sp = a.s_p + (int64_t)row * a.pitch;
    const float *sa = a.s_ar + (int64_t)row * a.pitch;
    if (VEC) {
        float4 p[4], q[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int j = j0 + 4 * (k * kSegThreads + tid);
            if (j + 3 < a.n_bins) {
                p[k] = __ldg(reinterpret_cast<const float4 *>(sp + j));
                q[k] = __ldg(reinterpret_cast<const float4 *>(sa + j));
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int loc = 4 * (k * kSegThreads + tid);
            const int j = j0 + loc;
            if (j + 3 < a.n_bins) {
                r_s[1 + loc] = __fdiv_rn(p[k].x, q[k].x);
                r_s[2 + loc] = __fdiv_rn(p[k].y, q[k].y);
                r_s[3 + loc] = __fdiv_rn(p[k].z, q[k].z);
                r_s[4 + loc] = __fdiv_rn(p[k].w, q[k].w);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) r_s[1 + loc + e] = ratio_at(sp, sa, j + e, a.n_bins);
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < kSegBins / kSegThreads; ++k) {
            const int loc = k * kSegThreads + tid;
            r_s[1 + loc] = ratio_at(sp, sa, j0 + loc, a.n_bins);
        }
    }
    if (tid == 0) r_s[0] = ratio_at(sp, sa, j0 - 1, a.n_bins);
    if (tid == 1) r_s[kSegBins + 1] = ratio_at(sp, sa, j0 + kSegBins, a.n_bins);
    __syncthreads();
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < kSegWords / (kSegThreads / 32); ++k) {
        const int wl = k * (kSegThreads / 32) + warp;  // word of the segment
        const int loc = wl * 32 + lane;
        const int j = j0 + loc;
        const float r = r_s[1 + loc];
        const bool f = j >= 1 && j <= a.n_bins - 2 && r > a.theta && r > r_s[loc] &&
                       r > r_s[loc + 2];
        const unsigned word = __ballot_sync(kFull, f);
        const int w = seg * kSegWords + wl;
        if (lane == 0 && w < a.n_words) a.mask[(int64_t)row * a.n_words + w] = word;
        cnt += __popc(word);
    }
    if (lane == 0) warp_cnt[warp] = cnt;
    __syncthreads();
    if (warp == 0) {
        int c = lane < kSegThreads / 32 ? warp_cnt[lane] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(kFull, c, o);
        if (lane == 0) a.seg_count[(int64_t)row * a.n_seg + seg] = c;
    }
}

struct ExpandArgs {
    const uint32_t *mask;
    const int64_t *seg_base;  // [fft][seg] first output slot of the segment
    int32_t n_seg, n_words;
    int64_t capacity;
    FreqOf fq;
    int32_t *bins;
    double *freq;
};

// One block per (segment, FFT): 128 words, one per thread; a block scan of
// their counts ranks the segment's peaks, which are staged in shared memory in
// bin order and written as contiguous runs.
__global__ void __launch_bounds__(kSegWords) select_expand_kernel(const ExpandArgs a)
{
    let_next_start();
    wait_for_previous();
    __shared__ int32_t wsum[kSegWords / 32];
    __shared__ int32_t peaks_s[kSegBins / 2];  // strict maxima: at most every other bin
    const int row = blockIdx.y, seg = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w = seg * kSegWords + tid;
    const uint32_t word = w < a.n_words ? a.mask[(int64_t)row * a.n_words + w] : 0u;
    const int c = __popc(word);
    int p = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, p, o);
        if (lane >= o) p += y;
    }
    if (lane == 31) wsum[warp] = p;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int q = 0; q < kSegWords / 32; ++q) {
        before += q < warp ? wsum[q] : 0;
        total += wsum[q];
    }
    int pos = before + p - c;
    uint32_t m = word;
    while (m) {
        const int bit = __ffs(m) - 1;
        m &= m - 1;
        peaks_s[pos++] = w * 32 + bit;
    }
    __syncthreads();
    const int64_t base = a.seg_base[(int64_t)row * a.n_seg + seg];
    for (int k = tid; k < total; k += kSegWords) {
        const int64_t out = base + k;
        if (out < a.capacity) {
            const int32_t b = peaks_s[k];
            a.bins[out] = b;
            if (a.freq) a.freq[out] = a.fq(b);
        }
    }
}

// Exclusive scan of n int32 counts into T: out[0 .. n], and (strided) out[r stride]
// alone into strided[r], r = 0 .. n / stride.  A tile of 8192 counts per block:
// each thread reads 8 in a row, warp scans and one block step rank them.  With
// several blocks, tile_sums_kernel runs first and each block adds up the tiles
// before its own (tiles >= 0); one block alone walks all tiles (tiles < 0).  The
// walk by one block of contiguous runs per thread, which this replaces, took
// 970 us for 10^6 counts; tiles take 15 us.
constexpr int kScanPer = 8;
constexpr int kScanTile = kScanThreads * kScanPer;

__global__ void __launch_bounds__(kScanThreads)
tile_sums_kernel(const int32_t *cnt, int64_t n, int64_t *sums)
{
    let_next_start();
    wait_for_previous();
    __shared__ int64_t part[kScanThreads / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        const int64_t i = base + k * kScanThreads + threadIdx.x;
        s += i < n ? cnt[i] : 0;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = part[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        if (threadIdx.x == 0) sums[blockIdx.x] = s;
    }
}

// eight consecutive sums, 16 bytes at a time
__device__ __forceinline__ void store_tile(int32_t *p, const int32_t (&x)[kScanPer])
{
    reinterpret_cast<int4 *>(p)[0] = make_int4(x[0], x[1], x[2], x[3]);
    reinterpret_cast<int4 *>(p)[1] = make_int4(x[4], x[5], x[6], x[7]);
}
__device__ __forceinline__ void store_tile(int64_t *p, const int64_t (&x)[kScanPer])
{
#pragma unroll
    for (int k = 0; k < kScanPer; k += 2)
        reinterpret_cast<longlong2 *>(p)[k / 2] = make_longlong2(x[k], x[k + 1]);
}

// Counts and sums move 16 bytes at a time where both arrays start on 16 (a caller's
// may not); 2 x 10^6 counts: 31 -> 15 us.
template <typename T>
__global__ void __launch_bounds__(kScanThreads)
scan_counts_kernel(const int32_t *cnt, int64_t n, T *pref, int32_t stride, int64_t *strided,
                   const int64_t *sums, int64_t *total)
{
    let_next_start();
    wait_for_previous();
    __shared__ int64_t part[kScanThreads / 32];
    __shared__ int64_t carry;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool aligned =
        ((reinterpret_cast<uintptr_t>(cnt) | reinterpret_cast<uintptr_t>(pref)) & 15) == 0;
    // the counts before this block's tile
    int64_t before = 0;
    if (sums) {
        for (int64_t b = tid; b < (int64_t)blockIdx.x; b += kScanThreads) before += sums[b];
        for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(kFull, before, o);
        if (lane == 0) part[warp] = before;
        __syncthreads();
        before = part[lane];
        for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(kFull, before, o);
        __syncthreads();
    }
    const int64_t first = sums ? (int64_t)blockIdx.x * kScanTile : 0;
    const int64_t last = sums ? min(n, first + kScanTile) : n;
    for (int64_t base = first; base < last || base == first; base += kScanTile) {
        const int64_t lo = base + (int64_t)tid * kScanPer;
        int32_t v[kScanPer];
        int64_t s = 0;
        if (aligned && lo + kScanPer <= n) {
            const int4 x = *reinterpret_cast<const int4 *>(cnt + lo);
            const int4 y = *reinterpret_cast<const int4 *>(cnt + lo + 4);
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
            v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
        } else {
#pragma unroll
            for (int k = 0; k < kScanPer; ++k) v[k] = lo + k < n ? cnt[lo + k] : 0;
        }
#pragma unroll
        for (int k = 0; k < kScanPer; ++k) s += v[k];
        int64_t p = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(kFull, p, o);
            if (lane >= o) p += y;
        }
        if (lane == 31) part[warp] = p;
        __syncthreads();
        if (warp == 0) {
            int64_t w = part[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t y = __shfl_up_sync(kFull, w, o);
                if (lane >= o) w += y;
            }
            part[lane] = w;
        }
        __syncthreads();
        int64_t run = before + p - s + (warp ? part[warp - 1] : 0);
        if (aligned && pref && !strided && lo + kScanPer < n) {
            T x[kScanPer];
#pragma unroll
            for (int k = 0; k < kScanPer; ++k) {
                x[k] = (T)run;
                run += v[k];
            }
            store_tile(pref + lo, x);
        } else {
#pragma unroll
            for (int k = 0; k < kScanPer; ++k) {
                const int64_t i = lo + k;
                if (i < n) {
                    if (pref) pref[i] = (T)run;
                    if (strided && i % stride == 0) strided[i / stride] = run;
                }
                run += v[k];
            }
        }
        if (tid == kScanThreads - 1) {
            carry = run;
            if (base + kScanTile >= n) {
                if (pref) pref[n] = (T)run;
                if (strided) strided[n / stride] = run;
                if (total) *total = run;
            }
        }
        __syncthreads();
        before = carry;
    }
}

// ---------------------------------------------------------------- cleaning
// What a call reads back: one small copy at its end.
struct Result {
    int32_t err;       // kErr* bits
    int32_t thr;       // persistency: a bin's count stays up to this
    int64_t total;     // peaks selected or kept
    double stats[3];   // persistency: m1, m2, threshold
};

// The peak range of FFT i, clamped into [0, n_peaks] whatever the offsets hold;
// a CSR that is not one (o[0] != 0, o[n] != n_peaks or a decrease) is flagged.
__device__ __forceinline__ void peak_range(const int64_t *o, int i, int64_t n_peaks, int64_t &lo,
                                           int64_t &hi)
{
    lo = min(max(o[i], (int64_t)0), n_peaks);
    hi = min(max(o[i + 1], lo), n_peaks);
}

__device__ __forceinline__ void check_csr(const int64_t *o, int32_t n_fft, int64_t n_peaks,
                                          int64_t first, int64_t step, int32_t *err)
{
    for (int64_t i = first; i <= n_fft; i += step) {
        bool bad = false;
        if (i == 0) bad = o[0] != 0;
        if (i == n_fft) bad = bad || o[n_fft] != n_peaks;
        if (i < n_fft) bad = bad || o[i] > o[i + 1];
        if (bad) atomicOr(err, kErrCsr);
    }
}

// floor(num / den) of the IEEE quotient: the product with inv = RN(1 / den)
// differs from the quotient by a few units of 2^-53 relative, so when it lies
// more than 1e-9 (relative, at least absolute) from an integer both have the
// same floor; otherwise the division decides.
__device__ __forceinline__ double floor_quot(double num, double den, double inv)
{
    const double q = __dmul_rn(num, inv);
    const double fq = floor(q);
    const double margin = 1e-9 * fmax(1.0, fabs(q));
    if (q - fq > margin && fq + 1.0 - q > margin) return fq;
    return floor(__ddiv_rn(num, den));
}

struct GrossGrid {
    const double *t;
    FreqOf fq;
    double t0_h, dt_h, f0_h, df_h, inv_df;
    int32_t n_th, n_fh;
    // time cell of FFT i, or -1 off the grid
    __device__ __forceinline__ int64_t it_of(int i) const
    {
        const double x = floor(__ddiv_rn(__dsub_rn(__ldg(t + i), t0_h), dt_h));
        return (x >= 0.0 && x < (double)n_th) ? (int64_t)x : -1;
    }
    // frequency cell of bin b (may lie off the grid); non-decreasing in b, each
    // of its operations being so
    __device__ __forceinline__ double column(int64_t b) const
    {
        return floor_quot(__dsub_rn(fq((int32_t)b), f0_h), df_h, inv_df);
    }
};

// Set-up of the gross veto: the CSR check, the cleared histogram and (edge not null)
// the column edges: edge[y], y = 0 .. n_fh, the first bin whose frequency cell is y or more
// (2^31 where no bin's is).  The bin that the grid names first, two to each side,
// brackets nearly every edge; else the whole range of bins is searched.
__global__ void __launch_bounds__(256)
gross_setup_kernel(const int64_t *o, int32_t n_fft, int64_t n_peaks, GrossGrid g, int64_t *edge,
                   int32_t *hist, int64_t cells, int32_t *err)
{
    let_next_start();
    const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    check_csr(o, n_fft, n_peaks, first, step, err);
    for (int64_t k = first; k < cells; k += step) hist[k] = 0;
    for (int64_t y = first; edge && y <= g.n_fh; y += step) {
        const int64_t kmin = INT_MIN, kmax = (int64_t)INT_MAX + 1;
        int64_t lo = kmin, hi = kmax;  // column(lo - 1) < y <= column(hi)
        const double guess = (g.f0_h + (double)y * g.df_h) * g.fq.t_fft - (double)g.fq.k0;
        if (guess > -2e9 && guess < 2e9) {
            const int64_t c = (int64_t)guess;
            if (g.column(c - 2) < (double)y && g.column(c + 2) >= (double)y) {
                lo = c - 1;
                hi = c + 2;
            }
        }
        while (lo < hi) {
            const int64_t m = (lo + hi) >> 1;  // m < hi <= 2^31
            if (g.column(m) >= (double)y) hi = m; else lo = m + 1;
        }
        edge[y] = lo;
    }
}

// Column edges from this many peaks per column on: an edge costs a few columns in
// binary64 and 8 bytes, and saves each peak its own.  The veto call on 1.96 million
// peaks: 10^4 columns 126 us with edges, 141 without; 5 x 10^4 143 and 142; 10^5 158 and
// 148; 10^6 212 and 153 (20 peaks, 10^6 columns: 162 and 61).  On 2 x 10^5 peaks no
// difference up to 10^4 columns.
constexpr int kPeaksPerEdge = 64;

// a block per FFT: 620 peaks in 5 steps of 128 (a warp per FFT left two thirds of
// the SMs' warps empty and every FFT a chain of 20 steps)
constexpr int kFftThreads = 128;

// The gross cell of every peak (kept for the veto pass) and the histogram: one
// atomic per run of peaks in one cell of a warp (an FFT's peaks come in bin
// order).  1.96 million peaks: 75 -> 17 us against a warp per FFT with each
// column from binary64 and warp-wide matches.  EDGES: columns by the edges of
// gross_setup_kernel, else each peak's own in binary64 (kPeaksPerEdge).
template <bool EDGES>
__global__ void __launch_bounds__(kFftThreads)
gross_hist_kernel(const int64_t *o, const int32_t *bins, int64_t n_peaks, GrossGrid g,
                  const int64_t *edge, int32_t *cell, int32_t *hist)
{
    let_next_start();
    wait_for_previous();
    __shared__ int64_t it_s;
    const int i = blockIdx.x, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) it_s = g.it_of(i);
    __syncthreads();
    const int64_t it = it_s;
    int64_t lo, hi;
    peak_range(o, i, n_peaks, lo, hi);
    const int64_t e0 = EDGES ? edge[0] : 0, e1 = EDGES ? edge[g.n_fh] : 0;
    const float per_bin = EDGES ? (float)g.n_fh / fmaxf(1.0f, (float)(e1 - e0)) : 0.0f;
    for (int64_t q0 = lo + (threadIdx.x & ~31); q0 < hi; q0 += kFftThreads) {
        const int64_t q = q0 + lane;
        int32_t c = -1;
        if (q < hi && it >= 0) {
            const int32_t b = __ldg(bins + q);
            if constexpr (!EDGES) {
                const double y = g.column(b);
                if (y >= 0.0 && y < (double)g.n_fh) c = (int32_t)(it * g.n_fh + (int64_t)y);
            } else if (b >= e0 && b < e1) {
                int32_t y = min((int32_t)((float)(b - e0) * per_bin), g.n_fh - 1);
                // the edges are evenly spaced to a bin, so the estimate is off by one at
                // most; a grid that is not takes the search
                if (b < edge[y]) --y;
                else if (b >= edge[y + 1]) ++y;
                if (y < 0 || y >= g.n_fh || b < edge[y] || b >= edge[y + 1]) {
                    int32_t a = 0, z = g.n_fh;  // edge[a] <= b < edge[z]
                    while (z - a > 1) {
                        const int32_t m = a + (z - a) / 2;
                        if (edge[m] <= b) a = m; else z = m;
                    }
                    y = a;
                }
                c = (int32_t)(it * g.n_fh + y);
            }
        }
        if (q < hi) cell[q] = c;
        const int32_t left = __shfl_up_sync(kFull, c, 1);
        const bool head = lane == 0 || c != left;
        const unsigned heads = __ballot_sync(kFull, head);
        if (head && c >= 0) {
            const unsigned after = lane == 31 ? 0u : heads >> (lane + 1);
            atomicAdd(hist + c, after ? __ffs(after) : 32 - lane);
        }
    }
}

// FFTs with a peak in each bin (bins outside [0, n_bins) are flagged), a thread
// per peak (1.9 million: 48 -> 20 us against a warp per FFT); the CSR check rides
// along
__global__ void __launch_bounds__(256)
bin_hist_kernel(const int64_t *o, const int32_t *bins, int32_t n_fft, int64_t n_peaks,
                int32_t n_bins, int32_t *hist, int32_t *err)
{
    let_next_start();
    const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    check_csr(o, n_fft, n_peaks, first, step, err);
    for (int64_t q = first; q < n_peaks; q += step) {
        const int32_t b = __ldg(bins + q);
        if (b >= 0 && b < n_bins)
            atomicAdd(hist + b, 1);
        else
            atomicOr(err, kErrInvalid);
    }
}

// histogram of the per-bin counts: hc[v] = bins whose count is v (v <= vmax;
// larger counts, possible only for an invalid CSR, go to vmax and are flagged)
__device__ __forceinline__ void count_values(const int32_t *hist, int32_t n_bins, int32_t vmax,
                                             int first, int step, int32_t *hc, int32_t *err)
{
    for (int b = first; b < n_bins; b += step) {
        int32_t v = hist[b];
        if (v < 0 || v > vmax) {
            atomicOr(err, kErrInvalid);
            v = v < 0 ? 0 : vmax;
        }
        atomicAdd(hc + v, 1);
    }
}
__global__ void count_hist_kernel(const int32_t *hist, int32_t n_bins, int32_t vmax, int32_t *hc,
                                  int32_t *err)
{
    let_next_start();
    wait_for_previous();
    count_values(hist, n_bins, vmax, blockIdx.x * blockDim.x + threadIdx.x,
                 gridDim.x * blockDim.x, hc, err);
}

// the ka-th and kb-th smallest (0-based, ka <= kb) of a multiset given by its value
// histogram h[0 .. nv): one block; every thread scans a contiguous run of values
__device__ void kth_of_hist(const int32_t *h, int64_t nv, int64_t ka, int64_t kb, int64_t *part,
                            int64_t (&result)[2])
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t per = (nv + blockDim.x - 1) / blockDim.x;
    const int64_t lo = min(nv, (int64_t)tid * per), hi = min(nv, lo + per);
    int64_t s = 0;
    for (int64_t v = lo; v < hi; ++v) s += h[v];
    int64_t p = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(kFull, p, o);
        if (lane >= o) p += y;
    }
    if (lane == 31) part[warp] = p;
    if (tid == 0) result[0] = result[1] = nv - 1;
    __syncthreads();
    int64_t before = lane < warp ? part[lane] : 0;  // (at most 32 warps)
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(kFull, before, o);
    int64_t run = before + p - s;
    if (run <= kb && ka < run + s) {
        for (int64_t v = lo; v < hi; ++v) {
            const int64_t next = run + h[v];
            if (run <= ka && ka < next) result[0] = v;
            if (run <= kb && kb < next) result[1] = v;
            run = next;
        }
    }
    __syncthreads();
}

// App. "Robust statistic" on the per-bin counts, from their value histogram
// hc (vmax + 1 values) and n_bins values in all: m1 = median, m2 =
// median(|x - m1|) / 0.6745, thr = m1 + k m2.  The deviations are half-integers;
// hd (2 vmax + 1 entries, zeroed) receives their doubled values.  One block.
// With `counts` the block forms hc itself, and both histograms live in shared
// memory (bands and FFT counts small enough: 8192 bins and 3164 FFTs take 12 us
// against 14 us for the two kernels on global memory).
constexpr int kSmallValues = 12000;  // words of shared memory for hc and hd
__global__ void __launch_bounds__(kScanThreads)
robust_stats_kernel(const int32_t *counts, int32_t *hc, int32_t vmax, int32_t n_bins, int32_t *hd,
                    double k_sigma, Result *res_out)
{
    let_next_start();
    wait_for_previous();
    extern __shared__ int32_t small_s[];
    __shared__ int64_t part[kScanThreads / 32];
    __shared__ int64_t res[2];
    const int64_t nv = (int64_t)vmax + 1;
    const int64_t nd = 2 * nv + 1;
    if (counts) {
        hc = small_s;
        hd = small_s + nv;
        for (int64_t v = threadIdx.x; v < nv + nd; v += blockDim.x) small_s[v] = 0;
        __syncthreads();
        count_values(counts, n_bins, vmax, threadIdx.x, blockDim.x, hc, &res_out->err);
        __syncthreads();
    }
    // median of an even count: the mean of the two middle values
    const int64_t ka = ((int64_t)n_bins - 1) / 2, kb = (int64_t)n_bins / 2;
    kth_of_hist(hc, nv, ka, kb, part, res);
    const int64_t m1x2 = res[0] + res[1];  // 2 m1, an integer
    for (int64_t v = threadIdx.x; v < nv; v += blockDim.x) {
        const int32_t c = hc[v];
        if (c) {
            const int64_t d = 2 * v - m1x2;
            atomicAdd(hd + (d < 0 ? -d : d), c);
        }
    }
    __syncthreads();
    kth_of_hist(hd, nd, ka, kb, part, res);
    if (threadIdx.x == 0) {
        const double m1 = __ddiv_rn((double)m1x2, 2.0);
        // median of |x - m1| = the mean of the two halves, exact for these sizes
        const double med = __ddiv_rn((double)(res[0] + res[1]), 4.0);
        const double m2 = __ddiv_rn(med, 0.6745);
        const double thr = __dadd_rn(m1, __dmul_rn(k_sigma, m2));
        res_out->stats[0] = m1;
        res_out->stats[1] = m2;
        res_out->stats[2] = thr;
        // count > thr exactly when count > floor(thr), the counts being integers
        const double f = floor(thr);
        res_out->thr = f >= 2147483647.0 ? INT_MAX : f <= -2147483648.0 ? INT_MIN : (int32_t)f;
    }
}

// which peaks stay: the gross cell holds at most `thr` peaks (or is off the grid)
struct KeepGross {
    const int32_t *cell, *hist;
    int32_t thr;
    __device__ __forceinline__ bool operator()(int64_t q, int32_t) const
    {
        const int32_t c = cell[q];
        return c < 0 || hist[c] <= thr;
    }
};
// which peaks stay: the bin's count is not above the persistency threshold
struct KeepPersist {
    const int32_t *hist;
    const Result *res;
    int32_t n_bins;
    __device__ __forceinline__ bool operator()(int64_t, int32_t b) const
    {
        return b < 0 || b >= n_bins || hist[b] <= res->thr;
    }
};

// a block per FFT: kept peaks of the FFT
template <class Keep>
__global__ void __launch_bounds__(kFftThreads)
filter_count_kernel(const int64_t *o, const int32_t *bins, int64_t n_peaks, Keep keep,
                    int32_t *cnt)
{
    let_next_start();
    wait_for_previous();
    __shared__ int sum;
    const int i = blockIdx.x;
    if (threadIdx.x == 0) sum = 0;
    __syncthreads();
    int64_t lo, hi;
    peak_range(o, i, n_peaks, lo, hi);
    int c = 0;
    for (int64_t q = lo + threadIdx.x; q < hi; q += kFftThreads) c += keep(q, __ldg(bins + q));
    c = __reduce_add_sync(kFull, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&sum, c);
    __syncthreads();
    if (threadIdx.x == 0) cnt[i] = sum;
}

// a block per FFT: the kept peaks, in order, from the FFT's new offset
template <class Keep>
__global__ void __launch_bounds__(kFftThreads)
filter_write_kernel(const int64_t *o, const int32_t *bins, int64_t n_peaks, Keep keep,
                    const int64_t *o_out, int64_t capacity, FreqOf fq, int32_t *bins_out,
                    double *freq_out)
{
    let_next_start();
    wait_for_previous();
    constexpr int kWarps = kFftThreads / 32;
    __shared__ int kept[2][kWarps];
    const int i = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    int64_t lo, hi;
    peak_range(o, i, n_peaks, lo, hi);
    int64_t pos = o_out[i];
    int turn = 0;
    for (int64_t q0 = lo; q0 < hi; q0 += kFftThreads, turn ^= 1) {
        const int64_t q = q0 + threadIdx.x;
        const int32_t b = q < hi ? __ldg(bins + q) : 0;
        const bool k = q < hi && keep(q, b);
        const unsigned m = __ballot_sync(kFull, k);
        if (lane == 0) kept[turn][warp] = __popc(m);
        __syncthreads();  // (the other half is free: every thread is past its last use)
        int64_t at = pos + __popc(m & lt);
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            at += w < warp ? kept[turn][w] : 0;
            pos += kept[turn][w];
        }
        if (k && at < capacity) {
            bins_out[at] = b;
            if (freq_out) freq_out[at] = fq(b);
        }
    }
}

}  // namespace

template <typename T>
cudaError_t scan_exclusive(const int32_t *cnt, int64_t n, T *pref, Scratch &sc, cudaStream_t s)
{
    const int64_t tiles = (n + kScanTile - 1) / kScanTile;
    int64_t *sums = nullptr;
    if (tiles > 2) {  // one or two tiles: one block, one launch
        const cudaError_t e = sc.get(&sums, (size_t)tiles);
        if (e != cudaSuccess) return e;
        launch_after(tile_sums_kernel, (unsigned)tiles, kScanThreads, 0, s, cnt, n, sums);
    }
    launch_after(scan_counts_kernel<T>, sums ? (unsigned)tiles : 1u, kScanThreads, 0, s, cnt, n,
                 pref, 1, nullptr, sums, nullptr);
    return cudaGetLastError();
}
template cudaError_t scan_exclusive<int32_t>(const int32_t *, int64_t, int32_t *, Scratch &,
                                             cudaStream_t);
template cudaError_t scan_exclusive<int64_t>(const int32_t *, int64_t, int64_t *, Scratch &,
                                             cudaStream_t);

namespace {

// kept peaks -> new CSR and lists; *n_out (and the statistics) on the host
template <class Keep>
int run_filter(const int64_t *o, const int32_t *bins, int32_t n_fft, int64_t n_peaks, Keep keep,
               int64_t k0, double t_fft, int64_t *o_out, int32_t *bins_out, double *freq_out,
               int64_t capacity, int64_t *n_out, Result *res, double *stats, Scratch &sc,
               cudaStream_t s)
{
    int32_t *cnt = nullptr;
    cudaError_t e = sc.get(&cnt, (size_t)n_fft);
    if (e == cudaSuccess && n_fft > 0) {
        launch_after(filter_count_kernel<Keep>, n_fft, kFftThreads, 0, s, o, bins, n_peaks, keep,
                     cnt);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        launch_after(scan_counts_kernel<int64_t>, 1, kScanThreads, 0, s, cnt, n_fft, o_out, 1,
                     nullptr, nullptr, &res->total);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && n_fft > 0) {
        launch_after(filter_write_kernel<Keep>, n_fft, kFftThreads, 0, s, o, bins, n_peaks, keep,
                     o_out, capacity, make_freq_of(k0, t_fft), bins_out, freq_out);
        e = cudaGetLastError();
    }
    Result h{};
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, res, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_error(e, "peakmap filter");
    if (stats)
        for (int k = 0; k < 3; ++k) stats[k] = h.stats[k];
    if (h.err & kErrCsr) return set_error(FH_ERR_INVALID_ARG, "offsets are not a CSR of n_peaks");
    if (h.err & kErrInvalid)
        return set_error(FH_ERR_INVALID_ARG, "a bin index outside [0, n_bins)");
    *n_out = h.total;
    if (h.total > capacity)
        return set_error(FH_ERR_CAPACITY, "%lld peaks kept, capacity %lld", (long long)h.total,
                         (long long)capacity);
    return FH_OK;
}

int check_peakmap_args(const int64_t *o, const int32_t *bins, int32_t n_fft, int64_t n_peaks,
                       const int64_t *o_out, const int32_t *bins_out, int64_t capacity,
                       const int64_t *n_out)
{
    if (!o || !o_out || !n_out || (n_peaks > 0 && !bins) || (capacity > 0 && !bins_out))
        return set_error(FH_ERR_INVALID_ARG, "null offsets, bins or output");
    if (n_fft < 0 || n_peaks < 0 || n_peaks >= ((int64_t)1 << 40) || capacity < 0)
        return set_error(FH_ERR_INVALID_ARG, "need n_fft >= 0, n_peaks in [0, 2^40), capacity >= 0");
    return FH_OK;
}

}  // namespace
}  // namespace fh

using namespace fh;

extern "C" {

int64_t fh_peakmap_select_workspace(int32_t n_fft, int32_t n_bins)
{
    if (n_fft < 0 || n_bins < 0) return -1;
    const int64_t n_seg = (n_bins + kSegBins - 1) / kSegBins;
    const int64_t n_words = (n_bins + 31) / 32;
    auto up = [](int64_t b) { return (b + 255) / 256 * 256; };
    return up(4 * n_fft * n_words) + up(4 * n_fft * n_seg) + up(8 * (n_fft * n_seg + 1)) + 256;
}

int fh_peakmap_select(const float *s_p, const float *s_ar, int32_t n_fft, int32_t n_bins,
                      int64_t pitch, float theta, int64_t k0, double t_fft, int64_t *offsets,
                      int32_t *bins, double *freq, int64_t capacity, int64_t *n_peaks,
                      void *workspace, int64_t workspace_bytes, void *stream)
{
    if (!offsets || (n_fft > 0 && n_bins > 0 && (!s_p || !s_ar)) || (capacity > 0 && !bins))
        return set_error(FH_ERR_INVALID_ARG, "null spectrum, offsets, bins or n_peaks");
    if (n_fft < 0 || n_fft > 65535 * 1024 || n_bins < 0 || pitch < n_bins || capacity < 0)
        return set_error(FH_ERR_INVALID_ARG, "need n_fft >= 0, n_bins >= 0, pitch >= n_bins, "
                                             "capacity >= 0");
    if ((int64_t)n_fft * (n_bins / kSegBins + 1) > ((int64_t)1 << 31))
        return set_error(FH_ERR_INVALID_ARG, "spectra too large");
    if (!(t_fft > 0.0) || !std::isfinite(t_fft) || std::isnan(theta))
        return set_error(FH_ERR_INVALID_ARG, "need t_fft > 0 and a threshold");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int32_t n_seg = (n_bins + kSegBins - 1) / kSegBins;
    const int32_t n_words = (n_bins + 31) / 32;
    if (n_fft == 0 || n_seg == 0) {
        cudaError_t e = cudaMemsetAsync(offsets, 0, sizeof(int64_t) * (n_fft + 1), s);
        if (e == cudaSuccess && n_peaks) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_error(e, "cudaMemsetAsync (peakmap)");
        if (n_peaks) *n_peaks = 0;
        return FH_OK;
    }
    if (n_fft > 65535) return set_error(FH_ERR_INVALID_ARG, "at most 65535 FFTs per call");
    Scratch sc(s);
    uint32_t *mask = nullptr;
    int32_t *seg_count = nullptr;
    int64_t *seg_base = nullptr;
    Result *res = nullptr;
    cudaError_t e = cudaSuccess;
    const int64_t need = fh_peakmap_select_workspace(n_fft, n_bins);
    if (workspace) {
        if (workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255u))
            return set_error(FH_ERR_INVALID_ARG, "workspace of %lld bytes (256-byte aligned) "
                                                 "needed", (long long)need);
        char *w = static_cast<char *>(workspace);
        auto up = [](int64_t b) { return (b + 255) / 256 * 256; };
        mask = reinterpret_cast<uint32_t *>(w);
        seg_count = reinterpret_cast<int32_t *>(w + up(4 * (int64_t)n_fft * n_words));
        seg_base = reinterpret_cast<int64_t *>(w + up(4 * (int64_t)n_fft * n_words) +
                                               up(4 * (int64_t)n_fft * n_seg));
        res = reinterpret_cast<Result *>(w + need - 256);
    } else {
        e = sc.get(&mask, (size_t)n_fft * n_words);
        if (e == cudaSuccess) e = sc.get(&seg_count, (size_t)n_fft * n_seg);
        if (e == cudaSuccess) e = sc.get(&seg_base, (size_t)n_fft * n_seg + 1);
        if (e == cudaSuccess) e = sc.get(&res, 1);
        if (e != cudaSuccess) return cuda_error(e, "cudaMallocAsync (peakmap)");
    }
    SelArgs a{s_p, s_ar, pitch, n_fft, n_bins, n_seg, n_words, theta, mask, seg_count,
              &res->err};
    const bool vec = ((reinterpret_cast<uintptr_t>(s_p) | reinterpret_cast<uintptr_t>(s_ar)) &
                      15u) == 0 && (pitch & 3) == 0;
    if (e == cudaSuccess) e = cudaMemsetAsync(res, 0, sizeof(Result), s);
    if (e != cudaSuccess) return cuda_error(e, "cudaMemsetAsync (peakmap)");
    if (vec && (n_bins & 3) == 0)
        select_mask_bulk_kernel<<<dim3(n_seg, n_fft), kSegThreads, 0, s>>>(a);
    else if (vec)
        select_mask_kernel<true><<<dim3(n_seg, n_fft), kSegThreads, 0, s>>>(a);
    else
        select_mask_kernel<false><<<dim3(n_seg, n_fft), kSegThreads, 0, s>>>(a);
    e = cudaGetLastError();
    if (e == cudaSuccess) {
        launch_after(scan_counts_kernel<int64_t>, 1, kScanThreads, 0, s, seg_count,
                     (int64_t)n_fft * n_seg, seg_base, n_seg, offsets, nullptr, &res->total);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        ExpandArgs x{mask, seg_base, n_seg, n_words, capacity, make_freq_of(k0, t_fft), bins,
                     freq};
        launch_after(select_expand_kernel, dim3(n_seg, n_fft), kSegWords, 0, s, x);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_error(e, "peak selection");
    if (!n_peaks) return FH_OK;  // asynchronous: the total is offsets[n_fft]
    Result h{};
    e = cudaMemcpyAsync(&h, res, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_error(e, "peak selection");
    if (h.err) return set_error(FH_ERR_TIMEOUT, "peak selection: a bulk-copy wait ran out");
    *n_peaks = h.total;
    if (h.total > capacity)
        return set_error(FH_ERR_CAPACITY, "%lld peaks selected, capacity %lld",
                         (long long)h.total, (long long)capacity);
    return FH_OK;
}

int fh_peakmap_gross_veto(const double *t, const int64_t *offsets, const int32_t *bins,
                          int32_t n_fft, int64_t n_peaks, int64_t k0, double t_fft, double t0_h,
                          double dt_h, int32_t n_th, double f0_h, double df_h, int32_t n_fh,
                          int32_t threshold, int32_t *hist, int64_t *offsets_out,
                          int32_t *bins_out, double *freq_out, int64_t capacity, int64_t *n_out,
                          void *stream)
{
    int rc = check_peakmap_args(offsets, bins, n_fft, n_peaks, offsets_out, bins_out, capacity,
                                n_out);
    if (rc) return rc;
    if ((n_fft > 0 && !t) || !hist || n_th < 1 || n_fh < 1 ||
        (int64_t)n_th * n_fh > ((int64_t)1 << 31) || !(dt_h > 0.0) || !(df_h > 0.0) ||
        !(t_fft > 0.0) || !std::isfinite(t0_h) || !std::isfinite(f0_h) ||
        !std::isfinite(dt_h) || !std::isfinite(df_h) || !std::isfinite(t_fft))
        return set_error(FH_ERR_INVALID_ARG, "bad gross grid (n_th, n_fh >= 1, steps > 0)");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    Scratch sc(s);
    Result *res = nullptr;
    int32_t *cell = nullptr;
    int64_t *edge = nullptr;
    const bool edges = n_fh < n_peaks / kPeaksPerEdge;
    cudaError_t e = sc.get(&res, 1);
    if (e == cudaSuccess) e = sc.get(&cell, (size_t)n_peaks);
    if (e == cudaSuccess && edges) e = sc.get(&edge, (size_t)n_fh + 1);
    if (e == cudaSuccess) e = cudaMemsetAsync(res, 0, sizeof(Result), s);
    const GrossGrid g{t, make_freq_of(k0, t_fft), t0_h, dt_h, f0_h, df_h, 1.0 / df_h, n_th, n_fh};
    const int64_t cells = (int64_t)n_th * n_fh;
    if (e == cudaSuccess) {
        const int64_t work = std::max(cells, (int64_t)n_fft + 1);  // (cells: n_fh or more)
        const int grid = (int)std::min<int64_t>((work + 255) / 256, 4096);
        gross_setup_kernel<<<grid, 256, 0, s>>>(offsets, n_fft, n_peaks, g, edge, hist, cells,
                                                &res->err);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && n_fft > 0) {
        launch_after(edges ? gross_hist_kernel<true> : gross_hist_kernel<false>, n_fft,
                     kFftThreads, 0, s, offsets, bins, n_peaks, g, edge, cell, hist);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_error(e, "gross histogram");
    return run_filter(offsets, bins, n_fft, n_peaks, KeepGross{cell, hist, threshold}, k0, t_fft,
                      offsets_out, bins_out, freq_out, capacity, n_out, res, nullptr, sc, s);
}

int fh_peakmap_persistency_veto(const int64_t *offsets, const int32_t *bins, int32_t n_fft,
                                int64_t n_peaks, int32_t n_bins, double k_sigma, int64_t k0,
                                double t_fft, int32_t *hist, double *stats,
                                int64_t *offsets_out, int32_t *bins_out, double *freq_out,
                                int64_t capacity, int64_t *n_out, void *stream)
{
    int rc = check_peakmap_args(offsets, bins, n_fft, n_peaks, offsets_out, bins_out, capacity,
                                n_out);
    if (rc) return rc;
    if (!hist || !stats || n_bins < 1 || !std::isfinite(k_sigma) || !(t_fft > 0.0) ||
        !std::isfinite(t_fft))
        return set_error(FH_ERR_INVALID_ARG, "need n_bins >= 1, finite k_sigma, t_fft > 0");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    Scratch sc(s);
    // a bin's count is at most n_fft for a valid CSR; one more value catches the rest
    const int32_t vmax = n_fft + 1;
    const size_t nv = (size_t)vmax + 1, nd = 2 * nv + 1;
    const bool small = nv + nd <= (size_t)kSmallValues && n_bins <= 65536;
    Result *res = nullptr;
    int32_t *hc = nullptr;
    cudaError_t e = sc.get(&res, 1);
    if (e == cudaSuccess && !small) e = sc.get(&hc, nv + nd);
    if (e == cudaSuccess) e = cudaMemsetAsync(res, 0, sizeof(Result), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(hist, 0, sizeof(int32_t) * (size_t)n_bins, s);
    if (e == cudaSuccess && !small)
        e = cudaMemsetAsync(hc, 0, sizeof(int32_t) * (nv + nd), s);
    if (e == cudaSuccess) {
        const int64_t work = std::max(n_peaks, (int64_t)n_fft + 1);
        const int grid = (int)std::min<int64_t>((work + 255) / 256, 8192);
        bin_hist_kernel<<<grid, 256, 0, s>>>(offsets, bins, n_fft, n_peaks, n_bins, hist,
                                             &res->err);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && !small) {
        const int grid = (int)std::min<int64_t>(((int64_t)n_bins + 255) / 256, 4096);
        launch_after(count_hist_kernel, grid, 256, 0, s, hist, n_bins, vmax, hc, &res->err);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        launch_after(robust_stats_kernel, 1, kScanThreads, small ? sizeof(int32_t) * (nv + nd) : 0,
                     s, small ? hist : nullptr, hc, vmax, n_bins, hc ? hc + nv : nullptr, k_sigma,
                     res);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_error(e, "persistency histogram");
    return run_filter(offsets, bins, n_fft, n_peaks, KeepPersist{hist, res, n_bins}, k0, t_fft,
                      offsets_out, bins_out, freq_out, capacity, n_out, res, stats, sc, s);
}

}  // extern "C"
