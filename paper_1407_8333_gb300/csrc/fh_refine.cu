// fh_refine: the refined-grid frequency-Hough search around coarse candidates
// (Sec. "Refined Grid in the parameter space").
//
// For each coarse candidate (cell b_c, row j_c of the plan's grid) the
// transform runs again on a small grid: the same K-over-resolved cells, +-1
// coarse bin around the candidate (cells b_c - K .. b_c + K); a spin-down step
// refined by K_fdot, 2 K_fdot rows below the coarse value and 2 K_fdot - 1
// above (refined row 0 on coarse row j_c - 2: shift S0_i + (j_c - 2) D_i, step
// D'_i = floor((fdot_step / K_fdot) c_i 2^32)); and the caller's refined sky
// directions.  One refined candidate is kept per coarse one: the largest count
// over all refined directions, rows and cells (ties: smallest direction, then
// row, then cell).
//
// Per call: the coarse shift tables (prep kernel) and, with device-side checks, the
// frequencies' order; then one kernel over (candidate, share of the FFTs): per FFT the
// contiguous range of peaks that can reach the refined band (a conservative
// frequency window, two binary searches), and per (peak of a range, refined
// direction) the position, exactly as the coarse correction forms it, and its
// stripe start on every refined row, counted in a histogram of starts in shared
// memory; last a kernel that sums the starts over K cells and picks.  A candidate's
// ranges hold a few tenths of a peak per FFT, so what is left of the work is the
// ranges themselves; positions are formed in lists of (peak, direction), a lane
// each, because a lane per FFT would leave three quarters of a warp idle.
// (The general transform on compacted peakmaps, which this replaces, needed a
// host round trip for the compaction, 178,200 blocks of positions and a launch per
// 12 candidates: 50 candidates x 9 directions on 3164 FFTs took
// 460 us of kernels and as much again on the host.)
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fh_internal.h"

using namespace fh;

namespace {

constexpr unsigned kFull = 0xffffffffu;

struct RefineArgs {
    const double *t, *freq, *v, *sky;  // sky: [cand][n_ref][3]
    const int64_t *offsets, *S0, *D;   // sanitised CSR; coarse shift tables
    const int32_t *cell, *row;
    int32_t n_fft, k_over, n_rows, n_ref;
    int32_t cand0, dir0, n_dir;        // the launch's first candidate and directions
    int32_t dirs_per, rows_per;        // directions and rows of one block's histogram
    int32_t ffts_per;                  // FFTs of one block
    double f0_min, kt, t_ref, step_ref, cshift;
    double half_inv_kt;                // 0.5 / kt
    int32_t *starts;  // [cand][direction][row][3 K] of the launch: stripe starts, zeroed
    int32_t *err;
};

constexpr int kRefThreads = 256;
constexpr int kRefList = 64;  // (FFT, peak) entries a warp collects before it places them

// Refined band of candidate c in refined cells [0, 2K + 1): a stripe starting at
// s touches it iff s in [1 - K, 2K].  With the refined shifts X_j = S0r + j D'
// (j < n_rows), positions A in [min_j X_j + (1 - K) 2^32, max_j X_j + (2K + 1)
// 2^32) can touch it; one extra cell on each side covers rounding.  A position
// is about ((f r - f0_min) KT + 0.5 - 0.5 K) 2^32 with r = 1 / (1 + v.n), so
// the frequencies f = u (1 + v.n) of the peaks that can take part lie between
// the extremes of that product over u in [u_lo, u_hi] and v.n between its
// least and largest value over the block's refined directions (a bilinear
// form: the extremes are at the corners).  v.n is formed in binary32 and widened by
// a bound of its error; the margin of a cell is far above the other roundings.
// The exact position of each peak of the range then decides.
//
// The binary64 pipe (1.68 results per SM and clock) bounds the kernel, so the ranges
// leave it what they must: the shifts in integers, the sky rounded to binary32 once
// per block, no division, the searches on the frequencies' bits.  50 candidates x 9
// directions on 3164 FFTs: 67 us with all of that in binary64, 43 us now.
//
// grid (candidates, shares of ffts_per FFTs, (direction, row) groups of one
// histogram).  A warp takes 32 FFTs at a time (lane <-> FFT), lists their peaks, and
// places list x directions, a lane each.
__global__ void __launch_bounds__(kRefThreads) refine_kernel(const RefineArgs a)
{
    let_next_start();
    wait_for_previous();
    extern __shared__ int32_t hist[];  // [direction][row][3 K], then the sky
    __shared__ int32_t list_fft[kRefThreads / 32][kRefList];
    __shared__ int64_t list_peak[kRefThreads / 32][kRefList];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = a.cand0 + blockIdx.x;
    const int row_groups = (a.n_rows + a.rows_per - 1) / a.rows_per;
    const int d0 = (int)(blockIdx.z / row_groups) * a.dirs_per;
    const int r0 = (int)(blockIdx.z % row_groups) * a.rows_per;
    const int nd = min(a.dirs_per, a.n_dir - d0), nr = min(a.rows_per, a.n_rows - r0);
    const int K = a.k_over, E = 3 * K;
    const int words = nd * nr * E;
    for (int w = threadIdx.x; w < words; w += kRefThreads) hist[w] = 0;
    const int64_t lo_cell = (int64_t)a.cell[c] - K;
    const int64_t j_off = (int64_t)a.row[c] - 2;
    const double *sky = a.sky + 3 * ((int64_t)c * a.n_ref + a.dir0);
    float *sky32 = reinterpret_cast<float *>(hist + a.dirs_per * a.rows_per * E);
    for (int w = threadIdx.x; w < 3 * nd; w += kRefThreads) sky32[w] = (float)sky[3 * d0 + w];
    __syncthreads();
    int32_t ev = 0;
    const int f_begin = blockIdx.y * a.ffts_per;
    const int f_end = min(a.n_fft, f_begin + a.ffts_per);

    // the listed peaks in every direction of the group, a lane each
    auto place = [&](int n) {
        __syncwarp();
        for (int q = lane; q < n * nd; q += 32) {
            const int e = q / nd, d = q - e * nd;
            const int i = list_fft[warp][e];
            const double *n3 = sky + 3 * (d0 + d);
            const double px = __dmul_rn(a.v[3 * (int64_t)i + 0], n3[0]);
            const double py = __dmul_rn(a.v[3 * (int64_t)i + 1], n3[1]);
            const double pz = __dmul_rn(a.v[3 * (int64_t)i + 2], n3[2]);
            const double den = __dadd_rn(1.0, __dadd_rn(__dadd_rn(px, py), pz));
            const double u = __dmul_rn(a.freq[list_peak[warp][e]], __drcp_rn(den));
            const double y = __dmul_rn(__dsub_rn(u, a.f0_min), a.kt);
            const double x = __dadd_rn(y, a.cshift);
            // |x| < 2^28 exactly when the biased exponent is below 1023 + 28
            if (((__double_as_longlong(x) >> 52) & 0x7FF) >= 1051) ev |= kErrRange;
            const double cc = __dmul_rn(__dsub_rn(a.t[i], a.t_ref), a.kt);
            const int64_t dr = floor_times_2p32(__dmul_rn(a.step_ref, cc));
            // start of the stripe on row r0, its cell 0 at start 1 - K
            int64_t X = floor_times_2p32(x) - (a.S0[i] + j_off * a.D[i]) -
                        (int64_t)r0 * dr + ((int64_t)(K - 1) - lo_cell) * 4294967296LL;
            int32_t *h = hist + d * nr * E;
            for (int r = 0; r < nr; ++r, X -= dr, h += E) {
                const int32_t L = (int32_t)(X >> 32);
                if ((uint32_t)L < (uint32_t)E) atomicAdd(h + L, 1);
            }
        }
        __syncwarp();
    };

    const double absmax = fabs(__dmul_rn((double)(a.n_rows - 1), a.step_ref));
    int listed = 0;
    for (int base = f_begin + 32 * warp; base < f_end; base += kRefThreads) {
        const int i = base + lane;
        int64_t p = 0, p_end = 0;
        if (i < f_end) {
            // the refined drift and its range check, as the shift tables form them
            const double cc = __dmul_rn(__dsub_rn(a.t[i], a.t_ref), a.kt);
            if (!(fabs(cc) * absmax < (double)kFixedLimit)) ev |= kErrRange;
            const int64_t dr = floor_times_2p32(__dmul_rn(a.step_ref, cc));
            const int64_t s0r = a.S0[i] + j_off * a.D[i] + lo_cell * 4294967296LL;
            const int64_t last = (int64_t)(a.n_rows - 1) * dr;
            // the band's two ends in half cells from f0_min: the cells below and above
            // the extreme shifts, (1 - K) - 1 and (2 K + 1) + 1, less 0.5 - 0.5 K (in 64
            // bits: a row far outside the plan's shifts by up to 2^31 cells)
            const int64_t x_lo = (s0r + (last < 0 ? last : 0)) >> 32;
            const int64_t x_hi = ((s0r + (last > 0 ? last : 0)) >> 32) + 1;
            const double u_lo = __fma_rn((double)(2 * x_lo - K - 1), a.half_inv_kt, a.f0_min);
            const double u_hi = __fma_rn((double)(2 * x_hi + 5 * K + 3), a.half_inv_kt, a.f0_min);
            const float vx = (float)a.v[3 * (int64_t)i], vy = (float)a.v[3 * (int64_t)i + 1],
                        vz = (float)a.v[3 * (int64_t)i + 2];
            float lo32 = 0.f, hi32 = 0.f;
            for (int d = 0; d < nd; ++d) {
                const float vn =
                    vx * sky32[3 * d] + vy * sky32[3 * d + 1] + vz * sky32[3 * d + 2];
                lo32 = d ? fminf(lo32, vn) : vn;
                hi32 = d ? fmaxf(hi32, vn) : vn;
            }
            // the sum of three products of rounded factors is off by less than
            // 4 x 2^-23 of the sum of their magnitudes (|n| <= 1.000001)
            const float wide = 5e-7f * (fabsf(vx) + fabsf(vy) + fabsf(vz)) + 1e-37f;
            const double g_lo = 1.0 + (double)(lo32 - wide), g_hi = 1.0 + (double)(hi32 + wide);
            double f_lo, f_hi;
            if (__double2hiint(u_lo) > 0 && __double2hiint(g_lo) > 0) {  // all positive
                f_lo = u_lo * g_lo;
                f_hi = u_hi * g_hi;
            } else {
                f_lo = fmin(fmin(u_lo * g_lo, u_lo * g_hi), fmin(u_hi * g_lo, u_hi * g_hi));
                f_hi = fmax(fmax(u_lo * g_lo, u_lo * g_hi), fmax(u_hi * g_lo, u_hi * g_hi));
            }
            // (frequencies are positive: their bits order as they do)
            const long long b_lo = __double_as_longlong(f_lo), b_hi = __double_as_longlong(f_hi);
            const long long *fb = reinterpret_cast<const long long *>(a.freq);
            p = a.offsets[i];
            p_end = a.offsets[i + 1];
            int64_t b = p_end;
            while (p < b) {  // first peak with f >= f_lo
                const int64_t m = (p + b) >> 1;
                if (fb[m] < b_lo) p = m + 1; else b = m;
            }
            int64_t e = p;
            b = p_end;
            while (e < b) {  // first peak with f > f_hi
                const int64_t m = (e + b) >> 1;
                if (fb[m] <= b_hi) e = m + 1; else b = m;
            }
            p_end = e;
        }
        // every lane lists one peak per turn
        for (;;) {
            const unsigned have = __ballot_sync(kFull, p < p_end);
            if (!have) break;
            if (listed + 32 > kRefList) {
                place(listed);
                listed = 0;
            }
            if (p < p_end) {
                const int k = listed + __popc(have & ((1u << lane) - 1u));
                list_fft[warp][k] = i;
                list_peak[warp][k] = p;
                ++p;
            }
            listed += __popc(have);
        }
    }
    place(listed);
    ev = (int32_t)__reduce_or_sync(kFull, (unsigned)ev);
    if (lane == 0 && ev) atomicOr(a.err, ev);
    __syncthreads();
    // into the candidate's starts (other shares of the FFTs add theirs)
    for (int w = threadIdx.x; w < words; w += kRefThreads) {
        const int n = hist[w];
        if (n) {
            const int d = w / (nr * E), rest = w - d * nr * E;
            atomicAdd(a.starts +
                          (((int64_t)blockIdx.x * a.n_dir + d0 + d) * a.n_rows + r0) * E + rest,
                      n);
        }
    }
}

struct PickArgs {
    const int32_t *starts;        // [cand][direction][row][3 K]
    const int32_t *cell, *row;
    int32_t n_rows, k_over, n_fft;
    int32_t cand0, dir0, n_dir;   // the launch's first candidate and directions
    int32_t *best;                // nullable: [cand] count, (direction, row), cell so far
    int32_t last;                 // no further directions: write the candidate
    double f0_min, kt, fdot_min, fdot_step, fdot_step_ref, p0;
    fh_candidate *out;
};

// One block per candidate: the best (count desc, direction asc, row asc, cell asc)
// of its refined maps.  A thread takes a (direction, row) at a time and slides a
// K-cell window of starts along its 2K + 1 cells (cell b counts the starts at
// b .. b + K - 1); later pairs and cells replace only by a larger count.
constexpr int kPickThreads = 256;
__global__ void __launch_bounds__(kPickThreads) refine_pick_kernel(const PickArgs a)
{
    let_next_start();
    wait_for_previous();
    __shared__ int32_t best_s[kPickThreads / 32][3];  // count, (direction, row), cell
    const int c = a.cand0 + blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int K = a.k_over, E = 3 * K, n = a.n_dir * a.n_rows;
    const int32_t *st = a.starts + (int64_t)blockIdx.x * n * E;
    int bc = -1, bq = 0x7fffffff, bb = 0x7fffffff;
    for (int q = threadIdx.x; q < n; q += kPickThreads) {
        const int32_t *h = st + (int64_t)q * E;
        int cnt = 0;
        for (int L = 0; L < K; ++L) cnt += h[L];
        for (int b = 0;; ++b) {
            if (cnt > bc) {
                bc = cnt;
                bq = a.dir0 * a.n_rows + q;
                bb = b;
            }
            if (b == 2 * K) break;
            cnt += h[b + K] - h[b];
        }
    }
    auto take = [&](int c2, int q2, int b2) {
        if (c2 > bc || (c2 == bc && (q2 < bq || (q2 == bq && b2 < bb)))) {
            bc = c2;
            bq = q2;
            bb = b2;
        }
    };
    for (int o = 16; o > 0; o >>= 1) {
        const int c2 = __shfl_down_sync(kFull, bc, o), q2 = __shfl_down_sync(kFull, bq, o),
                  b2 = __shfl_down_sync(kFull, bb, o);
        take(c2, q2, b2);
    }
    if (lane == 0) {
        best_s[warp][0] = bc;
        best_s[warp][1] = bq;
        best_s[warp][2] = bb;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < kPickThreads / 32; ++w) take(best_s[w][0], best_s[w][1], best_s[w][2]);
    if (a.best) {
        int32_t *m = a.best + 3 * (int64_t)c;
        if (a.dir0 > 0) take(m[0], m[1], m[2]);
        m[0] = bc;
        m[1] = bq;
        m[2] = bb;
    }
    if (!a.last) return;
    const int bd = bq / a.n_rows, bj = bq - bd * a.n_rows;
    fh_candidate r;
    r.subband = c;
    r.rank = 0;
    if (bc < 0) {
        r.dir = r.row = r.cell = r.count = -1;
        r.f0 = r.fdot = r.cr = 0.0;
    } else {
        const int cell = a.cell[c] - a.k_over + bb;
        r.dir = bd;
        r.row = bj;
        r.cell = cell;
        r.count = bc;
        r.f0 = __dadd_rn(a.f0_min, __ddiv_rn(__dadd_rn((double)cell, 0.5), a.kt));
        const double fdot_lo =
            __dadd_rn(a.fdot_min, __dmul_rn((double)(a.row[c] - 2), a.fdot_step));
        r.fdot = __dadd_rn(fdot_lo, __dmul_rn((double)bj, a.fdot_step_ref));
        const double np0 = __dmul_rn((double)a.n_fft, a.p0);
        const double sd = __dsqrt_rn(__dmul_rn(np0, __dsub_rn(1.0, a.p0)));
        r.cr = __ddiv_rn(__dsub_rn((double)bc, np0), sd);
    }
    a.out[c] = r;
}

}  // namespace

namespace fh {

int refine_impl(const fh_plan_desc &d, int n_sm, const fh_peakmap *pm,
                const double *v_over_c, const int32_t *cand_cell, const int32_t *cand_row,
                int32_t n_cand, const double *sky_ref, int32_t n_ref, int32_t k_fdot,
                fh_candidate *out, bool host_checks, cudaStream_t s)
{
    const double kt = (double)d.k_over * d.t_fft;
    const int32_t n = pm->n_fft;
    const int64_t np = pm->n_peaks;
    const int K = d.k_over;
    const int32_t n_rows = 4 * k_fdot;
    const double step_ref = d.fdot_step / (double)k_fdot;
    // the inputs are checked on the host, or (FH_CHECKS_DEVICE) by the kernels
    if (host_checks) {
        const int rc = validate_host_inputs(d, kt, pm, v_over_c, sky_ref, n_cand * n_ref);
        if (rc) return rc;
    }
    for (int32_t c = 0; c < n_cand; ++c)
        if ((int64_t)cand_cell[c] - K < -(int64_t(1) << 27) ||
            (int64_t)cand_cell[c] + K >= (int64_t(1) << 27) || cand_row[c] < -(1 << 27) ||
            cand_row[c] >= (1 << 27))
            return set_error(FH_ERR_RANGE, "candidate %d outside the plan's fixed-point range", c);

    Scratch sc(s);
    double *t = nullptr, *freq = nullptr, *v = nullptr, *sky = nullptr;
    int64_t *off = nullptr, *S0 = nullptr, *D = nullptr;
    int32_t *cc = nullptr, *cr = nullptr;
    cudaError_t e = cudaSuccess;
    e = sc.get(&t, (size_t)n);
    if (e == cudaSuccess) e = sc.get(&freq, (size_t)np);
    if (e == cudaSuccess) e = sc.get(&v, 3 * (size_t)n);
    if (e == cudaSuccess) e = sc.get(&sky, 3 * (size_t)n_cand * n_ref);
    if (e == cudaSuccess) e = sc.get(&off, (size_t)n + 1);
    int64_t *off_raw = nullptr;
    if (e == cudaSuccess && !host_checks) e = sc.get(&off_raw, (size_t)n + 1);
    if (e == cudaSuccess) e = sc.get(&S0, (size_t)n);
    if (e == cudaSuccess) e = sc.get(&D, (size_t)n);
    if (e == cudaSuccess) e = sc.get(&cc, (size_t)n_cand);
    if (e == cudaSuccess) e = sc.get(&cr, (size_t)n_cand);
    // A block's histogram of starts in shared memory: all directions and rows where
    // they fit in 40 KB, else groups of directions, else of rows.  In memory, the
    // starts of as many candidates and directions at a time as 1 GiB holds (and as
    // give a grid at most 65535 groups), or as half of that, and so on, where memory is
    // short.
    const int32_t E = 3 * K;
    const int64_t per_dir = (int64_t)n_rows * E, room = 40 * 1024 / 4;
    RefineArgs ra{};
    ra.rows_per = (int32_t)std::max<int64_t>(1, std::min<int64_t>(n_rows, room / E));
    const int64_t row_groups = (n_rows + ra.rows_per - 1) / ra.rows_per;
    // what is read back (the candidates, then the error word) and what starts at zero
    // beside it (largest |D|, stripe starts), in one block
    const size_t out_bytes = sizeof(fh_candidate) * (size_t)n_cand;
    int32_t dir_batch = 1, cand_batch = 1;
    size_t n_starts = 0;
    char *zero = nullptr;
    int32_t *best = nullptr;
    for (int64_t most = (int64_t)1 << 28; e == cudaSuccess; most /= 2) {
        dir_batch = (int32_t)std::max<int64_t>(
            1, std::min<int64_t>({n_ref, most / per_dir, 65535 / row_groups}));
        cand_batch = (int32_t)std::max<int64_t>(
            1, std::min<int64_t>(n_cand, most / (per_dir * dir_batch)));
        n_starts = (size_t)cand_batch * dir_batch * per_dir;
        e = sc.get(&zero, out_bytes + 64 + 4 * n_starts);
        if (e != cudaErrorMemoryAllocation || (dir_batch == 1 && cand_batch == 1)) break;
        cudaGetLastError();
        e = cudaSuccess;
    }
    ra.dirs_per = (int32_t)std::max<int64_t>(
        1, std::min<int64_t>(dir_batch, room / ((int64_t)ra.rows_per * E + 3)));  // + its sky
    if (e == cudaSuccess && dir_batch < n_ref) e = sc.get(&best, 3 * (size_t)n_cand);
    if (e != cudaSuccess) return cuda_error(e, "cudaMallocAsync (refinement)");
    fh_candidate *d_out = reinterpret_cast<fh_candidate *>(zero);
    int32_t *err = reinterpret_cast<int32_t *>(zero + out_bytes);
    unsigned long long *dmax = reinterpret_cast<unsigned long long *>(zero + out_bytes + 16);
    int32_t *starts = reinterpret_cast<int32_t *>(zero + out_bytes + 64);
    struct {
        void *dst;
        const void *src;
        size_t bytes;
    } cp[] = {{t, pm->t_fft, 8 * (size_t)n},
              {freq, pm->freq, 8 * (size_t)np},
              {v, v_over_c, 24 * (size_t)n},
              {sky, sky_ref, 24 * (size_t)n_cand * n_ref},
              {host_checks ? off : off_raw, pm->offsets, 8 * ((size_t)n + 1)},
              {cc, cand_cell, 4 * (size_t)n_cand},
              {cr, cand_row, 4 * (size_t)n_cand}};
    for (auto &x : cp)
        if (x.bytes && e == cudaSuccess)
            e = cudaMemcpyAsync(x.dst, x.src, x.bytes, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(zero, 0, out_bytes + 64 + 4 * n_starts, s);
    // coarse shift tables
    PrepArgs pa{};
    pa.offsets_in = host_checks ? nullptr : off_raw;  // sanitised into off by the checks
    pa.offsets_out = off;
    pa.validate = host_checks ? 0 : 1;
    pa.t = t;
    pa.v = v;
    pa.sky = sky;
    pa.n_fft = n;
    pa.n_dir = n_cand * n_ref;
    pa.n_fdot = d.n_fdot;
    pa.n_peaks = np;
    pa.t_ref = d.t_ref;
    pa.kt = kt;
    pa.fdot_min = d.fdot_min;
    pa.fdot_step = d.fdot_step;
    pa.S0 = S0;
    pa.D = D;
    pa.dmax = dmax;  // (not needed here)
    pa.err = err;
    if (e == cudaSuccess) e = launch_prep(pa, s);
    // device checks: every peak's frequency too (the positions below cover only
    // the peaks near each candidate, and the range searches need sorted FFTs)
    if (e == cudaSuccess && !host_checks)
        e = launch_validate_device_inputs(t, freq, off, v, sky, n, n_cand * n_ref, err, s);
    if (e != cudaSuccess) return cuda_error(e, "refinement set-up");
    // Refined maps are refused where a tile of 2 K + 1 cells with the guard of the
    // refined drift exceeds a block's shared memory.  (Looked at while the copies run, 4 us
    // in 3164 FFTs; they read the caller's page-locked arrays, so a refused call waits for
    // them.)
    {
        double m = 0.0;
        for (int32_t i = 0; i < n; ++i) {
            const double x = std::fabs(step_ref * ((pm->t_fft[i] - d.t_ref) * kt));
            if (x > m && x < 1e9) m = x;  // non-finite times are left to the checks
        }
        const int32_t guard = guard_for((unsigned long long)(m * 4294967296.0) + 4);
        int dev = 0;
        cudaGetDevice(&dev);
        if (transform_smem_bytes(2 * K + 1, K, FH_MODE_START, 16, guard) >
            (size_t)max_optin_smem(dev)) {
            e = cudaStreamSynchronize(s);
            return cuda_error(e != cudaSuccess ? e : cudaErrorInvalidValue,
                              "refined map in shared memory");
        }
    }
    const size_t smem = 4 * (size_t)ra.dirs_per * ((size_t)ra.rows_per * E + 3);
    // shares of the FFTs: two waves of four blocks per SM, at least a block's 256 each
    const int64_t blocks = (int64_t)std::min(n_cand, cand_batch) * row_groups *
                           ((dir_batch + ra.dirs_per - 1) / ra.dirs_per);
    const int64_t shares = std::max<int64_t>(
        1, std::min<int64_t>(8 * (int64_t)n_sm / blocks, (n + kRefThreads - 1) / kRefThreads));
    ra.ffts_per = (int32_t)(((n + shares - 1) / shares + 31) / 32 * 32);
    ra.t = t;
    ra.freq = freq;
    ra.v = v;
    ra.sky = sky;
    ra.offsets = off;
    ra.S0 = S0;
    ra.D = D;
    ra.cell = cc;
    ra.row = cr;
    ra.n_fft = n;
    ra.k_over = K;
    ra.n_rows = n_rows;
    ra.n_ref = n_ref;
    ra.f0_min = d.f0_min;
    ra.kt = kt;
    ra.t_ref = d.t_ref;
    ra.step_ref = step_ref;
    ra.cshift = 0.5 - 0.5 * (double)K;
    ra.half_inv_kt = 0.5 / kt;
    ra.starts = starts;
    ra.err = err;
    PickArgs pk{};
    pk.starts = starts;
    pk.cell = cc;
    pk.row = cr;
    pk.n_rows = n_rows;
    pk.k_over = K;
    pk.n_fft = n;
    pk.f0_min = d.f0_min;
    pk.kt = kt;
    pk.fdot_min = d.fdot_min;
    pk.fdot_step = d.fdot_step;
    pk.fdot_step_ref = step_ref;
    pk.p0 = d.p0;
    pk.out = d_out;
    pk.best = best;
    for (int32_t c0 = 0; c0 < n_cand; c0 += cand_batch)
        for (int32_t b0 = 0; b0 < n_ref; b0 += dir_batch) {
            const int32_t nc = std::min(cand_batch, n_cand - c0);
            if (c0 > 0 || b0 > 0) e = cudaMemsetAsync(starts, 0, 4 * n_starts, s);
            if (e != cudaSuccess) return cuda_error(e, "cudaMemsetAsync (refinement)");
            ra.cand0 = pk.cand0 = c0;
            ra.dir0 = pk.dir0 = b0;
            ra.n_dir = pk.n_dir = std::min(dir_batch, n_ref - b0);
            pk.last = b0 + ra.n_dir == n_ref;
            if (n > 0) {
                const unsigned groups =
                    (unsigned)((ra.n_dir + ra.dirs_per - 1) / ra.dirs_per * row_groups);
                dim3 grid(nc, (n + ra.ffts_per - 1) / ra.ffts_per, groups);
                launch_after(refine_kernel, grid, kRefThreads, smem, s, ra);
            }
            launch_after(refine_pick_kernel, nc, kPickThreads, 0, s, pk);
            e = cudaGetLastError();
            if (e != cudaSuccess) return cuda_error(e, "refinement");
        }
    std::vector<char> back(out_bytes + 4);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(back.data(), zero, back.size(), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_error(e, "refinement pick");
    std::memcpy(out, back.data(), out_bytes);
    int32_t h_err = 0;
    std::memcpy(&h_err, back.data() + out_bytes, 4);
    if (h_err) return device_error_code(h_err);
    return FH_OK;
}

}  // namespace fh
