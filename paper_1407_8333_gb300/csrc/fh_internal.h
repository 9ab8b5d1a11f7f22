// Internal declarations of libfh (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "fh.h"

namespace fh {

// Spin-down rows per slab: one row per lane of a warp.  The transform's
// shared-memory histogram is laid out [cell][row] with a row stride of 32
// words, so lane l (row l) always hits bank l and the +1 atomics of one warp
// instruction never conflict, wherever the 32 stripes start.
constexpr int kRows = 32;
constexpr int kMaxBatchJobs = 12;
constexpr int64_t kFixedLimit = int64_t(1) << 28;  // |cells| bound for 32.32 fixed point
// window table entry of an FFT whose window start or count does not fit 16 bits:
// the transform looks that window up by binary search instead
constexpr uint32_t kWinLookup = 0xFFFFFFFFu;

// error bits written by the device-side input checks
enum : int32_t { kErrUnsorted = 1, kErrRange = 2, kErrInvalid = 4, kErrCsr = 8 };

#ifdef __CUDACC__
// floor(x 2^32) for |x| < 2^28, exactly: x = m 2^(e - 1075) with m the
// significand (hidden bit included for normal numbers), so x 2^32 =
// m 2^(e - 1043), a left shift by at most 7 bits, or a right shift whose
// discarded bits round a negative value down.  Out-of-range inputs give some
// value; the caller flags them.
__device__ __forceinline__ int64_t floor_times_2p32(double x)
{
    const uint64_t bits = (uint64_t)__double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7FF);
    const uint64_t m = (bits & 0xFFFFFFFFFFFFFull) | (ex ? (uint64_t(1) << 52) : 0);
    const int sh = (ex ? ex : 1) - 1043;
    uint64_t q;
    bool frac;
    if (sh >= 0) {
        q = m << (sh < 10 ? sh : 10);
        frac = false;
    } else {
        const int rs = -sh;
        q = rs < 64 ? m >> rs : 0;
        frac = rs < 64 ? (m & ((uint64_t(1) << rs) - 1)) != 0 : m != 0;
    }
    return (bits >> 63) ? -(int64_t)q - (frac ? 1 : 0) : (int64_t)q;
}

// Programmatic dependent launch: a kernel launched by launch_after may be set up, and
// its blocks become resident, while the kernel before it on the stream drains;
// wait_for_previous(), before its first access to memory, holds it until that one has
// completed (and so, as every kernel of a chain waits, all before it).  The first
// kernel of a chain is launched plainly and has no wait.  A kernel that calls
// let_next_start() allows its successor in once all its own blocks have got there.
// Without a kernel before it, or in a plain launch, both do nothing.
// The read-only path (__ldg, const __restrict__ parameters) is for data that no kernel
// writes while the reader is resident: the caller's inputs, and for the transform the
// correction's output too, because the window pre-pass lets it in only after its own
// wait (without a pre-pass it is launched plainly).  What the kernel just before, or
// one that it overlaps, writes is read by ordinary loads.
// Worth 1 - 2 us per launch of a chain: a step of four kernels on 200 FFTs
// 45.2 -> 42.6 us, the selection and vetoes of 150 days (13 launches) 262 -> 250,
// clustering and coincidences of 10^5 candidates (30 launches) 560 -> 513.
__device__ __forceinline__ void wait_for_previous()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void let_next_start()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... Q>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                         Q &&...args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
#endif

// One direction set of one plan, as the transform kernel sees it.
struct TransformJob {
    const int64_t *A;        // positions, [dir][n_peaks] (absolute directions)
    const int64_t *offsets;  // n_fft + 1, valid CSR
    const int64_t *S0;       // n_fft
    const int64_t *D;        // n_fft
    uint64_t *profile;       // [dir][n_f0] (absolute directions)
    int32_t *maps;           // nullable, [dir - dir_begin][n_fdot][n_f0]
    const unsigned long long *dmax;  // max_i |D_i| (32.32 cells per row), from a3
    const int32_t *err;      // the job's device error word: the unclamped walk, which
                             // trusts the peak windows (sorted positions), runs only
                             // while it is 0
    const int32_t *weights;  // nullable (plain map): adaptive integer weights, [dir][n_fft]
                             // (absolute directions); each update adds its FFT's weight
    int64_t count_bound;     // no count of the job's maps exceeds it
    const uint32_t *windows; // nullable: precomputed peak windows per
                             // [dir - dir_begin][slab][tile][fft], each the first peak
                             // relative to the FFT's first (low 16 bits) and the count
                             // (high 16 bits), or kWinLookup: looked up (binary search)
    int32_t *dense;          // nullable: set by the window pre-pass when some FFT has two
                             // peaks within one cell (the packed counters then do not
                             // apply: each direction of a pair is walked on its own)
    int32_t dir_pairs;       // 1: items cover directions 2u and 2u + 1 with two 16-bit
                             // counts per shared word (plain START map, every job of a
                             // launch alike); the window table is per pair
    int32_t *unit_delta;     // (dir_pairs) per absolute index of a pair's first direction, the
                             // largest cell distance between a peak's two positions (+2),
                             // from the window pre-pass (zeroed with the positions)
    int32_t delta_alloc;     // (dir_pairs) the part of the guard that holds that distance;
                             // a pair beyond it takes the clamped walk
    int32_t row_pairs;       // 1 (plain START map of one direction, not with dir_pairs):
                             // slabs of 64 rows, rows j0 + r and j0 + 32 + r in the low and
                             // high halves of one shared word; the window table is per
                             // 64-row slab and the guard holds 63 rows of drift
    int64_t n_peaks;
    int64_t item_begin;      // first work item of this job in the launch
    int64_t n_items;         // units * n_slabs * n_tiles
    int32_t n_fft, n_f0, n_fdot, k_over;
    int32_t tile_cells;      // W
    int32_t n_slabs, n_tiles;
    int32_t dir_begin, n_dir;
    // runs of FFTs of the transform's warps (launch_transform): warp w's first run is
    // [w run0, (w + 1) run0), run r >= warps the run1 FFTs from run_base + r run1
    int32_t run0, run1, run_base;
};

struct JobTable {
    int32_t n_jobs;
    TransformJob job[kMaxBatchJobs];
};

struct SelectArgs {
    const uint64_t *profile; // [dir][n_f0]
    fh_candidate *out;       // [dir - dir_begin][n_sb][top_k]
    int32_t n_f0, subband_cells, top_k, excl, sep, n_thr, n_sb;
    int32_t dir_begin, n_dir, n_fft;
    double f0_min, kt, fdot_min, fdot_step, p0;
    const int64_t *s1, *s2;  // nullable (plain map): per absolute direction, sums of the
                             // adaptive weights and of their squares
};

// ---- launchers (fh_kernels.cu); all return cudaGetLastError() ----
// Per-call set-up in one block: (a) if offsets_in is given, the sanitised
// CSR copy of it (clamped to [0, n_peaks], non-decreasing, first 0, last
// n_peaks; kErrCsr if anything changed); (b) the spin-down shift tables S0, D
// of every FFT and the largest |D| (atomicMax into *dmax, which starts at 0);
// (c) if validate: t finite and strictly increasing, |v| < 0.1 componentwise,
// sky components within 1.000001.
struct PrepArgs {
    const int64_t *offsets_in;  // device CSR to sanitise, or null (offsets_out already valid)
    int64_t *offsets_out;
    const double *t, *v, *sky;
    int32_t n_fft, n_dir, n_fdot, validate;
    int64_t n_peaks;
    double t_ref, kt, fdot_min, fdot_step;
    int64_t *S0, *D;
    unsigned long long *dmax;
    int32_t *err;
};
cudaError_t launch_prep(const PrepArgs &a, cudaStream_t s);
// a1 - a3 in one launch: prep's work (a.offsets_in sanitised into
// a.offsets_out, shift tables, checks) and the positions of every (direction,
// peak) of the peakmap described by a, frequencies freq
cudaError_t launch_correct(const PrepArgs &a, const double *freq, double f0_min,
                           int32_t k_over, int64_t *A, double *out_r, cudaStream_t s);

// fh_refine on the plan's grid d (host inputs, host output; synchronises)
int refine_impl(const fh_plan_desc &d, int n_sm, const fh_peakmap *pm, const double *v_over_c,
                const int32_t *cand_cell, const int32_t *cand_row, int32_t n_cand,
                const double *sky_ref, int32_t n_ref, int32_t k_fdot, fh_candidate *out,
                bool host_checks, cudaStream_t s);
// the error of a device error word (0: FH_OK)
int device_error_code(int32_t bits);
cudaError_t launch_validate_device_inputs(const double *t, const double *freq,
                                          const int64_t *offsets, const double *v,
                                          const double *sky, int32_t n_fft, int32_t n_dir,
                                          int32_t *err, cudaStream_t s);
// Guard cells kept below and above a tile so that, in the fast path, no
// update of a slab needs a bounds clamp: enough for a drift of span_rows (the
// slab's rows - 1) x max|D| cells.  guard_for(dmax, rows - 1) is what a job
// needs; a launch allocates one guard for all its jobs and jobs needing more
// take the clamped path.
__host__ __device__ int32_t guard_for(unsigned long long dmax, int32_t span_rows = kRows - 1);
// smem bytes the transform needs for tile width W (and mode)
size_t transform_smem_bytes(int32_t tile_cells, int32_t k_over, int32_t mode, int32_t nwarps,
                            int32_t guard);
// How many blocks of the transform kernel of a launch shape fit an SM with `smem`
// bytes each (below 1: not launchable).  The first use of a shape opts its kernel
// in to the device's largest dynamic shared memory (never less: other plans may be
// using the same kernel with more).  The cache belongs to one plan or server; it
// saves the driver calls of the shapes used last.
struct LaunchCache {
    struct Entry {
        int32_t shape = -1, blocks = 0;
        size_t smem = 0;
    } entry[8];
    int32_t next = 0;
};
int transform_blocks_per_sm(LaunchCache &cache, int32_t mode, int32_t nwarps, bool weighted,
                            int pack, bool maps, size_t smem);
// sched: null (every block takes every grid-th item) or two device words that
// are zero at the launch (a counter handing out items after each block's
// first, and a count of finished blocks); the kernel's last block zeroes them
// again, so launches on one stream can share them (not concurrent launches).
cudaError_t launch_transform(int32_t mode, const JobTable &tbl, int64_t total_items,
                             int32_t grid, int32_t nwarps, size_t smem, int32_t guard,
                             cudaStream_t s, unsigned int *sched = nullptr);
// Peak windows of every (direction, slab, tile, FFT) of a job, written to
// job.windows (the job's other fields as for the transform).
cudaError_t launch_windows(const TransformJob &job, uint32_t *windows, cudaStream_t s);
cudaError_t launch_select(const SelectArgs &a, cudaStream_t s);
// Adaptive map's count bound: bound[d] += sum_i W[d][i] c_{d,i}, c_{d,i} = the
// most positions of FFT i (direction d) inside a half-open window of K cells
// (bound: n_dir words, zeroed by the caller).
cudaError_t launch_weight_bound(const int64_t *A, const int64_t *offsets, const int32_t *W,
                                int32_t n_fft, int32_t n_dir, int64_t n_peaks, int32_t k_over,
                                unsigned long long *bound, cudaStream_t s);
// binary64 multiply + add chains, grid blocks of 512 threads, 16 operations
// per thread per iteration
cudaError_t launch_fp64_bench(int32_t iters, int32_t grid, double *sink, cudaStream_t s);
cudaError_t launch_smem_atomic_bench(int32_t variant, int32_t iters, int32_t grid,
                                     unsigned long long *sink, cudaStream_t s);

// The pool that calls take their scratch from on the current device (fh_api.cu;
// null where it could not be made: the device's default pool serves then).
cudaMemPool_t scratch_pool();

// Device buffers of one call, taken stream-ordered and returned stream-ordered
// when the object goes out of scope.
struct Scratch {
    cudaStream_t s;
    cudaMemPool_t pool;
    std::vector<void *> bufs;
    explicit Scratch(cudaStream_t st) : s(st), pool(scratch_pool()) {}
    Scratch(const Scratch &) = delete;
    Scratch &operator=(const Scratch &) = delete;
    template <typename T>
    cudaError_t get(T **p, size_t n)
    {
        void *q = nullptr;
        const size_t bytes = (n ? n : 1) * sizeof(T);
        const cudaError_t e = pool ? cudaMallocFromPoolAsync(&q, bytes, pool, s)
                                   : cudaMallocAsync(&q, bytes, s);
        if (e == cudaSuccess) bufs.push_back(q);
        *p = static_cast<T *>(q);
        return e;
    }
    ~Scratch()
    {
        for (void *b : bufs) cudaFreeAsync(b, s);
    }
};

// Exclusive scan of n int32 counts into pref[0 .. n] (fh_peakmap.cu).
template <typename T>
cudaError_t scan_exclusive(const int32_t *cnt, int64_t n, T *pref, Scratch &sc, cudaStream_t s);

// ---- host helpers (fh_api.cu) ----
int set_error(int code, const char *fmt, ...);
int cuda_error(cudaError_t e, const char *what);
int max_optin_smem(int device);
int32_t default_tile(const fh_plan_desc &d, int device, int32_t mode, int32_t nwarps,
                     int32_t guard);
// guard for a plan when the FFT times are not known on the host: the drift of
// a grid with fdot_step = 1/(T_FFT T_obs) over +-T_obs/2 is K/2 cells per row
int32_t default_guard(const fh_plan_desc &d);
// guard for FFT start times held in host memory (exact drift of the grid)
int32_t host_guard(const fh_plan_desc &d, double kt, const double *t, int32_t n_fft);
// the drift bounds behind those guards: max |D_i| in 32.32 cells per row
unsigned long long default_drift(const fh_plan_desc &d);
unsigned long long host_drift(const fh_plan_desc &d, double kt, const double *t, int32_t n_fft);
// Whether a plain START map of n_dir directions may pair them (two 16-bit
// counts per shared word): its stripe-start counts fit 16 bits by its size
// (n_fft < 2^16; the window pre-pass checks the peaks' spacing), its counts
// keep the reduction key below 2^31 (K n_fft < 2^25) and a tile fits with the
// guard of drift bound `drift` plus the pair allowance pair_delta(d).
bool pairs_apply(const fh_plan_desc &d, int device, int32_t n_fft, int32_t n_dir,
                 unsigned long long drift);
// Whether one direction (n_dir == 1) of a plain START map may pair the two
// 32-row halves of 64-row slabs in the counters' 16-bit halves: the same
// 16-bit and key conditions as for direction pairs, and a tile fits with the
// guard of 63 rows of drift.
bool rows_apply(const fh_plan_desc &d, int device, int32_t n_fft, int32_t n_dir,
                unsigned long long drift);
// Cells of guard kept for the distance between a peak's positions in the two
// directions of a pair: neighbouring directions of a sky grid at the Doppler
// resolution differ by about one input bin (K cells); 2 K + 4 leaves room.
int32_t pair_delta(const fh_plan_desc &d);
int validate_desc(const fh_plan_desc &d);
// host-memory inputs: CSR, ordering, finiteness and the 32.32 fixed-point range
int validate_host_inputs(const fh_plan_desc &d, double kt, const fh_peakmap *pm, const double *v,
                         const double *sky, int32_t n_dir);

}  // namespace fh
