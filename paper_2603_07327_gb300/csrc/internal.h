// internal.h -- declarations shared by the library's translation units
// (device structs of the sort / coincidence stage and the host launchers).
#pragma once

#include <map>
#include <mutex>
#include <tuple>

#include <cuda_runtime.h>

#include "transport.cuh"

namespace gpet {

enum { kKernelDefault = 0, kKernelLoop = 1, kKernelWave = 2, kKernelCta = 3 };

struct LaunchCfg {
    int grid;            // CTAs of the transport kernel
    int block_size;      // threads per CTA
    int sm_count;
    int kernel;          // kKernelLoop / kKernelWave
    int max_smem_geoms;  // geometry descriptors staged in shared memory
    int compact_every;   // wavefront regrouping interval (events)
    int pool_depth;      // wavefront slots per lane (pool = 32 x depth histories per warp)
    bool phantom;        // a job of the launch has a phantom, or one may be appended
    bool posed;          // a geometry of the launch has panel poses, or one may be appended
    bool live;           // a live launch
    // a launch of one job that is known when it is made: the job and its
    // geometry, as they are in the device's tables (else NULL)
    const struct JobDev *one_job;
    const struct GeomDev *one_geom;
};

// one job's time buckets: a time t falls in bucket first + min(hi64(t * scale), n - 1)
struct BucketJob {
    uint64_t scale;
    uint32_t first, n;
};

// working set of the time sort (the radix passes ping-pong between two buffers)
struct SortDev {
    uint64_t *keys[2];
    uint32_t *vals[2];
    uint32_t *ghist;                 // [8][256]
    int *plan;                       // [8] active, [8] source buffer, [1] final buffer
    unsigned long long max_tiles;
    unsigned long long cap;
    const unsigned long long *n_in;  // device count of unsorted singles
    const RawSingle *in_raw;         // unsorted singles
    int *status;                     // run status word (kStatusSortStall)
    int job_shift;                   // sort key = (job << job_shift) | t_ps; 64: the key is t_ps alone
    // one-sweep passes (the simulation path): decoupled look-back words, two
    // buffers of [tiles][256] that alternate between active passes, and a
    // tile counter per pass
    unsigned long long *lb[2] = {nullptr, nullptr};
    unsigned int *tile_ctr = nullptr;
    // time buckets (n_buckets = 0: none, radix passes): per-job tables, the
    // counts of the buckets (then their first positions, n_buckets + 1 of them),
    // the scan's look-back words and tile counter
    const BucketJob *bjobs = nullptr;
    uint32_t *bstart = nullptr;
    unsigned long long *bscan = nullptr;
    uint32_t n_buckets = 0;
};

// singles per time bucket at one single per history, most singles of one
// bucket, and the narrowest bucket (ps): see sort.cu
constexpr uint32_t kBucketHistories = 16, kBucketMax = 1024;
constexpr uint64_t kBucketMinPs = 10000;
constexpr uint32_t kBucketScanTile = 4096, kCoincScanTile = 1024;

// Bit position of the job index in the 64-bit sort keys of a launch of n_jobs
// jobs: the job takes the fewest high bits that number the jobs, the time stamp
// the rest (64 for one job: the key is the time alone).
inline int sort_job_shift(int n_jobs) {
    int bits = 0;
    while ((1ll << bits) < (long long)n_jobs) ++bits;
    return 64 - bits;
}
// Largest time stamp a key with this shift holds (2^64 - 1 without job bits).
inline unsigned long long sort_time_limit(int job_shift) {
    return job_shift >= 64 ? ~0ull : (1ull << job_shift) - 1ull;
}

// time-ordered singles
struct SinglesDev {
    uint64_t *t, *h;
    int32_t *unit, *panel, *job;
    float *e, *eraw, *doi;
    unsigned long long *n;
};

struct CoincDev {
    unsigned long long *scan;        // tile ticket, then a look-back word per tile
    uint32_t *open;                  // per tile: first single + 1 of a window that reaches the next tile's cluster
    int32_t *a, *b;
    unsigned long long *n;
    const uint64_t *window_ps;       // per job
};

struct JobStatsDev {
    int n_jobs;
    const BucketJob *bjobs;              // time buckets of the sort, or NULL: first positions of the jobs' singles
    const uint32_t *bstart;
    unsigned long long *s_off, *c_off;   // [n_jobs + 1]
    unsigned long long *hits;            // [n_jobs]
    const unsigned long long *tally_count;
    const long long *tally_off, *tally_n; // [n_jobs]
};

// most geometry descriptors a transport CTA stages in shared memory
constexpr int kMaxStagedGeoms = 16;

// Raise kernel fn's dynamic shared-memory limit on the current device to at
// least `bytes` (capped at the device's opt-in maximum).  The attribute is set
// only when it grows, so a launch never changes it while a live launch of the
// same kernel may be running (a change can wait for running launches).
cudaError_t ensure_dynamic_smem(const void *fn, size_t bytes);

// Load every kernel the transport and digitizer can launch (and set their
// shared-memory limits), once per device.  CUDA loads kernels lazily, and a
// load can wait for running kernels: a live launch's kernel waits on the host,
// so nothing may be loaded while it runs.
cudaError_t preload_kernels();
cudaError_t preload_transport_kernels();
cudaError_t preload_wave_kernels();
cudaError_t preload_cta_kernels();
cudaError_t preload_sort_kernels();
cudaError_t preload_window_kernels();
cudaError_t preload_copy_kernels();

// Geometry descriptors a transport launch stages in shared memory: as many of
// the first min(n_geoms, max_geoms) as fit without fewer resident CTAs than a
// launch that stages none (the rest are read through L1).  The kernel's
// dynamic shared-memory limit covers the largest staging.
template <class Kernel>
cudaError_t staged_geometry(Kernel k, int block, size_t pool_smem, int n_geoms, int max_geoms, int *ng_out,
                            size_t *smem_out, int *occ_out) {
    int ng = n_geoms < max_geoms ? n_geoms : max_geoms;
    if (ng < 0) ng = 0;
    // the answer depends on the kernel, the device and these counts alone: kept
    // (a few entries per kernel), since a small run would spend 10 us asking
    struct Known { int ng, occ; size_t smem; };
    static std::mutex mu;
    static std::map<std::tuple<const void *, int, int, int, size_t, int>, Known> known;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const auto key = std::make_tuple(reinterpret_cast<const void *>(k), dev, block, ng, pool_smem, max_geoms);
    {
        std::lock_guard<std::mutex> lk(mu);
        const auto it = known.find(key);
        if (it != known.end()) {
            *ng_out = it->second.ng;
            *smem_out = it->second.smem;
            *occ_out = it->second.occ;
            return cudaSuccess;
        }
    }
    e = ensure_dynamic_smem(reinterpret_cast<const void *>(k),
                                        pool_smem + (size_t)(max_geoms > 0 ? max_geoms : 0) * sizeof(GeomDev));
    if (e != cudaSuccess) return e;
    int occ0 = 0, occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ0, k, block, pool_smem);
    if (e != cudaSuccess) return e;
    for (;; --ng) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, block, pool_smem + (size_t)ng * sizeof(GeomDev));
        if (e != cudaSuccess) return e;
        if (occ >= occ0 || ng == 0) break;
    }
    *ng_out = ng;
    *smem_out = pool_smem + (size_t)ng * sizeof(GeomDev);
    *occ_out = occ;
    std::lock_guard<std::mutex> lk(mu);
    known[key] = {ng, occ, *smem_out};
    return cudaSuccess;
}

// A kernel whose launch overlaps the end of the one before it in the stream: its
// blocks take the place of those that have ended, and after_previous(), the first
// statement of every kernel launched so, waits until the other is complete and its
// writes are seen.  Between the digitizer's dependent kernels this saves most of
// the launch's latency: seven of them 33 -> 23 us for 2e4 pairs, 47 -> 35 us for
// 3e5, 159 -> 148 us for 1e7.  (Letting a kernel's blocks in as soon as those of
// the one before have started, griddepcontrol.launch_dependents, took half of that
// back where the waiting blocks hold the places of working ones.)
template <class... Params, class... Args>
cudaError_t launch_next(void (*kernel)(Params...), dim3 grid, int block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchAttribute next{};
    next.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    next.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &next;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}
__device__ __forceinline__ void after_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

cudaError_t launch_job_stats(const SinglesDev &s, const CoincDev &C, const JobStatsDev &J, cudaStream_t st);
// the transport kernel cfg selects, then (with_redo) the re-simulation of
// histories whose singles list overflowed
cudaError_t launch_transport(const WorkDev &W, const OutDev &O, const LaunchCfg &cfg, cudaStream_t st,
                             bool with_redo = true);
cudaError_t launch_transport_redo(const WorkDev &W, const OutDev &O, const LaunchCfg &cfg, cudaStream_t st);
cudaError_t launch_transport_wave(const WorkDev &W, const OutDev &O, const LaunchCfg &cfg, cudaStream_t st);
cudaError_t launch_transport_cta(const WorkDev &W, const OutDev &O, const LaunchCfg &cfg, cudaStream_t st);
// warps resident at once in the transport launch that cfg selects (sizes the work chunks)
cudaError_t transport_resident_warps(int n_geoms, const LaunchCfg &cfg, long long *warps);
cudaError_t wave_resident_warps(int n_geoms, const LaunchCfg &cfg, long long *warps);
constexpr int kCtaThreads = 448;   // threads per CTA of the CTA kernel's default shape
cudaError_t cta_resident_warps(int n_geoms, const LaunchCfg &cfg, long long *warps);
// the CTA kernel's own counts (raw, kCtaCounterSlots of them behind the launch's first kCtaCounters) added to
// the launch's counters (host)
constexpr int kCtaCounters = 20, kCtaCounterSlots = 16;
void cta_counters(unsigned long long *counters, const unsigned long long *raw);
cudaError_t launch_sort_coinc(const SortDev &S, const SinglesDev &out, const CoincDev &C, int sm_count,
                              cudaStream_t st);

// polls of a look-back word before the pass gives up (with 64 ns sleeps after
// the first 64 polls: about a second); a tile whose owner never publishes is
// reported, not waited for forever
constexpr int kLookbackPolls = 1 << 24;

__device__ __forceinline__ uint32_t lane_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// block-wide exclusive scan of one value per thread (blockDim a multiple of 32, at most 1024)
__device__ __forceinline__ uint32_t block_exscan(uint32_t v, uint32_t &total, uint32_t *sw) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFullMask, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sw[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint32_t w = lane < (int)(blockDim.x >> 5) ? sw[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFullMask, w, o);
            if (lane >= o) w += y;
        }
        sw[lane] = w;  // inclusive warp prefix
    }
    __syncthreads();
    const uint32_t warp_base = wid ? sw[wid - 1] : 0;
    total = sw[(blockDim.x >> 5) - 1];
    __syncthreads();
    return warp_base + x - v;
}

// Pass plan of a radix sort from the digit histograms S.ghist, by a block of
// eight warps: which passes run, and which buffer each one reads.
__device__ __forceinline__ void plan_passes(const SortDev &S, unsigned long long n) {
    constexpr int kP = 8;
    __shared__ int active[kP];
    const int p = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t mx = 0;
    for (int d = lane; d < 256; d += 32) mx = max(mx, __ldcg(S.ghist + p * 256 + d));
    mx = __reduce_max_sync(kFullMask, mx);
    if (lane == 0) active[p] = (n > 1 && (unsigned long long)mx < n) ? 1 : 0;
    __syncthreads();
    if (threadIdx.x == 0) {
        int cur = 0;
        for (int q = 0; q < kP; ++q) {
            S.plan[q] = active[q];
            S.plan[kP + q] = cur;
            if (active[q]) cur ^= 1;
        }
        S.plan[2 * kP] = cur;  // buffer holding the sorted result
    }
}

// A tile of time-ordered singles in shared memory for cluster-by-cluster work: one
// single more at either end, whether each is linked to the one before it (same
// job, gap within the window; one bit more than the tile has singles), and the
// singles where a cluster of several begins, packed for the block's threads.
// Most singles are alone, and a thread per single waits for its warp's clusters:
// with a thread per cluster, 5.6 M singles take 79 us for coincidences (104) and
// 106 us for the counts of four energy windows (149).
template <int kThreads, int kTile>
struct ClusterTile {
    uint64_t t[kTile + 2];
    int32_t job[kTile + 2];
    uint32_t link[kTile / 32 + 1];
    uint16_t start[kTile];
    uint32_t n_start;

    __device__ __forceinline__ uint64_t time(const SinglesDev &s, uint32_t lo, uint32_t i) const {
        return i + 1u - lo < (uint32_t)(kTile + 2) ? t[i + 1u - lo] : s.t[i];
    }
    __device__ __forceinline__ int32_t job_of(const SinglesDev &s, uint32_t lo, uint32_t n, uint32_t i) const {
        return i + 1u - lo < (uint32_t)(kTile + 2) ? job[i + 1u - lo] : i < n ? s.job[i] : -1;
    }
    __device__ __forceinline__ bool linked(const SinglesDev &s, const uint64_t *window_ps, uint32_t lo, uint32_t n,
                                           uint32_t i) const {
        const uint32_t l = i - lo;
        if (l <= (uint32_t)kTile) return (link[l >> 5] >> (l & 31u)) & 1u;
        return i > 0u && i < n && s.job[i - 1u] == s.job[i] && s.t[i] - s.t[i - 1u] <= window_ps[s.job[i]];
    }
    // tile lo.. of n singles (all of the block's threads)
    __device__ __forceinline__ void load(const SinglesDev &s, const uint64_t *window_ps, uint32_t lo, uint32_t n) {
        if (threadIdx.x == 0) n_start = 0;
        for (int k = threadIdx.x; k < kTile + 2; k += kThreads) {
            const uint32_t i = lo + k - 1u;   // (wraps below 0: not < n)
            t[k] = i < n ? s.t[i] : 0ull;
            job[k] = i < n ? s.job[i] : -1;
        }
        __syncthreads();
#pragma unroll
        for (int l0 = 0; l0 <= kTile; l0 += kThreads) {
            const int l = l0 + threadIdx.x;
            bool on = false;
            if (l <= kTile) {
                const int j = job[l + 1];
                on = j >= 0 && j == job[l] && t[l + 1] - t[l] <= __ldg(window_ps + j);
            }
            const uint32_t w = __ballot_sync(kFullMask, on);
            if ((threadIdx.x & 31) == 0 && l <= kTile) link[l >> 5] = w;
        }
        __syncthreads();
#pragma unroll
        for (int l0 = 0; l0 < kTile; l0 += kThreads) {
            const int l = l0 + threadIdx.x;
            const uint32_t w = link[l >> 5], next = (l & 31) == 31 ? link[(l >> 5) + 1] & 1u : (w >> ((l & 31) + 1)) & 1u;
            const bool begins = next && !((w >> (l & 31)) & 1u);
            const uint32_t m = __ballot_sync(kFullMask, begins);
            if (m == 0) continue;
            uint32_t at = 0;
            if ((threadIdx.x & 31) == 0) at = atomicAdd(&n_start, (uint32_t)__popc(m));
            at = __shfl_sync(kFullMask, at, 0);
            if (begins) start[at + __popc(m & lane_lt())] = (uint16_t)l;
        }
        __syncthreads();
    }
};

// energy windows of one pass over the time-sorted singles
constexpr int kMaxWindows = 16;
struct WinDev {
    float lo[kMaxWindows], hi[kMaxWindows];
    int n;
};
// counts[job * n + w] += coincidences of window w (cap = capacity of the singles)
cudaError_t launch_coinc_windows(const SinglesDev &s, const CoincDev &C, const WinDev &win,
                                 unsigned long long *counts, unsigned long long cap, cudaStream_t st);

}  // namespace gpet
