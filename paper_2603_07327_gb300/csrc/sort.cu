// sort.cu -- digitizer back end: time sort of singles by 64-bit key, gather
// into time order, coincidence sorting (Sec. 2.3 timing window).
//
// Keys are (job << shift) | t_ps, with the job in the fewest high bits that
// number the launch's jobs (none for one job), so a batch of jobs sorts as
// independent segments and a single run sorts on the whole 64-bit time.  The
// transport writes them beside the records.  Runs whose decay times spread
// over buckets of at least kBucketMinPs sort by time buckets (below).  The rest
// -- very high activities, live launches, digitize-only runs -- take a
// least-significant-digit radix sort with 8-bit digits: one fused pass builds
// the eight digit histograms, a plan kernel drops the passes whose digit is the
// same for every key (high time bytes, unused job bits), and every remaining
// pass is one kernel (k_onesweep: tiles claimed in order, each tile's digit
// offsets from the global histogram and a decoupled look-back over the tiles
// before it: the published one-sweep radix sort of Adinets and Merrill, 2022, on
// the single-pass scan of Merrill and Garland, 2016).  Stable ranks inside a tile come from the lanes of a warp with the
// same digit (the intersection of bit-plane ballots), in input order.  A pass's
// input tiles are streamed into shared memory by the bulk-copy engine
// (cp.async.bulk completing on an mbarrier), one tile ahead of the tile being
// ranked.  (The allocation-free sort is a kernel of its own, sort_noalloc.cu.)
// The element count is read on the device, so the whole chain is enqueued
// without a host round trip.
#include "internal.h"

namespace gpet {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 16;
constexpr int kTile = kSortThreads * kSortItems;  // 4096 keys per tile
constexpr int kPasses = 8;
static_assert(kSortThreads == 256, "one thread per 8-bit digit in the pass's prefix step");

__device__ __forceinline__ unsigned long long sort_n(const SortDev &S) {
    const unsigned long long n = *S.n_in;
    return n < S.cap ? n : S.cap;
}

// Values (the identity permutation) and the eight digit histograms of the
// keys (smem, then global atomics).  The keys themselves were written by the
// transport's finish event, next to each single's record.
__global__ void __launch_bounds__(kSortThreads) k_make_keys(SortDev S) {
    after_previous();
    __shared__ uint32_t h[kPasses][256];
    for (int i = threadIdx.x; i < kPasses * 256; i += blockDim.x) (&h[0][0])[i] = 0;
    __syncthreads();
    const unsigned long long n = sort_n(S);
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const uint64_t key = __ldg(S.keys[0] + i);
        S.vals[0][i] = (uint32_t)i;
#pragma unroll
        for (int p = 0; p < kPasses; ++p) atomicAdd(&h[p][(key >> (8 * p)) & 0xFF], 1u);
    }
    // the first active pass's look-back words (each pass clears the next one's)
    if (S.lb[0]) {
        const unsigned long long words = (n + kTile - 1) / kTile * 256;
        for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < words;
             i += (unsigned long long)gridDim.x * blockDim.x)
            S.lb[0][i] = 0ull;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kPasses * 256; i += blockDim.x) {
        const uint32_t v = (&h[0][0])[i];
        if (v) atomicAdd(S.ghist + i, v);
    }
}

// which passes run, and which buffer each one reads (one warp per pass)
__global__ void __launch_bounds__(kPasses * 32) k_plan(SortDev S) { after_previous(); plan_passes(S, sort_n(S)); }

// Tile of a radix pass in shared memory.  Ranks come in (warp, round, lane) order, which
// is input order.  The tile is first rebuilt in shared memory in digit order,
// then written out from there: consecutive threads write consecutive slots of
// one digit's run, so the global stores coalesce (a direct store from the
// ranking registers would send each of a warp's 32 keys to its own sector).
struct ScatterSmem {
    uint64_t keys[kTile];
    uint32_t vals[kTile];
    uint32_t wh[kSortThreads / 32][256];
    uint32_t gdelta[256];   // global run start - local run start (mod 2^32)
    uint32_t sw[32];
};
// Staged form: while a tile is ranked and written, the bulk-copy engine
// streams the CTA's next tile (keys and indices) into shared memory, so each
// CTA keeps 48 KB of reads in flight through all of its tile's work instead
// of waiting for its loads at the start of every tile.
struct ScatterStage {
    uint64_t keys[kTile];
    uint32_t vals[kTile];
    unsigned long long bar;  // mbarrier: the copy of the staged tile has landed
};
constexpr size_t kScatterSmemStaged = sizeof(ScatterSmem) + sizeof(ScatterStage);
constexpr uint32_t kStageBytes = kTile * (sizeof(uint64_t) + sizeof(uint32_t));
static_assert(sizeof(ScatterSmem) % 16 == 0, "staging buffer must start on a 16-byte boundary");
static_assert((kTile * sizeof(uint32_t)) % 16 == 0 && (kTile * sizeof(uint64_t)) % 16 == 0,
              "bulk copies move multiples of 16 bytes");
// mbarrier waits give up after this many polls (each poll may suspend the
// thread for a bounded time); a tile copy that never lands is reported, not
// waited for forever
constexpr int kStageWaitPolls = 1 << 22;

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ bool stage_wait(uint32_t bar, uint32_t parity) {
    for (int it = 0; it < kStageWaitPolls; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// one thread: expect the tile's bytes on the barrier, start both copies
__device__ __forceinline__ void stage_issue(ScatterStage &sg, const uint64_t *kin, const uint32_t *vin,
                                            unsigned long long t) {
    const uint32_t bar = smem_addr(&sg.bar);
    // the staging buffer was last read by ordinary loads; order them before
    // the copy engine's writes
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(kStageBytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_addr(sg.keys)), "l"(kin + t * kTile), "r"((uint32_t)(kTile * sizeof(uint64_t))), "r"(bar)
        : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_addr(sg.vals)), "l"(vin + t * kTile), "r"((uint32_t)(kTile * sizeof(uint32_t))), "r"(bar)
        : "memory");
}

// Decoupled look-back words of the one-sweep passes: the kind in the top two
// bits (a tile's own count of a digit, or the count of that digit over all
// tiles up to and including it), the count below.  A word is written whole
// (one aligned 64-bit store), so a reader sees 0 or a complete word.
constexpr unsigned long long kLbAgg = 1ull << 62, kLbIncl = 2ull << 62, kLbCount = (1ull << 62) - 1ull;
__device__ __forceinline__ void lb_store(unsigned long long *p, unsigned long long v) {
    *reinterpret_cast<volatile unsigned long long *>(p) = v;
}
__device__ __forceinline__ unsigned long long lb_load(const unsigned long long *p) {
    return *reinterpret_cast<const volatile unsigned long long *>(p);
}

// One radix pass in one kernel (the simulation path): tiles are claimed in
// order from a counter; a tile's digit counts come from its own ranking, and
// its global run starts from the digits' bases (the global histogram) plus
// the counts of the tiles before it, found by looking back over their
// published words until an inclusive count.  Every tile a CTA waits on was
// claimed earlier by a running CTA, and waits only on tiles before it, so the
// waits end.  Tiles are staged into shared memory one ahead by the bulk-copy
// engine.
__global__ void __launch_bounds__(kSortThreads, 2) k_onesweep(SortDev S, int p) {
    after_previous();
    if (!S.plan[p]) return;
    extern __shared__ __align__(16) unsigned char scatter_raw[];
    ScatterSmem &sm = *reinterpret_cast<ScatterSmem *>(scatter_raw);
    ScatterStage &sg = *reinterpret_cast<ScatterStage *>(scatter_raw + sizeof(ScatterSmem));
    __shared__ uint32_t dbase[256];
    __shared__ uint32_t thist[256];  // the tile's own digit counts
    __shared__ unsigned long long tile_sh[2];  // the tile being sorted, the one claimed next
    const int src = S.plan[kPasses + p];
    const unsigned long long n = sort_n(S);
    const unsigned long long tiles = (n + kTile - 1) / kTile;
    const unsigned long long full_tiles = n / kTile;
    constexpr int kWarps = kSortThreads / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t *kin = src ? S.keys[1] : S.keys[0];
    const uint32_t *vin = src ? S.vals[1] : S.vals[0];
    uint64_t *kout = src ? S.keys[0] : S.keys[1];
    uint32_t *vout = src ? S.vals[0] : S.vals[1];
    unsigned long long *lbc = src ? S.lb[1] : S.lb[0];  // this pass's words
    unsigned long long *lbn = src ? S.lb[0] : S.lb[1];  // the next active pass's, cleared here
    {
        // the digits' bases: exclusive scan of this pass's global histogram
        uint32_t tot;
        dbase[threadIdx.x] = block_exscan(S.ghist[p * 256 + threadIdx.x], tot, sm.sw);
    }
    uint32_t parity = 0;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&sg.bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        const unsigned long long t0 = atomicAdd(S.tile_ctr + p, 1u);
        tile_sh[0] = t0;
        tile_sh[1] = tiles;
        if (t0 < full_tiles) stage_issue(sg, kin, vin, t0);
    }
    __syncthreads();
    for (;;) {
        const unsigned long long t = tile_sh[0];
        if (t >= tiles) break;
        for (int i = threadIdx.x; i < kWarps * 256; i += blockDim.x) (&sm.wh[0][0])[i] = 0;
        thist[threadIdx.x] = 0;
        const unsigned long long wb = t * kTile + (unsigned long long)w * (32 * kSortItems);
        uint64_t k[kSortItems];
        uint32_t v[kSortItems];
        uint32_t rank[kSortItems];
        if (t < full_tiles) {
            const bool ok = stage_wait(smem_addr(&sg.bar), parity);
            if (!__syncthreads_and(ok)) {
                if (threadIdx.x == 0) {
                    atomicOr(S.status, kStatusSortStall);
                    stage_wait(smem_addr(&sg.bar), parity);  // let the copy in flight land
                }
                return;
            }
            parity ^= 1u;
            const int lb = w * (32 * kSortItems) + lane;
#pragma unroll
            for (int j = 0; j < kSortItems; ++j) {
                k[j] = sg.keys[lb + j * 32];
                v[j] = sg.vals[lb + j * 32];
            }
        } else {
#pragma unroll
            for (int j = 0; j < kSortItems; ++j) {
                const unsigned long long i = wb + (unsigned long long)j * 32 + lane;
                k[j] = i < n ? __ldg(kin + i) : 0ull;
                v[j] = i < n ? __ldg(vin + i) : 0u;
            }
        }
        __syncthreads();  // the staging buffer is free and the histograms are cleared
        if (threadIdx.x == 0) {
            // claim the next tile and stream it in while this one is sorted
            const unsigned long long nt = atomicAdd(S.tile_ctr + p, 1u);
            tile_sh[1] = nt;
            if (nt < full_tiles) stage_issue(sg, kin, vin, nt);
        }
        // The tile's digit counts first, published before the ranking, so that
        // the tiles after it rarely find its word missing.
#pragma unroll
        for (int j = 0; j < kSortItems; ++j) {
            const unsigned long long i = wb + (unsigned long long)j * 32 + lane;
            if (i < n) atomicAdd(&thist[(uint32_t)((k[j] >> (8 * p)) & 0xFF)], 1u);
        }
        __syncthreads();
        unsigned long long *row = lbc + t * 256;
        const uint32_t cnt = thist[threadIdx.x];
        lb_store(row + threadIdx.x, (t == 0 ? kLbIncl : kLbAgg) | cnt);
#pragma unroll
        for (int j = 0; j < kSortItems; ++j) {
            const unsigned long long i = wb + (unsigned long long)j * 32 + lane;
            const bool ok = i < n;
            const uint32_t d = ok ? (uint32_t)((k[j] >> (8 * p)) & 0xFF) : 256u;
            uint32_t peers = kFullMask;
#pragma unroll
            for (int bit = 0; bit < 8; ++bit) {
                const uint32_t m = __ballot_sync(kFullMask, (d >> bit) & 1u);
                peers &= ((d >> bit) & 1u) ? m : ~m;
            }
            if (t >= full_tiles) {  // the last, partial tile: separate the lanes past the end
                const uint32_t m = __ballot_sync(kFullMask, d >> 8);
                peers &= (d >> 8) ? m : ~m;
            }
            const uint32_t before = (d < 256u) ? sm.wh[w][d] : 0u;
            rank[j] = before + __popc(peers & lane_lt());
            __syncwarp();
            if (d < 256u && (peers & lane_lt()) == 0) sm.wh[w][d] = before + __popc(peers);
            __syncwarp();
        }
        __syncthreads();
        uint32_t lstart;
        {
            const int d = threadIdx.x;  // kSortThreads == 256 digits
            uint32_t c = 0;
#pragma unroll
            for (int ww = 0; ww < kWarps; ++ww) {
                const uint32_t x = sm.wh[ww][d];
                sm.wh[ww][d] = c;
                c += x;
            }
            uint32_t tot;
            lstart = block_exscan(c, tot, sm.sw);
#pragma unroll
            for (int ww = 0; ww < kWarps; ++ww) sm.wh[ww][d] += lstart;
        }
        __syncthreads();
        // the tile in digit order in shared memory; its global offsets follow
#pragma unroll
        for (int j = 0; j < kSortItems; ++j) {
            const unsigned long long i = wb + (unsigned long long)j * 32 + lane;
            if (i < n) {
                const uint32_t lp = sm.wh[w][(uint32_t)((k[j] >> (8 * p)) & 0xFF)] + rank[j];
                sm.keys[lp] = k[j];
                sm.vals[lp] = v[j];
            }
        }
        // Look back: add the counts of the tiles before this one, eight words
        // per round trip, newest first, until an inclusive count.
        int fail = 0;
        {
            const int d = threadIdx.x;
            unsigned long long excl = 0;
            if (t > 0) {
                constexpr int kWin = 8;
                unsigned long long j = t;  // tiles [0, j) not yet added
                bool found = false;
                int polls = 0;
                while (!found && !fail) {
                    unsigned long long wv[kWin];
#pragma unroll
                    for (int q = 0; q < kWin; ++q)
                        wv[q] = (unsigned long long)q < j ? lb_load(lbc + (j - 1 - q) * 256 + d) : kLbIncl;
#pragma unroll
                    for (int q = 0; q < kWin; ++q) {
                        if (found || fail || (unsigned long long)q >= j) break;
                        unsigned long long x = wv[q];
                        while ((x >> 62) == 0) {
                            if (++polls > kLookbackPolls) { fail = 1; break; }
                            if (polls > 64) __nanosleep(64);
                            x = lb_load(lbc + (j - 1 - q) * 256 + d);
                        }
                        if (fail) break;
                        excl += x & kLbCount;
                        if ((x >> 62) == 2) found = true;
                    }
                    j = j > (unsigned long long)kWin ? j - kWin : 0;
                    if (j == 0 && !found) fail = 1;  // tile 0 always publishes an inclusive count
                }
                if (!fail) lb_store(row + d, kLbIncl | (excl + cnt));
            }
            sm.gdelta[d] = dbase[d] + (uint32_t)excl - lstart;
            lbn[t * 256 + d] = 0ull;
        }
        if (__syncthreads_or(fail)) {
            if (threadIdx.x == 0) {
                atomicOr(S.status, kStatusSortStall);
                if (tile_sh[1] < full_tiles) stage_wait(smem_addr(&sg.bar), parity);  // the copy in flight
            }
            return;
        }
        const unsigned long long rem = n - t * kTile;
        const int tn = rem < (unsigned long long)kTile ? (int)rem : kTile;
        bool stray = false;
        for (int i = threadIdx.x; i < tn; i += kSortThreads) {
            const uint64_t key = sm.keys[i];
            const uint32_t pos = sm.gdelta[(uint32_t)((key >> (8 * p)) & 0xFF)] + (uint32_t)i;
            if (pos < n) {
                kout[pos] = key;
                vout[pos] = sm.vals[i];
            } else {
                stray = true;  // an offset past the keys: reported, never written
            }
        }
        if (stray) atomicOr(S.status, kStatusSortStall);
        __syncthreads();
        if (threadIdx.x == 0) tile_sh[0] = tile_sh[1];
        __syncthreads();
    }
}

static cudaError_t scatter_smem_attr() {
    return ensure_dynamic_smem(reinterpret_cast<const void *>(k_onesweep), kScatterSmemStaged);
}

// ---------------------------------------------------------------------------
// Time buckets.  Decay times are uniform over a run's span (their model), so a
// linear map of the time spreads a job's singles evenly over its buckets, and
// the sort is four passes whatever the key's length, where the radix sort takes
// one per varying byte: count the buckets (each single keeps its rank of
// arrival there), turn the counts into first positions, place each single's
// index, and order each bucket by comparing its few singles with one another
// while they are gathered into the time-ordered arrays.  Keys order by time,
// then by arrival (the single's index), as the stable radix sort orders them.
// A bucket covers kBucketHistories histories' share of the span: up to about
// that many singles, 3 on average in a sweep ring.  With 32 histories the
// comparisons took 239 us for the 5.6 M singles of a sensitivity map; 32, 16 and 8
// of them: digitizer of 10 M pairs 134, 128 and 133 us (more counters), of 3 M in
// the h2r ring 159, 148 and 140, of 60 M 700, 697 and 723.  More than kBucketMax in one
// (times that are not uniform after all) sets kStatusBuckets, and the run is
// repeated with the radix passes.
// What bounds the passes is latency at 1e5 singles and the random accesses to
// counters and records beyond: 239 B of DRAM per single of 1.6e8 pairs, where the
// radix sort with 48-byte records moved 362.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t bucket_of(const SortDev &S, uint64_t key) {
    const int job = S.job_shift < 64 ? (int)(key >> S.job_shift) : 0;
    const uint64_t t = S.job_shift < 64 ? key & ((1ull << S.job_shift) - 1ull) : key;
    const uint64_t scale = __ldg(reinterpret_cast<const unsigned long long *>(&S.bjobs[job].scale));
    const uint2 fn = __ldg(reinterpret_cast<const uint2 *>(&S.bjobs[job].first));
    return fn.x + (uint32_t)min(__umul64hi(t, scale), (unsigned long long)(fn.y - 1u));
}

__global__ void __launch_bounds__(256) k_bucket_count(SortDev S) {
    after_previous();
    const unsigned long long n = sort_n(S), step = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long i0 = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += 4 * step) {
        uint32_t r[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {   // (four counters in flight per thread)
            const unsigned long long i = i0 + j * step;
            if (i < n) r[j] = atomicAdd(S.bstart + bucket_of(S, __ldg(S.keys[0] + i)), 1u);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned long long i = i0 + j * step;
            if (i < n) S.vals[0][i] = r[j];
        }
    }
}

// Sum of the totals of the tiles before `tile`, by its first warp: its own
// total is published, then the words of earlier tiles are read, 32 a round trip
// and newest first, to an inclusive sum; the tile's own inclusive sum follows.
// Tiles are claimed in order and wait only for earlier ones, so the waits end;
// false when a word did not come within the wait limit.
__device__ __forceinline__ bool warp_lookback(unsigned long long *words, uint32_t tile, uint32_t total, uint32_t &base) {
    const uint32_t lane = threadIdx.x & 31;
    if (lane == 0) lb_store(words + tile, (tile == 0 ? kLbIncl : kLbAgg) | total);
    base = 0;
    bool ok = true;
    for (uint32_t j = tile; j > 0 && ok;) {
        unsigned long long w = kLbIncl;   // (before tile 0: nothing)
        if (lane < j) {
            const unsigned long long *p = words + (j - 1 - lane);
            w = lb_load(p);
            for (int polls = 0; (w >> 62) == 0 && polls < kLookbackPolls; ++polls) {
                if (polls > 64) __nanosleep(64);
                w = lb_load(p);
            }
        }
        ok = !__any_sync(kFullMask, (w >> 62) == 0);
        const uint32_t incl = __ballot_sync(kFullMask, (w >> 62) == 2);
        const uint32_t last = incl ? (uint32_t)__ffs(incl) - 1u : 31u;
        base += __reduce_add_sync(kFullMask, lane <= last ? (uint32_t)(w & kLbCount) : 0u);
        j = incl ? 0u : j - 32u;
    }
    if (lane == 0 && tile > 0) lb_store(words + tile, kLbIncl | (unsigned long long)(base + total));
    return ok;
}

// bucket counts to first positions, in place (n_buckets + 1 of them): one pass,
// tiles in the order of a ticket, each tile's base by looking back
__global__ void __launch_bounds__(1024) k_bucket_scan(SortDev S) {
    after_previous();
    __shared__ uint32_t sw[32];
    __shared__ uint32_t tile_sh, base_sh;
    __shared__ int fail_sh;
    if (threadIdx.x == 0) tile_sh = (uint32_t)atomicAdd(S.bscan, 1ull);
    __syncthreads();
    const uint32_t tile = tile_sh, m = S.n_buckets + 1u;
    const uint64_t b = (uint64_t)tile * kBucketScanTile + 4u * threadIdx.x;
    uint32_t v[4], sum = 0, most = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        v[j] = b + j < m ? S.bstart[b + j] : 0u;
        sum += v[j];
        most = max(most, v[j]);
    }
    if (__syncthreads_or(most > kBucketMax) && threadIdx.x == 0) atomicOr(S.status, kStatusBuckets);
    uint32_t tot;
    uint32_t x = block_exscan(sum, tot, sw);
    if (threadIdx.x < 32) {
        uint32_t base = 0;
        const bool ok = warp_lookback(S.bscan + 1, tile, tot, base);
        if (threadIdx.x == 0) {
            if (!ok) atomicOr(S.status, kStatusSortStall);
            base_sh = base;
            fail_sh = !ok;
        }
    }
    __syncthreads();
    if (fail_sh) return;
    x += base_sh;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (b + j < m) S.bstart[b + j] = x;
        x += v[j];
    }
}

// each single's index to its bucket's next place, in order of arrival
__global__ void __launch_bounds__(256) k_bucket_place(SortDev S) {
    after_previous();
    const unsigned long long n = sort_n(S);
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t pos = S.bstart[bucket_of(S, __ldg(S.keys[0] + i))] + S.vals[0][i];
        if (pos < n) S.vals[1][pos] = (uint32_t)i;   // (always, unless the scan gave up)
    }
}

// Singles a CTA orders: the buckets that start in its stretch of positions.  Two
// a thread: the pass is a chain of dependent loads (index, key, bucket, record),
// so it wants many CTAs with few singles each.
constexpr int kBucketCta = 512;
constexpr int kBucketRoom = kBucketCta + (int)kBucketMax;

// a single, its sort key and its record from the transport, to place i of the
// time-ordered arrays
__device__ __forceinline__ void gather_one(const SortDev &S, uint64_t key, uint32_t slot, const SinglesDev &out,
                                           unsigned long long i) {
    const uint4 *r = reinterpret_cast<const uint4 *>(S.in_raw + slot);
    const uint4 a = __ldg(r), b = __ldg(r + 1);
    const bool jobs = S.job_shift < 64;
    out.t[i] = jobs ? key & ((1ull << S.job_shift) - 1ull) : key;
    out.job[i] = jobs ? (int32_t)(key >> S.job_shift) : 0;
    out.h[i] = ((uint64_t)a.y << 32) | a.x;
    out.unit[i] = (int32_t)a.z;
    out.panel[i] = (int32_t)a.w;
    out.e[i] = __uint_as_float(b.x);
    out.eraw[i] = __uint_as_float(b.y);
    out.doi[i] = __uint_as_float(b.z);
}

// first place at or after x where a bucket starts
__device__ __forceinline__ uint32_t bucket_edge(const SortDev &S, unsigned long long x, unsigned long long n) {
    if (x >= n) return (uint32_t)n;
    const uint32_t b = bucket_of(S, __ldg(S.keys[0] + S.vals[1][x]));
    const uint32_t s = S.bstart[b];
    return s == (uint32_t)x ? s : S.bstart[b + 1];
}

__global__ void __launch_bounds__(256) k_bucket_sort(SortDev S, SinglesDev out) {
    after_previous();
    __shared__ uint64_t key[kBucketRoom];
    __shared__ uint32_t idx[kBucketRoom];
    __shared__ uint32_t edge[2];
    const unsigned long long n = sort_n(S);
    // (a failed run hands nothing on: its arrays are not written)
    const bool failed = *reinterpret_cast<volatile int *>(S.status) & (kStatusBuckets | kStatusSortStall);
    if (blockIdx.x == 0 && threadIdx.x == 0) *out.n = failed ? 0ull : n;
    if (failed) return;
    for (unsigned long long x = (unsigned long long)blockIdx.x * kBucketCta; x < n; x += (unsigned long long)gridDim.x * kBucketCta) {
        if (threadIdx.x < 2) edge[threadIdx.x] = bucket_edge(S, x + threadIdx.x * kBucketCta, n);
        __syncthreads();
        const uint32_t p0 = edge[0], m = min(edge[1] - p0, (uint32_t)kBucketRoom);
        for (uint32_t i0 = threadIdx.x; i0 < m; i0 += 512) {
            const uint32_t i1 = i0 + 256;
            const uint32_t v0 = S.vals[1][p0 + i0], v1 = i1 < m ? S.vals[1][p0 + i1] : v0;
            const uint64_t k0 = __ldg(S.keys[0] + v0), k1 = __ldg(S.keys[0] + v1);
            idx[i0] = v0;
            key[i0] = k0;
            if (i1 < m) {
                idx[i1] = v1;
                key[i1] = k1;
            }
        }
        __syncthreads();
        for (uint32_t i0 = threadIdx.x; i0 < m; i0 += 512) {
            uint32_t lo[2], hi[2], v[2];
            uint64_t k[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint32_t i = i0 + 256 * q < m ? i0 + 256 * q : i0;
                k[q] = key[i];
                v[q] = idx[i];
                const uint32_t b = bucket_of(S, k[q]);
                lo[q] = S.bstart[b] - p0;
                hi[q] = min(S.bstart[b + 1] - p0, m);
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t at = lo[q];
                for (uint32_t j = lo[q]; j < hi[q]; ++j) {
                    const uint64_t kj = key[j];
                    at += kj < k[q] || (kj == k[q] && idx[j] < v[q]);
                }
                lo[q] = at;
            }
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (i0 + 256 * q < m) gather_one(S, k[q], v[q], out, p0 + lo[q]);
        }
        __syncthreads();
    }
}

// singles into time order, after the radix passes
__global__ void k_gather(SortDev S, SinglesDev out) {
    after_previous();
    const unsigned long long n = sort_n(S);
    const int fin = S.plan[2 * kPasses];
    const uint32_t *perm = fin ? S.vals[1] : S.vals[0];
    const uint64_t *key = fin ? S.keys[1] : S.keys[0];
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        gather_one(S, key[i], perm[i], out, i);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *out.n = n;
}

// Coincidence sorting.  A cluster is a maximal run of time-sorted singles of
// one job whose consecutive gaps are <= window; windows never cross cluster
// ends, so each cluster is processed alone: the earliest unconsumed single opens
// [t0, t0 + window]; exactly two singles in different panels make a coincidence;
// all singles in the window are consumed.
// One pass over tiles of singles: a thread per cluster that begins in the tile
// replays it up to the tile's end, and one goes on with the cluster that reaches
// into the tile from the window that the tile before left open.  The work is then
// that of one walk over the singles however long a cluster is, and a tile waits
// for those before it only through the words that they leave it.  (Walking back to
// the cluster's start took 392 ms for one cluster of 9.5e5 singles, and with the
// square of the tiles more for larger ones; now 2.1 ms.)  The pairs found
// in the tile are written after those of the tiles before it, whose number comes
// by look-back.  (Flags, counts, a scan and the writes as kernels of their own
// took 41 us for 1.6e6 singles and 18 us for any small number.)
constexpr int kCoincThreads = 256, kCoincPer = 4, kCoincTile = kCoincThreads * kCoincPer;
static_assert(kCoincTile == (int)kCoincScanTile, "look-back words are allocated per tile");

// The first single of the window that the tile before left open (its word is that
// single's index + 1), or false when the word did not come within the wait limit.
// That tile is done or being worked on, and leaves the word after at most a walk
// over its singles and the same wait: tiles are claimed in order.
__device__ __forceinline__ bool wait_open(const uint32_t *word, uint32_t &a) {
    uint32_t w = *reinterpret_cast<const volatile uint32_t *>(word);
    for (int polls = 0; w == 0u && polls < kLookbackPolls; ++polls) {
        if (polls > 64) __nanosleep(64);
        w = *reinterpret_cast<const volatile uint32_t *>(word);
    }
    a = w - 1u;
    return w != 0u;
}

__global__ void __launch_bounds__(kCoincThreads) k_coinc(SinglesDev s, CoincDev C, int *status) {
    after_previous();
    __shared__ ClusterTile<kCoincThreads, kCoincTile> tl;
    __shared__ uint32_t flag[kCoincTile / 32];
    __shared__ uint32_t sw[32], tile_sh, base_sh;
    __shared__ int fail_sh;
    const uint32_t n = (uint32_t)*s.n, tiles = (n + kCoincTile - 1) / kCoincTile;
    for (;;) {
        if (threadIdx.x == 0) {
            tile_sh = (uint32_t)atomicAdd(C.scan, 1ull);
            fail_sh = 0;
        }
        if (threadIdx.x < kCoincTile / 32) flag[threadIdx.x] = 0;
        __syncthreads();
        const uint32_t tile = tile_sh;
        if (tile >= tiles) break;
        const uint32_t lo = tile * kCoincTile, hi = min(lo + kCoincTile, n);
        tl.load(s, C.window_ps, lo, n);
        auto linked = [&](uint32_t i) { return tl.linked(s, C.window_ps, lo, n, i); };
        // the clusters that begin in the tile, and the one that reaches into it
        const uint32_t before = linked(lo) ? 1u : 0u;
        for (uint32_t c = threadIdx.x; c < tl.n_start + before; c += kCoincThreads) {
            // the window's first single, and the first one of the tile that may lie beyond the window
            uint32_t a = lo, b = lo;
            if (c < tl.n_start) {
                a += tl.start[c];
                b = a + 1u;
            } else if (!wait_open(C.open + tile - 1u, a)) {
                fail_sh = 1;
                break;
            }
            const int job = tl.job[b - lo];
            const uint64_t W = __ldg(C.window_ps + job);
            for (;;) {
                // (the singles of one job within W of a are those that follow it up to some place)
                const uint64_t ta = tl.time(s, lo, a);
                auto within = [&](uint32_t i) { return tl.job_of(s, lo, n, i) == job && tl.time(s, lo, i) - ta <= W; };
                if (a >= lo && within(a + 1u) && !within(a + 2u) && s.panel[a] != s.panel[a + 1u])
                    atomicOr(&flag[(a - lo) >> 5], 1u << ((a - lo) & 31));
                // the place by steps that double, then halve: most windows hold two singles, some a thousand
                uint32_t step = 1;
                while (b + step <= hi && within(b + step - 1u)) {
                    b += step;
                    step *= 2u;
                }
                while (step /= 2u)
                    if (b + step <= hi && within(b + step - 1u)) b += step;
                if (!linked(b)) break;   // the cluster's end
                if (b == hi) {           // the tile's: the window is the next one's to go on with
                    *reinterpret_cast<volatile uint32_t *>(C.open + tile) = a + 1u;
                    break;
                }
                a = b++;
            }
        }
        __syncthreads();
        if (fail_sh) {
            if (threadIdx.x == 0) atomicOr(status, kStatusSortStall);
            break;
        }
        uint32_t f = (flag[threadIdx.x * kCoincPer >> 5] >> (threadIdx.x * kCoincPer & 31)) & ((1u << kCoincPer) - 1u);
        uint32_t tot;
        uint32_t at = block_exscan(__popc(f), tot, sw);
        if (threadIdx.x < 32) {
            uint32_t base = 0;
            const bool ok = warp_lookback(C.scan + 1, tile, tot, base);
            if (threadIdx.x == 0) {
                if (!ok) atomicOr(status, kStatusSortStall);
                if (ok && hi == n) *C.n = base + tot;
                base_sh = base;
                fail_sh = !ok;
            }
        }
        __syncthreads();
        if (fail_sh) break;
        at += base_sh;
        for (; f; f &= f - 1) {
            const int32_t a = (int32_t)(lo + threadIdx.x * kCoincPer + __ffs(f) - 1);
            C.a[at] = a;
            C.b[at++] = a + 1;
        }
    }
}

// Per-job statistics of a (batched) run: start of each job's segment in the
// time-sorted singles and in the coincidences (both are ordered by job, the
// high bits of the sort key), and the job's hit count from its tallies.
// One warp searches each of the two (32 probes a round: 4 dependent loads for
// 1e6 singles where a bisection by one thread takes 20) while the others sum.
template <class JobOf>
__device__ __forceinline__ unsigned long long warp_lower_bound(unsigned long long n, int j, JobOf job_of) {
    unsigned long long lo = 0, hi = n;   // first i with job_of(i) >= j lies in [lo, hi]
    while (lo < hi) {
        const unsigned long long step = (hi - lo + 32) / 33;
        const unsigned long long p = lo + step * ((threadIdx.x & 31) + 1) - 1;
        const uint32_t below = __popc(__ballot_sync(kFullMask, p < hi && job_of(p) < j));
        const unsigned long long l = lo + step * below, h = l + step - 1;
        hi = below == 32 || h > hi ? hi : h;
        lo = l < hi ? l : hi;
    }
    return lo;
}

// (the tallies in slices: one block per job took 11 us for 67 k crystals, eight
// and a ninth for the segments take 4)
constexpr int kStatsSlices = 8;
__global__ void __launch_bounds__(1024) k_job_stats(SinglesDev s, CoincDev C, JobStatsDev J) {
    after_previous();
    const int j = blockIdx.x;
    if (blockIdx.y == kStatsSlices) {
        const unsigned long long ns = *s.n, nc = *C.n;
        const int wid = threadIdx.x >> 5;
        if (wid == 0) {   // first coincidence whose first single has job >= j
            const unsigned long long lo = j == 0 ? 0 : warp_lower_bound(nc, j, [&](unsigned long long i) { return s.job[C.a[i]]; });
            if (threadIdx.x == 0) J.c_off[j] = lo;
        } else if (wid == 1) {   // first single with job >= j
            const unsigned long long lo = j == 0 ? 0
                                          : J.bjobs ? J.bstart[J.bjobs[j].first]
                                                    : warp_lower_bound(ns, j, [&](unsigned long long i) { return s.job[i]; });
            if (threadIdx.x == 32) J.s_off[j] = lo;
        }
        if (threadIdx.x == 0 && j == J.n_jobs - 1) {
            J.s_off[J.n_jobs] = ns;
            J.c_off[J.n_jobs] = nc;
        }
        return;
    }
    // hits of job j = sum of its per-crystal counts (hits is cleared before a run)
    unsigned long long acc = 0;
    const unsigned long long *t = J.tally_count + J.tally_off[j];
    const long long nt = J.tally_n[j];
#pragma unroll 8
    for (long long i = (long long)blockIdx.y * 1024 + threadIdx.x; i < nt; i += 1024 * kStatsSlices) acc += t[i];
    __shared__ unsigned long long red[32];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFullMask, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = red[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFullMask, acc, o);
        if (threadIdx.x == 0 && acc) atomicAdd(J.hits + j, acc);
    }
}

cudaError_t launch_job_stats(const SinglesDev &s, const CoincDev &C, const JobStatsDev &J, cudaStream_t st) {
    return launch_next(k_job_stats, dim3(J.n_jobs, kStatsSlices + 1), 1024, 0, st, s, C, J);
}

cudaError_t launch_sort_coinc(const SortDev &S, const SinglesDev &out, const CoincDev &C, int sm_count,
                              cudaStream_t st) {
    // the staged passes report a stalled copy or look-back in the status word
    if (!S.status || !S.lb[0] || !S.lb[1] || !S.tile_ctr) return cudaErrorInvalidValue;
    cudaError_t e = scatter_smem_attr();
    if (e != cudaSuccess) return e;
    const int grid = sm_count * 4;
    if (S.n_buckets) {
        const unsigned long long want = (S.cap + kBucketCta - 1) / kBucketCta;
        const int bg = (int)(want < (unsigned long long)sm_count * 8 ? want : (unsigned long long)sm_count * 8);
        e = launch_next(k_bucket_count, bg, 256, 0, st, S);
        if (e == cudaSuccess) e = launch_next(k_bucket_scan, (S.n_buckets + kBucketScanTile) / kBucketScanTile, 1024, 0, st, S);
        if (e == cudaSuccess) e = launch_next(k_bucket_place, bg, 256, 0, st, S);
        if (e == cudaSuccess) e = launch_next(k_bucket_sort, bg, 256, 0, st, S, out);
    } else {
        e = cudaMemsetAsync(S.ghist, 0, sizeof(uint32_t) * kPasses * 256, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(S.tile_ctr, 0, sizeof(unsigned int) * kPasses, st);
        if (e != cudaSuccess) return e;
        e = launch_next(k_make_keys, sm_count * 4, kSortThreads, 0, st, S);
        if (e == cudaSuccess) e = launch_next(k_plan, 1, kPasses * 32, 0, st, S);
        // two CTAs per SM are resident; more would only claim tiles later
        const int tg = (int)(S.max_tiles < (unsigned long long)sm_count * 2 ? (S.max_tiles ? S.max_tiles : 1)
                                                                            : (unsigned long long)sm_count * 2);
        for (int p = 0; p < kPasses && e == cudaSuccess; ++p)
            e = launch_next(k_onesweep, tg, kSortThreads, kScatterSmemStaged, st, S, p);
        if (e == cudaSuccess) e = launch_next(k_gather, grid, 256, 0, st, S, out);
    }
    if (e != cudaSuccess) return e;
    const unsigned long long ct = (S.cap + kCoincTile - 1) / kCoincTile;
    const int cg = (int)(ct < (unsigned long long)sm_count * 8 ? ct : (unsigned long long)sm_count * 8);
    return launch_next(k_coinc, cg, kCoincThreads, 0, st, out, C, S.status);
}

// load the digitizer's kernels and set their shared-memory limits (internal.h)
cudaError_t preload_sort_kernels() {
    const void *fns[] = {reinterpret_cast<const void *>(k_make_keys), reinterpret_cast<const void *>(k_plan),
                         reinterpret_cast<const void *>(k_onesweep), reinterpret_cast<const void *>(k_bucket_count),
                         reinterpret_cast<const void *>(k_bucket_scan), reinterpret_cast<const void *>(k_bucket_place),
                         reinterpret_cast<const void *>(k_bucket_sort),
                         reinterpret_cast<const void *>(k_gather), reinterpret_cast<const void *>(k_coinc),
                         reinterpret_cast<const void *>(k_job_stats)};
    cudaFuncAttributes fa;
    for (const void *f : fns) {
        const cudaError_t e = cudaFuncGetAttributes(&fa, f);
        if (e != cudaSuccess) return e;
    }
    return scatter_smem_attr();
}

}  // namespace gpet
