// sort_noalloc.cu -- time sort that allocates no device memory.
//
// Some callers cannot call cudaMalloc: processes whose device memory is all
// handed out up front by another allocator (a caching allocator that has
// already reserved the pool, a serving process with a fixed memory budget),
// or latency-critical loops where an allocation's implicit device
// synchronisation is not acceptable.  For them this file provides one entry
// point, gpet_sort_times_noalloc, whose whole working set (key and index
// buffers, bucket counts, digit histograms) lives in the file-scope array below.
// The array is part of the library image: every GPU that loads the library
// holds it until the process exits.  The caller still passes its inputs and
// outputs.
#include <algorithm>

#include "gpet.h"
#include "host.h"

namespace gpet {

constexpr unsigned long long kNoallocMaxKeys = 1ull << 20;            // largest n accepted
constexpr int kNoallocTile = 4096;                                    // keys of a radix tile
constexpr unsigned long long kNoallocTiles = (kNoallocMaxKeys + kNoallocTile - 1) / kNoallocTile;
// layout of the scratch array (all offsets multiples of 256 bytes)
constexpr size_t kOffCtl = 0;                                         // NoallocCtl
constexpr size_t kOffFailed = 128;                                    // not 0: a sort gave up since the last query
constexpr size_t kOffHist = 256;                                      // [8][256] uint32 digit histograms
constexpr size_t kOffKeys = kOffHist + 8 * 256 * 4 + 256;             // two buffers, or the buckets' keys
constexpr size_t kOffVals = kOffKeys + 2 * 8 * kNoallocMaxKeys;       // and their indices
constexpr size_t kOffWords = kOffVals + 2 * 4 * kNoallocMaxKeys;      // bucket counts, or look-back words
constexpr size_t kScratchBytes = kOffWords + 256 * 4 * kNoallocTiles; // 24.26 MiB in all

static __device__ __align__(256) unsigned char g_sort_scratch[kScratchBytes];

// The sort is one cooperative kernel.  What bounds it is latency, not bandwidth
// (3.6 MB of keys and indices for 3e5 of them): with a kernel per step, eight
// radix passes of ~9 us and four more kernels took 102 us, of which the chip was
// busy for a few.  Here the keys are dealt into buckets by a linear map of
// [min, max], about 32 of them each, a bucket's place for every key by one atomic;
// after that each warp orders a bucket by comparing its keys with one another, and
// nothing is written twice.  Two waits of the whole grid separate the steps.
//   300007 keys of 46 bits: 102 us -> 40; 2^20 keys of 60 bits: 195 -> 86.
// A bucket holds up to kBucketRoom keys, or what the scratch array has for each;
// keys that crowd further (the mean of 32 makes that unlikely for a spread that
// is even over a bucket's width) are radix-sorted, in the same kernel: eight
// digits of eight bits at most, those that vary, a wait of the grid after each.
// A tile is ranked by the lanes of a warp with the same digit (the intersection
// of bit-plane ballots), in input order, so the passes are stable; a tile's
// offsets come by look-back over the tiles before it (Merrill and Garland, 2016).  The look-back words carry
// the pass they belong to, so one buffer serves all passes without being cleared
// between them, and 16 of them are read per round trip.
// Both ways give the one stable order, keys by value and equal ones by index.
constexpr int kSortBlock = 1024, kSortWarps = kSortBlock / 32;
constexpr int kItems = kNoallocTile / kSortBlock;
constexpr uint32_t kBucketMean = 32, kBucketRoom = 128, kMaxBuckets = 1u << 15;
// More than kSampleMost of 1024 sampled keys in one bucket (of 32 that the sample
// does not tell apart) send the input to the radix passes at once: a bucket that
// takes a twentieth of the keys is full, and the atomics of its keys wait for one
// another (0.6 ns each).  Not worth asking below kSampleFrom keys.
constexpr uint32_t kSampleMost = 48, kSampleFrom = 8192;
constexpr uint32_t kWordAgg = 1u << 26, kWordIncl = 2u << 26, kWordCount = (1u << 26) - 1u;
static_assert(kMaxBuckets * 4 <= 256 * 4 * kNoallocTiles, "the bucket counts lie where the look-back words do");
static_assert(kMaxBuckets * kBucketMean <= 2 * kNoallocMaxKeys && kMaxBuckets * kBucketMean >= kNoallocMaxKeys,
              "room for twice the mean, and a mean no larger than meant");

// polls of a wait of the whole grid before it gives up (several seconds; a test
// makes it none)
#ifndef GPET_GRID_WAIT_POLLS
#define GPET_GRID_WAIT_POLLS kLookbackPolls
#endif
constexpr int kGridWaitPolls = GPET_GRID_WAIT_POLLS;

struct NoallocCtl {
    unsigned long long nmin, max;   // of the keys: ~min, max
    unsigned int arrived;           // blocks, over all waits of the grid
    unsigned int crowded;           // a bucket is full
};
static_assert(sizeof(NoallocCtl) <= kOffFailed, "a call clears the control block, not the word behind it");
struct NoallocArgs {
    const uint64_t *t_in;
    uint64_t *t_out;
    uint32_t *perm;                 // or NULL
    uint32_t n;
    NoallocCtl *ctl;
    unsigned int *failed;
    uint32_t *ghist, *words;
    uint64_t *keys;
    uint32_t *vals;
};
struct TileSmem {
    uint64_t keys[kNoallocTile];
    uint32_t vals[kNoallocTile];
    uint32_t wh[kSortWarps][256];
    uint32_t gdelta[256], thist[256];
};
struct BucketSmem {
    uint64_t keys[kSortWarps][kBucketRoom];
    uint32_t vals[kSortWarps][kBucketRoom];
    uint32_t first[kSortBlock], count[kSortBlock];
};
constexpr size_t kNoallocSmem = sizeof(TileSmem) > sizeof(BucketSmem) ? sizeof(TileSmem) : sizeof(BucketSmem);

// All blocks have come here `turn` times (they are resident together: the launch
// is cooperative).  False if the wait ran out, after which the block gives up; the
// caller learns of it from gpet_sort_times_noalloc_status.
__device__ __forceinline__ bool grid_wait(const NoallocArgs &A, unsigned turn) {
    __syncthreads();
    int fail = 0;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&A.ctl->arrived, 1u);
        int polls = 0;
        while (*reinterpret_cast<volatile unsigned *>(&A.ctl->arrived) < turn * gridDim.x)
            if (++polls > kGridWaitPolls) { fail = 1; break; }
        if (fail) atomicOr(A.failed, 1u);
        __threadfence();
    }
    return !__syncthreads_or(fail);
}

// One radix tile: keys t * 4096.. of buffer `src`, stably by digit p, to the
// other buffer.  The blocks take tiles in rising order, so the tiles that a
// look-back waits for are done or being worked on.
__device__ __forceinline__ bool sort_tile(const NoallocArgs &A, TileSmem &sm, uint32_t *sw, int p, int src, uint32_t t) {
    const uint32_t n = A.n;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t *kin = A.keys + (src ? kNoallocMaxKeys : 0);
    const uint32_t *vin = A.vals + (src ? kNoallocMaxKeys : 0);
    uint64_t *kout = A.keys + (src ? 0 : kNoallocMaxKeys);
    uint32_t *vout = A.vals + (src ? 0 : kNoallocMaxKeys);
    for (int i = threadIdx.x; i < kSortWarps * 256; i += kSortBlock) (&sm.wh[0][0])[i] = 0;
    if (threadIdx.x < 256) sm.thist[threadIdx.x] = 0;
    __syncthreads();
    // the digits' bases: exclusive scan of this pass's global histogram
    uint32_t tot;
    const uint32_t dbase = block_exscan(threadIdx.x < 256 ? __ldcg(A.ghist + p * 256 + threadIdx.x) : 0u, tot, sw);
    const uint32_t wb = t * kNoallocTile + (uint32_t)w * (32 * kItems) + (uint32_t)lane;
    uint64_t k[kItems];
    uint32_t v[kItems], rank[kItems];
    // (through L2: other blocks wrote the buffer in this kernel)
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
        const uint32_t i = wb + 32 * j;
        k[j] = i < n ? __ldcg(kin + i) : 0ull;
        v[j] = i < n ? __ldcg(vin + i) : 0u;
    }
    // the tile's digit counts, published before the ranking
#pragma unroll
    for (int j = 0; j < kItems; ++j)
        if (wb + 32 * j < n) atomicAdd(&sm.thist[(uint32_t)((k[j] >> (8 * p)) & 0xFF)], 1u);
    __syncthreads();
    const uint32_t tag = (uint32_t)(p + 1) << 28;
    volatile uint32_t *row = A.words + (size_t)t * 256;
    const uint32_t cnt = threadIdx.x < 256 ? sm.thist[threadIdx.x] : 0u;
    if (threadIdx.x < 256) row[threadIdx.x] = tag | (t == 0 ? kWordIncl : kWordAgg) | cnt;
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
        const uint32_t d = wb + 32 * j < n ? (uint32_t)((k[j] >> (8 * p)) & 0xFF) : 256u;
        uint32_t peers = kFullMask;
#pragma unroll
        for (int bit = 0; bit < 9; ++bit) {   // (the ninth separates the lanes past the end)
            const uint32_t m = __ballot_sync(kFullMask, (d >> bit) & 1u);
            peers &= ((d >> bit) & 1u) ? m : ~m;
        }
        const uint32_t before = d < 256u ? sm.wh[w][d] : 0u;
        rank[j] = before + __popc(peers & lane_lt());
        __syncwarp();
        if (d < 256u && (peers & lane_lt()) == 0) sm.wh[w][d] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    uint32_t c = 0;
    if (threadIdx.x < 256) {
#pragma unroll
        for (int ww = 0; ww < kSortWarps; ++ww) {
            const uint32_t x = sm.wh[ww][threadIdx.x];
            sm.wh[ww][threadIdx.x] = c;
            c += x;
        }
    }
    const uint32_t lstart = block_exscan(c, tot, sw);
    if (threadIdx.x < 256) {
#pragma unroll
        for (int ww = 0; ww < kSortWarps; ++ww) sm.wh[ww][threadIdx.x] += lstart;
    }
    __syncthreads();
    // the tile in digit order in shared memory; its global offsets follow
#pragma unroll
    for (int j = 0; j < kItems; ++j)
        if (wb + 32 * j < n) {
            const uint32_t lp = sm.wh[w][(uint32_t)((k[j] >> (8 * p)) & 0xFF)] + rank[j];
            sm.keys[lp] = k[j];
            sm.vals[lp] = v[j];
        }
    int fail = 0;
    if (threadIdx.x < 256) {
        const uint32_t d = threadIdx.x;
        uint32_t excl = 0;
        constexpr int kWin = 16;
        int polls = 0;
        for (uint32_t j = t; j > 0 && !fail;) {   // tiles [0, j) not yet added
            uint32_t wv[kWin];
            const volatile uint32_t *q0 = A.words + d;
#pragma unroll
            for (int q = 0; q < kWin; ++q) wv[q] = (uint32_t)q < j ? q0[(size_t)(j - 1 - q) * 256] : 0u;
            bool found = false;
#pragma unroll
            for (int q = 0; q < kWin; ++q) {
                if (found || fail || (uint32_t)q >= j) break;
                uint32_t x = wv[q];
                while ((x >> 28) != (uint32_t)(p + 1)) {
                    if (++polls > kLookbackPolls) { fail = 1; break; }
                    if (polls > 64) __nanosleep(64);
                    x = q0[(size_t)(j - 1 - q) * 256];
                }
                if (fail) break;
                excl += x & kWordCount;
                found = (x & kWordIncl) != 0;
            }
            j = found ? 0u : (j > (uint32_t)kWin ? j - kWin : 0u);
        }
        if (!fail && t > 0) row[d] = tag | kWordIncl | (excl + cnt);
        sm.gdelta[d] = dbase + excl - lstart;
    }
    // (a tile whose look-back gave up writes nothing: the output is then incomplete)
    if (__syncthreads_or(fail)) {
        if (threadIdx.x == 0) atomicOr(A.failed, 1u);
        return false;
    }
    const uint32_t tn = min(n - t * kNoallocTile, (uint32_t)kNoallocTile);
    for (uint32_t i = threadIdx.x; i < tn; i += kSortBlock) {
        const uint64_t key = sm.keys[i];
        const uint32_t pos = sm.gdelta[(uint32_t)((key >> (8 * p)) & 0xFF)] + i;
        if (pos < n) {
            kout[pos] = key;
            vout[pos] = sm.vals[i];
        }
    }
    __syncthreads();
    return true;
}

// the keys by radix passes (turn: waits of the grid so far)
__device__ __noinline__ void radix_sort(const NoallocArgs &A, TileSmem &sm, uint32_t *sw, unsigned turn) {
    const uint32_t n = A.n, stride = gridDim.x * kSortBlock, first = blockIdx.x * kSortBlock + threadIdx.x;
    const uint32_t tiles = (n + kNoallocTile - 1) / kNoallocTile;
    uint32_t *h = &sm.wh[0][0];   // [8][256]
    for (int i = threadIdx.x; i < 8 * 256; i += kSortBlock) h[i] = 0;
    __syncthreads();
    for (uint32_t i = first; i < n; i += stride) {
        const uint64_t key = A.t_in[i];
        A.keys[i] = key;
        A.vals[i] = i;
#pragma unroll
        for (int p = 0; p < 8; ++p) atomicAdd(&h[p * 256 + ((key >> (8 * p)) & 0xFF)], 1u);
    }
    for (uint32_t i = first; i < tiles * 256; i += stride) A.words[i] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < 8 * 256; i += kSortBlock)
        if (h[i]) atomicAdd(A.ghist + i, h[i]);
    if (!grid_wait(A, ++turn)) return;
    // the digits that vary (every block finds the same ones)
    __shared__ int varies[8];
    if (threadIdx.x < 256) {
        const int p = threadIdx.x >> 5, lane = threadIdx.x & 31;
        uint32_t mx = 0;
        for (int d = lane; d < 256; d += 32) mx = max(mx, __ldcg(A.ghist + p * 256 + d));
        mx = __reduce_max_sync(kFullMask, mx);
        if (lane == 0) varies[p] = mx < n;
    }
    __syncthreads();
    int src = 0;
    for (int p = 0; p < 8; ++p) {
        if (!varies[p]) continue;
        for (uint32_t t = blockIdx.x; t < tiles; t += gridDim.x)
            if (!sort_tile(A, sm, sw, p, src, t)) return;
        src ^= 1;
        if (!grid_wait(A, ++turn)) return;
    }
    for (uint32_t i = first; i < n; i += stride) {
        A.t_out[i] = __ldcg(A.keys + (src ? kNoallocMaxKeys : 0) + i);
        if (A.perm) A.perm[i] = __ldcg(A.vals + (src ? kNoallocMaxKeys : 0) + i);
    }
}

__global__ void __launch_bounds__(kSortBlock, 1) k_noalloc_sort(const __grid_constant__ NoallocArgs A) {
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ uint32_t sw[32];
    __shared__ unsigned long long red[2][32];
    __shared__ unsigned long long scale_sh;
    const uint32_t n = A.n, stride = gridDim.x * kSortBlock, first = blockIdx.x * kSortBlock + threadIdx.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t nb = min(max(n / kBucketMean, 1u), kMaxBuckets);
    const uint32_t room = min(kBucketRoom, (uint32_t)(2 * kNoallocMaxKeys) / nb);
    constexpr int kAhead = 4;   // keys a thread has in flight
    // 1. the keys' range; counts and histograms cleared
    for (uint32_t i = first; i < nb; i += stride) A.words[i] = 0u;
    for (uint32_t i = first; i < 8 * 256; i += stride) A.ghist[i] = 0u;
    unsigned long long lo = 0, hi = 0;   // ~min, max
    for (uint32_t i0 = first; i0 < n; i0 += kAhead * stride) {
        unsigned long long k[kAhead];
#pragma unroll
        for (int q = 0; q < kAhead; ++q) k[q] = A.t_in[i0 + q * stride < n ? i0 + q * stride : i0];
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            lo = max(lo, ~k[q]);
            hi = max(hi, k[q]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = max(lo, __shfl_xor_sync(kFullMask, lo, o));
        hi = max(hi, __shfl_xor_sync(kFullMask, hi, o));
    }
    if (lane == 0) {
        red[0][wid] = lo;
        red[1][wid] = hi;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        unsigned long long m = 0;
        for (int w = 0; w < kSortWarps; ++w) m = max(m, red[threadIdx.x][w]);
        atomicMax(threadIdx.x ? &A.ctl->max : &A.ctl->nmin, m);
    }
    // (a sample over the whole input, the same for every block)
    const bool sampled = n > kSampleFrom;
    const unsigned long long sample = A.t_in[sampled ? (uint32_t)((unsigned long long)threadIdx.x * n / kSortBlock) : 0u];
    if (!grid_wait(A, 1)) return;
    // 2. each key to its bucket: hi64((key - min) * scale), or key - min where
    // there are no more values than buckets (scale 0)
    const unsigned long long mn = ~__ldcg(&A.ctl->nmin);
    if (threadIdx.x == 0) {
        const unsigned long long range = __ldcg(&A.ctl->max) - mn;
        // (a little below nb * 2^64 / range, so that the last key's bucket exists
        // whatever the rounding)
        scale_sh = range < nb ? 0ull : __float2ull_rz((float)nb * (0.999998f * 18446744073709551616.0f / __ull2float_ru(range)));
    }
    uint32_t *seen = reinterpret_cast<uint32_t *>(raw);
    seen[threadIdx.x] = 0;
    __syncthreads();
    const unsigned long long scale = scale_sh;
    auto bucket = [&](unsigned long long key) {
        const unsigned long long x = key - mn;
        return (uint32_t)min(scale ? __umul64hi(x, scale) : x, (unsigned long long)(nb - 1u));
    };
    bool crowded = false;
    if (sampled) crowded = atomicAdd(seen + bucket(sample) % kSortBlock, 1u) >= kSampleMost;
    if (__syncthreads_or(crowded)) {   // (every block sees this, or none)
        radix_sort(A, *reinterpret_cast<TileSmem *>(raw), sw, 1);
        return;
    }
    for (uint32_t i0 = first; i0 < n; i0 += kAhead * stride) {
        unsigned long long k[kAhead];
        uint32_t b[kAhead], r[kAhead];
#pragma unroll
        for (int q = 0; q < kAhead; ++q) k[q] = A.t_in[i0 + q * stride < n ? i0 + q * stride : i0];
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            b[q] = bucket(k[q]);
            r[q] = i0 + q * stride < n ? atomicAdd(A.words + b[q], 1u) : room;
        }
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            if (r[q] < room) {
                A.keys[b[q] * room + r[q]] = k[q];
                A.vals[b[q] * room + r[q]] = i0 + q * stride;
            } else if (i0 + q * stride < n) {
                crowded = true;
            }
        }
    }
    if (__syncthreads_or(crowded) && threadIdx.x == 0) atomicOr(&A.ctl->crowded, 1u);
    if (!grid_wait(A, 2)) return;
    if (__ldcg(&A.ctl->crowded)) {
        radix_sort(A, *reinterpret_cast<TileSmem *>(raw), sw, 2);
        return;
    }
    // 3. a stretch of buckets per block (a multiple of four: the counts before it
    // are read four at a time), a bucket at a time per warp
    BucketSmem &S = *reinterpret_cast<BucketSmem *>(raw);
    const uint32_t per = ((nb + gridDim.x - 1) / gridDim.x + 3u) & ~3u;
    const uint32_t b0 = blockIdx.x * per, b1 = min(b0 + per, nb);
    if (b0 >= nb) return;
    uint32_t before = 0, base = 0, total;
    for (uint32_t i = threadIdx.x * 4; i < b0; i += kSortBlock * 4) {
        const uint4 c = __ldcg(reinterpret_cast<const uint4 *>(A.words + i));
        before += c.x + c.y + c.z + c.w;
    }
    block_exscan(before, base, sw);
    for (uint32_t c0 = b0; c0 < b1; c0 += kSortBlock) {
        const uint32_t mine = c0 + threadIdx.x < b1 ? __ldcg(A.words + c0 + threadIdx.x) : 0u;
        S.first[threadIdx.x] = base + block_exscan(mine, total, sw);
        S.count[threadIdx.x] = mine;
        __syncthreads();
        const uint32_t nc = min(b1 - c0, (uint32_t)kSortBlock);
        for (uint32_t c = wid; c < nc; c += kSortWarps) {
            const uint32_t m = S.count[c], at = S.first[c], src = (c0 + c) * room;
            for (uint32_t j = lane; j < m; j += 32) {
                S.keys[wid][j] = __ldcg(A.keys + src + j);
                S.vals[wid][j] = __ldcg(A.vals + src + j);
            }
            __syncwarp();
            for (uint32_t j = lane; j < m; j += 32) {
                const uint64_t key = S.keys[wid][j];
                const uint32_t val = S.vals[wid][j];
                uint32_t rank = at;
                for (uint32_t i = 0; i < m; ++i) {
                    const uint64_t o = S.keys[wid][i];
                    rank += o < key || (o == key && S.vals[wid][i] < val);
                }
                A.t_out[rank] = key;
                if (A.perm) A.perm[rank] = val;
            }
            __syncwarp();
        }
        base += total;
        __syncthreads();
    }
}

}  // namespace gpet

using namespace gpet;

extern "C" int gpet_sort_times_noalloc(const uint64_t *d_t_in, uint64_t n, uint64_t *d_t_out, uint32_t *d_perm_out,
                                       void *stream) {
    if (n > kNoallocMaxKeys)
        return gpet_fail(GPET_ERR_INVALID_ARG, "gpet_sort_times_noalloc: n = %llu exceeds its maximum of %llu keys",
                         (unsigned long long)n, kNoallocMaxKeys);
    if (n == 0) return GPET_OK;
    if (!d_t_in || !d_t_out) return gpet_fail(GPET_ERR_INVALID_ARG, "gpet_sort_times_noalloc: NULL input or output");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return gpet_cuda_fail(e, "cudaGetDevice");
    // The host-side name of the array is not a device address: ask the runtime
    // for the address of the current device's copy.  The first lookup on a
    // device loads the module that holds the array (modules load lazily), which
    // is when its device memory is taken; later lookups read the loaded
    // module's symbol table.  Looking it up on every call, rather than caching
    // it, keeps the address right after a cudaDeviceReset reloads the module.
    void *sym = nullptr;
    e = cudaGetSymbolAddress(&sym, g_sort_scratch);
    if (e != cudaSuccess) return gpet_cuda_fail(e, "cudaGetSymbolAddress(sort scratch)");
    unsigned char *base = static_cast<unsigned char *>(sym);
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return gpet_cuda_fail(e, "cudaDeviceGetAttribute");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    NoallocArgs A;
    A.t_in = d_t_in;
    A.t_out = d_t_out;
    A.perm = d_perm_out;
    A.n = (uint32_t)n;
    A.ctl = reinterpret_cast<NoallocCtl *>(base + kOffCtl);
    A.failed = reinterpret_cast<unsigned int *>(base + kOffFailed);
    A.ghist = reinterpret_cast<uint32_t *>(base + kOffHist);
    A.keys = reinterpret_cast<uint64_t *>(base + kOffKeys);
    A.vals = reinterpret_cast<uint32_t *>(base + kOffVals);
    A.words = reinterpret_cast<uint32_t *>(base + kOffWords);
    const void *fn = reinterpret_cast<const void *>(k_noalloc_sort);
    e = ensure_dynamic_smem(fn, kNoallocSmem);
    if (e == cudaSuccess) e = cudaMemsetAsync(A.ctl, 0, sizeof(NoallocCtl), st);
    // one block per multiprocessor at most (all of them run at once), 512 keys a block at least; fewer where the
    // stream has a part of the device's multiprocessors
    unsigned blocks = (unsigned)std::min<uint64_t>((uint64_t)sms, (n + 511) / 512);
    void *args[] = {&A};
    while (e == cudaSuccess) {
        e = cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(kSortBlock), args, kNoallocSmem, st);
        if (e != cudaErrorCooperativeLaunchTooLarge || blocks == 1) break;
        cudaGetLastError();
        e = cudaSuccess;
        blocks /= 2;
    }
    if (e != cudaSuccess) return gpet_cuda_fail(e, "gpet_sort_times_noalloc launch");
    return GPET_OK;
}

extern "C" int gpet_sort_times_noalloc_status(void *stream) {
    void *sym = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&sym, g_sort_scratch);
    if (e != cudaSuccess) return gpet_cuda_fail(e, "cudaGetSymbolAddress(sort scratch)");
    unsigned char *word = static_cast<unsigned char *>(sym) + kOffFailed;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned int failed = 0;
    e = cudaMemcpyAsync(&failed, word, sizeof(failed), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && failed) e = cudaMemsetAsync(word, 0, sizeof(failed), st);
    if (e != cudaSuccess) return gpet_cuda_fail(e, "gpet_sort_times_noalloc_status");
    if (failed) return gpet_fail(GPET_ERR_CUDA, "a wait of gpet_sort_times_noalloc ran out: its output is incomplete");
    return GPET_OK;
}
