// transport_cta.cu -- warp-autonomous wavefront transport kernel over a pool
// of history slots that a CTA shares.
//
// A CTA keeps its history slots in shared memory and one 32-bit mask per
// (phase, lane class): bit i of mask[p][l] says that slot i of lane class l
// waits in phase p.  A slot stays with its lane class (slot i of class l is
// always served by lane l of some warp), so every state access is free of bank
// conflicts.  Each warp, on its own, takes the phase in which most of its lanes
// have a slot, claims one slot per lane (an atomic AND on the mask), runs that
// phase's event, and hands each slot on to its next phase (an atomic OR).  There
// is no barrier: a warp that waits for memory or for its slowest lane delays no
// other.
//
// What bounds it is instruction issue: no DRAM traffic to speak of, and the
// state never leaves the SM.  Three things make that work:
//   - Events are cut where their lanes would diverge.  A Woodcock step only
//     finds the collision; sampling it (one Kahn trial, rotation, record) is an
//     event of its own with its lanes packed, and a rejected trial waits for the
//     next one.  The finish event digitizes one single per lane, where a loop
//     over a history's singles waits for the warp's longest list.
//   - The code of all events together is small (46 KB, the hot part less), since
//     the warps of an SM are in different phases at once: one flight routine with
//     one slab-test loop for every kind of flight, one Philox draw and one sine
//     and cosine for all events that need them, cold paths out of line.  At 74 KB
//     the same scheme lost half of its issue slots to instruction fetch (7.6 of
//     14 warp-cycles per issue; now 1.4 of 9), and events that a whole CTA runs
//     together behind a barrier lost them to the barrier (6.0 of 13.5).
//   - First flights of a pair's two photons are one event (the same ray in both
//     directions), which keeps photon 1's panel and distances in the slot until
//     its turn; a photon that leaves through a panel's back, where no other panel
//     can be, ends without a flight event.
//   - A history's singles are a chain of entries that the slots of a lane class
//     share, so a list has no length of its own to overflow: only a class without
//     a free entry leaves a history to the redo kernel, which simulates it again,
//     and has a slot less from then on.  Nothing waits for an entry.  With lists of
//     six, that kernel's few serial histories took 30 us of every launch of 1e6
//     pairs and more (1e6 pairs in the 12-panel ring 207 us, now 175; 2e6 in four
//     heads 235, now 213; 24 designs in one launch 1.44 ms, now 1.38).
// Photons of a pair run one after the other, and events are those of
// transport.cuh, so the histories equal the other kernels' bit for bit.
//
// Measured on a GB300, transport of one sweep position of 1e7 pairs: 2.52 ms
// with the phase chosen per CTA behind a barrier and per-warp pools, 1.28 ms
// with this scheme alone, 1.03 ms with what the comments below add.
#include "internal.h"
#include "transport.cuh"

namespace gpet {

namespace {

// one more phase here than in transport.cuh: a collision to be sampled
constexpr uint32_t kPhInteract = 7;
constexpr int kPhCount = 8;
constexpr uint32_t kPhGivenUp = kPhSource;  // (the decay is the idle phase's event here)
constexpr int kEntries = 48;  // singles entries of a lane class, for all of its slots
constexpr int kKeptSlots = 8;  // slots of a lane class that are never given up

// state words of a slot; the last four only where a job has a phantom
enum : int { kSh0 = 0, kSh1,
             kSjob,             // job; [16:23) photon 1's first panel + 1 (0: it enters none);
                                // [23:29) first entry + 1 of the history's singles list (0: empty)
             kSox, kSoy, kSoz,
             kSx, kSy, kSz, kSdx, kSdy, kSdz, kSE,
             kSpath,            // path; distance to the panel of a photon 0 that has not entered it yet
             kStrem,            // distance to the panel's exit; crystal id of a collision to be sampled
             kSin1, kSrem1,     // photon 1's distance to its first panel, and through it
             kSrw,              // azimuth word (top 23 bits) of a collision and its Kahn trials (low 9 bits);
                                // distance to the next panel of a photon between panels
             kSpk,
             kSx0, kSy0, kSz0, kSph };
constexpr int kWordsPlain = kSx0, kWordsPhantom = kSph + 1;
constexpr int kJobPanel1 = 16, kJobList = 23;

// packed word: [0:7) panel + 1, [7:14) last panel + 1
// (in a panel: not 0 where the photon has still to enter it; a collision: bit 7
// counts 512 Kahn trials), [14] photon, [15] the list has singles, [18] list
// overflowed, [19] photon 1 starts in the phantom, [20] photon not in its first
// panel yet (its state is the decay's), [21:31) detector steps, [31]
// photoelectric absorption
constexpr int kPkLast = 7, kPkStep = 21;
constexpr uint32_t kPkPanel = 0x7Fu, kPkLastMask = 0x7Fu << kPkLast, kPkGamma = 1u << 14, kPkSing = 1u << 15,
                   kPkOvf = 1u << 18, kPkPhantom1 = 1u << 19, kPkFresh = 1u << 20, kPkStepMask = 0x3FFu << kPkStep,
                   kPkPhoto = 1u << 31;
static_assert(kMaxSteps < 1024 && kMaxPanels < 127 && kMaxTrials <= 1024 && kEntries < 63, "packed word fields");

// event counters: slots 0..7 count the events of each phase (decays in 0,
// lanes fed in 1); lane i of a warp keeps counter i
enum : int { kNLanes = 1, kNScrStart = 8, kNScrFlight, kNEntered, kNHits, kNTrials, kNSingles, kNFin, kNIter, kNCount };
// Lanes with a slot in a warp's last phase for which it stays with that phase.  Where
// the code is longer than the instruction cache likes, fewer lanes are the better
// price: 5 M pairs in the hot-rod phantom with 10, 14, 18, 22, 26 of them 1.477,
// 1.479, 1.499, 1.533, 1.582 ms; 10 M in ring A 1.107, 1.071, 1.052, 1.045, 1.056.
constexpr int sticky_lanes(bool phantom) { return phantom ? 14 : 22; }
constexpr uint32_t kMaxSpins = 1u << 24;  // waits for a slot (over a second) before a warp gives up
constexpr unsigned kFlushEvery = 1u << 20;  // events; below 2^32 counts in as many of any kind

template <int SLOTS, bool PH>
struct CtaPool {
    static constexpr int kWords = PH ? kWordsPhantom : kWordsPlain;
    static constexpr int kN = SLOTS * 32;
    uint32_t st[kWords * kN];
    uint32_t e_unit[kEntries * 32];
    float e_e[kEntries * 32];
    uint32_t e_dt[kEntries * 32];
    float e_ew[kEntries * 32];
    uint8_t e_next[kEntries * 32];   // next entry + 1 of the history's list (0: the last); four of a lane in a word
};

// place of entry e in e_next
__device__ __forceinline__ uint32_t next_at(uint32_t e, int lane) { return ((e >> 2) * 32u + lane) * 4u + (e & 3u); }
// the free entries of a lane class (the entry's last reads come before)
__device__ __forceinline__ void free_entry(uint32_t (*efree)[32], int lane, uint32_t e) {
    asm volatile("" ::: "memory");
    atomicOr(&efree[e >> 5][lane], 1u << (e & 31u));
}
// a free entry, or kEntries
__device__ __forceinline__ uint32_t take_entry(uint32_t (*efree)[32], int lane) {
#pragma unroll 1
    for (int w = 0; w < 2; ++w) {
        uint32_t f = *reinterpret_cast<volatile uint32_t *>(&efree[w][lane]);
#pragma unroll 1
        while (f) {
            const uint32_t b = f & (0u - f);
            const uint32_t old = atomicAnd(&efree[w][lane], ~b);
            if (old & b) return (uint32_t)(32 * w) + 31u - (uint32_t)__clz((int)b);
            f = old & ~b;
        }
    }
    return (uint32_t)kEntries;
}

// frees a history's whole list, whose first entry + 1 is in jobw (out of line: rarely run,
// and its code in the collision's place made 10 M pairs in ring A 1.061 ms, not 1.028)
__device__ __noinline__ uint32_t free_list(uint32_t (*efree)[32], const uint8_t *e_next, int lane, uint32_t jobw) {
    for (uint32_t next = (jobw >> kJobList) & 63u; next;) {
        const uint32_t e = next - 1u;
        next = e_next[next_at(e, lane)];
        free_entry(efree, lane, e);
    }
    return jobw & ~(63u << kJobList);
}

// Photon of packed word pk is done: the slot's next phase.  Photon 0 hands
// over to photon 1, which starts in the phantom, at the panel its first flight
// found (panel1 = panel + 1), or not at all (0); a history without singles has
// nothing to digitize, its slot is free.
__device__ __forceinline__ uint32_t photon_end(uint32_t &pk, uint32_t panel1) {
    const bool first = !(pk & kPkGamma), ph1 = pk & kPkPhantom1;
    pk &= kPkSing | kPkOvf;
    if (first && (ph1 || panel1)) {
        pk |= kPkGamma | (ph1 ? 0u : kPkFresh | panel1);
        return ph1 ? kPhPhantom : kPhPanel;
    }
    return pk ? kPhFinish : kPhIdle;
}

// n more of event counter i, kept by lane i (a function, so that every lane evaluates n)
__device__ __forceinline__ void count(uint32_t &acc, int i, uint32_t n) {
    if ((int)(threadIdx.x & 31) == i) acc += n;
}

// The warp's next chunk, for its refill state in shared memory (out of line: called once
// in several decay events, and inline it took the step code's place
// in the instruction cache; 60 M pairs in two ring geometries: 6.33 ms against 6.64)
template <bool kLive>
__device__ __noinline__ bool next_chunk_out(const WorkDev &W, Refill &R) {
    Refill r;   // field by field: a copy of the whole would go through local memory
    r.pend = R.pend; r.jc0 = R.jc0; r.jend = R.jend; r.base = R.base; r.nh = R.nh;
    r.next = R.next; r.end = R.end;
    r.job = R.job;
    __syncwarp();
    const bool got = next_chunk<kLive>(W, r);
    if ((threadIdx.x & 31) == 0) {
        R.next = r.next; R.end = r.end;
        R.pend = r.pend; R.jc0 = r.jc0; R.jend = r.jend; R.base = r.base; R.nh = r.nh;
        R.job = r.job;
        R.exhausted = r.exhausted; R.waiting = r.waiting;
    }
    __syncwarp();
    return got;
}

// a crystal interaction into the optional hit list (tests, depth studies)
__device__ __noinline__ void keep_hit(const OutDev &O, const JobDev &J, const GeomDev &g, uint64_t h, int job,
                                      uint32_t gamma, uint32_t step, int crystal, float dep, uint32_t dtp, float x,
                                      float y, float z) {
    PState s;
    s.h = h;
    s.t0 = decay_time(J, draw(J.seed, h, kTagSource, 0u, 0u, 0u));
    s.gamma = gamma;
    s.job = job;
    s.x = x; s.y = y; s.z = z;
    const int c = crystal % g.crystals_per_module;   // the layer, from the id within the module
    int layer = 0;
    while (layer + 1 < g.n_layers && c >= g.layers[layer + 1].loff) ++layer;
    store_hit(O, s, crystal, layer, step, dep, dtp);
}

}  // namespace

// kPhantom: jobs with a phantom may occur; kPosed: geometries with panel poses
// may.  kLive: a live launch (chunks the host appends while the kernel runs,
// bounded idle waits, per-job singles buffers).  Separate instantiations, so
// that a fixed launch without them carries none of their instructions,
// registers and state words.
// kTab: where an event finds its job and geometry.
// - kTabOne: the launch has one job, which with its geometry comes in the kernel's
//   parameters: what every lane reads alike is then an operand of the instruction
//   that uses it (the random draws' key schedule is the warp's, too), where a
//   launch of several jobs loads it lane by lane.  Tables that lanes index by
//   panel, layer or material stay in shared memory, since lanes that read
//   different constants read them one after the other.  10 M pairs in ring A
//   1.127 ms without it, 1.080 with; 5 M in the hot-rod phantom 1.64, 1.51; 3 M in
//   the h2r ring 0.783, 0.743; 2e4 in the tiny ring 53 us, 51.
// - kTabStaged: several jobs, and all of the launch's geometries are staged in
//   shared memory: read there, where the general form reads through a pointer to
//   either memory.  60 M pairs in two rings 6.25 ms without it, 6.03 with; a map of
//   6.4 M pairs in two rings 2.04, 1.98.  (The jobs staged as well: 6.13.)
// - kTabJobs: any launch.
enum : int { kTabJobs = 0, kTabOne = 1, kTabStaged = 2 };
template <int kTab>
struct CtaTables {
    int ng_smem;   // geometries staged in shared memory
};
template <>
struct CtaTables<kTabOne> {
    JobDev J;
    GeomDev g;
};
template <int kTab>
__device__ __forceinline__ int staged(const CtaTables<kTab> &T) { return T.ng_smem; }
__device__ __forceinline__ int staged(const CtaTables<kTabOne> &) { return 1; }
template <int kTab>
__device__ __forceinline__ const JobDev &job_of(const CtaTables<kTab> &, const WorkDev &W, uint32_t j) { return W.jobs[j]; }
__device__ __forceinline__ const JobDev &job_of(const CtaTables<kTabOne> &T, const WorkDev &, uint32_t) { return T.J; }
template <int kTab>
__device__ __forceinline__ const GeomDev &geom_of(const CtaTables<kTab> &T, const GeomDev *sgeom, const WorkDev &W, int i) {
    return kTab == kTabStaged || i < T.ng_smem ? sgeom[i] : W.geoms[i];
}
__device__ __forceinline__ GeomOne geom_of(const CtaTables<kTabOne> &T, const GeomDev *sgeom, const WorkDev &, int) {
    return GeomOne{T.g, sgeom[0]};
}

template <int WARPS, int SLOTS, int CTAS, bool kPhantom, bool kPosed, bool kLive, int kTab>
__global__ void __launch_bounds__(WARPS * 32, CTAS) k_transport_cta(const __grid_constant__ WorkDev W,
                                                                   const __grid_constant__ OutDev O,
                                                                   const __grid_constant__ CtaTables<kTab> T) {
    const int ng_smem = staged(T);
    static_assert(SLOTS <= 32, "one mask bit per slot");
    using Pool = CtaPool<SLOTS, kPhantom>;
    constexpr int kN = Pool::kN;
    extern __shared__ __align__(16) uint8_t smem[];
    GeomDev *sgeom = reinterpret_cast<GeomDev *>(smem);
    Pool &P = *reinterpret_cast<Pool *>(sgeom + ng_smem);
    __shared__ uint32_t mask[kPhCount][32];
    __shared__ uint32_t efree[2][32];
    __shared__ Refill refills[WARPS];
    stage_geometry(W, sgeom, ng_smem);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x < 32) {
#pragma unroll
        for (int p = 0; p < kPhCount; ++p) mask[p][lane] = p == kPhIdle ? 0xFFFFFFFFu >> (32 - SLOTS) : 0u;
        efree[0][lane] = 0xFFFFFFFFu;
        efree[1][lane] = 0xFFFFFFFFu >> (64 - kEntries);
    }
    if (lane == 0) refill_init(refills[wid]);
    __syncthreads();
    LiveIdle idle;
    live_idle_reset(idle);
    uint32_t *const st = P.st;
    bool done = false;    // no histories to come for this warp
    uint32_t acc = 0;     // lane i: event counter i
    uint32_t ph = kPhIdle, spins = 0;
    bool waiting = false, alone = false;   // live: the next chunk is not published; no slot in any other phase
#define ST(w) st[(w) * kN + q]
#define STF(w) __uint_as_float(st[(w) * kN + q])
#define STORE3(w, a, b, c) (ST(w) = __float_as_uint(a), ST((w) + 1) = __float_as_uint(b), ST((w) + 2) = __float_as_uint(c))

    for (unsigned it = 1;; ++it) {
        // 1. the phase: the last one again while most lanes have a slot in it,
        // else the one with the most lanes (ties to the later one, so that
        // histories end before others begin)
        uint32_t m = *reinterpret_cast<volatile uint32_t *>(&mask[ph][lane]);
        if ((ph == kPhIdle && (done || (kLive && waiting))) || __popc(__ballot_sync(kFullMask, m != 0)) < sticky_lanes(kPhantom)) {
            uint32_t best = 0;
            alone = true;
#pragma unroll
            for (int p = 0; p < kPhCount; ++p) {
                if (p == (int)kPhGivenUp || (p == 2 && !kPhantom)) continue;
                const uint32_t v = *reinterpret_cast<volatile uint32_t *>(&mask[p][lane]);
                uint32_t n = (p == kPhIdle && done) ? 0u : (uint32_t)__popc(__ballot_sync(kFullMask, v != 0));
                // a live launch's warp whose next chunk is not published yet asks for
                // it every eighth time, or when there is nothing else to do
                if (kLive && p == kPhIdle && waiting && (it & 7u)) n = min(n, 1u);
                if (kLive && p != kPhIdle && n) alone = false;
                best = max(best, n ? (n << 3) | (uint32_t)p : 0u);
            }
            if (best == 0) {
                // every slot that this warp could take is in other warps' hands,
                // which hand it on or, with no histories to come, see to its end
                if (done) break;
                if (++spins > kMaxSpins) {
                    if (lane == 0) atomicOr(O.status, kStatusBadPhase);
                    break;
                }
                __nanosleep(64);
                continue;
            }
            spins = 0;
            ph = best & 7u;
            m = *reinterpret_cast<volatile uint32_t *>(&mask[ph][lane]);
        }
        // 2. claim one slot of the phase per lane (each warp from another bit on)
        const uint32_t rot = (uint32_t)(wid * 5) & 31u;
        uint32_t bit = 0;
        bool active = false;
#pragma unroll 1
        for (int t = 0; t < 2; ++t) {   // (a lane whose bit went to another warp tries once more)
            if (!active && m) {
                const uint32_t mr = __funnelshift_r(m, m, rot);
                const uint32_t low = mr & (0u - mr);
                bit = __funnelshift_l(low, low, rot);
                const uint32_t old = atomicAnd(&mask[ph][lane], ~bit);
                active = old & bit;
                m = old & ~bit;
            }
            if (!__any_sync(kFullMask, !active && m)) break;
        }
        const uint32_t am = __ballot_sync(kFullMask, active);
        if (am == 0) continue;
        __threadfence_block();
        const int q = active ? (31 - __clz((int)bit)) * 32 + lane : lane;
        count(acc, kNIter, 1);
        count(acc, kNLanes, __popc(am));
        if (it % kFlushEvery == 0) {   // (32-bit counts never wrap: see kFlushEvery)
            if (lane < kNCount && acc) atomicAdd(O.counters + kCtaCounters + lane, (unsigned long long)acc);
            acc = 0;
        }
        // 3. the event
        uint32_t jobw = 0, pk = 0, to = kPhIdle;
        uint64_t h = 0;
        bool run = active;   // lanes with a history
        if (ph == kPhIdle) {
            Refill &rf = refills[wid];
            // consecutive histories of the warp's chunks to the claimed lanes
            uint32_t need = am;
            run = false;
#pragma unroll 1
            do {
                const uint64_t next = rf.next, avail = rf.end - next;
                const uint32_t rank = __popc(need & lanemask_lt());
                const uint32_t take = (uint32_t)min(avail, (uint64_t)__popc(need));
                if (((need >> lane) & 1u) && rank < take) {
                    run = true;
                    h = next + rank;
                    jobw = (uint32_t)rf.job;
                }
                __syncwarp();
                if (lane == 0) rf.next = next + take;
                need &= ~__ballot_sync(kFullMask, run);
                __syncwarp();
            } while (need && next_chunk_out<kLive>(W, rf));
            done = rf.exhausted;
            waiting = rf.waiting;
        } else if (active) {
            jobw = ST(kSjob);
            pk = ST(kSpk);
            h = ((uint64_t)ST(kSh1) << 32) | ST(kSh0);
        }
        const JobDev &J = job_of(T, W, jobw & 0xFFFFu);
        decltype(auto) geom = geom_of(T, sgeom, W, J.geom);
        const GeomDev &g = fields(geom);
        const uint32_t gamma = (pk & kPkGamma) ? 1u : 0u;
        if (ph == kPhFlight || ph == kPhFlightOut) {
            // Flights to the next panel: the first ones of both photons from the
            // decay point (but one that the axial screen ended), or of one photon
            // out of a panel or the phantom.
            uint32_t n_fl = 0, n_in = 0, n_scr = 0;
            if (run) {
                const bool out = ph == kPhFlightOut;
                const bool pair = !out && (!kPhantom || ST(kSph) == 0);
                float x, y, z, dx, dy, dz;
                if (pair) {
                    x = kPhantom ? STF(kSx0) : J.src_pos[0];
                    y = kPhantom ? STF(kSy0) : J.src_pos[1];
                    z = kPhantom ? STF(kSz0) : J.src_pos[2];
                    const float sg = gamma ? -1.0f : 1.0f;
                    dx = sg * STF(kSox); dy = sg * STF(kSoy); dz = sg * STF(kSoz);
                } else {
                    x = STF(kSx); y = STF(kSy); z = STF(kSz);
                    dx = STF(kSdx); dy = STF(kSdy); dz = STF(kSdz);
                }
                const int skip = out ? (int)((pk & kPkLastMask) >> kPkLast) - 1 : -1;
                uint32_t p0 = 0, p1 = 0, second = gamma;
#pragma unroll 1
                for (;;) {
                    float t_in, t_out;
                    const int k = flight<kPosed>(geom, x, y, z, dx, dy, dz, skip, t_in, t_out);
                    n_fl++;
                    n_scr += k == kFlightScreened ? 1u : 0u;
                    if (k >= 0) {
                        n_in++;
                        (second ? p1 : p0) = (uint32_t)(k + 1);
                        const int wi = !pair ? kSrw : second ? kSin1 : kSpath, wr = pair && second ? kSrem1 : kStrem;
                        st[wi * kN + q] = __float_as_uint(t_in);
                        st[wr * kN + q] = __float_as_uint(t_out - t_in);
                    }
                    // photon 1 of a pair next (pk's fresh flag: the screen ended it)
                    if (!pair || second || (pk & kPkFresh)) break;
                    second = 1;
                    dx = -dx; dy = -dy; dz = -dz;
                }
                if (pair) {
                    ST(kSjob) = jobw | (p1 << kJobPanel1);
                    pk = p0 ? kPkFresh | p0 : (p1 ? kPkFresh | kPkGamma | p1 : 0u);
                    to = pk ? kPhPanel : kPhIdle;
                } else {
                    if (kPhantom) ST(kSph) = 0;
                    const uint32_t k1 = p0 | p1;
                    if (k1) {
                        pk = (pk & ~kPkPanel) | kPkLastMask | k1;   // enters it at its next step
                        to = kPhPanel;
                    } else {
                        to = photon_end(pk, (jobw >> kJobPanel1) & 0x7Fu);
                    }
                }
                ST(kSpk) = pk;
            }
            // (at most two a lane)
            const uint32_t n = __reduce_add_sync(kFullMask, n_fl | (n_in << 8) | (n_scr << 16));
            count(acc, ph, n & 0xFFu);
            count(acc, kNEntered, (n >> 8) & 0xFFu);
            count(acc, kNScrFlight, n >> 16);
        } else {
            // The other events begin with a draw, made here for all of them.
            const bool in_panel = !kPhantom || (pk & kPkPanel);
            uint32_t c2 = kTagSource << 28, c3 = 0, rw = 0, e = 0, next = 0, unit = 0;
            const uint32_t step = (pk & kPkStepMask) >> kPkStep;
            if (ph == kPhPanel) {
                c2 = (kTagDetector << 28) | (gamma << 27) | step;
            } else if (kPhantom && ph == kPhPhantom) {
                c2 = (kTagPhantom << 28) | (gamma << 27) | (run ? ST(kSph) : 0u);
            } else if (ph == kPhInteract) {
                rw = ST(kSrw);
                c2 = (in_panel ? (kTagDetector << 28) | (step - 1u) : (kTagPhantom << 28) | (ST(kSph) - 1u)) | (gamma << 27);
                c3 = 1u + (rw & 511u) + ((pk >> kPkLast) & 1u) * 512u;
            } else if (ph == kPhFinish) {
                e = ((jobw >> kJobList) & 63u) - 1u;
                if (!run || !(pk & kPkSing)) e = 0;   // overflowed: it has no list
                unit = P.e_unit[e * 32 + lane];
                next = P.e_next[next_at(e, lane)];
                c2 = kTagDigi << 28;
                c3 = unit;
            }
            const uint4 r = philox4x32_10(make_uint4((uint32_t)h, (uint32_t)(h >> 32), c2, c3),
                                          make_uint2((uint32_t)J.seed, (uint32_t)(J.seed >> 32)));
            if (ph == kPhPanel || (kPhantom && ph == kPhPhantom)) {
                // one Woodcock step in the panel or the phantom
                uint32_t n_left = 0;
                if (run) {
                    const bool panel = !kPhantom || ph == kPhPanel;
                    PState s;
                    s.panel = (int)(pk & kPkPanel) - 1;
                    const uint32_t sph = kPhantom ? ST(kSph) : 0u;
                    const bool fresh = panel ? (pk & kPkFresh) != 0 : sph == 0;
                    if (fresh) {   // starts at its decay point
                        s.x = kPhantom ? STF(kSx0) : J.src_pos[0];
                        s.y = kPhantom ? STF(kSy0) : J.src_pos[1];
                        s.z = kPhantom ? STF(kSz0) : J.src_pos[2];
                        const float sg = gamma ? -1.0f : 1.0f;
                        s.dx = sg * STF(kSox); s.dy = sg * STF(kSoy); s.dz = sg * STF(kSoz);
                        s.E = kE0;
                        s.path = 0.0f;
                        ST(kSE) = __float_as_uint(kE0);
                    } else {
                        s.x = STF(kSx); s.y = STF(kSy); s.z = STF(kSz);
                        s.dx = STF(kSdx); s.dy = STF(kSdy); s.dz = STF(kSdz);
                        s.E = STF(kSE);
                        s.path = STF(kSpath);
                    }
                    bool moved = fresh;   // the direction is not the slot's
                    s.trem = __uint_as_float(st[(fresh && gamma ? kSrem1 : kStrem) * kN + q]);
                    if (panel && (pk & (kPkFresh | kPkLastMask))) {
                        const int wi = !fresh ? kSrw : gamma ? kSin1 : kSpath;
                        enter_panel<kPosed>(geom, s.panel, __uint_as_float(st[wi * kN + q]), s);
                        pk &= ~(kPkFresh | kPkLastMask);
                        moved = true;
                    }
                    const bool late = (panel ? step : sph) >= (uint32_t)kMaxSteps;
                    Loc L;
                    L.crystal = -1;
                    bool left_ring = false;
                    // a branch each for panel and phantom (5 M pairs in the hot-rod phantom: 1.65 ms
                    // against 1.71); a live launch, whose code is the longest, takes one for both
                    // (a served burst: 2.89 ms against 3.03)
                    int what;
                    if (kLive) what = woodcock_step<3, kPosed>(J, geom, W, r, s, panel, L, left_ring);
                    else if (panel) what = woodcock_step<1, kPosed>(J, geom, W, r, s, true, L, left_ring);
                    else what = woodcock_step<2, kPosed>(J, geom, W, r, s, false, L, left_ring);
                    if (panel) pk += late ? 0u : 1u << kPkStep;
                    else ST(kSph) = sph + 1u;
                    to = ph;
                    ST(kStrem) = what >= kStepPhoto ? (uint32_t)L.crystal : __float_as_uint(s.trem);
                    if (moved || what == kStepExit) STORE3(kSdx, s.dx, s.dy, s.dz);
                    bool ends = !panel && what == kStepPhoto;
                    if (what == kStepExit) {
                        if (!panel) {
                            to = kPhFlight;
                        } else if (left_ring) {
                            // its flight would end it: counted as one, without the event
                            ends = true;
                            n_left = 1;
                            const float c0 = fmaf(s.x, s.x, s.y * s.y), a = fmaf(s.dx, s.dx, s.dy * s.dy);
                            if (a > 0.0f && !(c0 < g.R2 * 0.9999f) && outside_screened(g, a, fmaf(s.x, s.dx, s.y * s.dy), c0))
                                n_left = 1u | 1u << 16;
                        } else {
                            pk = (pk & ~kPkPanel) | ((pk & kPkPanel) << kPkLast);
                            to = kPhFlightOut;
                        }
                    } else if (what != kStepVirtual) {
                        ST(kSrw) = r.w & ~511u;
                        pk = (pk & ~kPkPhoto) | (what == kStepPhoto ? kPkPhoto : 0u);
                        to = kPhInteract;   // panel field 0: in the phantom
                    }
                    if (ends) {
                        to = photon_end(pk, (jobw >> kJobPanel1) & 0x7Fu);
                        if (kPhantom) ST(kSph) = 0;
                    }
                    STORE3(kSx, s.x, s.y, s.z);
                    ST(kSpath) = __float_as_uint(s.path);
                    ST(kSpk) = pk;
                    if (late) {   // step cap hit: abandon the history (and its entries), flag the run
                        atomicOr(O.status, kStatusTimeout);
                        to = kPhIdle;
                    }
                }
                count(acc, ph, __popc(am));
                n_left = __reduce_add_sync(kFullMask, n_left);
                count(acc, kPhFlightOut, n_left & 0xFFFFu);
                count(acc, kNScrFlight, n_left >> 16);
            } else {
                // decay, collision and finish take one azimuth
                float sp, cp;
                sincospif(2.0f * u01(ph == kPhInteract ? rw : ph == kPhFinish ? r.y : r.w), &sp, &cp);
                if (ph == kPhInteract) {
                    // the collision found by a step: one Kahn trial an event, a photon
                    // whose trial is rejected stays
                    uint32_t n_hits = 0, n_trials = 0;
                    if (run) {
                        const bool photo = (pk & kPkPhoto) && in_panel;
                        const float E = STF(kSE);
                        float xm1 = 0.f;
                        bool accept = true;
                        if (!photo) {
                            const float k = E * kInvMec2;
                            accept = kahn_try(r, k, 1.0f + 2.0f * k, 9.0f + 2.0f * k, xm1);
                            n_trials = accept ? c3 : 0u;
                        }
                        to = kPhInteract;
                        if (!accept) {
                            if (c3 >= (uint32_t)kMaxTrials) {
                                atomicOr(O.status, kStatusTimeout);
                                to = kPhIdle;
                            }
                            ST(kSrw) = (rw & ~511u) | (c3 & 511u);
                            pk = (pk & ~kPkLastMask) | ((c3 >> 9) << kPkLast);
                        } else {
                            const float x = STF(kSx), y = STF(kSy), z = STF(kSz);
                            const float Ep = E / (1.0f + xm1);
                            const bool dead = photo || Ep < J.e_cut;
                            const float dep = dead ? E : E * xm1 / (1.0f + xm1);
                            const int crystal = in_panel ? (int)ST(kStrem) : -1;
                            if (crystal >= 0) {
                                // a crystal interaction: the history's singles, tallies, optional hit list
                                const uint32_t dtp = (uint32_t)floorf(STF(kSpath) * kInvCmmPerPs);
                                unit = (uint32_t)crystal;
                                if (g.readout_level == 0) unit = (pk & kPkPanel) - 1u;
                                else if (g.readout_level == 1) unit = (uint32_t)crystal / (uint32_t)g.crystals_per_module;
                                // the list's entry of this unit, or its last one
                                uint32_t ei = kEntries * 32, last = 0;
                                next = (jobw >> kJobList) & 63u;
#pragma unroll 1
                                while (next) {
                                    last = next--;
                                    const uint32_t u = P.e_unit[next * 32 + lane];
                                    if (u == unit) ei = next * 32 + lane;
                                    next = P.e_next[next_at(next, lane)];
                                }
                                if (ei < kEntries * 32) {
                                    P.e_e[ei] += dep;
                                    P.e_ew[ei] += dep * x;
                                    P.e_dt[ei] = min(P.e_dt[ei], dtp);
                                } else if (!(pk & kPkOvf)) {
                                    e = take_entry(efree, lane);
                                    if (e < (uint32_t)kEntries) {
                                        ei = e * 32 + lane;
                                        P.e_unit[ei] = unit;
                                        P.e_e[ei] = dep;
                                        P.e_ew[ei] = dep * x;
                                        P.e_dt[ei] = dtp;
                                        P.e_next[next_at(e, lane)] = 0;
                                        if (last) P.e_next[next_at(last - 1u, lane)] = (uint8_t)(e + 1u);
                                        else ST(kSjob) = jobw | ((e + 1u) << kJobList);
                                        pk |= kPkSing;
                                    } else {
                                        // simulated again by the redo kernel; its entries are the others' now
                                        pk = (pk & ~kPkSing) | kPkOvf;
                                        ST(kSjob) = free_list(efree, P.e_next, lane, jobw);
                                    }
                                }
                                n_hits = 1;
                                atomicAdd(J.tally_count + crystal, 1ull);
                                atomicAdd(J.tally_efx + crystal, (unsigned long long)__float2ull_rn(dep * kEfxScale));
                                if (O.hit_cap)
                                    keep_hit(O, J, g, h, (int)(jobw & 0xFFFFu), gamma, step - 1u, crystal, dep, dtp, x, y, z);
                            }
                            pk &= ~kPkLastMask;
                            if (dead) {
                                to = photon_end(pk, (jobw >> kJobPanel1) & 0x7Fu);
                                if (kPhantom) ST(kSph) = 0;
                            } else {
                                // rotation in the panel frame with v as polar reference: for the ring
                                // (w, u, v) is a rotation of (x, y, z) about the axis, so this equals the
                                // global rotation; a posed panel takes its own v axis
                                float dx = STF(kSdx), dy = STF(kSdy), dz = STF(kSdz);
                                rotate_dir(dx, dy, dz, xm1 / (E * kInvMec2), sp, cp);
                                STORE3(kSdx, dx, dy, dz);
                                ST(kSE) = __float_as_uint(Ep);
                                if (in_panel) ST(kStrem) = __float_as_uint(panel_exit(g, x, y, z, dx, dy, dz));
                                to = in_panel ? kPhPanel : kPhPhantom;
                            }
                        }
                        ST(kSpk) = pk;
                    }
                    count(acc, kNHits, __popc(__ballot_sync(kFullMask, n_hits)));
                    count(acc, kNTrials, __reduce_add_sync(kFullMask, n_trials));
                } else if (ph == kPhIdle) {
                    // decay: the pair's direction, and what its photons do first
                    uint32_t n_scr = 0;
                    if (run) {
                        float x0, y0, z0, ox, oy, oz;
                        sample_decay<kPhantom>(J, h, r, sp, cp, x0, y0, z0, ox, oy, oz);
                        to = kPhFlight;
                        if (kPhantom && J.has_phantom && in_phantom(J, x0, y0, z0)) {
                            to = kPhPhantom;
                            pk = kPkPhantom1;
                        } else {
                            if (start_screened<kPosed>(g, x0, y0, z0, ox, oy, oz)) {
                                n_scr = 1;
                                pk = kPkGamma;     // (for the flight event: photon 1's flight only)
                            }
                            if (start_screened<kPosed>(g, x0, y0, z0, -ox, -oy, -oz)) {
                                pk |= kPkFresh;    // (photon 0's flight only)
                                if (++n_scr == 2) to = kPhIdle;
                            }
                        }
                        ST(kSh0) = (uint32_t)h;
                        ST(kSh1) = (uint32_t)(h >> 32);
                        ST(kSjob) = jobw;
                        STORE3(kSox, ox, oy, oz);
                        ST(kSpk) = pk;
                        if (kPhantom) {
                            STORE3(kSx0, x0, y0, z0);
                            ST(kSph) = 0;
                        }
                    }
                    const uint32_t got = __popc(__ballot_sync(kFullMask, run));
                    count(acc, kPhIdle, got);
                    count(acc, kNScrStart, __reduce_add_sync(kFullMask, n_scr));
                    if (kLive) {
                        if (got || !alone) {
                            live_idle_reset(idle);
                        } else if (!done) {
                            // no chunk published: the launch's host has nothing yet
                            int status = kStatusOk;
                            if (__any_sync(kFullMask, live_idle_wait(idle, status, W, O))) {
                                if (lane == 0) atomicOr(O.status, kStatusLiveStall);
                                done = true;
                            }
                        }
                    }
                } else {
                    // digitizer: one single of the history's list, in list order
                    const bool ovf = run && (pk & kPkOvf), one = run && !ovf;
                    append_overflow(O, ovf, h, (int)(jobw & 0xFFFFu), kFullMask);
                    SingleOut so;
                    so.keep = false;
                    if (one) {
                        const uint32_t ei = e * 32 + lane;
                        blur_single(J, r, sp, cp, unit, P.e_e[ei], P.e_dt[ei], P.e_ew[ei], so);
                        free_entry(efree, lane, e);
                    }
                    append_single<kLive, true>(W.geoms, O, J, (int)(jobw & 0xFFFFu), h, 0, so, kFullMask);
                    const bool last = ovf || !next;
                    if (run && !last) ST(kSjob) = (jobw & ~(63u << kJobList)) | (next << kJobList);
                    to = last ? kPhIdle : kPhFinish;
                    // An overflow tells that the class has more histories in flight than entries
                    // for them: the slot is given up (no event serves the phase it goes to), but
                    // for the class's first ones.  Overflows (on the CPU) at 2.6 hits per pair, without and with
                    // the rule: 2.0 and 0.6 % of 15 M histories; at 3.8 hits 21 and 1.9 %, at 11 hits
                    // 75 and 26 %; at one hit none.
                    if (ovf && (bit >> kKeptSlots)) to = kPhGivenUp;
                    count(acc, kNFin, __popc(__ballot_sync(kFullMask, run && last)));
                    count(acc, kNSingles, __popc(__ballot_sync(kFullMask, one)));
                }
            }
        }
        // 4. hand the slots on to their next phases, their state first
        __threadfence_block();
        if (active) atomicOr(&mask[to][lane], bit);
        __syncwarp();
    }
#undef ST
#undef STF
#undef STORE3
    if (lane < kNCount && acc) atomicAdd(O.counters + kCtaCounters + lane, (unsigned long long)acc);
}

// The launch shapes: 448 threads by default, or 128, 256 or 512
// (gpet_options.block_size); slots of a lane class without and with the
// phantom's state words, and CTAs an SM.  Measured on a sweep position (1e7
// pairs, transport ms) and on the hot-rod phantom (5e6 pairs) when the scheme was
// new, and again at 1.04 ms with the same order (15 warps 1.09): 12 warps 1.31 and
// 1.97, 14 warps 1.28 and 1.89, 15 warps 1.27 and 1.88 (two CTAs an SM each);
// 8 warps 1.66 (two CTAs) and 1.57 (three); 20 warps (one CTA) 1.68.
template <int WARPS>
struct Shape;
template <> struct Shape<4> { static constexpr int kPlain = 12, kPhantom = 10, kCtas = 4; };
template <> struct Shape<8> { static constexpr int kPlain = 18, kPhantom = 16, kCtas = 3; };
template <> struct Shape<14> { static constexpr int kPlain = 32, kPhantom = 28, kCtas = 2; };
template <> struct Shape<16> { static constexpr int kPlain = 32, kPhantom = 28, kCtas = 2; };

// the kernel that cfg and kTab select, and the size of its pool
template <int WARPS, int kTab>
static const void *cta_kernel(const LaunchCfg &cfg, size_t *pool) {
    using S = Shape<WARPS>;
    *pool = cfg.phantom ? sizeof(CtaPool<S::kPhantom, true>) : sizeof(CtaPool<S::kPlain, false>);
    if constexpr (kTab == kTabJobs)
        if (cfg.live) return (const void *)k_transport_cta<WARPS, S::kPhantom, S::kCtas, true, true, true, kTab>;
    if (cfg.phantom)
        return cfg.posed ? (const void *)k_transport_cta<WARPS, S::kPhantom, S::kCtas, true, true, false, kTab>
                         : (const void *)k_transport_cta<WARPS, S::kPhantom, S::kCtas, true, false, false, kTab>;
    return cfg.posed ? (const void *)k_transport_cta<WARPS, S::kPlain, S::kCtas, false, true, false, kTab>
                     : (const void *)k_transport_cta<WARPS, S::kPlain, S::kCtas, false, false, false, kTab>;
}

// (the other shapes and live launches have the general form alone)
static bool has_tab(const LaunchCfg &cfg) { return !cfg.live && cfg.block_size == kCtaThreads; }
static_assert(kCtaThreads != 128 && kCtaThreads != 256 && kCtaThreads != 512, "the other shapes take the job table");

static const void *cta_kernel(const LaunchCfg &cfg, int tab, int *threads, size_t *pool) {
    switch (cfg.block_size) {
        case 128: *threads = 128; return cta_kernel<4, kTabJobs>(cfg, pool);
        case 256: *threads = 256; return cta_kernel<8, kTabJobs>(cfg, pool);
        case 512: *threads = 512; return cta_kernel<16, kTabJobs>(cfg, pool);
        default: *threads = kCtaThreads;
    }
    constexpr int kW = kCtaThreads / 32;
    return tab == kTabOne ? cta_kernel<kW, kTabOne>(cfg, pool) : tab == kTabStaged ? cta_kernel<kW, kTabStaged>(cfg, pool)
                                                                                  : cta_kernel<kW, kTabJobs>(cfg, pool);
}

// A launch's kernel, its form of the tables, threads, dynamic shared memory,
// CTAs and staged geometries
struct CtaLaunch {
    const void *k;
    int tab, threads, ctas, ng;
    size_t smem;
};
static cudaError_t cta_shape(int n_geoms, const LaunchCfg &cfg, CtaLaunch &L) {
    L.tab = !has_tab(cfg) ? kTabJobs : cfg.one_job ? kTabOne : kTabStaged;
    int occ = 0;
    for (;; L.tab = kTabJobs) {
        size_t pool = 0;
        L.k = cta_kernel(cfg, L.tab, &L.threads, &pool);
        cudaError_t e = staged_geometry(L.k, L.threads, pool, n_geoms, cfg.max_smem_geoms, &L.ng, &L.smem, &occ);
        if (e != cudaSuccess) return e;
        // (all geometries fit beside the pool, one of them always does)
        if (L.tab == kTabJobs || (L.ng >= n_geoms && occ >= 1)) break;
    }
    if (occ < 1) return cudaErrorInvalidConfiguration;
    L.ctas = cfg.sm_count * occ;
    return cudaSuccess;
}

// resident warps of the launch that launch_transport_cta makes
cudaError_t cta_resident_warps(int n_geoms, const LaunchCfg &cfg, long long *warps) {
    CtaLaunch L{};
    cudaError_t e = cta_shape(n_geoms, cfg, L);
    *warps = (long long)L.ctas * (L.threads / 32);
    return e;
}

cudaError_t launch_transport_cta(const WorkDev &W, const OutDev &O, const LaunchCfg &cfg, cudaStream_t st) {
    CtaLaunch L{};
    cudaError_t e = cta_shape(W.n_geoms, cfg, L);
    if (e != cudaSuccess) return e;
    CtaTables<kTabJobs> many{L.ng};
    CtaTables<kTabStaged> all{L.ng};
    CtaTables<kTabOne> one;
    if (L.tab == kTabOne) one = {*cfg.one_job, *cfg.one_geom};
    void *tables = L.tab == kTabOne ? (void *)&one : L.tab == kTabStaged ? (void *)&all : (void *)&many;
    void *args[] = {const_cast<WorkDev *>(&W), const_cast<OutDev *>(&O), tables};
    return cudaLaunchKernel(L.k, dim3(L.ctas), dim3(L.threads), args, L.smem, st);
}

void cta_counters(unsigned long long *c, const unsigned long long *raw) {
    static_assert((int)kNCount == kCtaCounterSlots, "one raw slot per count");
    c[0] += raw[kPhPanel];
    c[1] += raw[kPhFlight] + raw[kPhFlightOut] + raw[kNScrStart];
    c[2] += raw[kNTrials];
    c[3] += raw[kNEntered];
    c[4] += raw[kPhPhantom];
    c[5] += raw[kNHits];
    c[6] += raw[kNIter];
    c[7] += raw[kNLanes];
    c[8] += raw[kNScrStart] + raw[kNScrFlight];
    c[9] += raw[kNSingles];
    // events per phase: slots 10 + phase
    c[10 + kPhSource] += raw[kPhIdle];
    c[10 + kPhPhantom] += raw[kPhPhantom];
    c[10 + kPhFlight] += raw[kPhFlight];
    c[10 + kPhPanel] += raw[kPhPanel];
    c[10 + kPhFinish] += raw[kNFin];
    c[10 + kPhFlightOut] += raw[kPhFlightOut];
}

// load every instantiation and set its shared-memory limit (internal.h)
cudaError_t preload_cta_kernels() {
    for (int block : {128, 256, kCtaThreads, 512})
        for (int form = 0; form < 5; ++form) {
            LaunchCfg cfg{};
            cfg.block_size = block;
            cfg.phantom = form & 1;
            cfg.posed = form & 2;
            cfg.live = form == 4;
            for (int tab = 0; tab < (has_tab(cfg) ? 3 : 1); ++tab) {
                int threads = 0;
                size_t pool = 0;
                const void *k = cta_kernel(cfg, tab, &threads, &pool);
                cudaError_t e = ensure_dynamic_smem(k, pool + (size_t)kMaxStagedGeoms * sizeof(GeomDev));
                if (e != cudaSuccess) return e;
            }
        }
    return cudaSuccess;
}

}  // namespace gpet
