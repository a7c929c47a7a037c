// pool.cpp -- the slot-pool transport kernel's own source, one CTA of it, on the
// CPU (warp_fibers.h), for a ring of twelve panels of one crystal material, run
// under two schedules of its warps.  What a history does may not depend on the
// schedule: both runs have the same tallies, and a history that overflowed in
// neither has the same singles in both.
// Arguments: warps (4, 8, 14, 16; 114: 14, with the phantom's state words), pairs,
// Compton and photoelectric coefficient at 511 keV (1/cm), depth (mm), crystal
// pitch (mm), half-length of the ring (mm), cutoff (keV), readout level, seed of
// the schedules, length of a decay's, collision's or finish event against the
// others', most warp passes per pair.
// Prints per schedule: end (0: every warp ended, 2: pass limit), status, histories
// begun, hits, singles kept, histories that overflowed, events, lanes; then the
// number of disagreements between the two.
#include "warp_fibers.h"

namespace gpet { alignas(128) unsigned char smem[1 << 20]; }
#include "cta_kernel.inc"

using namespace gpet;

static WorkDev W{};
static OutDev O{};
static CtaTables<kTabOne> T;

template <int WARPS, int SLOTS, bool PH>
static void cta() { k_transport_cta<WARPS, SLOTS, 1, PH, false, false, kTabOne>(W, O, T); }

int main(int argc, char **argv) {
    if (argc < 13) return 1;
    auto arg = [&](int i) { return std::atof(argv[i]); };
    const int shape = std::atoi(argv[1]), n = std::atoi(argv[2]);
    const float depth = (float)arg(5), pitch = (float)arg(6), half_v = (float)arg(7), R = 55.0f, half_u = 14.5f;
    GeomDev g{};
    g.n_panels = 12; g.n_layers = 1; g.n_materials = 2; g.modules_u = g.modules_v = 1; g.readout_level = std::atoi(argv[9]);
    g.R = R; g.W = depth; g.half_u = half_u; g.half_v = half_v;
    g.msu = g.mpu = 2 * half_u; g.msv = g.mpv = 2 * half_v;
    g.inv_mpu = 1 / g.mpu; g.inv_mpv = 1 / g.mpv;
    g.mu_c511[1] = (float)arg(3); g.mu_pe511[1] = (float)arg(4);
    const float ro = R + depth;
    g.R2 = R * R; g.rout2 = (ro * ro + half_u * half_u) * 1.000001f; g.beta = std::atan2(half_u, R);
    g.dphi = (float)(2 * M_PI / 12); g.inv_dphi = 1 / g.dphi; g.w_clear = 3.0e38f;
    for (int k = 0; k < 12; ++k) g.cs[k] = {(float)std::cos(2 * M_PI * k / 12), (float)std::sin(2 * M_PI * k / 12)};
    LayerDev &L = g.layers[0];
    L.w1 = depth; L.pitch_u = L.pitch_v = pitch; L.inv_pitch_u = L.inv_pitch_v = 1 / pitch;
    L.ghi_u = L.ghi_v = pitch; L.n_u = (int)(g.msu / pitch); L.n_v = (int)(g.msv / pitch); L.crystal_mat = 1;
    g.crystals_per_module = L.n_u * L.n_v;
    g.n_crystals = 12 * g.crystals_per_module;

    JobDev J{};
    J.seed = 7; J.n_decays = J.n_hist = n; J.t_span_ps = 1000000000000ull; J.e_cut = (float)arg(8);
    J.e_hi = 1e9f; J.src_pos[2] = 3;
    // Klein-Nishina cross-section over its value at 511 keV
    auto kn = [](double k) {
        const double q = 1 + 2 * k, ln = std::log(q);
        return (1 + k) / (k * k) * (2 * (1 + k) / q - ln / k) + ln / (2 * k) - (1 + 3 * k) / (q * q);
    };
    W.ln_emin = std::log(kXsEmin);
    const double h = (std::log(511.0) - W.ln_emin) / kXsIntervals;
    std::vector<float> gtab(kXsIntervals + 1);
    for (int i = 0; i <= kXsIntervals; ++i) gtab[i] = (float)(kn(std::exp(W.ln_emin + h * i) / 511.0) / kn(1.0));
    W.gtab = gtab.data(); W.inv_h = (float)(1 / h);

    fibers::slow_events = arg(11);
    std::vector<unsigned long long> count[2], efx[2];
    std::vector<uint64_t> singles[2];
    std::vector<char> overflowed[2];
    long long bad = 0;
    for (int run = 0; run < 2; ++run) {
        count[run].resize(g.n_crystals); efx[run].resize(g.n_crystals);
        J.tally_count = count[run].data(); J.tally_efx = efx[run].data();
        const unsigned chunk = 256;
        unsigned long long starts[2] = {0, (n + chunk - 1) / chunk}, next = 0, n_s = 0, n_h = 0, n_o = 0;
        unsigned long long counters[kCtaCounters + kCtaCounterSlots] = {};
        int status = 0;
        std::vector<RawSingle> raw((size_t)n * 48);
        std::vector<uint64_t> keys(raw.size()), ovf_h(n);
        std::vector<int> ovf_job(n);
        W.jobs = &J; W.n_jobs = 1; W.geoms = &g; W.n_geoms = 1; W.chunk_start = starts; W.total_chunks = starts[1];
        W.next_chunk = &next; W.chunk_size = chunk;
        O.s_raw = raw.data(); O.n_singles = &n_s; O.s_cap = raw.size(); O.s_keys = keys.data(); O.key_shift = 64;
        O.n_hits = &n_h; O.ovf_h = ovf_h.data(); O.ovf_job = ovf_job.data(); O.n_ovf = &n_o; O.ovf_cap = n;
        O.counters = counters; O.status = &status;
        T.J = J;
        T.g = g;
        void (*f)() = shape == 4 ? cta<4, 12, false> : shape == 8 ? cta<8, 18, false> : shape == 16 ? cta<16, 32, false>
                      : shape == 114 ? cta<14, 28, true> : cta<14, 32, false>;
        const int end = fibers::run(shape % 100, f, (uint64_t)std::atoll(argv[10]) + run, (uint64_t)(arg(12) * n));
        if (end == 0) cta_counters(counters, counters + kCtaCounters);
        unsigned long long hits = 0;
        for (unsigned long long c : count[run]) hits += c;
        std::printf("%d %d %llu %llu %llu %llu %llu %llu\n", end, status, counters[10 + kPhSource], hits, n_s, n_o,
                    counters[6], counters[7]);
        if (end) return 0;
        // a history's singles, whatever their order
        singles[run].resize(n);
        overflowed[run].resize(n);
        for (unsigned long long i = 0; i < n_s; ++i) {
            uint64_t x = keys[i] * 0x9E3779B97F4A7C15ull;
            for (uint32_t v : {(uint32_t)raw[i].unit, __float_as_uint(raw[i].e_raw), __float_as_uint(raw[i].e),
                               __float_as_uint(raw[i].doi)})
                x = (x ^ v) * 0xD6E8FEB86659FD93ull;
            singles[run][raw[i].h] += x;
        }
        for (unsigned long long i = 0; i < n_o; ++i) {
            bad += overflowed[run][ovf_h[i]]++;          // listed once,
            bad += singles[run][ovf_h[i]] != 0;          // and without singles of its own
        }
        bad += hits != counters[5];
    }
    bad += count[0] != count[1] || efx[0] != efx[1];
    for (int i = 0; i < n; ++i) bad += !overflowed[0][i] && !overflowed[1][i] && singles[0][i] != singles[1][i];
    std::printf("%lld\n", bad);
    return 0;
}
