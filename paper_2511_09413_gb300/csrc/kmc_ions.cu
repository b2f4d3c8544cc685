// kmc_ions.cu -- single-device launches of the ion-list tile (kmc_ions.cuh) and the
// choice of a device's tile.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "kmc_ions.cuh"

namespace kmc {

namespace {

// 4 CTAs of 256 threads per SM (64 registers).  With 5 (48 registers) the
// replicated 512-site device ran 4-11 % slower, with 3 (80) 4 % slower.  Rails of
// more than 32 entries a lane are of 1,025 sites and more, whose site table and
// columns leave room for 20 warps on an SM at most: they run in CTAs of up to as
// many (96 registers), so that the table is held once.  2,500 rails of 2,048 sites
// (16.4 warps an SM, half of them in a second wave in CTAs of 8): 5.1 -> 3.5 ms for
// 300 steps in one wave of CTAs of 17.
bool ion_wide(int kind) { return kind >= kWordKinds + 8; }
int ion_most_smem(int kind) { return ion_wide(kind) ? kGradSmem : 200 * 1024; }
template <class M>
constexpr int kIonWarps = sizeof(M) > 4 ? 20 : 8;
template <int P, bool ACC, bool OPEN, class M, int AHEAD = OPEN ? kIonAhead : 4>
__global__ void __launch_bounds__(32 * kIonWarps<M>, sizeof(M) > 4 ? 1 : 4) ion_kernel(const __grid_constant__ SweepArgs a, const int *gate)
{
    extern __shared__ __align__(16) uint8_t smem[];
    if (gate && *gate != 0) return;     // the occupancy words advance this device
    const int64_t tile_rail0 = (int64_t)blockIdx.x * (blockDim.x >> 5) * (32 / P);
    ion_tile<P, ACC, OPEN, M, false, AHEAD>(a, a.rk0, a.rk1, a.t0, a.n_steps, a.flush, tile_rail0, smem);
}

// Slots of a lane's column, two more than the rows its bits can count (one that
// the draw loop reads ahead, one that an end entry may take before the entries
// are dealt out again): blocking rails keep their ion counts (at most n_max), an
// open rail holds at most one entry per site.  0: more rows than bits.
int ion_rows(int P, int L, bool open, int64_t n_max, int bits)
{
    const int even = (int)(((open ? (int64_t)L : n_max) + P - 1) / P);   // a lane's even share
    if (even > bits) return 0;
    return std::min(even + (open ? 2 : 0), even <= 32 ? 32 : bits) + 2;
}
int ion_rows(int P, int L, bool open, int64_t n_max)
{
    return ion_rows(P, L, open, n_max, P == 32 ? 64 : 32);
}

}  // namespace

// Blocking rails on 32 lanes with at most four ions to a lane (two slots more)
static bool ion_few(int P, bool open, int rcap) { return P == 32 && !open && rcap <= 6; }

IonLayout ion_layout(int P, int Z, int L, bool open, bool persite, int rcap, bool grad, bool acc, bool rule)
{
    const uint32_t G = 32u / (uint32_t)P, rows = ((uint32_t)Z << (persite && !acc ? 2 : 0)) + (open ? 5u : 1u);
    const uint32_t words = G * (uint32_t)((L + 31) >> 5) * 4u;   // occupancy words, staged in the bounds
    const uint32_t gz = G * (uint32_t)Z;
    const uint32_t pz = (uint32_t)align16(4u * G * (uint32_t)(Z + 1));
    IonLayout y;
    y.tab = 16u * (uint32_t)(L + 2);
    y.row = rows * 16u;
    y.p0b = ion_fixed(P) + (uint32_t)align16(std::max(G * y.row, words));
    y.pb = y.p0b + (persite ? (uint32_t)align16(8u * gz) : 0u);
    y.st = y.pb + pz;
    y.hit = y.st + 128u * kIonSlots;
    y.g = y.hit + 128u * (acc ? (rule ? 1u : 0u) : open || ion_few(P, open, rcap) ? (uint32_t)kIonAhead : 4u) * (grad || rcap > 34 ? 2u : 1u);
    y.col = y.g + (grad ? 2688u + 64u * G + (uint32_t)align16(8u * G * (uint32_t)(Z + 1)) + 48u * gz : 0u);
    y.bytes = y.col + (uint32_t)rcap * 128u;
    return y;
}

// The tile and its lanes per rail.
//
// Ion lists against occupancy words (one GB300, site-updates/s, words first):
// with the accept path 6.6e11 -> 1.29e12 at 65,536 x 512 rails 20 % full, 3.9e11
// -> 5.7e11 at 8,192 x 1,000 half full, 4.0e11 -> 4.2e11 at 70 %; without it
// 8.5e11 -> 8.6e11 at 8,192 x 1,000 and 7.6e11 -> 8.4e11 at 16,384 x 512 half
// full, 8.4e11 -> 7.3e11 at 60 % (blocked ions draw in vain, and there is little
// rebuilding to save).  Rails of a few sites have next to no ions, and the words
// put 32 of them on a warp (4 sites: 2.7e11 -> 1.2e11; 8: 1.1e11 -> 1.6e11).
//
// (The handle knows the filling of step 0 only; a long launch looks again, tile_gate.)
//
// Few lanes per rail spread a step's fixed work (bounds, refresh, votes) over
// more ions of a lane and waste less of the last row; they also make fewer
// warps.  6,000 warps fill the GPU (152 SMs x 32) with something to spare for
// the last wave; with the accept path 3,600 in one wave of even CTAs do (8,192 x
// 1,000 on 16 lanes: 300 steps 3.16 -> 2.91 ms; without it 1.23 -> 1.25 ms for
// 200).  Below about six ions to a lane the fixed work costs more than half-empty
// SMs (32,768 x 128, 26 ions: 3.0e11 on 32 lanes, 4.1e11 on 16, 5.6e11 on 8,
// 6.0e11 on 4).
float tile_max_fill(bool acc) { return acc ? 0.7f : 0.5f; }

// The filling at which random rails run equally long on both tiles (16,384 x 512,
// 65,536 x 100 and 4,000 x 1,000: without the accept path 0.93 to 0.95 times the words' time
// on the lists at 55 %, 1.01 to 1.02 at 60 %; with it 0.81 to 0.91 at 70 %, 1.01 to 1.13 at
// 80 %), and the share of blocked ions where they stand in runs: without the accept
// path 0.86 to 1.03 at up to 0.3 and 1.13 to 1.26 at 0.5; with it 0.79 to 0.89 at 0.75 and up
// to 1.7 at 0.94.  Rails held together by a field are at 0.9 and more: 2 to 7 times.
struct TileLine {
    float fill, blocked;
};
static TileLine tile_line(bool acc) { return acc ? TileLine{0.75f, 0.9f} : TileLine{0.58f, 0.35f}; }

// The tile for a device as it stands, from 32 rails spread over it, a warp to each:
// *words = 1 for the occupancy words, when more than line.fill of their sites are
// occupied or more than line.blocked of their ions held on both sides, by an ion or a
// blocking electrode, 0 for the lists.  Both tiles are launched after it and one of
// them returns at once (2 us); the choice changes no result.  dst (may be null) receives
// the arguments.
static __global__ void __launch_bounds__(1024) tile_gate_kernel(const __grid_constant__ SweepArgs a, SweepArgs *dst,
                                                                TileLine line, int *words)
{
    __shared__ int ions, held;
    if (threadIdx.x == 0) {
        if (dst) *dst = a;
        ions = held = 0;
    }
    if (!words) return;
    __syncthreads();
    const uint8_t *row = a.occ + (int64_t)(threadIdx.x >> 5) * a.R / 32 * a.stride;
    const int wall = a.electrodes == 1 ? 0 : 1;
    int n = 0, b = 0;
    for (int k = (int)(threadIdx.x & 31u); k < a.L; k += 32) {
        const int left = k > 0 ? row[k - 1] : wall, right = k + 1 < a.L ? row[k + 1] : wall;
        n += row[k];
        b += row[k] & left & right;
    }
    n = __reduce_add_sync(0xffffffffu, n);
    b = __reduce_add_sync(0xffffffffu, b);
    if ((threadIdx.x & 31u) == 0u) {
        atomicAdd(&ions, n);
        atomicAdd(&held, b);
    }
    __syncthreads();
    if (threadIdx.x == 0)
        *words = (float)ions > line.fill * 32.0f * (float)a.L || (float)held > line.blocked * (float)ions ? 1 : 0;
}

cudaError_t tile_gate(const SweepArgs &a, SweepArgs *dst, bool acc, int *words, cudaStream_t s)
{
    tile_gate_kernel<<<1, words ? 1024 : 32, 0, s>>>(a, dst, tile_line(acc), words);
    return cudaGetLastError();
}

// Building the lists and writing them back takes as long as a few steps, and without
// the accept path the least that is drawn is four steps.  Lists' time over the words',
// 1, 2, 3, 4 and 8 steps without the accept path: 1.3, 1.05, 0.99, 0.92, 0.83 on 1,000 x 300, 1.5, 1.3,
// 1.13, 1.03, 0.9 on 16,384 x 512 open, 2.8, 2.1, 1.8, 1.5, 1.3 (1.16 for 16, 0.96 for 32) on 65,536 x 1,024 open
// with a warp to every rail; with it 1.4, 1.2, 1.05, 0.98 on 16,384 x 512, 1.5, 1.25, 1.14, 1.07 on
// 65,536 x 1,024 open, 0.9 on 1,000 x 300.  With many zones to a lane of the words the lists
// are faster from the first step on (65,536 x 100, 32 zones: 0.73).
int64_t words_up_to(const TileShape &t, int64_t rails, int L, int Z, bool acc)
{
    int wpl = 1;
    if (!t.ions || rails < 1000 || Z > 4 * sweep_pick_lpr(L, &wpl)) return 0;
    const bool own = t.lpr == 32 && rails >= 32768;     // a warp to a rail, several waves
    if (acc) return L >= 256 && rails >= 10000 ? (own ? 3 : 1) : 0;
    return own ? 16 : 3;
}

// Many rails of few sites and few zones.  The words put a rail of up to 32 sites on one
// lane and of up to 64 on two, where the lists take four and repeat a warp's fixed work
// two to eight times as often; zones bring the two together, as a warp evaluates those
// of all its rails.  65,536 rails, 64 steps, times of the lists over those of the words:
// closed with the accept path 1.7, 1.6, 1.4, 1.3 and 0.9 at 8 sites (1, 2, 4, 7 and 8 zones), 1.3, 1.2
// and 0.98 at 16 (1, 2, 4); open without it 2.0, 1.4, 1.05 and 0.65 at 16 (1, 4, 8, 10; 40 % full
// 2.2, 1.9, 1.5 and 0.94), 1.5 to 1.0 at 24 and 32 (1), 1.05 to 0.85 at 48 and 64; closed
// without it below 1 at all; open with it 1.6, 1.3 and 0.54 at 16 (1, 4, 10) under a slow
// voltage, but 0.7 and 0.4 under one that moves by 8 mV a step, whose draws the words' bands
// of 32 steps leave to their slow path: these stay on the lists.  With fewer rails the words
// leave SMs idle: from 24,000 on 1.1 to 1.5 at up to 16 sites and two zones, from 4,000 on 1.1
// to 1.4 at 8 closed ones with the accept path.
static bool words_for_few_sites(int64_t rails, int L, int Z, bool open, bool acc)
{
    int most = 0;       // zones
    if (acc && !open) most = rails >= 40000 ? (L < 16 ? 7 : L <= 32 ? 2 : 0) : rails >= 4000 && L < 16 ? 3 : 0;
    if (!acc && open) most = rails >= 40000 ? (L < 24 ? 9 : L <= 32 ? 2 : 0) : rails >= 20000 && L < 24 ? 2 : 0;
    return Z <= most;
}

// Without the accept path although a hop is likely (a caller's choice): on the lists
// every move costs the steps drawn ahead, so they win on few rails only (16,384 x 512
// closed 1.05 times the words' time at P0 = 0.17, 0.85 at 0.07; open 1.6 and 1.2, 1.04 at
// 0.02; 300 x 100 0.4).
static bool words_for_likely_hops(int64_t rails, bool open, double P0)
{
    return rails >= 4000 && P0 > (open ? 1.0 / 64.0 : 1.0 / 8.0);
}

TileShape pick_tile(int64_t rails, int64_t n_rails, int L, int Z, bool open, int64_t n_tot, int64_t n_max, bool acc, double P0)
{
    TileShape t{};
    const double mean = (double)n_tot / (double)n_rails;
    if (L >= 8 && mean <= tile_max_fill(acc) * L && !words_for_few_sites(rails, L, Z, open, acc) &&
        (acc || !words_for_likely_hops(rails, open, P0))) {
        int P = 32;
        while (P > 4) {
            const int64_t warps = rails * (P / 2) / 32;
            const bool enough = warps >= (acc ? 3600 : 6000) || (mean / P < 6.0 && warps >= 2400);
            if (!enough || ion_rows(P / 2, L, open, n_max) == 0) break;
            P >>= 1;
        }
        t.ions = 1;
        t.lpr = P;
        t.rcap = ion_rows(P, L, open, n_max);
        const int k = P == 4 ? 0 : P == 8 ? 1 : P == 16 ? 2 : t.rcap <= 34 ? 3 : 4;
        t.kind = kWordKinds + 2 * k + (open ? 1 : 0);
        return t;
    }
    t.wpl = 1;
    t.lpr = sweep_pick_lpr(L, &t.wpl);
    t.kind = sweep_kind(t.lpr, t.wpl);
    return t;
}

// One ion crossing boundary b changes P_b by one, so Q_b-1 and Q_b by a half and
// their mean by at most that much: no zone's Q_z - Qbar moves by more than a half,
// its exponent by |kappa alpha| / (2 L kT).  Exchanges with an electrode alternate
// in and out as long as the list keeps its entries, so they shift a rail by one at
// each end and are not counted; where that leaves no room they are.  Room for ten
// crossings, at most 0.25 (a fifth more draws to look at), at least 0.05.  Where an
// open rail is so short that not counting its exchanges takes more, up to 0.7: every
// exchange would use up room that a crossing needs (65,536 x 48 rails 40 % full, an
// exchange in most steps, 64 steps: 1.59 ms counting them, 0.79 not; 0.93 on the
// occupancy words).  e^s < 1 + s + s^2 and e^-s > 1 - s there.
static void ion_slack(SweepArgs &a, bool open)
{
    const double per = 0.505 * fabs((double)a.ka_f) * (double)a.inv_LkT;
    double slack = std::min(0.25, std::max(0.05, 10.0 * per));
    if (open && 0.99 * slack < 4.0 * per && 4.1 * per <= 0.7) slack = 4.1 * per;
    a.ion_slack = (float)slack;
    const int fits = per * 1000.0 < 0.99 * slack ? 1000 : (int)floor(0.99 * slack / per);
    a.ion_exchange = open && fits < 4 ? 1 : 0;
    a.ion_budget = open && fits >= 4 ? fits - 2 : fits;
}

size_t tile_args(SweepArgs &a, const TileShape &t, const kmc_params &p, bool persite, int warps, bool acc)
{
    if (!t.ions) return sweep_smem_bytes(t.lpr, t.wpl, p.n_zones, p.n_sites, warps, 0, acc);
    a.rcap = t.rcap;
    a.rcpZ = 65536u / (uint32_t)p.n_zones + 1u;
    ion_slack(a, p.electrodes == 1);
    a.cls_shift = persite && !acc ? 2 : 0;
    a.iy = ion_layout(t.lpr, p.n_zones, p.n_sites, p.electrodes == 1, persite, t.rcap, false, acc,
                      p.update_rule != 0);
    return a.iy.tab + (size_t)warps * a.iy.bytes;
}

// Warps per CTA of a launch over `warps` warps.  When all are
// resident at once the launch takes as long as the fullest SM sub-partition: the
// CTA size that leaves it the fewest warps, of equals the largest (4,000 warps of
// 16,000 x 200 rails: 8 to a sub-partition and 2.94 ms in CTAs of 8, 7 and 2.60 ms
// in CTAs of 7; 64 warps: 2 and 0.41 ms in CTAs of 8, 1 and 0.36 ms in CTAs of 4).
// In more than one wave 8 (16,384 x 1,024: 6.8 ms in CTAs of 8, 6.8 of 4, 7.6
// of 2, which repeat the site table more often), or of the wide CTAs those that
// hold the most warps on an SM.
int ion_cta_warps(const SweepArgs &a, int kind, int64_t warps)
{
    int dev = 0, sms = 0, sm = 0, cta = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&cta, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (cta <= 0) cta = 48 * 1024;
    sms = std::max(sms, 1);
    const bool wide = ion_wide(kind);
    int best = 1;
    int64_t least = INT64_MAX, most = 0;
    for (int w = wide ? kIonWarps<uint64_t> : kIonWarps<uint32_t>; w >= 1; --w) {
        const size_t smem = a.iy.tab + (size_t)w * a.iy.bytes;
        if (smem > (size_t)std::min(cta, ion_most_smem(kind))) continue;
        // the system takes 1 KB a CTA
        const int64_t resident = std::min<int64_t>((wide ? 20 : 32) / w, std::max(sm, cta) / (int64_t)(smem + 1024));
        const int64_t per_sm = ((warps + w - 1) / w + sms - 1) / sms;
        if (per_sm > resident) {
            if (least == INT64_MAX && (wide ? resident * w : w) > most) {
                most = wide ? resident * w : w;
                best = w;
            }
            continue;
        }
        const int64_t fullest = (per_sm * w + 3) / 4;
        if (fullest < least) {
            least = fullest;
            best = w;
        }
    }
    return best;
}

// The gradient pass's tile.  An FP64 warp instruction takes the SM's FP64 pipe for
// 16 cycles whatever the number of lanes at work, so the fewest lanes per rail are
// the best: a rail's zones then fill the lanes (10 zones on 4 lanes: 10 of 12) and
// its sums are formed once for 8 rails (65,536 x 512 rails: 56 us a step on 4
// lanes, 70 on 8, 91 on 16, 155 on 32).  More lanes only where fewer than 1,200
// warps would be left (4,096 rails: 9.0 us on 4, 7.3 on 8, 6.7 on 16, 11 on 32).
//
// The words take fewer lanes for a rail of few sites, so their warps repeat the fixed
// work less often; the lists evaluate fewer zones (only where an ion crossed a
// boundary), and a voltage that moves does not widen their bounds as much.  Lists' time
// over the words', 64 steps at 20 % filling under a slow voltage: 65,536 rails closed 1.9,
// 1.4, 1.05 and 0.8 at 32 sites (1, 2, 4 and 7 zones), 1.3, 1.3 and 0.95 at 64 (1, 2, 4), open 2.3, 1.7, 1.3
// and 0.97 at 32 and 1.4, 1.4, 1.15 at 64; 24,000 rails closed 1.4, 1.15 and 0.83 at 32 (1, 2, 4), open 1.5, 1.3
// and 0.95; open rails whose lists make two waves by their shared memory (10 zones) 1.3 at
// up to 32 sites and 1.0 to 1.4 at 64, in one wave (7 zones) 0.75.  On fewer rails, and on
// longer ones, each side wins somewhere (1,500 to 4,000 rails of one zone: 0.6 to 1.3 by
// filling and voltage): they stay on the lists.
static bool words_for_gradient(int64_t rails, int L, int Z, bool open, int64_t waves)
{
    if (rails < 16000 || L > 64) return false;
    if (open && waves > 1 && (rails < 40000 || L > 32) && Z <= 10) return true;
    return Z <= (rails >= 40000 ? (L <= 32 ? 4 : 2) : (L <= 32 ? 3 : 0));
}

TileShape pick_grad_tile(int64_t rails, int64_t n_rails, const kmc_params &p, int64_t n_tot, int64_t n_max)
{
    TileShape t{};
    const int L = p.n_sites;
    const bool open = p.electrodes == 1;
    if (L >= 8 && (double)n_tot <= tile_max_fill(true) * (double)n_rails * (double)L) {
        int P = 32;
        while (P > 4 && rails * (P / 2) / 32 >= 1200 && ion_rows(P / 2, L, open, n_max, 64) > 0) P >>= 1;
        t.ions = 1;
        t.lpr = P;
        t.rcap = ion_rows(P, L, open, n_max, 64);
        t.kind = kWordKinds + 2 * (P == 4 ? 0 : P == 8 ? 1 : P == 16 ? 2 : 3) + (open ? 1 : 0);
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        sms = std::max(1, sms);
        size_t most = 0, total = 0;
        grad_smem_limits(&most, &total, true);
        const int w = grad_warps(t, p, most, total, rails, sms);
        SweepArgs a;
        const int64_t resident = (int64_t)w * std::max<int>(1, std::min<int>((int)(total / (grad_tile_args(a, t, p, w) + 1024)), kGradWarps / w));
        const int64_t waves = (rails * P / 32 + sms * resident - 1) / (sms * resident);
        if (!words_for_gradient(rails, L, p.n_zones, open, waves)) return t;
        t = TileShape{};
    }
    t.lpr = sweep_pick_lpr(L, &t.wpl);
    t.kind = sweep_kind(t.lpr, t.wpl);
    return t;
}

void grad_smem_limits(size_t *most, size_t *total, bool ions)
{
    int dev = 0, cta = 0, sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&cta, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (cta <= 0) cta = 48 * 1024;
    if (sm < cta) sm = cta;
    *most = (size_t)std::min(cta, ions ? kGradSmem : 200 * 1024);
    *total = (size_t)sm;
}

// Warps per CTA of a shape's gradient launch over `rails` rails: as many resident
// on an SM as its shared memory (`total` bytes, `most` to a CTA, which costs 1 KB
// more than it asks for) allows, of equals the smaller CTA; when all warps are
// resident at once, the same number on every SM (16,384 x 512 rails on 4 lanes,
// 13.5 warps an SM: 14.4 us a step in one wave of 14, 20.4 us in CTAs of 8).
int grad_warps(const TileShape &t, const kmc_params &p, size_t most, size_t total, int64_t rails, int sms)
{
    SweepArgs a;
    int best = 1, resident = 0, largest = 1;
    for (int w = 1; w <= (t.ions ? kGradWarps : 8); ++w) {
        const size_t m = grad_tile_args(a, t, p, w);
        if (m > most) break;
        if (!t.ions && (w & (w - 1))) continue;
        largest = w;
        const int n = t.ions ? w * std::min<int>((int)(total / (m + 1024)), kGradWarps / w) : w;
        if (n > resident) {
            resident = n;
            best = w;
        }
    }
    const int64_t even = (rails * t.lpr / 32 + sms - 1) / std::max(1, sms);
    if (t.ions && even <= std::min(resident, largest)) return (int)std::max<int64_t>(1, even);
    return best;
}

size_t grad_tile_args(SweepArgs &a, const TileShape &t, const kmc_params &p, int warps)
{
    if (!t.ions) return grad_smem_bytes(t.lpr, t.wpl, p.n_zones, p.n_sites, warps);
    a.rcap = t.rcap;
    a.rcpZ = 65536u / (uint32_t)p.n_zones + 1u;
    a.iy = ion_layout(t.lpr, p.n_zones, p.n_sites, p.electrodes == 1, false, t.rcap, true, true, p.update_rule != 0);
    return a.iy.tab + (size_t)warps * a.iy.bytes;
}

cudaError_t ion_set_smem_limits()
{
    cudaError_t e = cudaFuncSetAttribute(ion_kernel<32, false, false, uint32_t, kIonAhead>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, ion_most_smem(kWordKinds));
    for (int k = kWordKinds; k < kShapeKinds; ++k)
        for (int acc = 0; acc < 2; ++acc) {
            const cudaError_t r = with_ions(k, acc != 0, [k](auto p, auto ac, auto open, auto m) {
                return cudaFuncSetAttribute(
                    ion_kernel<decltype(p)::value, decltype(ac)::value, decltype(open)::value, decltype(m)>,
                    cudaFuncAttributeMaxDynamicSharedMemorySize, ion_most_smem(k));
            });
            if (r != cudaSuccess) e = r;
        }
    const cudaError_t b = ion_batch_set_smem_limits(), g = ion_grad_set_smem_limits();
    return e != cudaSuccess ? e : b != cudaSuccess ? b : g;
}

cudaError_t ion_launch(const SweepArgs &a, const SweepLaunch &l, const int *gate, cudaStream_t s)
{
    if (!l.acc && ion_few(l.lpr, a.electrodes == 1, a.rcap)) {
        ion_kernel<32, false, false, uint32_t, kIonAhead><<<l.grid, l.warps * 32, l.smem, s>>>(a, gate);
        return cudaGetLastError();
    }
    return with_ions(l.kind, l.acc != 0, [&](auto p, auto acc, auto open, auto m) {
        ion_kernel<decltype(p)::value, decltype(acc)::value, decltype(open)::value, decltype(m)>
            <<<l.grid, l.warps * 32, l.smem, s>>>(a, gate);
        return cudaGetLastError();
    });
}

}  // namespace kmc
