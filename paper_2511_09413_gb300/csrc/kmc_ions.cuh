// kmc_ions.cuh -- the per-time-step sweep (arXiv 2511.09413, Supplementary
// S2.1.2 - S2.1.7) over ordered ion lists, hand-written for sm_103a.
//
// The state of a rail is the list of its ions' sites.  Ions never pass one
// another (S2.1.6), so the list stays ordered and an ion's neighbours are its
// predecessor and successor: exclusion is a gap of one site, a conflict a gap
// of two with both ions moving inward.  P lanes share a rail, 32 / P rails a
// warp; a lane holds consecutive ions in a column of shared memory that only
// it touches.  Against the occupancy words of kmc_sweep.cu nothing is rebuilt
// when an ion moves (no popcount scan, free-neighbour masks or compaction of
// candidates): every lane draws for its next ion in every iteration.  Ions
// with both neighbours occupied draw in vain, so fuller rails stay with the
// occupancy words (pick_tile, tile_gate).
//
//  * Zone sums.  The number of ions below each zone boundary, P_b, and
//    F = sum_b P_b w_b are updated when an ion crosses a boundary, and the
//    field of S2.1.8 and the decision bounds of Eqs. 3-6 are evaluated again
//    only then (or when a voltage window starts).
//  * Open electrodes.  The first entry of an open rail's list is at site 0 or,
//    when that site is empty, at the virtual site -1; an injection is its hop
//    to site 0 and an extraction the hop back, so the exchange (the most
//    frequent event of an open rail) moves an entry like any other hop.  Site
//    L - 1 mirrors this with the virtual site L.  The list grows or shrinks
//    only when an ion hops between a boundary site and its inner neighbour.
//  * Decisions are those of kmc_sweep.cu: integer bounds on the draw's high
//    word that provably enclose the FP64 probability, an FP64 band for the
//    draws between them and the exact evaluation for the last 1e-11.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <algorithm>
#include <type_traits>

#include "kmc_device.cuh"
#include "kmc_internal.h"

namespace kmc {

namespace {

constexpr uint32_t kM0 = 0xD2511F53u, kM1 = 0xCD9E8D57u;   // Philox multipliers

__device__ __forceinline__ uint64_t mul_wide(uint32_t x, uint32_t m)
{
    uint64_t p;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(x), "r"(m));
    return p;
}

// The words x1, x3 of one Philox4x32-10 block (the high words of the right and
// left draws).  The first two rounds split into a part of (step, rail) alone,
// formed once per step in (u1, u2, u3), and one multiply each of the site's;
// the last round needs only the low halves of its products.
struct StepDraw {
    uint32_t u1, u2, u3;
};
__device__ __forceinline__ StepDraw step_draw(uint32_t t, uint32_t rail, const uint32_t *rk0,
                                              const uint32_t *rk1)
{
    const uint64_t a = mul_wide(t, kM1);
    const uint32_t c0 = (uint32_t)(a >> 32) ^ rail ^ rk0[0];
    const uint64_t b = mul_wide(c0, kM0);
    StepDraw d;
    d.u1 = (uint32_t)a ^ rk0[1];
    d.u2 = (uint32_t)(b >> 32) ^ rk1[1];
    d.u3 = (uint32_t)b;
    return d;
}
// The site's part of the first two rounds: three words that depend on the site
// and the instance only.
__device__ __forceinline__ uint3 site_words(uint32_t site, uint32_t kc)
{
    const uint64_t a = mul_wide(site, kM0);
    const uint64_t b = mul_wide((uint32_t)(a >> 32) ^ kc, kM1);
    return make_uint3((uint32_t)(b >> 32), (uint32_t)b, (uint32_t)a);
}
__device__ __forceinline__ void site_draw(const StepDraw &d, uint32_t w0, uint32_t w1, uint32_t w2,
                                          const uint32_t *rk0, const uint32_t *rk1, uint32_t &xy, uint32_t &xw)
{
    uint32_t c0 = w0 ^ d.u1, c1 = w1;
    uint32_t c2 = w2 ^ d.u2, c3 = d.u3;
#pragma unroll
    for (int i = 2; i < 9; ++i) {
        const uint64_t p0 = mul_wide(c0, kM0), p1 = mul_wide(c2, kM1);
        c0 = (uint32_t)(p1 >> 32) ^ c1 ^ rk0[i];
        c1 = (uint32_t)p1;
        c2 = (uint32_t)(p0 >> 32) ^ c3 ^ rk1[i];
        c3 = (uint32_t)p0;
    }
    xy = c2 * kM1;
    xw = c0 * kM0;
}

// The site table (per CTA, one uint4 per position -1 .. L): the three words of
// site_words, and the position's entry, as the lists hold it: 16 times
// (position + 1), its own byte offset in the table, in the low 16 bits, above
// them the byte offset of its row of decision bounds.  Rows: one per zone, or four
// with per-site barriers (2^cls_shift), of an open rail four more for positions
// -1, 0, L - 1, L, and a dead row (nothing accepted) for the unused slots of a
// column.  With per-site barriers the table holds a zone's first row and an ion's
// entry adds the class of its site: P0 within a half, a quarter, an eighth of the
// zone's largest one or below.  At a spread of 20 meV the largest of a zone's 100
// sites is five times the mean, so bounds of whole zones let through six draws to
// look at for each that is accepted, those of classes 1.5.  Looking the words up takes two of
// the draw's 16 widening multiplies off the pipe that bounds the loop.
constexpr int kStep = 16;          // an entry's difference between neighbouring positions
__device__ __forceinline__ int pos_of(uint32_t e) { return (int)((e & 0xFFFFu) / kStep) - 1; }
__device__ __forceinline__ uint4 site_at(const uint8_t *tab, uint32_t e) { return *(const uint4 *)(tab + (e & 0xFFFFu)); }
// A warp's block: header of 64 bytes (band factor and mid voltage of the voltage
// window float [2], the bounds' widest band in its last word, the largest column, the step up to which draws are counted;
// in the gradient pass the doubles of IonScore from byte 24 on),
// int [G] each of F, N0, the sum of positions that the per-rail current counts
// from, and the rail, then the bounds.
constexpr uint32_t kIonHead = 64u;
__host__ __device__ constexpr uint32_t ion_fixed(int P) { return kIonHead + 16u * (32u / (uint32_t)P); }
// per-lane words ([kIonSlots][32]): entries of the column; distances from its
// first entry to the one before (low half) and from its last to the one after
// (high half), on the neighbouring lanes or the rail's ends; moves since the
// last flush
enum { kSlotN = 0, kSlotGaps = 1, kSlotMoves = 2, kIonSlots = 3 };
constexpr int kIonAhead = 8;       // steps drawn ahead without the accept path at most, four at a time

// The thread index, read anew.  Each phase of a step forms its addresses from
// it and takes its state from shared memory, so that no phase's registers are
// held through another: with one set of pointers for the whole launch the draw
// loop ran on spilled values.
__device__ __forceinline__ uint32_t tid_here()
{
    uint32_t v;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(v));
    return v;
}
// A lane's view of its warp's shared memory.  CLS: with per-site barriers the rows
// of bounds distinguish classes of sites (without the accept path: with it the look
// for a moved ion's class cost the replicated 512-site device 8 %).
template <int P, bool CLS>
struct IonView {
    static constexpr int G = 32 / P;
    const SweepArgs &a;
    uint32_t tid;
    uint8_t *sb;
    __device__ __forceinline__ IonView(const SweepArgs &args, uint8_t *smem) : a(args)
    {
        tid = tid_here();
        sb = smem + a.iy.tab + (tid >> 5) * a.iy.bytes;
    }
    __device__ __forceinline__ int lane() const { return (int)(tid & 31u); }
    __device__ __forceinline__ int seg() const { return (int)(tid & 31u) / P; }
    __device__ __forceinline__ int sl() const { return (int)(tid & (P - 1)); }
    // the lane's place in the tiles' order of rails, and its rail
    __device__ __forceinline__ int64_t place(int64_t tile_rail0) const { return tile_rail0 + (int64_t)(tid >> 5) * G + seg(); }
    __device__ __forceinline__ int64_t rail() const { return (int64_t)Fs()[3 * G]; }
    __device__ __forceinline__ int cls() const { return CLS ? a.cls_shift : 0; }
    // zone code of an entry: z + 1, and 0 / Z + 1 for the virtual sites -1 / L
    __device__ __forceinline__ int code(uint32_t e) const
    {
        const int row = (int)(e >> 20), q = row - (a.Z << cls());
        return q < 0 ? (row >> cls()) + 1 : (q < 2 ? q : a.Z + q - 2);
    }
    __device__ __forceinline__ int zone(uint32_t e) const { return min(max(code(e) - 1, 0), a.Z - 1); }
    // rows of the ends of an open rail
    __device__ __forceinline__ uint8_t *end_rows(int sg) const { return bounds(sg) + (a.Z << cls()) * 16; }
    // the entry at 16 (x + 1) of the site table for an ion of `rail`
    __device__ __forceinline__ uint32_t entry(const uint8_t *tab, uint32_t at, int64_t rail) const
    {
        uint32_t e = site_at(tab, at).w;
        if (cls() != 0 && (int)(e >> 20) < a.Z << cls()) {
            const int x = pos_of(at);
            e += ((__ldg(a.P0cls + rail * ((a.L + 15) >> 4) + (x >> 4)) >> (2 * (x & 15))) & 3u) << 20;
        }
        return e;
    }
    __device__ __forceinline__ float4 &band() const { return *(float4 *)sb; }
    // with the accept path: the widest band of the bounds, in units of a draw's high word
    __device__ __forceinline__ uint32_t &width() const { return *(uint32_t *)(sb + 12); }
    __device__ __forceinline__ int &kmax() const { return *(int *)(sb + 16); }
    __device__ __forceinline__ int &mark() const { return *(int *)(sb + 20); }
    // [0] F, [G] N0, [2 G] sum of positions, [3 G] rail (a.R: none)
    __device__ __forceinline__ int32_t *Fs(int sg) const { return (int32_t *)(sb + kIonHead) + sg; }
    __device__ __forceinline__ int32_t *Fs() const { return Fs(seg()); }
    __device__ __forceinline__ uint8_t *bounds(int sg) const { return sb + ion_fixed(P) + sg * (int)a.iy.row; }
    __device__ __forceinline__ uint8_t *bounds() const { return bounds(seg()); }
    __device__ __forceinline__ uint32_t *words() const { return (uint32_t *)(sb + ion_fixed(P)); }
    __device__ __forceinline__ float2 *p0b(int sg) const { return (float2 *)(sb + a.iy.p0b) + sg * a.Z; }
    __device__ __forceinline__ int32_t *Pb(int sg) const { return (int32_t *)(sb + a.iy.pb) + sg * (a.Z + 1); }
    __device__ __forceinline__ uint32_t &slot(int k) const { return ((uint32_t *)(sb + a.iy.st))[k * 32 + lane()]; }
    // without the accept path: rows that may be accepted, per step drawn ahead;
    // with it and the even/odd rule: rows at odd positions
    // (kIonAhead words, as many again for the rows from 32 on)
    __device__ __forceinline__ uint32_t &hits(int k) const { return ((uint32_t *)(sb + a.iy.hit))[k * 32 + lane()]; }
    __device__ __forceinline__ uint32_t *col() const { return (uint32_t *)(sb + a.iy.col); }
    __device__ __forceinline__ uint32_t *colp() const { return col() + lane(); }
    // gradient pass: [0] V of the cached probabilities, [1] exp(xV V), [2] xV:
    // dV_z -> ln B_z, [3] kC: dq -> d ln B_z / d kappa, [4] 0.5 / L
    __device__ __forceinline__ double *gh() const { return (double *)(sb + 24); }
    // per lane: W, K, G_W, G_K and (a rail's first lane) G_1
    __device__ __forceinline__ double &gacc(int k) const { return ((double *)(sb + a.iy.g))[k * 32 + lane()]; }
    // per lane: outcome bits, the counts before the lane and its first entry's index
    __device__ __forceinline__ uint64_t *gbits(int k) const { return (uint64_t *)(sb + a.iy.g + 1280u) + k * 32; }
    __device__ __forceinline__ uint64_t *gbefore() const { return (uint64_t *)(sb + a.iy.g + 2304u); }
    __device__ __forceinline__ int32_t *gstart() const { return (int32_t *)(sb + a.iy.g + 2560u); }
    // per rail: p of injection and extraction at site 0, of extraction and
    // injection at site L - 1, and their 1 / (1 - p)
    __device__ __forceinline__ double *gends(int sg) const { return (double *)(sb + a.iy.g + 2688u) + sg * 8; }
    __device__ __forceinline__ double *gends() const { return gends(seg()); }
    // per rail and boundary: counts below it; per rail and zone, double2 each:
    // 0 (q_R, q_L), 1 (d ln p_R / d kappa, d ln B / d kappa), 2 (p_R, p_L)
    __device__ __forceinline__ uint64_t *gbelow() const { return (uint64_t *)(sb + a.iy.g + 2688u + 64u * G) + seg() * (a.Z + 1); }
    __device__ __forceinline__ double2 *gzone(int k, int sg) const
    {
        return (double2 *)(sb + a.iy.g + 2688u + 64u * G + (uint32_t)align16(8u * G * (a.Z + 1))) + (k * G + sg) * a.Z;
    }
};
__device__ __forceinline__ int gap_first(uint32_t w) { return (int)(w & 0xFFFFu); }
__device__ __forceinline__ int gap_last(uint32_t w) { return (int)(w >> 16); }

// Bits of a lane's rows: 32 or 64.
__device__ __forceinline__ int count_bits(uint32_t m) { return __popc(m); }
__device__ __forceinline__ int count_bits(uint64_t m) { return __popcll(m); }
__device__ __forceinline__ int first_bit(uint32_t m) { return __ffs(m) - 1; }
__device__ __forceinline__ int first_bit(uint64_t m) { return __ffsll(m) - 1; }
template <class M>
__device__ __forceinline__ M low_bits(int n)      // n in [0, bits of M]
{
    return n < (int)(8 * sizeof(M)) ? (M(1) << n) - M(1) : ~M(0);
}

// Row j of a lane's column (n entries): the distances to its step-start
// neighbours and which of its trials are open (the neighbouring site free, or
// an open electrode; under the even/odd rule only across the active bond).
struct IonEntry {
    uint32_t e;
    int x, gL, gR;
    bool fL, fR;
};
__device__ __forceinline__ IonEntry ion_entry(const uint32_t *colp, int j, int n, uint32_t gaps, int rule,
                                              uint32_t t)
{
    IonEntry q;
    q.e = colp[j * 32];
    q.x = pos_of(q.e);
    q.gL = j > 0 ? q.x - pos_of(colp[(j - 1) * 32]) : gap_first(gaps);
    q.gR = j + 1 < n ? pos_of(colp[(j + 1) * 32]) - q.x : gap_last(gaps);
    q.fR = j < n && q.gR > 1;
    q.fL = j < n && q.gL > 1;
    if (rule != 0) {
        // the bond right of x is active when x = t (mod 2)
        const bool odd = ((q.x ^ (int)t) & 1) != 0;
        q.fR = q.fR && !odd;
        q.fL = q.fL && odd;
    }
    return q;
}

// A draw within the FP32 band of its probability: the FP64 band, then the exact
// path.  d* in: 2 for a trial to decide, else 0 or 1; out: 0 or 1.
template <int P, bool CLS>
__device__ __forceinline__ void ion_exact(const IonView<P, CLS> &c, int sg, int64_t r2, int pos, int zone,
                                          uint32_t t, int &dR, int &dL)
{
    constexpr int G = 32 / P;
    const SweepArgs &a = c.a;
    const int L = a.L, Z = a.Z;
    const DevConst *K = a.K;
    const int site = min(max(pos, 0), L - 1);
    const bool open = a.electrodes == 1;
    const int kindR = pos < 0 ? 1 : (open && pos == L - 1 ? 2 : 0);
    const int kindL = pos >= L ? 1 : (open && pos == 0 ? 2 : 0);
    const uint4 x = philox((uint32_t)site, a.rail_base + (uint32_t)r2, t, a.instance, a.rk0, a.rk1);
    const double V = a.V[t];
    const double P0k = a.P0bnd != nullptr ? a.P0site[r2 * L + site] : K->P0;
    const double baseR = kindR == 1 ? K->E_in : (kindR == 2 ? K->E_out : P0k);
    const double baseL = kindL == 1 ? K->E_in : (kindL == 2 ? K->E_out : P0k);
    const uint64_t wR = ((uint64_t)x.y << 32) | x.x, wL = ((uint64_t)x.w << 32) | x.z;
    const int32_t *Pb = c.Pb(sg);
    const int32_t *Fs = c.Fs(sg);
    unsigned ne = 0;
    // FP64 band (kmc_sweep.cu, slow_candidate): p to 1e-13 relative, so a draw
    // more than 1e-11 from it is decided.  m_z does not change when every P_b
    // is shifted by the same count, as an open rail's are.
    if (a.bgd) {
        const int m = (int)((uint32_t)L * (uint32_t)(Pb[zone] + Pb[zone + 1]) - (uint32_t)Fs[0]);
        const double dq = __fma_rn((double)m, K->half_invL, -a.bgd[r2 * Z + zone].y);
        const double xx = __dmul_rn(__fma_rn(-K->ka, dq, V), K->xs);
        if (fabs(xx) < 600.0) {
            const double Bf = exp(xx);
            const double invf = 1.0 / (1.0 + Bf);
            if (dR == 2) {
                const double d = __dsub_rn(__dmul_rn((double)(wR >> 11), 0x1.0p-53),
                                           __dmul_rn(__dmul_rn(baseR, invf), Bf));
                if (fabs(d) > 1e-11) {
                    dR = d <= 0.0 ? 1 : 0;
                    ++ne;
                }
            }
            if (dL == 2) {
                const double d = __dsub_rn(__dmul_rn((double)(wL >> 11), 0x1.0p-53),
                                           __dmul_rn(baseL, invf));
                if (fabs(d) > 1e-11) {
                    dL = d <= 0.0 ? 1 : 0;
                    ++ne;
                }
            }
        }
    }
    if (dR == 2 || dL == 2) {
        double B, inv;
        exact_zone(Pb, K, Z, L, Fs[G], a.bgd ? a.bgd + r2 * Z : nullptr, V, zone, &B, &inv);
        const int32_t rg = (int32_t)(a.rail_base + (uint32_t)r2);
        if (dR == 2) {
            const double p = __dmul_rn(__dmul_rn(baseR, inv), B);   // Eq. 6
            dR = exact_trial(wR, p, a.log, a.log_count, a.log_cap, rg, t, site, 0, kindR) ? 1 : 0;
            ++ne;
        }
        if (dL == 2) {
            const double p = __dmul_rn(baseL, inv);                  // Eq. 5
            dL = exact_trial(wL, p, a.log, a.log_count, a.log_cap, rg, t, site, 1, kindL) ? 1 : 0;
            ++ne;
        }
    }
    atomicAdd(&a.counters[1], (unsigned long long)ne);
}

// Distances across the lanes of a rail, for the columns as they stand (n entries
// on this lane).  wallL, wallR: the positions beyond a rail's ends.
template <int P, bool CLS>
__device__ __forceinline__ void ion_refresh(const IonView<P, CLS> &c, int n, int wallL, int wallR)
{
    const uint32_t *colp = c.colp();
    const int xF = n > 0 ? pos_of(colp[0]) : wallR;
    const int xL = n > 0 ? pos_of(colp[(n - 1) * 32]) : wallR;
    int up = __shfl_up_sync(FULL, xL, 1, P), dn = __shfl_down_sync(FULL, xF, 1, P);
    if (c.sl() == 0) up = wallL;
    if (c.sl() == P - 1) dn = wallR;
    c.slot(kSlotGaps) = (uint32_t)(xF - up) | (uint32_t)(dn - xL) << 16;
}

// Deals a warp's entries out evenly from the occupancy words (staged where the
// bounds are): M / P to a lane and one more to the first M % P lanes; the other
// slots are dead.  Sets the lane's state words and the largest column.
template <int P, bool OPEN, bool CLS>
__device__ __forceinline__ void ion_build(const IonView<P, CLS> &c, const uint8_t *tab, int64_t rail)
{
    const SweepArgs &a = c.a;
    const int L = a.L, W = (L + 31) >> 5, C = (W + P - 1) / P, sl = c.sl();
    const int w0 = min(sl * C, W), w1 = min(w0 + C, W);
    const uint32_t *words = c.words() + c.seg() * W;
    uint32_t *col = c.col();
    const uint32_t dead = (a.iy.row - 16u) << 16 | (uint32_t)kStep;
    for (int r = 0; r < a.rcap; ++r) col[r * 32 + c.lane()] = dead;
    int cnt = 0;
    for (int w = w0; w < w1; ++w) cnt += __popc(words[w]);
    int incl = cnt;
#pragma unroll
    for (int off = 1; off < P; off <<= 1) {
        const int v = __shfl_up_sync(FULL, incl, off, P);
        if (sl >= off) incl += v;
    }
    const int total = __shfl_sync(FULL, incl, P - 1, P);
    int vl = 0, vr = 0;
    if (OPEN && rail < a.R) {
        vl = (words[0] & 1u) ? 0 : 1;
        vr = ((words[(L - 1) >> 5] >> ((L - 1) & 31)) & 1u) ? 0 : 1;
    }
    const int M = total + vl + vr;
    const int base = M / P, rem = M - base * P;
    __syncwarp();
    auto place = [&](int i, int xb) {
        int l, r;
        if (i < rem * (base + 1)) {
            l = i / (base + 1);
            r = i - l * (base + 1);
        } else {
            const int i2 = i - rem * (base + 1);
            l = i2 / base;      // base > 0: M > rem (base + 1) here
            r = i2 - l * base;
            l += rem;
        }
        col[r * 32 + c.seg() * P + l] = c.entry(tab, (uint32_t)xb * kStep, rail);
    };
    int i = incl - cnt + vl;
    for (int w = w0; w < w1; ++w) {
        uint32_t m = words[w];
        while (m) {
            place(i++, 32 * w + __ffs(m));      // position + 1
            m &= m - 1;
        }
    }
    if (sl == 0 && vl) place(0, 0);
    if (sl == P - 1 && vr) place(M - 1, L + 1);
    __syncwarp();
    const int n = base + (sl < rem ? 1 : 0);
    if (sl == 0) *(uint4 *)(c.bounds() + a.iy.row - 16u) = make_uint4(0u, 0u, 0u, 0u);
    c.slot(kSlotN) = (uint32_t)n;
    const int km = __reduce_max_sync(FULL, n);
    if (c.lane() == 0) c.kmax() = km;
    ion_refresh<P>(c, n, OPEN ? -2 : -1, OPEN ? L + 1 : L);
    __syncwarp();
}

// The sum of the positions of a rail's entries (on all of its lanes).
template <int P, bool CLS>
__device__ __forceinline__ int ion_sum(const IonView<P, CLS> &c)
{
    const uint32_t *colp = c.colp();
    const int n = (int)c.slot(kSlotN);
    int v = 0;
    for (int r = 0; r < n; ++r) v += pos_of(colp[r * 32]);
#pragma unroll
    for (int off = P / 2; off >= 1; off >>= 1) v += __shfl_xor_sync(FULL, v, off, P);
    return v;
}

// The occupancy words of the lists (staged where the bounds are).
template <int P, bool CLS>
__device__ __forceinline__ void ion_to_words(const IonView<P, CLS> &c)
{
    const int L = c.a.L, W = (L + 31) >> 5;
    uint32_t *words = c.words();
    const uint32_t *colp = c.colp();
    __syncwarp();
    for (int i = c.lane(); i < 32 / P * W; i += 32) words[i] = 0u;
    __syncwarp();
    const int n = (int)c.slot(kSlotN);
    for (int r = 0; r < n; ++r) {
        const int x = pos_of(colp[r * 32]);
        if (x >= 0 && x < L) atomicOr(&words[c.seg() * W + (x >> 5)], 1u << (x & 31));
    }
    __syncwarp();
}

// Entry e at *at moves by m: its new entry, and when it crosses a zone boundary
// b the counts P_b and F, which lose (rightward) or gain one ion, and the zone
// counts of the next step, zc[b - 1] and zc[b] (null after the launch's last
// step).  Returns 0 when it crossed none, 1 for a boundary inside the rail, 2 for
// an end of the rail (an exchange with an electrode).
template <int P, bool CLS>
__device__ __forceinline__ int ion_commit(const IonView<P, CLS> &c, const uint8_t *tab, int64_t rail, uint32_t *at,
                                          uint32_t e, int m, unsigned long long *zc)
{
    const SweepArgs &a = c.a;
    const uint32_t en = c.entry(tab, (e & 0xFFFFu) + (uint32_t)(kStep * m), rail);
    *at = en;
    if (((e ^ en) >> 16) == 0u) return 0;
    const int k0 = c.code(e), k1 = c.code(en);
    if (k0 == k1) return 0;
    const int b = max(k0, k1) - 1;
    atomicAdd(&c.Pb(c.seg())[b], -m);
    atomicAdd(c.Fs(), -m * a.wsum[b]);
    if (zc) {
        if (b > 0) atomicAdd(zc + (b - 1), (unsigned long long)(long long)(-m));
        if (b < a.Z) atomicAdd(zc + b, (unsigned long long)(long long)m);
    }
    return b == 0 || b == a.Z ? 2 : 1;
}

// Under the even/odd rule with the accept path: the rows at odd positions.  A move
// flips its row's bit, so they are formed anew only when rows come or go.
template <int P, class M, bool CLS>
__device__ __forceinline__ M ion_odd(const IonView<P, CLS> &c)
{
    M m = c.hits(0);
    if (sizeof(M) > 4) m |= (M)c.hits(1) << (8 * sizeof(M) - 32);
    return m;
}
template <int P, class M, bool CLS>
__device__ __forceinline__ void ion_set_odd(const IonView<P, CLS> &c, M m)
{
    c.hits(0) = (uint32_t)m;
    if (sizeof(M) > 4) c.hits(1) = (uint32_t)(m >> (8 * sizeof(M) - 32));
}
template <int P, class M, bool CLS>
__device__ __forceinline__ void ion_parity(const IonView<P, CLS> &c)
{
    const int n = (int)c.slot(kSlotN);
    M m = 0;
    for (int r = 0; r < n; ++r)
        if (pos_of(c.colp()[r * 32]) & 1) m |= M(1) << r;
    ion_set_odd<P, M>(c, m);
}

// Zone z of rail slot sg as it stands (the field of S2.1.8, Eqs. 3-4) at the mid
// voltage of the window: B/(1+B) and 1/(1+B) in FP32 and the factors [lo, hi]
// that enclose the exact probabilities.  p lies within a factor 1 +- eps of its
// FP32 value, times [1 / eh, eh] over a voltage window.  With u = 2^-24, every one
// of the twelve roundings that lead to the exponent x is relative to at most
// S = (|V| + |kappa alpha| (P_z + P_z+1 + F / L + N0)) / (L kT), so x is off by
// less than 16 u S, and Eqs. 5-6 move by that relatively (their logarithmic
// derivatives with respect to x are at most 1); __expf adds (2 + 1.2 |x|) ulp, the
// division two, the other operations three.
struct IonZone {
    float sR, inv, lo, hi;
    bool ok;        // false: no bounds, every draw goes to the FP64 paths
};
template <int P, bool OPEN, bool CLS>
__device__ __forceinline__ IonZone ion_zone(const IonView<P, CLS> &c, int sg, int z)
{
    constexpr int G = 32 / P;
    const SweepArgs &a = c.a;
    const float eh = c.band().x, Vf = c.band().y;
    const int32_t *Pb = c.Pb(sg), *Fs = c.Fs(sg);
    // an open rail's counts are relative to its first boundary
    const int p0 = OPEN ? Pb[0] : 0;
    const int Pz = Pb[z] - p0, Pz1 = Pb[z + 1] - p0;
    const int F = OPEN ? (int)((uint32_t)Fs[0] - (uint32_t)p0 * (uint32_t)(2 * a.L)) : Fs[0];
    const float Ff = (float)F * a.inv_L, Nf = (float)Fs[G], Pf = (float)(Pz + Pz1);
    const float qd = 0.5f * (Pf - Ff) - Nf * a.cz[z];
    const float x = -(Vf - a.ka_f * qd) * a.inv_LkT;
    const float S = (fabsf(Vf) + fabsf(a.ka_f) * (Pf + Ff + Nf)) * a.inv_LkT;
    const float eps = 4e-6f + 5e-7f * fabsf(x) + 1.2e-6f * S;
    IonZone r{0.0f, 0.0f, 0.0f, 0.0f, fabsf(x) <= 40.0f && eps < 0.25f};
    if (r.ok) {
        const float B = __expf(x);
        r.inv = __fdividef(1.0f, 1.0f + B);
        r.sR = r.inv * B;
        r.lo = __fdividef(1.0f - eps, eh);
        r.hi = (1.0f + eps) * eh;
    }
    return r;
}

// A voltage window: steps from s on, at most 32, whose voltage stays near the
// first one's.  Evaluating at the window's mid voltage changes B/(1+B) and
// 1/(1+B) by a factor within [e^-h, e^h] (logarithmic derivatives at most 1).  With
// ACC every draw in that band is looked at, so a window's exponent stays within 2e-3
// and its bounds are cheap to evaluate beside a step's work.  Without ACC the bounds
// only choose the draws to look at, and a short window wastes the steps drawn ahead:
// it spans 0.1, and 0.3 over the steps drawn at once.  A fast ramp (2 V up and down in
// 1,000 steps) on 65,536 x 100 rails 20 % full with per-site barriers, 381 steps: 7.28 ms
// with 2e-3, 1.92 with (0.3, 0.03), 1.55 with (0.3, 0.1), the occupancy words 2.21; no
// difference on a slow one (in 100,000 steps).  Returns the first step after it.
template <int P, bool ACC, bool CLS>
__device__ __forceinline__ int ion_window(const IonView<P, CLS> &c, int64_t t0, int s, int n_steps)
{
    const SweepArgs &a = c.a;
    const int left = min(32, n_steps - s);
    const double v = a.V[t0 + s + min(c.lane(), left - 1)];
    const float v0 = __shfl_sync(FULL, (float)v, 0);
    const float near = ACC ? 2e-3f : c.lane() < kIonAhead ? 0.3f : 0.1f;
    const uint32_t far = __ballot_sync(FULL, fabsf((float)v - v0) * a.inv_LkT > near);
    const int len = min(left, far ? __ffs(far) - 1 : 32);
    float vlo = __double2float_rd(v), vhi = __double2float_ru(v);
    if (c.lane() >= len) vlo = vhi = v0;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        vlo = fminf(vlo, __shfl_xor_sync(FULL, vlo, off));
        vhi = fmaxf(vhi, __shfl_xor_sync(FULL, vhi, off));
    }
    const float h = 0.5f * (vhi - vlo) * a.inv_LkT;
    if (c.lane() == 0) {
        float4 &b = c.band();
        b.x = __expf(h) * (1.0f + 4e-6f + 2e-6f * h);
        b.y = 0.5f * (vlo + vhi);
    }
    return s + len;
}

// Decision bounds of the zones of the rail slots in `dirty` (bits; `all`: of every
// one).  With ACC they are upper bounds too, and the widest band between a bound and
// the draws that are surely accepted is kept beside them: a draw nearer to its bound
// than that is decided with its own zone and site.  Without ACC
// they only tell which draws may be accepted, for any state of an end entry and
// with room for a.ion_slack in the exponent, so that they hold while ions cross a
// few boundaries (a.ion_budget); the draws below them are decided with ion_zone.
__device__ __forceinline__ float ion_class(int k) { return __int_as_float((127 - k) << 23); }     // 2^-k
template <int P, bool ACC, bool OPEN, bool CLS>
__device__ __forceinline__ void ion_zones(const IonView<P, CLS> &c, uint32_t dirty, bool all)
{
    constexpr int G = 32 / P;
    const SweepArgs &a = c.a;
    const int Z = a.Z;
    __syncwarp();
    const int items = __popc(dirty) * Z;
    uint32_t wide = 0u;
    for (int i = c.lane(); i < items; i += 32) {
        const int k = (int)(((uint32_t)i * a.rcpZ) >> 16), z = i - k * Z;    // i / Z for i < 1024
        uint32_t m = dirty;
        for (int q = 0; q < k; ++q) m &= m - 1;
        const int sg = G == 1 ? 0 : __ffs(m) - 1;
        const IonZone r = ion_zone<P, OPEN>(c, sg, z);
        uint8_t *rm = c.bounds(sg) + (z << c.cls()) * 16, *ends = c.end_rows(sg);
        float blo = a.P0f_scalar, bhi = a.P0f_scalar;
        if (a.P0bnd != nullptr) {
            const float2 pp = c.p0b(sg)[z];
            blo = pp.x;
            bhi = pp.y;
        }
        if constexpr (!ACC) {
            const float top = r.hi * (1.0f + a.ion_slack + a.ion_slack * a.ion_slack);    // above e^slack
            const float bot = a.ion_exchange ? 0.0f : r.lo * (1.0f - a.ion_slack);
            uint2 b = make_uint2(FULL, FULL);
            if (r.ok) b = make_uint2(rej_thr(bhi * r.sR * top), rej_thr(bhi * r.inv * top));
            *(uint2 *)rm = b;
            for (int k = 1; k < 1 << c.cls(); ++k) {
                const float bk = bhi * ion_class(k) * (1.0f + 2.4e-7f);     // P0 rounded to FP32 chose the class
                if (r.ok) *(uint2 *)(rm + 16 * k) = make_uint2(rej_thr(bk * r.sR * top), rej_thr(bk * r.inv * top));
                else *(uint2 *)(rm + 16 * k) = b;
            }
            if (OPEN && (z == 0 || z == Z - 1)) {
                // end rows: the hop inward, then the bounds of the exchange with
                // the electrode, from the virtual site in, from the site out
                const float Ein = a.E_inf, Eout = a.E_outf;
                if (z == 0) {
                    uint4 in = make_uint4(FULL, FULL, FULL, 0u), out = in;
                    if (r.ok) {
                        in = make_uint4(b.x, 0u, rej_thr(Ein * r.sR * top), acc_thr(Ein * r.sR * bot));
                        out = make_uint4(b.x, 0u, rej_thr(Eout * r.inv * top), acc_thr(Eout * r.inv * bot));
                    }
                    *(uint4 *)ends = in;
                    *(uint4 *)(ends + 16) = out;
                }
                if (z == Z - 1) {
                    uint4 in = make_uint4(FULL, FULL, FULL, 0u), out = in;
                    if (r.ok) {
                        in = make_uint4(0u, b.y, rej_thr(Ein * r.inv * top), acc_thr(Ein * r.inv * bot));
                        out = make_uint4(0u, b.y, rej_thr(Eout * r.sR * top), acc_thr(Eout * r.sR * bot));
                    }
                    *(uint4 *)(ends + 32) = out;
                    *(uint4 *)(ends + 48) = in;
                }
            }
            continue;
        }
        const float sm = fmaxf(r.sR, r.inv);
        uint2 b = make_uint2(FULL, FULL);
        uint32_t w = FULL;
        if (r.ok) {
            b = make_uint2(rej_thr(bhi * r.sR * r.hi), rej_thr(bhi * r.inv * r.hi));
            w = rej_thr(bhi * sm * r.hi) - acc_thr(blo * sm * r.lo) + 2u;
        }
        *(uint2 *)rm = b;
        if (OPEN && (z == 0 || z == Z - 1)) {
            // electrode positions: outward trials are extractions, the virtual
            // sites' inward trials injections
            const float Ein = a.E_inf, Eout = a.E_outf, Em = fmaxf(Ein, Eout) * sm;
            if (r.ok) w = max(w, rej_thr(Em * r.hi) - acc_thr(Em * r.lo) + 2u);
            if (z == 0) {
                uint2 in = b, out = b;
                if (r.ok) {
                    in.x = rej_thr(Ein * r.sR * r.hi);
                    out.y = rej_thr(Eout * r.inv * r.hi);
                }
                *(uint2 *)ends = in;
                *(uint2 *)(ends + 16) = out;
            }
            if (z == Z - 1) {
                uint2 in = b, out = b;
                if (r.ok) {
                    in.y = rej_thr(Ein * r.inv * r.hi);
                    out.x = rej_thr(Eout * r.sR * r.hi);
                }
                *(uint2 *)(ends + 32) = out;
                *(uint2 *)(ends + 48) = in;
            }
        }
        wide = max(wide, w);
    }
    if constexpr (ACC) {
        wide = __reduce_max_sync(FULL, wide);
        if (c.lane() == 0) c.width() = all ? wide : max(wide, c.width());
    }
    __syncwarp();
}

// A draw that may be accepted, decided in the FP32 band of its own probability:
// the site's P0, or the electrode's.  d* out: 0, 1, or 2 when it lies in the band.
template <int P, bool OPEN, bool CLS>
__device__ __forceinline__ void ion_decide(const IonView<P, CLS> &c, const IonEntry &q, int64_t rail, uint32_t xy,
                                           uint32_t xw, int &dR, int &dL)
{
    const SweepArgs &a = c.a;
    const int L = a.L;
    const IonZone r = ion_zone<P, OPEN>(c, c.seg(), c.zone(q.e));
    float P0 = a.P0f_scalar;
    if (a.P0bnd != nullptr && (!OPEN || (q.x >= 0 && q.x < L))) P0 = __ldg(a.P0f + rail * L + q.x);
    float bR = P0, bL = P0;
    if (OPEN) {
        if (q.x < 0) bR = a.E_inf;
        if (q.x == 0) bL = a.E_outf;
        if (q.x == L - 1) bR = a.E_outf;
        if (q.x >= L) bL = a.E_inf;
    }
    dR = q.fR ? (r.ok ? bounded(xy, bR * r.sR, r.lo, r.hi) : 2) : 0;
    dL = q.fL ? (r.ok ? bounded(xw, bL * r.inv, r.lo, r.hi) : 2) : 0;
}

// Exchanges with the electrodes without the accept path.  They are the most
// frequent events of an open rail, and as long as no ion inside it moves they
// concern its end entries only, which then step in and out in turn.  ion_end_draws
// draws for both ends over the next kIonAhead steps, one lane to an end and step;
// its result, on the lane that holds the end entry: bits q of a step where an
// injection may (0..7) or surely will (8..15) be accepted, and an extraction (16..31).
template <int P, bool CLS>
__device__ __forceinline__ bool ion_end(const IonView<P, CLS> &c, bool &left, uint32_t *&at)
{
    const int n = (int)c.slot(kSlotN), sl = c.sl();
    left = sl == 0;
    at = c.colp();
    if (n <= 0) return false;
    if (left) return true;
    at += (n - 1) * 32;
    return sl == P - 1 || pos_of(*at) + gap_last(c.slot(kSlotGaps)) == c.a.L + 1;
}
template <int P, bool CLS>
__device__ __forceinline__ uint32_t ion_end_draws(const IonView<P, CLS> &c, const uint8_t *tab, uint32_t t, uint32_t prail,
                                                  const uint32_t *rk0, const uint32_t *rk1)
{
    const SweepArgs &a = c.a;
    uint32_t *at;
    bool left;
    const bool own = ion_end<P>(c, left, at);
    uint32_t f[4] = {};     // 16 bits each: the left end's steps, the right end's
#pragma unroll
    for (int pass = 0; pass < (P >= 16 ? 1 : 16 / P); ++pass) {
        const int ci = pass * P + (c.sl() & 15);
        const bool right = (ci & 8) != 0;
        const uint32_t tk = t + (uint32_t)(ci & 7);
        const uint4 w = site_at(tab, (uint32_t)(right ? a.L : 1) * kStep);
        uint32_t xy, xw;
        site_draw(step_draw(tk, prail, rk0, rk1), w.x, w.y, w.z, rk0, rk1, xy, xw);
        const uint8_t *rm = c.end_rows(c.seg()) + 8;
        const uint2 in = *(const uint2 *)(rm + (right ? 48 : 0)), out = *(const uint2 *)(rm + (right ? 32 : 16));
        const uint32_t xi = right ? xw : xy, xo = right ? xy : xw;
        // the even/odd rule: the bond right of x is active when x = t (mod 2)
        const bool act = a.rule == 0 || (((uint32_t)(right ? a.L - 1 : -1) ^ tk) & 1u) == 0u;
        const int sh = c.lane() - c.sl();
        constexpr uint32_t mine = P >= 16 ? 0xFFFFu : (1u << P) - 1u;
        f[0] |= ((__ballot_sync(FULL, act && xi <= in.x) >> sh) & mine) << (pass * P);
        f[1] |= ((__ballot_sync(FULL, act && xi < in.y) >> sh) & mine) << (pass * P);
        f[2] |= ((__ballot_sync(FULL, act && xo <= out.x) >> sh) & mine) << (pass * P);
        f[3] |= ((__ballot_sync(FULL, act && xo < out.y) >> sh) & mine) << (pass * P);
    }
    const int sh = left ? 0 : 8;
    const uint32_t r = ((f[0] >> sh) & 255u) | ((f[1] >> sh) & 255u) << 8 | ((f[2] >> sh) & 255u) << 16 | ((f[3] >> sh) & 255u) << 24;
    return own ? r : 0u;
}
// Steps q .. stop - 1 (after step s of the launch), in which nothing but exchanges
// can happen: carries them out, up to the first one that is not sure, and returns
// the step that has to be looked at, stop when there was none.  und: the end entry's
// bit if its exchange may be accepted in that step.
template <int P, class M, bool CLS>
__device__ __forceinline__ int ion_exchanges(const IonView<P, CLS> &c, const uint8_t *tab, int64_t t0, int s, int n_steps,
                                             int q, int stop, uint32_t bits, M &und)
{
    const SweepArgs &a = c.a;
    uint32_t *at;
    bool left;
    const bool own = ion_end<P>(c, left, at);
    const int x = own ? pos_of(*at) : 0;
    const bool full = left ? x >= 0 : x < a.L;
    uint32_t moved = 0u;
    int mine = stop;
    if (bits != 0u) {
        bool o = full;
        for (int k = q; k < stop; ++k) {
            const uint32_t b = bits >> (k + (o ? 16 : 0));
            if ((b & 0x101u) == 0x1u) {
                mine = k;
                break;
            }
            if (b & 1u) {
                moved |= 1u << k;
                o = !o;
            }
        }
    }
    stop = __reduce_min_sync(FULL, mine);
    moved &= (1u << stop) - 1u;
    if (__any_sync(FULL, moved != 0u)) {
        if (moved) {
            int m = full == left ? -1 : 1;
            const int cnt = __popc(moved);
            if (cnt & 1) {
                const int b = left ? 0 : a.Z;
                atomicAdd(&c.Pb(c.seg())[b], -m);
                atomicAdd(c.Fs(), -m * a.wsum[b]);
                *at = site_at(tab, (uint32_t)(x + 1 + m) * kStep).w;
            }
            c.slot(kSlotMoves) += (uint32_t)cnt;
            unsigned long long *const J = a.J + t0 + s, *const zc = a.Zc + (t0 + s + 1) * a.Z + (left ? 0 : a.Z - 1);
            for (uint32_t k = moved; k; k &= k - 1) {
                const int w = __ffs(k) - 1;
                atomicAdd(J + w, (unsigned long long)(long long)(-m));
                if (s + w + 1 < n_steps)
                    atomicAdd(zc + (int64_t)w * a.Z, (unsigned long long)(long long)(left ? m : -m));
                m = -m;
            }
        }
        __syncwarp();
        ion_refresh<P>(c, (int)c.slot(kSlotN), -2, a.L + 1);
        __syncwarp();
    }
    if (own) {
        const bool o = full != ((__popc(moved) & 1) != 0);
        if (stop < kIonAhead && ((bits >> (stop + (o ? 16 : 0))) & 1u) != 0u) und = left ? M(1) : M(1) << ((int)c.slot(kSlotN) - 1);
    }
    return stop;
}

// The list ends of open rails after a step's moves: the first entry stays at
// site -1 or 0, the last at L - 1 or L.  Returns (warp-uniform) 0 when no entry
// came or went, 1 when one did, 2 when the bounds were overwritten on the way.
template <int P, bool CLS>
__device__ __forceinline__ int ion_ends(const IonView<P, CLS> &c, const uint8_t *tab, int s, int64_t rail,
                                        uint32_t &draws)
{
    const SweepArgs &a = c.a;
    const int L = a.L, sl = c.sl();
    const uint32_t dead = (a.iy.row - 16u) << 16 | (uint32_t)kStep;
    uint32_t *colp = c.colp();
    const uint32_t gaps = c.slot(kSlotGaps);
    const int n0 = (int)c.slot(kSlotN);
    int n = n0;
    if (n > 0 && sl == 0) {
        const int xF = pos_of(colp[0]);
        if (xF > 0) {
            for (int r = n; r > 0; --r) colp[r * 32] = colp[(r - 1) * 32];
            colp[0] = site_at(tab, 0u).w;
            ++n;
            atomicAdd(&c.Fs()[2 * (32 / P)], -1);     // entries that come and go are no moves
        } else if (xF < 0) {
            const int x2 = n > 1 ? pos_of(colp[32]) : xF + gap_last(gaps);
            if (x2 == 0) {
                --n;
                for (int r = 0; r < n; ++r) colp[r * 32] = colp[(r + 1) * 32];
                colp[n * 32] = dead;
                atomicAdd(&c.Fs()[2 * (32 / P)], 1);
            }
        }
    }
    const int xe = n > 0 ? pos_of(colp[(n - 1) * 32]) : 0;
    if (n > 0 && (sl == P - 1 || xe + gap_last(gaps) == L + 1)) {        // the lane of the last entry
        if (xe < L - 1) {
            colp[n * 32] = site_at(tab, (uint32_t)(L + 1) * kStep).w;
            ++n;
            atomicAdd(&c.Fs()[2 * (32 / P)], L);
        } else if (xe == L) {
            const int x2 = n > 1 ? pos_of(colp[(n - 2) * 32]) : xe - gap_first(gaps);
            if (x2 == L - 1) {
                --n;
                colp[n * 32] = dead;
                atomicAdd(&c.Fs()[2 * (32 / P)], -L);
            }
        }
    }
    if (!__any_sync(FULL, n != n0)) return 0;
    // draws so far were of the old columns
    draws = __reduce_add_sync(FULL, (uint32_t)n0) * (uint32_t)(s + 1 - c.mark());
    __syncwarp();
    if (c.lane() == 0) c.mark() = s + 1;
    c.slot(kSlotN) = (uint32_t)n;
    // deal the entries out again when a lane ran empty, holds more than one
    // above its even share or has outgrown its bits
    int M = n;
#pragma unroll
    for (int off = P / 2; off >= 1; off >>= 1) M += __shfl_xor_sync(FULL, M, off, P);
    if (__any_sync(FULL, (n0 > 0 && n == 0) || n > min((M + P - 1) / P + 1, a.rcap - 2))) {
        ion_to_words<P>(c);
        ion_build<P, true>(c, tab, rail);
        return 2;
    }
    const int km = __reduce_max_sync(FULL, n);
    if (c.lane() == 0) c.kmax() = km;
    ion_refresh<P>(c, n, -2, L + 1);
    __syncwarp();
    return 1;
}

// ------------------------------------------------- gradient pass
// 0 <= n < 2^24 as a double, by widening its FP32 bits with integer operations:
// a conversion instruction would take the FP64 pipe, the bound of this pass.
__device__ __forceinline__ double count_to_double(int n)
{
    const uint32_t u = __float_as_uint((float)n);
    return __hiloint2double(n ? (int)((u >> 3) + 0x38000000u) : 0, (int)(u << 29));
}

// Constants and empty sums of the warp's rails.
template <int P, bool CLS>
__device__ __forceinline__ void ion_score_begin(const IonView<P, CLS> &c)
{
    const SweepArgs &a = c.a;
    const int L = a.L;
    const DevConst &K = *a.K;
    const double xV = -(K.d / K.t_dev) / K.kT;
    if (c.lane() == 0) {
        double *h = c.gh();
        h[0] = __longlong_as_double(0x7FF8000000000000ll);     // no cache
        h[2] = xV;
        h[3] = (a.alpha * K.d) / a.tdev_kT;
        h[4] = 0.5 / (double)L;
    }
    for (int k = 0; k < 5; ++k) c.gacc(k) = 0.0;
    __syncwarp();
}

// Probabilities (Eqs. 3-6, FP64) and score factors of the zones of the rail slots
// in `stale`: q = p / (1 - p) of both directions (0 for a certain trial, whose
// weight is then its outcome), and the kappa derivatives.  B_z is the product of
// exp(xV V), exp(xV kappa alpha D'_z) and the tabulated exponential of the
// integer zone sum m_z = L (P_z + P_z+1) - F; one reciprocal of x1 y2 y3 with
// x1 = 1 + B, y2 = x1 (1 - p_R), y3 = x1 (1 - p_L) serves all three quotients.
template <int P, bool OPEN, bool CLS>
__device__ __forceinline__ void ion_score_zones(const IonView<P, CLS> &c, uint32_t t, uint32_t stale)
{
    constexpr int G = 32 / P;
    const SweepArgs &a = c.a;
    const int Z = a.Z, L = a.L;
    const DevConst &K = *a.K;
    const double V = a.V[t];
    if (__double_as_longlong(V) != __double_as_longlong(c.gh()[0])) {
        __syncwarp();
        if (c.lane() == 0) {
            c.gh()[0] = V;
            c.gh()[1] = exp(__dmul_rn(c.gh()[2], V));
        }
        __syncwarp();
        stale = (uint32_t)((1ull << G) - 1u);
    }
    const int items = __popc(stale) * Z;
    for (int i = c.lane(); i < items; i += 32) {
        const int k = (int)(((uint32_t)i * a.rcpZ) >> 16), z = i - k * Z;
        uint32_t sm = stale;
        for (int q = 0; q < k; ++q) sm &= sm - 1;
        const int sg = G == 1 ? 0 : __ffs(sm) - 1;
        const int32_t *Pb = c.Pb(sg);
        const int m = (int)((uint32_t)L * (uint32_t)(Pb[z] + Pb[z + 1]) - (uint32_t)c.Fs(sg)[0]);
        const double2 bg = __ldg(a.bgN + (int64_t)c.Fs(sg)[G] * Z + z);
        const double *h = c.gh();
        const double dq = __fma_rn(h[4], (double)m, -bg.x);
        double B;
        if (a.etL != nullptr && fabs(__dmul_rn(h[2], V)) < 600.0) {
            const int u = m + a.etM;
            B = __dmul_rn(__dmul_rn(h[1], bg.y), __dmul_rn(__ldg(a.etH + (u >> 10)), __ldg(a.etL + (u & 1023))));
        } else {
            B = exp(__dmul_rn(__fma_rn(-K.ka, dq, V), h[2]));
        }
        const double cB = __dmul_rn(h[3], dq);                  // d ln B / d kappa
        const double x1 = __dadd_rn(1.0, B), P0B = __dmul_rn(K.P0, B);
        const double y2 = __dsub_rn(x1, P0B), y3 = __dsub_rn(x1, K.P0);
        const double y23 = __dmul_rn(y2, y3);
        const double xd = __dmul_rn(x1, y23);
        double inv, qR, qL;
        if (inside_bits(xd, 1e-300, 1e300)) {                   // both trials uncertain
            const double rp = recip_newton(xd);
            const double xr = __dmul_rn(x1, rp);                // 1 / (y2 y3)
            inv = __dmul_rn(y23, rp);
            qR = __dmul_rn(__dmul_rn(P0B, y3), xr);             // p_R / (1 - p_R) = P0 B / y2
            qL = __dmul_rn(__dmul_rn(K.P0, y2), xr);            // P0 / y3
        } else {                                                // a certain trial, or B out of range
            inv = __drcp_rn(x1);
            const double pL = __dmul_rn(K.P0, inv), pR = __dmul_rn(pL, B);
            qR = pR < 1.0 ? __dmul_rn(pR, __drcp_rn(__dsub_rn(1.0, pR))) : 0.0;
            qL = pL < 1.0 ? __dmul_rn(pL, __drcp_rn(__dsub_rn(1.0, pL))) : 0.0;
        }
        const double pL = __dmul_rn(K.P0, inv);                 // Eq. 5
        c.gzone(0, sg)[z] = make_double2(qR, qL);
        c.gzone(1, sg)[z] = make_double2(__dmul_rn(inv, cB), cB);
        c.gzone(2, sg)[z] = make_double2(__dmul_rn(pL, B), pL); // Eq. 6
        if (OPEN && (z == 0 || z == Z - 1)) {
            double *e = c.gends(sg);
            if (z == 0) {
                e[0] = __dmul_rn(__dmul_rn(K.E_in, inv), B);    // injection into 0
                e[1] = __dmul_rn(K.E_out, inv);                 // extraction at 0
                e[4] = e[0] < 1.0 ? __drcp_rn(__dsub_rn(1.0, e[0])) : 0.0;
                e[5] = e[1] < 1.0 ? __drcp_rn(__dsub_rn(1.0, e[1])) : 0.0;
            }
            if (z == Z - 1) {
                e[2] = __dmul_rn(__dmul_rn(K.E_out, inv), B);   // extraction at L - 1
                e[3] = __dmul_rn(K.E_in, inv);                  // injection into L - 1
                e[6] = e[2] < 1.0 ? __drcp_rn(__dsub_rn(1.0, e[2])) : 0.0;
                e[7] = e[3] < 1.0 ? __drcp_rn(__dsub_rn(1.0, e[3])) : 0.0;
            }
        }
    }
    __syncwarp();
}

// Score of one step's trials, before its moves.  fR, fL: the rows whose right and
// left trials are open (performed), aR, aL: those accepted.  Inner hops of a zone
// share p, so their summed weight A / (1 - p) - n q = A + (A - n) q needs only the
// counts of performed and accepted trials; a zone's ions are consecutive entries
// of the list (index P_b to P_b+1), so the counts below every boundary are a sum
// over the lanes before it and a population count within its lane.  The electrode
// trials of an open rail's end entries are added one by one.  The lanes of a rail
// take its zones in turn and keep their own shares of W, K and the estimator
// sums; only the step's coefficient (the zone counts' share less the current's
// innovation, a control variate of zero mean) is summed over them.
template <int P, bool OPEN, class M, bool CLS>
__device__ __forceinline__ void ion_score(const IonView<P, CLS> &c, uint32_t t, M fR, M fL, M aR, M aL)
{
    const SweepArgs &a = c.a;
    const int Z = a.Z, L = a.L, sl = c.sl();
    const bool wantE = a.wJ != nullptr;
    double Ws = 0.0, Ks = 0.0, Ep = 0.0;
    int Ei = 0;                     // accepted left less accepted right trials
    int vl = 0;                     // the list starts with the virtual site -1
    if (OPEN) {
        const int n = (int)c.slot(kSlotN);
        const uint32_t *colp = c.colp();
        const double *e = c.gends();
        if (n > 0 && sl == 0) {
            const double2 dk = c.gzone(1, c.seg())[0];
            if (pos_of(colp[0]) < 0) {      // injection into site 0
                vl = 1;
                const int hit = (int)(aR & 1);
                Ks = __dmul_rn(et_weight(hit, e[0], e[4]), dk.x);
                Ei -= hit;
                Ep = e[0];
                fR &= ~M(1);
                aR &= ~M(1);
            } else {                        // extraction through the left electrode
                const int hit = (int)(aL & 1);
                Ks = __dmul_rn(et_weight(hit, e[1], e[5]), __dsub_rn(dk.x, dk.y));
                Ei += hit;
                Ep = -e[1];
                fL &= ~M(1);
                aL &= ~M(1);
            }
        }
        const int xe = n > 0 ? pos_of(colp[(n - 1) * 32]) : 0;
        if (n > 0 && (sl == P - 1 || xe + gap_last(c.slot(kSlotGaps)) == L + 1)) {
            const double2 dk = c.gzone(1, c.seg())[Z - 1];
            const M bit = M(1) << (n - 1);
            if (xe == L) {                  // injection into site L - 1
                const int hit = (aL & bit) ? 1 : 0;
                Ks = __fma_rn(et_weight(hit, e[3], e[7]), __dsub_rn(dk.x, dk.y), Ks);
                Ei += hit;
                Ep = __dsub_rn(Ep, e[3]);
                fL &= ~bit;
                aL &= ~bit;
            } else {                        // extraction through the right electrode
                const int hit = (aR & bit) ? 1 : 0;
                Ks = __fma_rn(et_weight(hit, e[2], e[6]), dk.x, Ks);
                Ei -= hit;
                Ep = __dadd_rn(Ep, e[2]);
                fR &= ~bit;
                aR &= ~bit;
            }
        }
        vl = __shfl_sync(FULL, vl, 0, P);
    }
    // counts (performed and accepted, right and left, 16 bits each) and entries
    // of the lanes before
    const int n = (int)c.slot(kSlotN);
    const uint64_t own = (uint64_t)(uint32_t)(count_bits(fR) | count_bits(aR) << 16) |
                         (uint64_t)(uint32_t)(count_bits(fL) | count_bits(aL) << 16) << 32;
    uint64_t incl = own;
    int to = n;
#pragma unroll
    for (int off = 1; off < P; off <<= 1) {
        const uint64_t u = __shfl_up_sync(FULL, incl, off, P);
        const int v = __shfl_up_sync(FULL, to, off, P);
        if (sl >= off) {
            incl += u;
            to += v;
        }
    }
    c.gbits(0)[c.lane()] = fR;
    c.gbits(1)[c.lane()] = aR;
    c.gbits(2)[c.lane()] = fL;
    c.gbits(3)[c.lane()] = aL;
    c.gbefore()[c.lane()] = incl - own;
    c.gstart()[c.lane()] = to - n;
    __syncwarp();
    const int32_t *Pb = c.Pb(c.seg());
    for (int b = sl; b <= Z; b += P) {
        const int idx = Pb[b] - (OPEN ? Pb[0] : 0) + vl;
        int l = c.lane() - sl;
#pragma unroll
        for (int h = P / 2; h >= 1; h >>= 1)
            if (c.gstart()[l + h] <= idx) l += h;
        const M m = low_bits<M>(idx - c.gstart()[l]);
        const int cR = count_bits((M)c.gbits(0)[l] & m) | count_bits((M)c.gbits(1)[l] & m) << 16;
        const int cL = count_bits((M)c.gbits(2)[l] & m) | count_bits((M)c.gbits(3)[l] & m) << 16;
        c.gbelow()[b] = c.gbefore()[l] + ((uint64_t)(uint32_t)cR | (uint64_t)(uint32_t)cL << 32);
    }
    __syncwarp();
    // zones outside [lo, hi) have zero weight; a step without weights a zero share
    const int zr = a.fZa ? a.fZr[t] : 0;
    double d = 0.0;
    if (zr != 0 && sl == 0) d = -a.fZb[t];
    for (int z = sl; z < Z; z += P) {
        const uint64_t k = c.gbelow()[z + 1] - c.gbelow()[z];
        const int nR = (int)(k & 0xFFFFu), cR = (int)(k >> 16 & 0xFFFFu);
        const int nL = (int)(k >> 32 & 0xFFFFu), cL = (int)(k >> 48);
        if (nR | nL) {
            const double2 q = c.gzone(0, c.seg())[z], dk = c.gzone(1, c.seg())[z];
            const double wR = __fma_rn(-count_to_double(nR - cR), q.x, count_to_double(cR));
            const double wL = __fma_rn(-count_to_double(nL - cL), q.y, count_to_double(cL));
            const double w = __dadd_rn(wR, wL);
            Ws = __dadd_rn(Ws, w);
            // right trials (inv c), left trials (inv c - c)
            Ks = __fma_rn(w, dk.x, __fma_rn(-wL, dk.y, Ks));
            if (wantE) {
                // left trials' a - p less right trials' a - p
                const double2 p = c.gzone(2, c.seg())[z];
                Ei += cL - cR;
                Ep = __fma_rn(count_to_double(nR), p.x, __fma_rn(-count_to_double(nL), p.y, Ep));
            }
        }
        if (z >= (zr & 255) && z < (zr >> 8))
            d = __fma_rn(a.fZa[(int64_t)t * Z + z], count_to_double(Pb[z + 1] - Pb[z]), d);
    }
    if (wantE) d = __fma_rn(-a.wJ[t], __dadd_rn(Ep, (double)Ei), d);
    double W = c.gacc(0), K = c.gacc(1);
    if (zr != 0 || wantE) {
#pragma unroll
        for (int off = P / 2; off >= 1; off >>= 1) d = __dadd_rn(d, __shfl_xor_sync(FULL, d, off, P));
        if (nonzero_bits(d)) {
            c.gacc(2) = __fma_rn(d, W, c.gacc(2));
            c.gacc(3) = __fma_rn(d, K, c.gacc(3));
            if (sl == 0) c.gacc(4) = __dadd_rn(c.gacc(4), d);
        }
    }
    c.gacc(0) = __dadd_rn(W, Ws);
    c.gacc(1) = __dadd_rn(K, Ks);
}

// The current of step t pairs with the score of steps <= t.  Jl: this lane's net
// leftward crossings.
template <int P, bool CLS>
__device__ __forceinline__ void ion_score_current(const IonView<P, CLS> &c, uint32_t t, int Jl)
{
    const SweepArgs &a = c.a;
    if (!a.wJ) return;
    const double2 ab = a.fJab[t];
    if (!(nonzero_bits(ab.x) || nonzero_bits(ab.y))) return;
#pragma unroll
    for (int off = P / 2; off >= 1; off >>= 1) Jl += __shfl_xor_sync(FULL, Jl, off, P);
    const double fJ = __fma_rn(ab.x, (double)Jl, -ab.y);
    c.gacc(2) = __fma_rn(fJ, c.gacc(0), c.gacc(2));
    c.gacc(3) = __fma_rn(fJ, c.gacc(1), c.gacc(3));
    if (c.sl() == 0) c.gacc(4) = __dadd_rn(c.gacc(4), fJ);
}

// The rails' W, K, G_W, G_K: sums of their lanes' shares.
template <int P, bool CLS>
__device__ __forceinline__ void ion_score_end(const IonView<P, CLS> &c, int64_t rail)
{
    const SweepArgs &a = c.a;
    for (int k = 0; k < 5; ++k) {
        double v = c.gacc(k);
        if (k < 4)
#pragma unroll
            for (int off = P / 2; off >= 1; off >>= 1) v = __dadd_rn(v, __shfl_xor_sync(FULL, v, off, P));
        if (c.sl() == 0 && rail < a.R) a.gstate[rail * kGradState + k] = v;
    }
}

// One CTA's tile of rails advanced through steps [t0, t0 + n_steps): rails
// [tile_rail0, tile_rail0 + G * warps).  The draw loop only compares each
// entry's two words with its bounds and keeps the outcomes as bits of M, one
// per row.  With ACC (hop probabilities of order 1e-2 and above, several
// accepted draws per warp and step) it also keeps the least distance of a draw
// below its bound and which neighbours are one and two sites away, so that exclusion
// and conflicts are a few operations on bits.  That loop takes 100 cycles a row on a
// sub-partition, 69 of the multiplier and 73 of the ALU pipe; so an entry's halves
// are two loads instead of a mask and a shift, and the distance stands for the
// comparisons with two lower bounds (65,536 rails of 512 sites, 20 % full: 8.8 ->
// 8.4 ms for 300 steps).  Without ACC, the entries with a word
// below its upper bound are looked at one by one, and as moves are rare the loop
// draws for four steps at once: an entry is loaded once for four draws, and the four
// chains hide each other's latency.  AHEAD: twice four on open rails (16,384 x 1,024:
// 6.7 -> 6.5 ms) and where a lane holds four ions at most (64 x 100: 0.36 -> 0.32 ms),
// once on others, where every ion that moves is drawn for again for the steps left
// (8,192 x 1,000 30 % full: 1.21 -> 1.23 ms for twice).  An ion that moves is drawn for again for
// the steps left.  Steps with nothing but exchanges are left to ion_exchanges (the
// virtual site -1 draws for site 0, so they change no draw).  Against one step at a
// time, 1,000 steps at P0 = 3.8e-4: 64 rails of 100 sites 0.35 -> 0.16 ms, 16,000 of
// 200 3.2 -> 2.6 ms, 3,001 open ones of 777 3.0 -> 2.2 ms; 65,536 of 1,024 with
// per-site barriers 60 -> 50 ms.  GRAD: the gradient pass, which
// replays the sweep from its first occupancy with the score accumulated instead
// of the traces.
//
// The lanes of a warp go through as many rows as its fullest lane, so the rails that
// share a warp should hold equally many ions: a.order lists them by their first
// occupancy's counts, the fullest first (65,536 rails of 512 sites, 102 +- 9 ions, 8
// to a warp: 29 rows on average in the order of their indices, 26 in this one).
template <int P, bool ACC, bool OPEN, class M, bool GRAD = false, int AHEAD = OPEN ? kIonAhead : 4>
__device__ __forceinline__ void ion_tile(const SweepArgs &a, const uint32_t *rk0, const uint32_t *rk1,
                                         int64_t t0, int n_steps, int flush, int64_t tile_rail0,
                                         uint8_t *smem)
{
    constexpr int G = 32 / P;
    using View = IonView<P, !ACC>;
    uint8_t *tab = smem;    // site table of the CTA

    {
        const View c(a, smem);
        const int L = a.L, Z = a.Z, sl = c.sl();
        const int64_t place = c.place(tile_rail0);
        const bool active = place < a.R;
        const int64_t rail = !active ? a.R : a.order != nullptr ? a.order[place] : place;
        // ---- site table of the CTA
        for (int i = (int)c.tid; i < L + 2; i += blockDim.x) {
            const int k = min(max(i - 1, 0), L - 1);
            int row = 0;
            while (a.bnd[row + 1] <= k) ++row;
            row <<= c.cls();
            if (OPEN && i <= 1) row = (Z << c.cls()) + i;
            if (OPEN && i >= L) row = (Z << c.cls()) + 2 + (i - L);
            const uint3 w = site_words((uint32_t)k, a.instance ^ rk1[0]);
            ((uint4 *)tab)[i] = make_uint4(w.x, w.y, w.z, (uint32_t)(i * kStep) | (uint32_t)(row * 16) << 16);
        }
        // ---- occupancy words of the warp's rails, read once from HBM
        const int W = (L + 31) >> 5;          // words per rail
        const int C = (W + P - 1) / P;        // words per lane
        const int w0 = min(sl * C, W), w1 = min(w0 + C, W);
        uint32_t *words = c.words() + c.seg() * W;
        for (int w = w0; w < w1; ++w) {
            uint32_t bits = 0;
            if (active) {
                const uint8_t *row = a.occ + rail * a.stride + 32 * w;
                bits = pack16(*(const uint4 *)row);
                if (32 * w + 16 < a.stride) bits |= pack16(*(const uint4 *)(row + 16)) << 16;
                if (32 * w + 32 > L) bits &= (1u << (L - 32 * w)) - 1u;
            }
            words[w] = bits;
        }
        if (sl == 0) {
            c.Fs()[G] = active ? a.N0[rail] : 0;
            c.Fs()[3 * G] = (int32_t)rail;
        }
        if (a.P0bnd != nullptr)
            for (int z = sl; z < Z; z += P)
                c.p0b(c.seg())[z] = active ? a.P0bnd[rail * Z + z] : make_float2(0.0f, 0.0f);
        c.slot(kSlotMoves) = 0u;
        if (c.lane() == 0) c.mark() = 0;
        __syncthreads();
        if (place - c.seg() >= a.R) return;
        // ---- ions below each zone boundary and F
        for (int b = sl; b <= Z; b += P) {
            const int e = a.bnd[b];
            int m = 0;
            for (int w = 0; w < (e >> 5); ++w) m += __popc(words[w]);
            if (e & 31) m += __popc(words[e >> 5] & ((1u << (e & 31)) - 1u));
            c.Pb(c.seg())[b] = m;
        }
        __syncwarp();
        if (sl == 0) {
            int f = 0;
            for (int b = 0; b <= Z; ++b) f += c.Pb(c.seg())[b] * a.wsum[b];
            c.Fs()[0] = f;
        }
        // zone counts of the launch's first step (the changes of later ones follow)
        for (int z = sl; z < Z && !GRAD; z += P) {
            const int nz = c.Pb(c.seg())[z + 1] - c.Pb(c.seg())[z];
            if (nz != 0) atomicAdd(&a.Zc[t0 * Z + z], (unsigned long long)(long long)nz);
        }
        ion_build<P, OPEN>(c, tab, rail);
        const int sum = ion_sum<P>(c);
        if (sl == 0) c.Fs()[2 * G] = sum;
        __syncwarp();
        if (ACC && a.rule != 0) ion_parity<P, M>(c);
        if constexpr (GRAD) ion_score_begin<P>(c);
    }

    int wend = 0;          // first step after the voltage window of the bounds
    int spent = 0;         // boundary crossings since the bounds were evaluated
    uint32_t dirty = 0u;   // rail slots whose zone sums changed since their bounds were evaluated
    for (int c0 = 0; c0 < n_steps; c0 += flush) {
        const int c1 = min(n_steps, c0 + flush);
        for (int s = c0; s < c1;) {
            const uint32_t t = (uint32_t)(t0 + s);

            const bool window = s == wend;
            if (dirty != 0u || window) {
                const View c(a, smem);
                if (window) wend = ion_window<P, ACC>(c, t0, s, n_steps);
                ion_zones<P, ACC, OPEN>(c, window ? (uint32_t)((1ull << G) - 1u) : dirty, window);
                spent = 0;
            }
            const uint32_t stale = GRAD ? dirty : 0u;   // rail slots to score anew
            dirty = 0u;

            // ---- draws: accepted trials aR, aL (M bits per row), entries with a
            //      draw still to be decided, and rows whose successor is two
            //      sites away
            M aR = 0, aL = 0, und = 0, two = 0;
            M fR = 0, fL = 0;       // rows with open trials (gradient pass)
            uint32_t look = 0u, ends_at = 0u;   // without ACC: steps with a draw that may be accepted, exchanges
            {
                const View c(a, smem);
                const uint32_t prail = a.rail_base + (uint32_t)c.rail();
                const uint8_t *rm = c.bounds();
                const uint32_t *cp = c.colp();
                const uint32_t *const end = cp + c.kmax() * 32;
                if constexpr (ACC) {
                    const StepDraw sd = step_draw(t, prail, rk0, rk1);
                    M one = 0;
                    uint32_t e = *(const uint16_t *)cp, least = FULL;    // distance of a draw below its bound
                    for (int half = 0; half < (int)sizeof(M) / 4 && cp != end; ++half) {
                        // 32 rows at a time, their bits in one register each
                        const uint32_t *const to = end - cp > 32 * 32 ? cp + 32 * 32 : end;
                        uint32_t hR = 0u, hL = 0u, g1 = 0u, g2 = 0u, bit = 1u;
#pragma unroll 4
                        while (cp != to) {
                            const uint2 th = *(const uint2 *)(rm + ((const uint16_t *)cp)[1]);
                            cp += 32;
                            const uint32_t en = *(const uint16_t *)cp;  // the column has one slot more than rows in use
                            const uint32_t gap = en - e;
                            const uint4 w = *(const uint4 *)(tab + e);
                            uint32_t xy, xw;
                            site_draw(sd, w.x, w.y, w.z, rk0, rk1, xy, xw);
                            if (xy <= th.x) hR |= bit;
                            if (xw <= th.y) hL |= bit;
                            least = min(least, min(th.x - xy, th.y - xw));
                            if (gap == 1u * kStep) g1 |= bit;
                            if (gap == 2u * kStep) g2 |= bit;
                            bit <<= 1;
                            e = en;
                        }
                        aR |= (M)hR << (32 * half);
                        aL |= (M)hL << (32 * half);
                        one |= (M)g1 << (32 * half);
                        two |= (M)g2 << (32 * half);
                    }
                    const int n = (int)c.slot(kSlotN);
                    const uint32_t gaps = c.slot(kSlotGaps);
                    // the last entry's successor is on the next lane
                    const M last = n > 0 ? M(1) << (n - 1) : M(0), valid = low_bits<M>(n);
                    one = (one & (valid >> 1)) | (gap_last(gaps) == 1 ? last : 0);
                    two = (two & (valid >> 1)) | (gap_last(gaps) == 2 ? last : 0);
                    fR = valid & ~one;
                    fL = valid & ~(one << 1 | (gap_first(gaps) == 1 ? 1u : 0u));
                    aR &= fR;
                    aL &= fL;
                    if (a.rule != 0) {
                        M odd = ion_odd<P, M>(c);
                        if (t & 1u) odd = ~odd;
                        aR &= ~odd;
                        aL &= odd;
                    }
                    // some draw is within a bound's band: all that may be accepted are looked at
                    und = least <= c.width() ? aR | aL : 0;
                } else {
#pragma unroll 1
                    for (int q0 = 0; q0 < (AHEAD > 4 ? min(AHEAD, min(c1, wend) - s) : 1); q0 += 4) {
                        StepDraw sd[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) sd[q] = step_draw(t + (uint32_t)(q0 + q), prail, rk0, rk1);
                        cp = c.colp();
                        for (int half = 0; half < (int)sizeof(M) / 4; ++half) {
                            const uint32_t *const to = end - cp > 32 * 32 ? cp + 32 * 32 : end;
                            uint32_t h[4] = {}, bit = 1u;
#pragma unroll 1
                            while (cp != to) {
                                const uint32_t e = *cp;
                                cp += 32;
                                const uint4 w = site_at(tab, e);
                                const uint2 th = *(const uint2 *)(rm + (e >> 16));
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    uint32_t xy, xw;
                                    site_draw(sd[q], w.x, w.y, w.z, rk0, rk1, xy, xw);
                                    if (xy <= th.x || xw <= th.y) h[q] |= bit;
                                }
                                bit <<= 1;
                            }
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                c.hits(q0 + q + AHEAD * half) = h[q];
                                if (h[q]) look |= 1u << (q0 + q);
                            }
                        }
                    }
                    look = __reduce_or_sync(FULL, look);
                    if constexpr (OPEN) ends_at = ion_end_draws<P>(c, tab, t, prail, rk0, rk1);
                }
            }
            // ---- the steps drawn for, up to one whose draws are to be made again
            int ahead = ACC ? 1 : min(AHEAD, min(c1, wend) - s);
#pragma unroll 1
            for (int q = 0; q < ahead; ++q) {
            if constexpr (!ACC) {
                const uint32_t next = look >> q;
                int stop = next ? min(ahead, q + __ffs(next) - 1) : ahead;
                und = 0;
                const View c(a, smem);
                if (OPEN) stop = ion_exchanges<P, M>(c, tab, t0, s, n_steps, q, stop, ends_at, und);
                if (stop >= ahead) break;
                q = stop;
                und |= c.hits(q);
                if (sizeof(M) > 4) und |= (M)c.hits(q + AHEAD) << (8 * sizeof(M) - 32);
                aR = aL = two = 0;
            }
            const int sq = s + q;
            const uint32_t tq = t + (uint32_t)q;
            if (ACC && !GRAD && !__any_sync(FULL, (aR | aL | und) != 0)) continue;

            // ---- draws between their bounds (without ACC every draw that may be
            //      accepted): the site's own base probability in the FP32 band
            if (__any_sync(FULL, und != 0)) {
                M left = 0;
                {
                    const View c(a, smem);
                    const int64_t rail = c.rail();
                    const StepDraw sd = step_draw(tq, a.rail_base + (uint32_t)rail, rk0, rk1);
                    const int n = (int)c.slot(kSlotN);
                    const uint32_t gaps = c.slot(kSlotGaps);
                    for (; und; und &= und - 1) {
                        const M bit = und & (M(0) - und);
                        const IonEntry en = ion_entry(c.colp(), first_bit(und), n, gaps, a.rule, tq);
                        const uint4 w = site_at(tab, en.e);
                        uint32_t xy, xw;
                        site_draw(sd, w.x, w.y, w.z, rk0, rk1, xy, xw);
                        int dR, dL;
                        ion_decide<P, OPEN>(c, en, rail, xy, xw, dR, dL);
                        aR = dR == 1 ? aR | bit : aR & ~bit;
                        aL = dL == 1 ? aL | bit : aL & ~bit;
                        if (en.gR == 2) two |= bit;
                        if (dR == 2 || dL == 2) left |= bit;
                    }
                }
                // ---- draws within the band: FP64
                if (__any_sync(FULL, left != 0)) {
                    const View c(a, smem);
                    for (; left; left &= left - 1) {
                        const M bit = left & (M(0) - left);
                        const IonEntry en = ion_entry(c.colp(), first_bit(left), (int)c.slot(kSlotN),
                                                     c.slot(kSlotGaps), a.rule, tq);
                        int dR = en.fR ? 2 : 0, dL = en.fL ? 2 : 0;
                        ion_exact<P>(c, c.seg(), c.rail(), en.x, c.zone(en.e), tq, dR, dL);
                        aR = dR == 1 ? aR | bit : aR & ~bit;
                        aL = dL == 1 ? aL | bit : aL & ~bit;
                    }
                }
            }

            if constexpr (GRAD) {
                const View c(a, smem);
                ion_score_zones<P, OPEN>(c, t, stale);
                ion_score<P, OPEN, M>(c, t, fR, fL, aR, aL);
            }

            // ---- moves and the current: both trials accepted, the ion stays; two
            //      ions entering the site between them are both cancelled
            bool inner = false;      // a move inside the rail
            uint32_t more = 0u;      // steps in which it may move again
            int crossings = 0;       // zone boundaries crossed
            {
                const View c(a, smem);
                const M both = aR & aL;
                aR ^= both;
                aL ^= both;
                if (!__any_sync(FULL, (aR | aL) != 0)) {
                    if constexpr (GRAD) ion_score_current<P>(c, t, 0);
                    continue;
                }
                const int n = (int)c.slot(kSlotN), sl = c.sl();
                const uint32_t gaps = c.slot(kSlotGaps);
                const M clash = aR & (aL >> 1) & two;
                aR ^= clash;
                aL ^= clash << 1;
                // across lanes: the last entry's hop right and the next lane's first left
                const int lastR = n > 0 ? (int)(aR >> (n - 1)) & 1 : 0, firstL = (int)aL & 1;
                const int up = __shfl_up_sync(FULL, lastR, 1, P), dn = __shfl_down_sync(FULL, firstL, 1, P);
                if (sl > 0 && up && firstL && gap_first(gaps) == 2) aL ^= M(1);
                if (sl < P - 1 && dn && lastR && gap_last(gaps) == 2) aR ^= M(1) << (n - 1);
                const int nR = count_bits(aR), nL = count_bits(aL);
                uint32_t *colp = c.colp();
                for (M todo = aR | aL; todo; todo &= todo - 1) {
                    const int j = first_bit(todo);
                    const int r = ion_commit<P>(c, tab, c.rail(), colp + j * 32, colp[j * 32], (aR >> j) & 1 ? 1 : -1,
                                                !GRAD && sq + 1 < n_steps ? a.Zc + (t0 + sq + 1) * a.Z : nullptr);
                    if constexpr (ACC) {
                        crossings += r != 0 ? 1 : 0;
                    } else {
                        crossings += r == 2 ? a.ion_exchange : r;
                        if (r == 2) continue;
                        inner = true;
                        const uint32_t e = colp[j * 32], prail = a.rail_base + (uint32_t)c.rail();
                        const uint4 w = site_at(tab, e);
                        const uint2 th = *(const uint2 *)(c.bounds() + (e >> 16));
#pragma unroll 1
                        for (int k = q + 1; k < ahead; ++k) {
                            uint32_t xy, xw;
                            site_draw(step_draw(t + (uint32_t)k, prail, rk0, rk1), w.x, w.y, w.z, rk0, rk1, xy, xw);
                            if (xy <= th.x || xw <= th.y) {
                                c.hits(k + AHEAD * (j >> 5)) |= 1u << (j & 31);
                                more |= 1u << k;
                            }
                        }
                    }
                }
                if (ACC && a.rule != 0) ion_set_odd<P, M>(c, ion_odd<P, M>(c) ^ (aR | aL));
                if constexpr (GRAD) {
                    ion_score_current<P>(c, t, nL - nR);
                } else {
                    c.slot(kSlotMoves) += (uint32_t)(nR + nL);
                    const int Jw = __reduce_add_sync(FULL, nL - nR);
                    if (c.lane() == 0 && Jw != 0) atomicAdd(&a.J[t0 + sq], (unsigned long long)(long long)Jw);
                }
                ion_refresh<P>(c, n, OPEN ? -2 : -1, OPEN ? a.L + 1 : a.L);
                __syncwarp();
            }
            // an entry can come or go at an end only when one inside has moved
            int ends = 0;
            if (!ACC && __any_sync(FULL, inner)) {
                look |= __reduce_or_sync(FULL, more);
                inner = true;
            }
            if (OPEN && (ACC || inner)) {
                const View c(a, smem);
                uint32_t draws = 0u;
                ends = ion_ends<P>(c, tab, sq, c.rail(), draws);
                if (!GRAD && draws != 0u && c.lane() == 0) atomicAdd(&a.counters[0], (unsigned long long)draws);
            }
            if (ACC && OPEN && ends != 0 && a.rule != 0) {
                const View c(a, smem);
                ion_parity<P, M>(c);
            }
            if constexpr (ACC) {
                // lanes to rail slots
                const uint32_t cm = ends == 2 ? FULL : __ballot_sync(FULL, crossings != 0);
                if (G == 1) dirty = cm != 0u ? 1u : 0u;
                else
#pragma unroll
                    for (int k = 0; k < G; ++k)
                        if ((cm >> (k * P)) & ((1u << (P & 31)) - 1u)) dirty |= 1u << k;
            } else {
                if (__any_sync(FULL, crossings != 0)) spent += __reduce_add_sync(FULL, crossings);
                if (ends != 0) spent += 2;
                if (spent > a.ion_budget || ends == 2) dirty = (uint32_t)((1ull << G) - 1u);
                if (ends != 0 || dirty != 0u) ahead = q + 1;
            }
            }
            s += ahead;
        }
        // ---- flush this warp's counters and per-rail current
        if constexpr (!GRAD) {
            const View c(a, smem);
            __syncwarp();
            const uint32_t nd = __reduce_add_sync(FULL, c.slot(kSlotN)) * (uint32_t)(c1 - c.mark());
            const uint32_t nv = __reduce_add_sync(FULL, c.slot(kSlotMoves));
            // a rail's net leftward crossings: the decrease of its positions' sum
            const int sum = ion_sum<P>(c);
            __syncwarp();
            if (c.lane() == 0) {
                if (nd) atomicAdd(&a.counters[0], (unsigned long long)nd);
                if (nv) atomicAdd(&a.counters[2], (unsigned long long)nv);
                c.mark() = c1;
            }
            c.slot(kSlotMoves) = 0u;
            const int64_t rail = c.rail();
            if (c.sl() == 0) {
                const int v = c.Fs()[2 * G] - sum;
                c.Fs()[2 * G] = sum;
                if (a.Jr && rail < a.R && v != 0) a.Jr[rail] += v;
            }
            __syncwarp();
        }
    }

    if constexpr (GRAD) {
        const View c(a, smem);
        ion_score_end<P>(c, c.rail());
        return;
    }
    // ---- write the rails back
    {
        const View c(a, smem);
        ion_to_words<P>(c);
        const int W = (a.L + 31) >> 5, C = (W + P - 1) / P;
        const int w0 = min(c.sl() * C, W), w1 = min(w0 + C, W);
        const uint32_t *words = c.words() + c.seg() * W;
        const int64_t rail = c.rail();
        if (rail < a.R)
            for (int w = w0; w < w1; ++w) {
                const uint32_t o = words[w];
                uint8_t *row = a.occ + rail * a.stride + 32 * w;
                *(uint4 *)row = unpack16(o & 0xFFFFu);
                if (32 * w + 16 < a.stride) *(uint4 *)(row + 16) = unpack16(o >> 16);
            }
    }
}

// Calls f(lanes per rail, accept path, open electrodes, type of the row bits)
// for an ion-list kind.
template <class F>
cudaError_t with_ions(int kind, bool acc, F &&f)
{
    using std::integral_constant;
    using T = integral_constant<bool, true>;
    using N = integral_constant<bool, false>;
    const int k = kind - kWordKinds;
    const bool open = (k & 1) != 0;
    auto go = [&](auto p, auto m) {
        if (acc) return open ? f(p, T(), T(), m) : f(p, T(), N(), m);
        return open ? f(p, N(), T(), m) : f(p, N(), N(), m);
    };
    switch (k >> 1) {
    case 0: return go(integral_constant<int, 4>(), uint32_t());
    case 1: return go(integral_constant<int, 8>(), uint32_t());
    case 2: return go(integral_constant<int, 16>(), uint32_t());
    case 3: return go(integral_constant<int, 32>(), uint32_t());
    default: return go(integral_constant<int, 32>(), uint64_t());
    }
}

}  // namespace

}  // namespace kmc
