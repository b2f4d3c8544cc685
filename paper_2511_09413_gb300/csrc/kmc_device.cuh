// kmc_device.cuh -- device routines shared by the tile bodies (kmc_sweep.cu,
// kmc_ions.cu): the Philox4x32-10 draw, occupancy packing, the integer bounds
// of a decision and the exact FP64 decision path.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "kmc_internal.h"

namespace kmc {

namespace {

constexpr unsigned FULL = 0xffffffffu;

__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): per round two 32x32->64
// multiplies; the high halves are xor-ed with the other counter words and the
// round key.  The ten round keys are precomputed on the host.
__device__ __forceinline__ uint4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                        const uint32_t *rk0, const uint32_t *rk1)
{
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        // one widening multiply per product (both halves at once): 1 % faster
        // in the sweep and 2.5 % in the Philox-only probe than separate
        // low and high multiplies
        uint64_t p0, p1;
        asm("mul.wide.u32 %0, %1, %2;" : "=l"(p0) : "r"(c0), "r"(0xD2511F53u));
        asm("mul.wide.u32 %0, %1, %2;" : "=l"(p1) : "r"(c2), "r"(0xCD9E8D57u));
        const uint32_t lo0 = (uint32_t)p0, hi0 = (uint32_t)(p0 >> 32);
        const uint32_t lo1 = (uint32_t)p1, hi1 = (uint32_t)(p1 >> 32);
        c0 = hi1 ^ c1 ^ rk0[i];
        c1 = lo1;
        c2 = hi0 ^ c3 ^ rk1[i];
        c3 = lo0;
    }
    return make_uint4(c0, c1, c2, c3);
}

// 16 occupancy bytes (values 0/1) -> 16 bits; byte i -> bit i.
__device__ __forceinline__ uint32_t pack4(uint32_t v)
{
    return (((v & 0x01010101u) * 0x00204081u) >> 21) & 0xFu;
}
__device__ __forceinline__ uint32_t pack16(uint4 q)
{
    return pack4(q.x) | (pack4(q.y) << 4) | (pack4(q.z) << 8) | (pack4(q.w) << 12);
}
// 4 bits -> 4 bytes of 0/1
__device__ __forceinline__ uint32_t unpack4(uint32_t n)
{
    return (n * 0x00204081u) & 0x01010101u;
}
__device__ __forceinline__ uint4 unpack16(uint32_t b)
{
    return make_uint4(unpack4(b & 0xF), unpack4((b >> 4) & 0xF), unpack4((b >> 8) & 0xF),
                      unpack4((b >> 12) & 0xF));
}

// Conservative integer thresholds on the high 32 bits h of a 64-bit draw w
// (u = (w >> 11) 2^-53):  h < acc_thr(p_lo) implies u <= p;  h > rej_thr(p_hi)
// implies u > p, for any p in [p_lo, p_hi].
__device__ __forceinline__ uint32_t acc_thr(float p_lo)
{
    const uint32_t f = __float2uint_rd(p_lo * 4294967296.0f);
    return f > 0u ? f - 1u : 0u;
}
__device__ __forceinline__ uint32_t rej_thr(float p_hi)
{
    return __float2uint_ru(p_hi * 4294967296.0f);
}

// --------------------------------------------------------- exact FP64 path
// Exact FP64 zone quantities (B_z, 1/(1+B_z)) for zone zt of one rail, with
// the operation order of the oracle: excess C_z, enclosed charge Q_z, mean
// Qbar, dV_z (S2.1.8), dE_z (Eq. 3), B_z (Eq. 4).  Every operation is an
// explicitly rounded intrinsic so that no contraction changes the result.
__device__ __forceinline__ void exact_zone(const int32_t *Pb, const DevConst *Kp, int Z, int L,
                                        int32_t n0, const double2 *bgd, double V, int zt, double *B,
                                        double *inv)
{
    const DevConst &K = *Kp;
    const double Ld = (double)L;
    double run = 0.0, acc = 0.0, Qt = 0.0;
    for (int z = 0; z < Z; ++z) {
        const int w = K.bnd[z + 1] - K.bnd[z];
        const int Nz = Pb[z + 1] - Pb[z];
        // background N0 w_z / L: the rail's precomputed row when there is one
        const double bz = bgd ? bgd[z].x : __ddiv_rn(__dmul_rn((double)n0, (double)w), Ld);
        const double C = __dsub_rn((double)Nz, bz);
        const double Q = __dadd_rn(run, __dmul_rn(0.5, C));
        run = __dadd_rn(run, C);
        acc = __dadd_rn(acc, __dmul_rn((double)w, Q));
        if (z == zt) Qt = Q;
    }
    const double Qbar = __ddiv_rn(acc, Ld);
    const double dV = __dsub_rn(V, __dmul_rn(K.ka, __dsub_rn(Qt, Qbar)));
    const double dE = __ddiv_rn(__dmul_rn(dV, K.d), K.t_dev);
    const double b = exp(__ddiv_rn(-dE, K.kT));
    *B = b;
    *inv = __ddiv_rn(1.0, __dadd_rn(1.0, b));
}

// Exact decision u <= p for the 64-bit word w, with near-threshold logging.
__device__ __forceinline__ bool exact_trial(uint64_t w, double p, kmc_log_entry *log,
                                         unsigned long long *log_count, int64_t log_cap,
                                         int32_t rail, uint32_t step, int32_t site, int32_t dir,
                                         int32_t kind)
{
    const double u = __dmul_rn((double)(w >> 11), 0x1.0p-53);
    const double diff = __dsub_rn(u, p);
    if (fabs(diff) < 1e-12) {
        const unsigned long long slot = atomicAdd(log_count, 1ull);
        if ((int64_t)slot < log_cap) {
            kmc_log_entry e;
            e.rail = rail;
            e.step = step;
            e.site = site;
            e.dir = dir;
            e.kind = kind;
            e.pad = 0;
            e.diff = diff;
            log[slot] = e;
        }
    }
    return u <= p;
}

// Band factors: p_lo = p flo, p_hi = p fhi bracket the exact p.
__device__ __forceinline__ int bounded(uint32_t h, float p, float flo, float fhi)
{
    return h < acc_thr(p * flo) ? 1 : (h > rej_thr(p * fhi) ? 0 : 2);
}

// ------------------------------------------------- gradient pass helpers
// Tests on a double's bit pattern, on the integer pipe (FP64 compares take
// the FP64 pipe, the gradient pass's bottleneck): x != 0 (NaN counts as
// nonzero, as the FP64 test does), equality of two values that are never NaN
// (+0 and -0 differ: a stale mark at worst), and lo < x < hi for lo, hi
// positive and finite (positive doubles order as their bit patterns; negative
// values and NaN fall outside).
__device__ __forceinline__ bool nonzero_bits(double x)
{
    return ((unsigned long long)__double_as_longlong(x) << 1) != 0ull;
}
__device__ __forceinline__ bool same_bits(double x, double y)
{
    return __double_as_longlong(x) == __double_as_longlong(y);
}
__device__ __forceinline__ bool inside_bits(double x, double lo, double hi)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const unsigned long long l = (unsigned long long)__double_as_longlong(lo);
    const unsigned long long h = (unsigned long long)__double_as_longlong(hi);
    return u - (l + 1ull) < h - (l + 1ull);
}

// 1 / d for d > 0 (normal, finite) by Newton-Raphson on f(r) = 1/r - d from the
// hardware approximation (rcp.approx.ftz.f64, about 2^-22 relative): each
// step r <- r + r (1 - d r) squares the relative error, so two give full FP64
// accuracy up to a few ulp, enough for score weights.
__device__ __forceinline__ double recip_newton(double d)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    double e = __fma_rn(-d, r, 1.0);
    r = __fma_rn(r, e, r);
    e = __fma_rn(-d, r, 1.0);
    return __fma_rn(r, e, r);
}

// Score weight of one electrode trial of probability p, outcome hit, with
// r1 = 1 / (1 - p) (0 when p >= 1)
__device__ __forceinline__ double et_weight(int hit, double p, double r1)
{
    if (p >= 1.0) return (double)hit;
    return __fma_rn(-1.0, __dmul_rn(p, r1), __dmul_rn((double)hit, r1));
}
}  // namespace

}  // namespace kmc
