// synth.cu -- training profiles: seeded light curves generated on the device and folded
// at their true period (plus a random drift of at most `drift_bins` bins over the
// baseline) by a single-period fold.
//
// Light curve j (global index) has n_cadences samples at t_i = i * cadence from t0 = 0,
// flux = 1 + sigma z_i + signal(t_i) with z_i standard normal. Even j: a box transit
// (positive). Odd j, by (j / 2) mod 3: noise only, a sinusoid, or an eclipsing-binary-like
// pair of boxes (primary + secondary half a period later) -- the negatives.
// Random numbers come from Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11) keyed by the
// 64-bit seed: counter (j, 0, 0, 0xFFFFFFFF) and (j, 1, 0, 0xFFFFFFFF) give the light curve's
// parameters, counter (j, i / 4, 1, 0) the four normals of samples 4(i/4) .. 4(i/4)+3
// (Box-Muller on uniforms u = (x >> 8) 2^-24).
//
// Fold: one block per light curve, lanes taking four consecutive samples each (the four
// normals of one Philox call). What bounds it is instruction issue: the device's FP64 rate is
// one warp instruction per 64 cycles and scheduler, so a sample does no FP64 at all.
//  * tau_i = rint(fl(i cadence) 2^24) comes from a 64-bit fixed-point product i * cadence
//    2^(24+40), and the box membership from the fixed-point phase of the light curve's own
//    period; both know how far they can be off, and a sample that close to a rounding or box
//    edge (one in some 10^5) is decided by the FP64 formula itself, so every bin, count and
//    membership is that of the formula.
//  * flux: x is summed as integers, rint(x 2^e) with |x| 2^e < 2^29 (exact where |x| 2^e is 2^24 or
//    more), by shared-memory reductions: the low 15 bits, the rest and the count each have a word
//    per bin. Integer sums are exact and independent of their order; sum and sum of squares (of
//    the upper 26 bits, a 64-bit integer per lane, emptied into FP64 with the bin words) also give
//    the flux standard deviation.
//  * a sinusoid's phase is fixed point too, and its flux a sum of FP32 pairs.
// 4,096 curves of 65,536 samples: 12.5 ms with FP64 phases, fmod, moments and a 32-shuffle
// merge of equal bins per sample; now 1.32 ms.
#include <cmath>
#include <cstdint>

#include "gpfc_common.cuh"
#include "gpfc_synth.h"

namespace gpfc {

struct Philox4 {
    uint32_t v[4];
};

__host__ __device__ __forceinline__ Philox4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                          uint32_t k0, uint32_t k1)
{
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k0 += W0;
            k1 += W1;
        }
        const uint64_t p0 = (uint64_t)M0 * c0, p1 = (uint64_t)M1 * c2;
        const uint32_t hi0 = (uint32_t)(p0 >> 32), lo0 = (uint32_t)p0;
        const uint32_t hi1 = (uint32_t)(p1 >> 32), lo1 = (uint32_t)p1;
        const uint32_t n0 = hi1 ^ c1 ^ k0, n1 = lo1, n2 = hi0 ^ c3 ^ k1, n3 = lo0;
        c0 = n0;
        c1 = n1;
        c2 = n2;
        c3 = n3;
    }
    return Philox4{{c0, c1, c2, c3}};
}

__device__ __forceinline__ double unif64(uint32_t x) { return (double)(x >> 8) * (1.0 / 16777216.0); }
__device__ __forceinline__ float unif32(uint32_t x) { return (float)(x >> 8) * (1.0f / 16777216.0f); }

// Parameters of a light curve, derived by one warp and shared by its block.
struct LcParams {
    int kind;        // 0 transit, 1 noise, 2 sinusoid, 3 eclipsing binary
    int fixed;       // the fixed-point phases below hold for every sample
    double period, epoch, duration, fold_period;
    float sigma, depth, depth2, amp, amp_lo;  // (amp + amp_lo: to FP64's precision)
    uint32_t Fl, Fh;  // fold frequency, rint(2^40 / fold_period)
    uint32_t Gl, Gh;  // light curve's own frequency, rint(2^40 / period)
    uint32_t off;     // epoch / period in 2^-32 cycles
    uint32_t half;    // half the duration in 2^-32 cycles
    uint32_t guard;   // bound of the phase's error in 2^-32 cycles
    float cyc;        // 2^-24 / period: cycles per unit of tau
    float drift;      // cycles per 2^16 units of tau that 2^-40 (Gh 2^32 + Gl) falls short by
    float scale;      // 2^e
    int e;
    // the cadence in units of tau: integer part, fraction in 2^-64; and in 2^-20 (64-bit)
    uint32_t step_i;
    uint64_t step_f, step20;
    uint32_t tguard;  // bound of the fixed-point time's error in 2^-20 units of tau
};

// Called by one whole warp; lane 0's values are the light curve's.
__device__ LcParams lc_params(uint64_t seed, int64_t j, const gpfc_synth_params &sp, int lane)
{
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const Philox4 a = philox4x32_10((uint32_t)j, 0u, 0u, 0xFFFFFFFFu, k0, k1);
    const Philox4 b = philox4x32_10((uint32_t)j, 1u, 0u, 0xFFFFFFFFu, k0, k1);
    LcParams p{};
    p.kind = (j & 1) ? 1 + (int)((j >> 1) % 3) : 0;
    // the three log-uniform draws (sigma, depth, amplitude) on three lanes at once
    const double lo = lane == 0 ? sp.sigma_min : sp.depth_min, hi = lane == 0 ? sp.sigma_max : sp.depth_max;
    const double lu = exp(log(lo) + unif64(lane == 0 ? a.v[0] : (lane == 1 ? b.v[0] : b.v[2])) * log(hi / lo));
    const double sigma = __shfl_sync(0xffffffffu, lu, 0), depth = __shfl_sync(0xffffffffu, lu, 1);
    const double amp = __shfl_sync(0xffffffffu, lu, 2);
    // explicit round-to-nearest operations (no fused multiply-add), so that these values
    // are bit-identical to any IEEE-754 evaluation of the same formulas
    p.period = __dadd_rn(sp.p_min, __dmul_rn(unif64(a.v[1]), __dsub_rn(sp.p_max, sp.p_min)));
    p.epoch = __dmul_rn(unif64(a.v[2]), p.period);
    p.duration = __ddiv_rn(__dadd_rn(sp.dur_min_h, __dmul_rn(unif64(a.v[3]), __dsub_rn(sp.dur_max_h, sp.dur_min_h))),
                           24.0);
    const double depth2 = __dmul_rn(depth, __dadd_rn(0.2, __dmul_rn(0.8, unif64(b.v[1]))));
    const double T = __dmul_rn((double)sp.n_cadences, sp.cadence);
    const double df = __ddiv_rn(__dmul_rn(__dsub_rn(__dmul_rn(2.0, unif64(b.v[3])), 1.0), sp.drift_bins),
                                __dmul_rn(256.0, T));
    p.fold_period = __ddiv_rn(1.0, __dadd_rn(__ddiv_rn(1.0, p.period), df));
    p.sigma = (float)sigma;
    p.depth = (float)depth;
    p.depth2 = (float)depth2;
    p.amp = (float)amp;
    p.amp_lo = (float)(amp - (double)p.amp);
    const unsigned long long F = (unsigned long long)__double2ll_rn(__ddiv_rn(1099511627776.0, p.fold_period));
    p.Fl = (uint32_t)F;
    p.Fh = (uint32_t)(F >> 32);
    // |x| < 5.78 sigma (the largest Box-Muller radius for u >= 2^-24) plus the signal
    const double xmax = 5.78 * sigma + (p.kind == 2 ? amp : (p.kind == 0 ? depth : (p.kind == 3 ? depth + depth2 : 0.0)));
    p.e = max(-100, min(100, 28 - ilogb(xmax)));
    p.scale = (float)ldexp(1.0, p.e);
    // fixed-point phase of the light curve's own period: off by at most 2^-25 d of tau, half a
    // unit of 2^-40 c/d over T, and a few units of 2^-32 cycles
    const double freq = 1.0 / p.period;
    const unsigned long long G = (unsigned long long)__double2ll_rn(1099511627776.0 * freq);
    p.Gl = (uint32_t)G;
    p.Gh = (uint32_t)(G >> 32);
    p.drift = (float)((freq - (double)G * 9.094947017729282e-13) * 0.00390625);
    p.off = (uint32_t)__double2ll_rn(p.epoch * freq * 4294967296.0);
    const double half = 0.5 * p.duration * freq;
    p.half = (uint32_t)__double2ll_rn(fmin(half, 0.5) * 4294967296.0);
    const double guard = 4294967296.0 * (freq * 5.9604644775390625e-08 + T * 9.094947017729282e-13) + 16.0;
    p.guard = (uint32_t)fmin(guard, 1e9);
    p.cyc = (float)(freq * 5.9604644775390625e-08);
    // fixed-point time of four consecutive samples: the first exact to 2^-32 and cut to 2^-20
    // units of tau, three additions of a step cut to 2^-20; and the rounding of i * cadence in FP64
    const double c24 = sp.cadence * 16777216.0;
    const double tguard = 6.0 + 1048576.0 * (T * 16777216.0) * 2.220446049250313e-16;
    p.fixed = c24 < 8388608.0 && T * 16777216.0 < 4398046511104.0 && tguard < 65536.0 && freq < 1e6 && freq > 1e-6 &&
              guard < 1e6 && half < 0.49;
    p.tguard = p.fixed ? (uint32_t)tguard : 0u;
    p.step_i = p.fixed ? (uint32_t)c24 : 0u;
    p.step_f = p.fixed ? (uint64_t)((c24 - floor(c24)) * 18446744073709551616.0) : 0ull;
    p.step20 = p.fixed ? (uint64_t)(c24 * 1048576.0) : 0ull;
    return p;
}

// The box membership in FP64: |t - nearest mid-transit| < dur / 2.
__device__ __noinline__ bool in_box(double t, double period, double centre, double dur)
{
    const double half = __dmul_rn(0.5, period);
    const double d = fmod(__dadd_rn(__dsub_rn(t, centre), half), period);
    const double dd = __dsub_rn(d < 0.0 ? __dadd_rn(d, period) : d, half);
    return fabs(dd) < __dmul_rn(0.5, dur);
}

// The membership from the signed fixed-point phase about the mid-transit; 0 or 1, or 2 within
// the guard of an edge.
__device__ __forceinline__ int in_box_fixed(int32_t su, uint32_t half, uint32_t guard)
{
    const uint32_t a = su < 0 ? 0u - (uint32_t)su : (uint32_t)su;
    return a - half + guard <= 2u * guard ? 2 : (a < half ? 1 : 0);
}

__device__ __noinline__ long long tau_fp64(int i, double cadence)
{
    return __double2ll_rn(__dmul_rn(__dmul_rn((double)i, cadence), 16777216.0));
}

// sin(2 pi (u 2^-32 + du)), |du| small, as lead + mid + rest: u is reduced to within an eighth of a
// cycle of a quarter; there the sine is a = 2 pi f and the cosine 1 - a^2 / 2, up to a rest below 0.1,
// from the Taylor series (next terms below 2e-9 for |a| <= pi / 4).
__device__ __forceinline__ void sin_cycles(uint32_t u, float du, float &lead, float &mid, float &rest)
{
    const uint32_t quarter = (u + (1u << 29)) >> 30;
    const int32_t v = (int32_t)(u - (quarter << 30));
    const int32_t vh = v & ~63;  // (24 bits: exact in FP32)
    const float f = (float)vh * 2.3283064365386963e-10f, fl = fmaf((float)(v - vh), 2.3283064365386963e-10f, du);
    const float a = 6.2831855f * f;
    const float al = fmaf(6.2831855f, f, -a) + fmaf(-1.7484556e-7f, f, 6.2831855f * fl);
    const float q = a * a;
    // sin a - a, and cos a - (1 - q / 2) with what q is short of a^2
    const float s = a * q * fmaf(q, fmaf(q, fmaf(q, 2.7557319e-6f, -1.9841270e-4f), 8.3333333e-3f), -0.16666667f);
    const float c = fmaf(q * q, fmaf(q, fmaf(q, fmaf(q, -2.7557319e-7f, 2.4801587e-5f), -1.3888889e-3f), 4.1666667e-2f),
                         -0.5f * fmaf(a, a, -q));
    const bool cosine = quarter & 1u;
    lead = cosine ? 1.f : a;
    mid = cosine ? -0.5f * q : 0.f;
    rest = cosine ? fmaf(-al, a + s, c) : fmaf(al, fmaf(-0.5f, q, 1.f + c), s);
    if (quarter & 2u) {
        lead = -lead;
        mid = -mid;
        rest = -rest;
    }
}

// a + b as a pair (TwoSum)
__device__ __forceinline__ float two_sum(float a, float b, float &e)
{
    const float s = a + b, bb = s - a;
    e = (a - (s - bb)) + (b - bb);
    return s;
}

// Threads per light curve: 256, so that several blocks share an SM and one's set-up overlaps
// the others' samples; 1,024 where there are too few light curves to fill the SMs that way. Curves
// of few samples are set-up above all and take four blocks an SM, with 64 registers a thread: 4,096 of
// 1,000 samples 168 -> 143 us, of 65,536 1.32 -> 1.44 ms.
constexpr int kSynthThreads = 256, kSynthWide = 1024, kSynthShort = 4096;

// Samples between emptyings of the 32-bit bin words (|hi| <= 2^14 and lo < 2^15 a sample: sums up to
// 2^31 and below 2^32) and of a lane's squares (512 of 2^52 at most).
constexpr int kSynthSpan = 1 << 17;

template <bool POW2, int THREADS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS) synth_fold_kernel(SynthParams P, int shift)
{
    __shared__ uint32_t s_lo[256], s_hi[256], s_cnt[256];  // sum = hi 2^15 + lo, hi signed
    __shared__ LcParams s_lp;
    __shared__ long long s_m1[8];
    __shared__ double s_m2[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nb = P.nbins, n = P.sp.n_cadences, tid = threadIdx.x;
    const uint32_t k0 = (uint32_t)P.seed, k1 = (uint32_t)(P.seed >> 32);
    for (int64_t q = blockIdx.x; q < P.n; q += gridDim.x) {
        const int64_t j = P.first + q;
        if (warp == 0) {
            const LcParams l = lc_params(P.seed, j, P.sp, lane);
            if (lane == 0) s_lp = l;
        }
        if (tid < 256) s_lo[tid] = s_hi[tid] = s_cnt[tid] = 0u;
        __syncthreads();
        const LcParams &lp = s_lp;
        const int kind = lp.kind;
        const bool fixed = lp.fixed != 0, boxes = kind == 0 || kind == 3;
        const uint32_t Fl = lp.Fl, Fh = lp.Fh, Gl = lp.Gl, Gh = lp.Gh, half = lp.half, guard = lp.guard;
        const uint32_t step_i = lp.step_i, sfl = (uint32_t)lp.step_f, sfh = (uint32_t)(lp.step_f >> 32), tguard = lp.tguard;
        const uint64_t step20 = lp.step20;
        const float sigma = lp.sigma, scale = lp.scale;
        double m2 = 0.0;                       // sum of squares of this lane's integers, over 2^6
        long long tot = 0;                     // bin tid: sum and count
        uint32_t cnt = 0u;
        for (int64_t span = 0; span < n; span += kSynthSpan) {
            const int i_end = (int)min((int64_t)n, span + kSynthSpan);
            unsigned long long sq = 0ull;
            for (int64_t base = span + 128 * warp; base < i_end; base += 128 * nw) {
                const int i0 = (int)base + 4 * lane;  // this lane's four samples
                if (i0 >= i_end) break;               // (no warp-wide operation below)
                const Philox4 r = philox4x32_10((uint32_t)j, (uint32_t)(i0 >> 2), 1u, 0u, k0, k1);
                // time of sample i0 in 2^-20 units of tau
                const uint64_t p0 = (uint64_t)(uint32_t)i0 * sfl, p1 = (uint64_t)(uint32_t)i0 * sfh + (p0 >> 32);
                uint64_t tf = (((uint64_t)(uint32_t)i0 * step_i + (p1 >> 32)) << 20) | ((uint32_t)p1 >> 12);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float u1 = 1.0f - unif32(r.v[2 * h]);  // (0, 1]
                    const float u2 = unif32(r.v[2 * h + 1]);
                    const float rad = sqrtf(-2.0f * logf(u1));
                    float sn, cs;
                    sincospif(2.0f * u2, &sn, &cs);
#pragma unroll
                    for (int m = 0; m < 2; ++m, tf += step20) {
                        const int i = i0 + 2 * h + m;
                        if (i >= i_end) break;
                        // tau: the rounded fixed-point time, or FP64 near a half
                        const uint64_t tr = tf + (1ull << 19);
                        long long tau = (long long)(tr >> 20);
                        const uint32_t fr = (uint32_t)tr & 0xFFFFFu;
                        if (!fixed || fr - tguard > 0xFFFFFu - 2u * tguard) tau = tau_fp64(i, P.sp.cadence);
                        const uint32_t tl = (uint32_t)(unsigned long long)tau, th = (uint32_t)((unsigned long long)tau >> 32);
                        float x = sigma * (m ? rad * sn : rad * cs), xl = 0.f;
                        if (kind != 1) {
                            const uint32_t ph = (uint32_t)(((unsigned long long)tl * Gl +
                                                            ((unsigned long long)(th * Gl + tl * Gh) << 32)) >> 32);
                            const int32_t su = (int32_t)(ph - lp.off);
                            if (boxes) {
                                int in = fixed ? in_box_fixed(su, half, guard) : 2;
                                if (in == 2)
                                    in = in_box(__dmul_rn((double)i, P.sp.cadence), lp.period, lp.epoch, lp.duration);
                                if (in) x -= lp.depth;
                                if (kind == 3) {
                                    in = fixed ? in_box_fixed((int32_t)((uint32_t)su ^ 0x80000000u), half, guard) : 2;
                                    if (in == 2)
                                        in = in_box(__dmul_rn((double)i, P.sp.cadence), lp.period,
                                                    __dadd_rn(lp.epoch, __dmul_rn(0.5, lp.period)), lp.duration);
                                    if (in) x -= lp.depth2;
                                }
                            } else if (fixed) {
                                // phase with the part of the time below the unit of tau
                                const float dt = (float)((int32_t)fr - (1 << 19)) * 9.5367431640625e-07f;
                                const float t16 = (float)((th << 16) | (tl >> 16));  // tau / 2^16 < 2^26
                                float lead, mid, rest, e0, e1;
                                sin_cycles((uint32_t)su, fmaf(dt, lp.cyc, t16 * lp.drift), lead, mid, rest);
                                // the products and their sum with what FP32 cuts off, xl
                                const float p0 = lp.amp * lead, p1 = lp.amp * mid;
                                x = two_sum(two_sum(p0, p1, e0), fmaf(lp.amp, rest, fmaf(lp.amp_lo, lead + mid, x)), e1);
                                xl = (e0 + e1) + (fmaf(lp.amp, lead, -p0) + fmaf(lp.amp, mid, -p1));
                            } else {
                                const double t = __dmul_rn((double)i, P.sp.cadence);
                                x += (float)(((double)lp.amp + (double)lp.amp_lo) *
                                             sinpi(2.0 * (t - lp.epoch) / lp.period));
                            }
                        }
                        int xq = __float2int_rn(x * scale);
                        if (kind == 2) xq += __float2int_rn(xl * scale);
                        const int x26 = (xq + 4) >> 3;
                        sq += (unsigned long long)((long long)x26 * (long long)x26);
                        const unsigned long long phi = (unsigned long long)tl * Fl +
                                                       ((unsigned long long)(th * Fl + tl * Fh) << 32);
                        const uint32_t bin = POW2 ? (uint32_t)(phi >> 32) >> shift
                                                  : (uint32_t)__umul64hi(phi, (unsigned long long)nb);
                        atomicAdd(&s_lo[bin], (uint32_t)xq & 32767u);
                        atomicAdd(&s_hi[bin], (uint32_t)(xq >> 15));
                        atomicAdd(&s_cnt[bin], 1u);
                    }
                }
            }
            m2 += (double)sq;
            __syncthreads();
            if (tid < nb) {
                tot += ((long long)(int32_t)s_hi[tid] << 15) + (long long)s_lo[tid];
                cnt += s_cnt[tid];
                s_lo[tid] = s_hi[tid] = s_cnt[tid] = 0u;
            }
            __syncthreads();
        }
        const double unit = ldexp(1.0, -lp.e);
        if (tid < nb) {
            const size_t o = (size_t)q * nb + tid;
            if (P.folded)
                P.folded[o] = cnt ? (float)(1.0 + (double)tot * unit / (double)cnt) : __int_as_float(0x7fc00000);
            if (P.counts) P.counts[o] = (int32_t)cnt;
        }
        if (P.sigma_out) {
            for (int o = 16; o > 0; o >>= 1) {
                tot += __shfl_xor_sync(0xffffffffu, tot, o);
                m2 += __shfl_xor_sync(0xffffffffu, m2, o);
            }
            if (lane == 0) {
                if (warp < 8) s_m1[warp] = tot;  // (256 bins: the first eight warps)
                s_m2[warp] = m2;
            }
            __syncthreads();
            if (tid == 0) {
                long long a = 0;
                double b2 = 0.0;
                for (int w = 0; w < min(nw, 8); ++w) a += s_m1[w];
                for (int w = 0; w < nw; ++w) b2 += s_m2[w];
                const double nn = (double)n, mu = (double)a / nn;
                P.sigma_out[q] = (float)(sqrt(fmax(64.0 * b2 / nn - mu * mu, 0.0)) * unit);
            }
        }
        if (tid == 0 && P.label) P.label[q] = kind == 0 ? 1.f : 0.f;
        if (tid == 0 && P.period_out) P.period_out[q] = lp.fold_period;
        __syncthreads();
    }
}

// ------------------------------------------------------------------ the paper's vectors

// One thread per 4 bins of a vector (the 4 normals of one Philox call), 64 per vector of
// 256 bins; the vector's parameters are derived by every thread from the same counters.
__global__ void paper_vectors_kernel(VectorParams P)
{
    const uint32_t k0 = (uint32_t)P.seed, k1 = (uint32_t)(P.seed >> 32);
    const int per_vec = (P.nbins + 3) / 4;
    const int64_t total = P.n * per_vec;
    const gpfc_vector_params &v = P.vp;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total; g += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = g / per_vec;
        const int m = (int)(g - q * per_vec);
        const int64_t j = P.first + q;
        const Philox4 a = philox4x32_10((uint32_t)j, 0u, 2u, 0xFFFFFFFFu, k0, k1);
        const Philox4 b = philox4x32_10((uint32_t)j, 1u, 2u, 0xFFFFFFFFu, k0, k1);
        const bool positive = (j & 1) == 0;
        const bool inject = positive || ((j >> 1) & 1);
        const double sigma = exp(log(v.sigma_min) + unif64(a.v[0]) * log(v.sigma_max / v.sigma_min));
        double alpha = 0.0;
        if (positive) alpha = v.alpha_pos_min + unif64(a.v[1]) * (v.alpha_pos_max - v.alpha_pos_min);
        else if (inject) alpha = unif64(a.v[1]) * v.alpha_neg_max;
        const double qq = v.q_min + unif64(a.v[2]) * (v.q_max - v.q_min);
        const double r = unif64(a.v[3]);
        const double phi0 = unif64(b.v[0]);
        const double depth = alpha * sigma / sqrt((double)v.n_points * qq);
        const double sigma_bin = sigma * sqrt((double)P.nbins / (double)v.n_points);
        const double t14 = 2.0 * qq / (1.0 + r), t23 = r * t14;
        const Philox4 rr = philox4x32_10((uint32_t)j, (uint32_t)m, 3u, 0u, k0, k1);
        float z[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float u1 = 1.0f - unif32(rr.v[2 * h]);
            const float u2 = unif32(rr.v[2 * h + 1]);
            const float rad = sqrtf(-2.0f * logf(u1));
            float sn, cs;
            sincospif(2.0f * u2, &sn, &cs);
            z[2 * h] = rad * cs;
            z[2 * h + 1] = rad * sn;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int bin = 4 * m + u;
            if (bin >= P.nbins) break;
            const double x = ((double)bin + 0.5) / (double)P.nbins;
            double d = x - phi0;
            d = fabs(d - floor(d + 0.5));
            const double shape = d <= 0.5 * t23 ? 1.0 : (d < 0.5 * t14 ? (0.5 * t14 - d) / (0.5 * (t14 - t23)) : 0.0);
            P.folded[q * P.nbins + bin] = (float)(1.0 + sigma_bin * (double)z[u] - depth * shape);
        }
        if (m == 0) {
            if (P.label) P.label[q] = positive ? 1.f : 0.f;
            if (P.alpha) P.alpha[q] = (float)alpha;
            if (P.sigma_bin) P.sigma_bin[q] = (float)sigma_bin;
        }
    }
}

cudaError_t launch_paper_vectors(const VectorParams &p, int num_sms, cudaStream_t st)
{
    const int64_t total = p.n * ((p.nbins + 3) / 4);
    const int64_t want = (total + 255) / 256;
    const int grid = (int)(want < (int64_t)num_sms * 8 ? want : (int64_t)num_sms * 8);
    paper_vectors_kernel<<<grid, 256, 0, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_synth(const SynthParams &p, int num_sms, cudaStream_t st)
{
    const int threads = p.n < (int64_t)num_sms * 2 ? kSynthWide : kSynthThreads;
    const int grid = (int)(p.n < (int64_t)num_sms * 8 ? p.n : (int64_t)num_sms * 8);
    int shift = 32;
    while (shift > 0 && (1 << (32 - shift)) < p.nbins) --shift;
    const bool pow2 = (p.nbins & (p.nbins - 1)) == 0;
    auto launch = [&](auto k_pow2, auto k_any) {
        if (pow2) k_pow2<<<grid, threads, 0, st>>>(p, shift);
        else k_any<<<grid, threads, 0, st>>>(p, 0);
    };
    if (threads == kSynthWide)
        launch(synth_fold_kernel<true, kSynthWide, 0>, synth_fold_kernel<false, kSynthWide, 0>);
    else if (p.sp.n_cadences < kSynthShort)
        launch(synth_fold_kernel<true, kSynthThreads, 4>, synth_fold_kernel<false, kSynthThreads, 4>);
    else launch(synth_fold_kernel<true, kSynthThreads, 0>, synth_fold_kernel<false, kSynthThreads, 0>);
    return cudaGetLastError();
}

}  // namespace gpfc
