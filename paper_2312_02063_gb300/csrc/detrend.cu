// detrend.cu -- the pre-processing of Sec. 2.2 (Fig. 3) on the GPU: segmentation at time
// and flux gaps, a clipped least-squares cubic spline per segment with the knot spacing
// chosen by the Bayesian Information Criterion, division by the fit, and clipping of each
// segment's edges.
//
// Readings (the paper names the steps, not the spline or the criterion's form):
//  * a segment starts at sample i when t_i - t_{i-1} > time_gap or |f_i - f_{i-1}| >
//    flux_gap_sigma times the population standard deviation of the whole light curve;
//  * the spline is cubic with clamped end knots at the segment's first and last times and
//    interior knots at t0 + spacing j strictly inside; for each candidate spacing the fit
//    solves (B^T B + lambda D^T D) c = B^T f over the used points, D the second difference
//    of the coefficients and lambda = ridge trace(B^T B) / p, so a knot interval left
//    without points takes coefficients continued from its neighbours;
//  * clipping: residuals over the whole segment, sigma = RMS over the used points; the next
//    fit uses the unmasked points with |r| <= max(clip_sigma sigma, 1e-9 RMS(f)); repeat
//    until the used set repeats or max_iter fits have been made;
//  * the spacing with the smallest BIC = n ln(RSS / n) + p ln n wins (ties: the earlier);
//    a candidate with fewer used points than coefficients, or a normal matrix that is not
//    positive definite, is skipped;
//  * the output is f / spline for every point of a segment except its first and last
//    `edge` points (segments of 2 edge points or fewer are dropped), in time order.
//
// Layout: every per-point scratch array is indexed by the point's own index, and a
// segment's p <= n_s coefficients live at the indices of its own points, so segments
// never share scratch; each candidate spacing fitted at the same time has its own copy, 122 bytes a
// point (arrays whose lifetimes do not meet share it). Spacings go through in groups of as many
// copies as kDtScratch holds, one at least. Every reduction runs in a fixed order: the results do
// not depend on scheduling or grouping.
//
// What bounds it: FP64 instructions, one per warp and scheduler every 64 cycles whatever the
// number of active lanes, and the serial factorisation. So each (segment, spacing) is a block of
// its own (a full-length light curve has some hundred); the B-splines of a point, which do not
// change between the fits of one candidate, are evaluated once, with the reciprocal knot
// differences of an interval instead of six divisions a point; the normal equations are summed
// per knot interval, one thread for each of an interval's 14 sums; and the banded matrix is
// factored as L D L^T from both ends at once by two lanes, with a Newton reciprocal for each pivot
// (no square root, no division in the chain). 65,536 cadences with gaps, five spacings: 27.9 ms
// with one block per segment, bases evaluated again in each of up to ten fits and a Cholesky
// factorisation by one thread; now 1.33 ms.
#include <cmath>
#include <cstdint>

#include "gpfc_common.cuh"
#include "gpfc_detrend.h"

namespace gpfc {

constexpr int kDtThreads = 256;

// fixed-order block sum (warp shuffles, then the warp totals in order)
__device__ __forceinline__ double dt_block_sum(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < kDtThreads / 32; ++w) t += red[w];
    __syncthreads();
    return t;
}

__device__ __forceinline__ void dt_range(int64_t n, int64_t &i0, int64_t &i1)
{
    const int64_t per = (n + gridDim.x - 1) / gridDim.x;
    i0 = (int64_t)blockIdx.x * per;
    i1 = min(n, i0 + per);
    if (i0 > n) i0 = n;
}

// pass 1: per-block sums of f; pass 2: per-block sums of (f - mean)^2
__global__ void __launch_bounds__(kDtThreads) dt_moment_kernel(DetrendParams p, int pass)
{
    __shared__ double red[kDtThreads / 32];
    __shared__ double s_mean;
    if (pass == 2 && threadIdx.x == 0) {
        double tot = 0.0;
        for (int g = 0; g < (int)gridDim.x; ++g) tot += p.partial[g];
        s_mean = tot / (double)p.n;
    }
    __syncthreads();
    int64_t i0, i1;
    dt_range(p.n, i0, i1);
    double acc = 0.0;
    for (int64_t i = i0 + threadIdx.x; i < i1; i += kDtThreads) {
        const double v = (double)p.f[i];
        acc += pass == 1 ? v : (v - s_mean) * (v - s_mean);
    }
    const double t = dt_block_sum(acc, red);
    if (threadIdx.x == 0) p.partial[(pass - 1) * gridDim.x + blockIdx.x] = t;
}

__device__ __forceinline__ double dt_sigma(const DetrendParams &p, int G)
{
    double v = 0.0;
    for (int g = 0; g < G; ++g) v += p.partial[G + g];
    return sqrt(v / (double)p.n);
}

__device__ __forceinline__ bool dt_break(const DetrendParams &p, int64_t i, double fgap)
{
    if (i == 0) return true;
    return (p.t[i] - p.t[i - 1] > p.time_gap) || (fabs((double)p.f[i] - (double)p.f[i - 1]) > fgap);
}

// segment starts: pass 1 counts per block, pass 2 writes them in order
__global__ void __launch_bounds__(kDtThreads) dt_starts_kernel(DetrendParams p, int pass)
{
    __shared__ double s_fgap;
    __shared__ int64_t s_base;
    __shared__ int s_warp[kDtThreads / 32];
    if (threadIdx.x == 0) {
        s_fgap = p.flux_gap_sigma * dt_sigma(p, gridDim.x);
        s_base = pass == 2 ? p.blk_off[blockIdx.x] : 0;
    }
    __syncthreads();
    int64_t i0, i1;
    dt_range(p.n, i0, i1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t count = 0;
    for (int64_t c0 = i0; c0 < i1; c0 += kDtThreads) {
        const int64_t i = c0 + threadIdx.x;
        const bool br = i < i1 && dt_break(p, i, s_fgap);
        const unsigned m = __ballot_sync(0xffffffffu, br);
        if (lane == 0) s_warp[warp] = __popc(m);
        __syncthreads();
        int before = 0, tot = 0;
        for (int w = 0; w < kDtThreads / 32; ++w) {
            if (w < warp) before += s_warp[w];
            tot += s_warp[w];
        }
        if (pass == 2 && br) p.seg_start[s_base + count + before + __popc(m & ((1u << lane) - 1u))] = i;
        count += tot;
        __syncthreads();
    }
    if (pass == 1 && threadIdx.x == 0) p.blk_count[blockIdx.x] = count;
}

// exclusive scan over at most a few thousand block counts (one block, fixed order)
__global__ void dt_scan_kernel(const int64_t *cnt, int64_t ncnt, int64_t *off, int64_t *total)
{
    if (threadIdx.x != 0) return;
    int64_t s = 0;
    for (int64_t g = 0; g < ncnt; ++g) {
        off[g] = s;
        s += cnt[g];
    }
    off[ncnt] = s;
    if (total) *total = s;
}

__global__ void dt_close_starts_kernel(DetrendParams p)
{
    if (threadIdx.x == 0) p.seg_start[*p.n_seg] = p.n;
}

// knot j of the clamped cubic knot vector of a segment [t0, t1] with m interior knots
__device__ __forceinline__ double dt_knot(int j, double t0, double t1, double sp, int m)
{
    return j < 4 ? t0 : (j < 4 + m ? t0 + sp * (double)(j - 3) : t1);
}

// Interval j (0 <= j <= m: knots k_{3+j} <= t < k_{4+j}, the segment's last time in the last
// interval) holding t.
__device__ __forceinline__ int dt_interval(double t, double t0, double sp, double inv_sp, int m)
{
    int j = (int)floor((t - t0) * inv_sp);  // interior knots t0 + sp i <= t: i = 1 .. j
    if (j < 0) j = 0;
    if (j > m) j = m;
    while (j > 0 && t0 + sp * (double)j > t) --j;
    while (j < m && t0 + sp * (double)(j + 1) <= t) ++j;
    return j;
}

// Reciprocal of a positive d: an FP32 quotient and two Newton steps, each doubling the correct
// bits (24 -> 48 -> all but the last rounding).
__device__ __forceinline__ double dt_rcp(double d)
{
    if (!(d > 1e-30 && d < 1e30)) return 1.0 / d;
    double x = (double)(1.0f / (float)d);
    x = fma(fma(-d, x, 1.0), x, x);
    x = fma(fma(-d, x, 1.0), x, x);
    return x;
}

// BIC of the segment that starts at point a with the group's spacing c (infinite: skipped), in the
// place of its matrix, which is done with.
__device__ __forceinline__ double &dt_bic(const DetrendParams &p, int c, int64_t a)
{
    return p.band[8 * ((size_t)c * p.n + a)];
}

// One end's elimination state: the last three rows' pivots and multipliers.
// A row i of a symmetric band matrix (half width 3), left-looking: with the eliminated rows i - k,
//   c_k = g(i, i-k) - sum over eliminated columns left of it,  l_k = c_k / d_{i-k},
//   d = g(i, i) - sum l_k c_k,  z = r_i - sum l_k z_{i-k}.
struct BandState {
    double inv1, inv2, inv3;  // 1 / d of rows i-1, i-2, i-3
    double z1, z2, z3;
    double l11, l12;          // row i-1: l_1, l_2
    double l21;               // row i-2: l_1
    __device__ void clear() { inv1 = inv2 = inv3 = z1 = z2 = z3 = l11 = l12 = l21 = 0.0; }
    __device__ __forceinline__ void reduce(double g1, double g2, double g3, double &c1, double &c2, double &c3) const
    {
        c3 = g3;
        c2 = fma(-l21, c3, g2);
        c1 = fma(-l11, c2, fma(-l12, c3, g1));
    }
    __device__ __forceinline__ void push(double inv, double z, double l1, double l2)
    {
        inv3 = inv2;
        inv2 = inv1;
        inv1 = inv;
        z3 = z2;
        z2 = z1;
        z1 = z;
        l21 = l11;
        l11 = l1;
        l12 = l2;
    }
};

// Solve the banded normal equations (G[i][d] = entry (i, i + d), right side r) into x. Lanes 0
// and 1 of one warp eliminate h rows from either end at once (the same code on mirrored indices),
// lane 1 hands its reduction of the next three rows over, lane 0 eliminates the rows between, and
// both substitute back. L keeps each row's multipliers and reciprocal pivot. False if a pivot
// is not positive.
__device__ bool dt_solve(double *G, double *r, double *L, double *x, int n, int lane)
{
    const int h = n >= 12 ? (n - 6) / 2 : 0;
    const bool rev = lane == 1;
    // mirrored row i is row n - 1 - i; its entry with mirrored row i - k
    auto at = [&](int i) { return rev ? n - 1 - i : i; };
    auto gk = [&](int i, int k) { return i < k ? 0.0 : (rev ? G[4 * (n - 1 - i) + k] : G[4 * (i - k) + k]); };
    BandState S;
    S.clear();
    int ok = 1;
    auto row = [&](int i, double g0, double g1, double g2, double g3, double ri) {
        double c1, c2, c3;
        S.reduce(g1, g2, g3, c1, c2, c3);
        const double l1 = c1 * S.inv1, l2 = c2 * S.inv2, l3 = c3 * S.inv3;
        const double d = fma(-l1, c1, fma(-l2, c2, fma(-l3, c3, g0)));
        const double z = fma(-l1, S.z1, fma(-l2, S.z2, fma(-l3, S.z3, ri)));
        if (!(d > 0.0)) ok = 0;
        const double inv = dt_rcp(d);
        double *Li = L + 4 * at(i);
        Li[0] = inv;
        Li[1] = l1;
        Li[2] = l2;
        Li[3] = l3;
        x[at(i)] = z;
        S.push(inv, z, l1, l2);
    };
    const int mine = lane < 2 ? h : 0;
    double n0 = 0.0, n1 = 0.0, n2 = 0.0, n3 = 0.0, nr = 0.0;  // the next row, loaded ahead
    auto fetch = [&](int i) {
        n0 = G[4 * at(i)];
        n1 = gk(i, 1);
        n2 = gk(i, 2);
        n3 = gk(i, 3);
        nr = r[at(i)];
    };
    if (lane < 2) fetch(0);
    for (int i = 0; i < mine; ++i) {
        const double g0 = n0, g1 = n1, g2 = n2, g3 = n3, ri = nr;
        fetch(i + 1);  // (h <= n - 6: row h exists)
        row(i, g0, g1, g2, g3, ri);
    }
    if (lane == 1 && h > 0) {
        // rows h, h+1, h+2 less the eliminated ones' part
        double c1, c2, c3;
        const double i1 = S.inv1, i2 = S.inv2, i3 = S.inv3;
        S.reduce(gk(h, 1), gk(h, 2), gk(h, 3), c1, c2, c3);
        const double e2 = gk(h + 1, 3), e1 = fma(-S.l11, e2, gk(h + 1, 2));  // row h+1: columns h-2, h-1
        const double f1 = gk(h + 2, 3);                                      // row h+2: column h-1
        const int a0 = n - 1 - h, a1 = a0 - 1, a2 = a0 - 2;
        G[4 * a0] -= c1 * c1 * i1 + c2 * c2 * i2 + c3 * c3 * i3;
        G[4 * a1] -= e1 * e1 * i1 + e2 * e2 * i2;
        G[4 * a2] -= f1 * f1 * i1;
        G[4 * a1 + 1] -= e1 * c1 * i1 + e2 * c2 * i2;  // (a1, a0)
        G[4 * a2 + 2] -= f1 * c1 * i1;                 // (a2, a0)
        G[4 * a2 + 1] -= f1 * e1 * i1;                 // (a2, a1)
        r[a0] -= c1 * i1 * S.z1 + c2 * i2 * S.z2 + c3 * i3 * S.z3;
        r[a1] -= e1 * i1 * S.z1 + e2 * i2 * S.z2;
        r[a2] -= f1 * i1 * S.z1;
    }
    __syncwarp();
    if (lane == 0) {
        for (int i = h; i < n - h; ++i) {
            fetch(i);
            row(i, n0, n1, n2, n3, nr);
        }
    }
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) return false;
    if (lane == 0) {  // the rows between: x_i = z_i / d_i - sum l(i+k, i) x_{i+k}
        for (int i = n - h - 1; i >= h; --i) {
            double v = x[i] * L[4 * i];
            for (int k = 1; k <= 3 && i + k < n - h; ++k) v = fma(-L[4 * (i + k) + k], x[i + k], v);
            x[i] = v;
        }
    }
    __syncwarp();
    if (lane < 2 && h > 0) {
        // row h + k - 1's multipliers on the columns eliminated at this end: lane 0's are in L (its
        // elimination went on through them); lane 1's are formed again from the band
        double x1 = x[at(h)], x2 = x[at(h + 1)], x3 = x[at(h + 2)];
        double m11, m12, m13, m22, m23, m33;  // l(h, h-1..h-3), l(h+1, h-1..h-2), l(h+2, h-1)
        if (lane == 0) {
            m11 = L[4 * h + 1];
            m12 = L[4 * h + 2];
            m13 = L[4 * h + 3];
            m22 = L[4 * (h + 1) + 2];
            m23 = L[4 * (h + 1) + 3];
            m33 = L[4 * (h + 2) + 3];
        } else {
            double c1, c2, c3;
            S.reduce(gk(h, 1), gk(h, 2), gk(h, 3), c1, c2, c3);
            m11 = c1 * S.inv1;
            m12 = c2 * S.inv2;
            m13 = c3 * S.inv3;
            const double e2 = gk(h + 1, 3);
            m22 = fma(-S.l11, e2, gk(h + 1, 2)) * S.inv1;
            m23 = e2 * S.inv2;
            m33 = gk(h + 2, 3) * S.inv1;
        }
        // multipliers l(i+1, i), l(i+2, i), l(i+3, i) of the row being solved
        for (int i = h - 1; i >= 0; --i) {
            const double *Li = L + 4 * at(i);
            double k1, k2, k3;
            if (i == h - 1) k1 = m11, k2 = m22, k3 = m33;
            else if (i == h - 2) k1 = L[4 * at(i + 1) + 1], k2 = m12, k3 = m23;
            else if (i == h - 3) k1 = L[4 * at(i + 1) + 1], k2 = L[4 * at(i + 2) + 2], k3 = m13;
            else k1 = L[4 * at(i + 1) + 1], k2 = L[4 * at(i + 2) + 2], k3 = L[4 * at(i + 3) + 3];
            const double v = fma(-k1, x1, fma(-k2, x2, fma(-k3, x3, x[at(i)] * Li[0])));
            x[at(i)] = v;
            x3 = x2;
            x2 = x1;
            x1 = v;
        }
    }
    return true;
}

// Knot intervals whose sums a block holds at a time: enough for most segments (a quarter of a
// mission at half a day); longer ones go through in tiles, three intervals summed again for each.
constexpr int kDtRows = kDtThreads;

// The clipped fit of one segment with one knot spacing (of the group's): a block each.
__global__ void __launch_bounds__(kDtThreads) dt_fit_kernel(DetrendParams p)
{
    __shared__ double s_part[14 * (kDtRows + 3)];
    __shared__ double red[kDtThreads / 32];
    __shared__ int s_m, s_ok, s_changed, s_cnt[kDtThreads / 32];
    __shared__ double s_lambda;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t nseg = *p.n_seg;
    for (int64_t item = blockIdx.x; item < nseg * p.group; item += gridDim.x) {
        const int64_t s = item / p.group;
        const int c = (int)(item - s * p.group);
        const int64_t a = p.seg_start[s], b = p.seg_start[s + 1];
        const int ns = (int)(b - a);
        const size_t o = (size_t)c * p.n + a;  // this candidate's copy of the segment's scratch
        if (ns <= 2 * (int64_t)p.edge) {
            if (tid == 0) dt_bic(p, c, a) = INFINITY;
            continue;
        }
        const double *t = p.t + a;
        const float *f = p.f + a;
        double4 *N = p.basis + o;
        // the knot intervals' reciprocal differences (at most ns - 3 intervals of 6) are used up before
        // the matrix is formed, its factor before the fit is evaluated
        double *G = p.band + 8 * o, *LB = G + 4 * (size_t)ns, *iv = G, *trend = LB;
        double *rhs = p.rhs + o, *coef = p.coef + o;
        int32_t *iv_of = p.interval + o, *first = p.first + o + (int64_t)c;  // [intervals + 1] <= ns + 1
        uint8_t *used = p.used + o, *used2 = p.used2 + o;
        const double t0 = t[0], t1 = t[ns - 1];
        const double sp = p.sp[p.sp0 + c], inv_sp = 1.0 / sp;
        __syncthreads();  // every thread has left the previous item
        if (tid == 0) {
            // interior knots t0 + sp i < t1 (at most 2^30, and no more than make ns coefficients
            // and one: the candidate is skipped then anyway)
            const double q = fmin((t1 - t0) * inv_sp, (double)ns);
            int m = max(0, (int)q);
            while (m > 0 && !(t0 + sp * (double)m < t1)) --m;
            while (m < ns && t0 + sp * (double)(m + 1) < t1) ++m;
            s_m = m;
        }
        __syncthreads();
        const int m = s_m, np_ = m + 4;
        bool valid = np_ <= ns;  // else fewer points than coefficients
        double bic = INFINITY;
        if (valid) {
            // reciprocals of an interval's six knot differences, in the order dt_basis uses them
            for (int j = tid; j <= m; j += kDtThreads) {
                const int mu = 3 + j;
                int e = 0;
                for (int d = 1; d <= 3; ++d)
                    for (int q = 0; q < d; ++q, ++e) {
                        const double den = dt_knot(mu + q + 1, t0, t1, sp, m) - dt_knot(mu + 1 - d + q, t0, t1, sp, m);
                        iv[6 * j + e] = den != 0.0 ? 1.0 / den : 0.0;
                    }
            }
            // (filled for every interval, so that times out of order leave no index out of range)
            for (int q = tid; q <= m + 1; q += kDtThreads) first[q] = ns;
            __syncthreads();
            // each point's interval and its four nonzero cubic B-splines (de Boor's triangular
            // recursion); the first point of every interval
            for (int i = tid; i < ns; i += kDtThreads) {
                const double ti = t[i];
                const int j = dt_interval(ti, t0, sp, inv_sp, m);
                const int jp = i > 0 ? dt_interval(t[i - 1], t0, sp, inv_sp, m) : -1;
                for (int q = jp + 1; q <= j; ++q) first[q] = i;
                iv_of[i] = j;
                const double *w = iv + 6 * j;
                const int mu = 3 + j;
                double B[4], left[4], right[4];
                B[0] = 1.0;
                int e = 0;
#pragma unroll
                for (int d = 1; d <= 3; ++d) {
                    left[d] = ti - dt_knot(mu + 1 - d, t0, t1, sp, m);
                    right[d] = dt_knot(mu + d, t0, t1, sp, m) - ti;
                    double saved = 0.0;
#pragma unroll
                    for (int q = 0; q < d; ++q, ++e) {
                        const double temp = B[q] * w[e];
                        B[q] = fma(right[q + 1], temp, saved);
                        saved = left[d - q] * temp;
                    }
                    B[d] = saved;
                }
                N[i] = make_double4(B[0], B[1], B[2], B[3]);
                used[i] = p.mask ? (uint8_t)(p.mask[a + i] == 0) : 1;
            }
            __syncthreads();
            for (int it = 0; it < p.max_iter; ++it) {
                // used count
                int cu = 0;
                for (int i = tid; i < ns; i += kDtThreads) cu += used[i];
                cu = __reduce_add_sync(0xffffffffu, cu);
                if (lane == 0) s_cnt[warp] = cu;
                __syncthreads();
                int nused = 0;
                for (int w = 0; w < kDtThreads / 32; ++w) nused += s_cnt[w];
                if (nused < np_) {
                    valid = false;
                    break;
                }
                double tr = 0.0;
                for (int r0 = 0; r0 < np_; r0 += kDtRows) {
                    // an interval's sums over its used points: N_x N_y (x <= y) and N_x f
                    const int j0 = max(0, r0 - 3), j1 = min(m + 1, r0 + kDtRows);
                    for (int e = tid; e < 14 * (j1 - j0); e += kDtThreads) {
                        const int j = j0 + e / 14, k = e % 14;
                        const int i0 = first[j], i1 = first[j + 1];
                        const int x = k < 4 ? 0 : (k < 7 ? 1 : (k < 9 ? 2 : (k < 10 ? 3 : k - 10)));
                        const int y = k < 4 ? k : (k < 7 ? k - 3 : (k < 9 ? k - 5 : 3));
                        const double *Nd = reinterpret_cast<const double *>(N);
                        double acc = 0.0;
                        if (k < 10) {
                            for (int i = i0; i < i1; ++i)
                                if (used[i]) acc = fma(Nd[4 * (size_t)i + x], Nd[4 * (size_t)i + y], acc);
                        } else {
                            for (int i = i0; i < i1; ++i)
                                if (used[i]) acc = fma(Nd[4 * (size_t)i + x], (double)f[i], acc);
                        }
                        s_part[e] = acc;
                    }
                    __syncthreads();
                    // rows of the normal equations from the intervals they reach over (B_r is the q-th
                    // spline of interval r - q), and the trace
                    const int r = r0 + tid;
                    if (r < np_) {
                        double g[4] = {0.0, 0.0, 0.0, 0.0}, v = 0.0;
                        for (int q = 3; q >= 0; --q) {
                            const int j = r - q;
                            if (j < 0 || j > m) continue;
                            const double *w = s_part + 14 * (j - j0);
                            const int at = q == 0 ? 0 : (q == 1 ? 4 : (q == 2 ? 7 : 9));
                            for (int d = 0; q + d <= 3; ++d) g[d] += w[at + d];
                            v += w[10 + q];
                        }
                        for (int d = 0; d < 4; ++d) G[4 * (size_t)r + d] = g[d];
                        rhs[r] = v;
                        tr += g[0];
                    }
                    __syncthreads();  // the sums are read before the next rows' replace them
                }
                const double trace = dt_block_sum(tr, red);
                if (tid == 0) s_lambda = p.ridge * trace / (double)np_;
                __syncthreads();
                // + lambda D^T D: (D^T D)[j][j+d] = sum over rows r of D (coefficients r..r+2
                // weighted 1, -2, 1) of D[r][j] D[r][j+d]
                for (int j = tid; j < np_; j += kDtThreads) {
                    for (int d = 0; d <= 2; ++d) {
                        if (j + d >= np_) break;
                        int v = 0;
                        for (int r = j + d - 2; r <= j; ++r) {
                            if (r < 0 || r > np_ - 3) continue;
                            const int w1 = j - r == 1 ? -2 : 1, e = j + d - r, w2 = e == 1 ? -2 : 1;
                            v += w1 * w2;
                        }
                        G[4 * (size_t)j + d] += s_lambda * (double)v;
                    }
                }
                if (tid == 0) s_changed = 0;
                __syncthreads();
                if (warp == 0) {
                    const bool ok = dt_solve(G, rhs, LB, coef, np_, lane);
                    if (lane == 0) s_ok = ok;
                }
                __syncthreads();
                if (!s_ok) {
                    valid = false;
                    break;
                }
                // the fit at every point of the segment, residual statistics over the used ones
                double rr = 0.0, ff = 0.0;
                for (int i = tid; i < ns; i += kDtThreads) {
                    const double4 n4 = N[i];
                    const double *cf = coef + iv_of[i];
                    const double v = fma(cf[3], n4.w, fma(cf[2], n4.z, fma(cf[1], n4.y, cf[0] * n4.x)));
                    trend[i] = v;
                    if (used[i]) {
                        const double fi = (double)f[i], r = fi - v;
                        rr = fma(r, r, rr);
                        ff = fma(fi, fi, ff);
                    }
                }
                const double rss = dt_block_sum(rr, red);
                const double fss = dt_block_sum(ff, red);
                const double nu = (double)nused;
                const double thr = fmax(p.clip_sigma * sqrt(rss / nu), 1e-9 * sqrt(fss / nu));
                int ch = 0;
                for (int i = tid; i < ns; i += kDtThreads) {
                    const uint8_t free_ = p.mask ? (uint8_t)(p.mask[a + i] == 0) : 1;
                    const uint8_t nx = free_ && fabs((double)f[i] - trend[i]) <= thr;
                    used2[i] = nx;
                    ch |= nx != used[i];
                }
                if (ch) s_changed = 1;
                __syncthreads();
                if (!s_changed || it == p.max_iter - 1) {
                    bic = rss > 0.0 ? nu * log(rss / nu) + (double)np_ * log(nu) : -INFINITY;
                    break;  // the last fit's own point set is `used`
                }
                uint8_t *sw = used;  // (each thread goes on with the points it wrote)
                used = used2;
                used2 = sw;
                __syncthreads();
            }
        }
        if (tid == 0) dt_bic(p, c, a) = valid ? bic : INFINITY;
    }
}

// The spacing of each segment (of this group's and the best of the groups before, bic_in, or NULL)
// and the light curve over its fit: kDtParts blocks a segment.
constexpr int kDtParts = 8;
__global__ void __launch_bounds__(kDtThreads) dt_choose_kernel(DetrendParams p, const double *bic_in, double *bic_out)
{
    const int64_t nseg = *p.n_seg;
    for (int64_t item = blockIdx.x; item < nseg * kDtParts; item += gridDim.x) {
        const int64_t s = item / kDtParts;
        const int part = (int)(item - s * kDtParts);
        const int64_t a = p.seg_start[s], b = p.seg_start[s + 1], ns = b - a;
        int best = -1;
        double bic = bic_in ? bic_in[s] : INFINITY;
        for (int c = 0; c < p.group; ++c) {
            const double v = dt_bic(p, c, a);
            if (v < bic) {
                bic = v;
                best = c;
            }
        }
        const double *trend = p.band + 8 * ((size_t)max(best, 0) * p.n + a) + 4 * (size_t)ns;
        const int64_t i1 = ns * (part + 1) / kDtParts;
        if (best >= 0 || !bic_in)
            for (int64_t i = ns * part / kDtParts + threadIdx.x; i < i1; i += kDtThreads)
                p.det[a + i] = best >= 0 ? (float)((double)p.f[a + i] / trend[i]) : 0.f;
        if (part == 0 && threadIdx.x == 0) {
            if (bic_out) bic_out[s] = bic;
            p.seg_keep[s] = bic < INFINITY ? ns - 2 * (int64_t)p.edge : 0;
        }
    }
}

// kept counts -> output offsets and the output length (one thread, fixed order)
__global__ void dt_offsets_kernel(DetrendParams p)
{
    if (threadIdx.x != 0) return;
    const int64_t nseg = *p.n_seg;
    int64_t o = 0;
    for (int64_t s = 0; s < nseg; ++s) {
        p.seg_off[s] = o;
        o += p.seg_keep[s];
    }
    *p.n_out = o;
}

__global__ void dt_write_kernel(DetrendParams p)
{
    const int64_t nseg = *p.n_seg;
    for (int64_t s = blockIdx.x; s < nseg; s += gridDim.x) {
        const int64_t keep = p.seg_keep[s];
        if (keep == 0) continue;
        const int64_t a = p.seg_start[s] + p.edge, o = p.seg_off[s];
        for (int64_t k = threadIdx.x; k < keep; k += blockDim.x) {
            p.t_out[o + k] = p.t[a + k];
            p.f_out[o + k] = p.det[a + k];
            if (p.seg_out) p.seg_out[o + k] = (int32_t)s;
        }
    }
}

cudaError_t launch_detrend(const DetrendParams &p, int num_sms, cudaStream_t st)
{
    const int G = p.blocks;
    dt_moment_kernel<<<G, kDtThreads, 0, st>>>(p, 1);
    dt_moment_kernel<<<G, kDtThreads, 0, st>>>(p, 2);
    dt_starts_kernel<<<G, kDtThreads, 0, st>>>(p, 1);
    dt_scan_kernel<<<1, 32, 0, st>>>(p.blk_count, G, p.blk_off, p.n_seg);
    dt_starts_kernel<<<G, kDtThreads, 0, st>>>(p, 2);
    dt_close_starts_kernel<<<1, 32, 0, st>>>(p);
    for (int c = 0, turn = 0; c < p.n_sp; c += p.group, ++turn) {
        DetrendParams q = p;
        q.sp0 = c;
        q.group = p.n_sp - c < p.group ? p.n_sp - c : p.group;
        dt_fit_kernel<<<num_sms * 4, kDtThreads, 0, st>>>(q);
        dt_choose_kernel<<<num_sms * 4, kDtThreads, 0, st>>>(q, c > 0 ? p.best[turn & 1] : nullptr,
                                                             p.best[(turn + 1) & 1]);
    }
    dt_offsets_kernel<<<1, 32, 0, st>>>(p);
    dt_write_kernel<<<num_sms * 2, kDtThreads, 0, st>>>(p);
    return cudaGetLastError();
}

}  // namespace gpfc
