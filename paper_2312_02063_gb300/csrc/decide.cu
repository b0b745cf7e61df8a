// decide.cu -- per-star decision over a periodogram of scores.
//
// For each star's scores (one per trial period): mean and population standard deviation
// of the finite scores; SDE = (max - mean) / sd (Eq. 3; 0 when sd is 0); peaks as in
// Sec. 4.2: maximal runs of consecutive periods scoring above mean + k_sigma sd that are
// at least min_width periods wide, each with its height (largest score, first occurrence);
// the best peak (highest, ties to the smaller index) and the highest max_peaks peaks,
// each flagged against the best peak's period for harmonics (Fig. 14 notes them): 1 for
// the best, +m if P = m Pb, -m if P = Pb / m (m = 2..4), else 0.
//
// A star is taken by one block of kPkThreads threads, or by a cluster of them that split its
// periods and meet through distributed shared memory. Statistics are FP64 sums in a fixed
// order. For the runs, thread t owns the runs that start in its contiguous chunk of periods and
// follows a run past the chunk's end until it closes; qualifying runs go to the candidate
// list of the cluster's first block (the first kPkCap of them; the best peak and the count are
// exact in any case). What bounds it: FP64 instructions (one per warp and scheduler every 64
// cycles), five a period; one block takes 0.60 ms for 250,000 periods, a cluster of sixteen 0.09 ms.
#include <cmath>
#include <cooperative_groups.h>
#include <cstdint>

#include "gpfc_common.cuh"
#include "gpfc_decide.h"

namespace gpfc {

constexpr int kPkThreads = 1024;
constexpr int kPkCap = 2048;

// Block reductions through one warp (every warp adding all partials would cost 32 FP64
// instructions a warp); the value is returned to all threads.
template <class T, class Op>
__device__ __forceinline__ T pk_block_reduce(T v, T *red, T zero, Op op)
{
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < kPkThreads / 32 ? red[lane] : zero;
        for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (lane == 0) red[0] = v;
    }
    __syncthreads();
    return red[0];
}
template <class T>
__device__ __forceinline__ T pk_block_sum(T v, T *red)
{
    return pk_block_reduce(v, red, (T)0, [](T a, T b) { return a + b; });
}
__device__ __forceinline__ unsigned long long pk_block_max(unsigned long long v, unsigned long long *red)
{
    return pk_block_reduce(v, red, 0ull, [](unsigned long long a, unsigned long long b) { return a > b ? a : b; });
}

__device__ __forceinline__ float key_value(unsigned long long key)
{
    const uint32_t ord = (uint32_t)(key >> 32);
    const uint32_t u = (ord & 0x80000000u) ? (ord & 0x7fffffffu) : ~ord;
    return __uint_as_float(u);
}
__device__ __forceinline__ int64_t key_index(unsigned long long key)
{
    return (int64_t)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull));
}

// C blocks (a cluster, or one block) per star at a time.
template <int C>
__global__ void __launch_bounds__(kPkThreads, 1) peaks_kernel(const PeakParams p)
{
    namespace cg = cooperative_groups;
    __shared__ double red_d[kPkThreads / 32];
    __shared__ float red_f[kPkThreads / 32];
    __shared__ int red_i[kPkThreads / 32];
    __shared__ unsigned long long red_k[kPkThreads / 32];
    __shared__ float c_h[kPkCap];
    __shared__ int c_i[kPkCap];
    __shared__ int c_w[kPkCap];
    __shared__ int c_n, c_peaks[C];  // candidates; qualifying runs and best key of each block
    __shared__ unsigned long long c_best[C];
    __shared__ double part_sum, part_ss;  // this block's partial sums, read by the cluster
    __shared__ int part_cnt;
    __shared__ float part_mx;
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = C > 1 ? (int)cluster.block_rank() : 0;
    auto meet = [&]() {
        if (C > 1) cluster.sync();
        else __syncthreads();
    };
    auto of = [&](auto *ptr, int r) { return C > 1 ? cluster.map_shared_rank(ptr, r) : ptr; };
    for (int s = blockIdx.x / C; s < p.nstars; s += gridDim.x / C) {
        const int64_t gb = p.grid_off ? p.grid_off[s] : 0, ge = p.grid_off ? p.grid_off[s + 1] : p.np;
        const float *sc = p.score + gb;
        const int64_t len = ge - gb;
        const int64_t lo = len * rank / C, hi = len * (rank + 1) / C;  // this block's periods
        if (threadIdx.x == 0) c_n = 0;
        // statistics of the finite scores
        double sum = 0.0;
        int cnt = 0;
        for (int64_t k = lo + threadIdx.x; k < hi; k += kPkThreads) {
            const float v = sc[k];
            if (isfinite(v)) {
                sum += (double)v;
                ++cnt;
            }
        }
        sum = pk_block_sum(sum, red_d);
        cnt = pk_block_sum(cnt, red_i);
        if (threadIdx.x == 0) {
            part_sum = sum;
            part_cnt = cnt;
        }
        meet();
        int ntot = 0;
        double tot = 0.0;
#pragma unroll 1
        for (int r = 0; r < C; ++r) {
            tot += *of(&part_sum, r);
            ntot += *of(&part_cnt, r);
        }
        const double mean = ntot > 0 ? tot / (double)ntot : NAN;
        double ss = 0.0;
        float mx = -INFINITY;
        for (int64_t k = lo + threadIdx.x; k < hi; k += kPkThreads) {
            const float v = sc[k];
            if (isfinite(v)) {
                const double d = (double)v - mean;
                ss += d * d;
                mx = fmaxf(mx, v);
            }
        }
        ss = pk_block_sum(ss, red_d);
        mx = pk_block_reduce(mx, red_f, -INFINITY, [](float a, float b) { return fmaxf(a, b); });
        if (threadIdx.x == 0) {
            part_ss = ss;
            part_mx = mx;
        }
        meet();
        ss = 0.0;
        mx = -INFINITY;
#pragma unroll 1
        for (int r = 0; r < C; ++r) {
            ss += *of(&part_ss, r);
            mx = fmaxf(mx, *of(&part_mx, r));
        }
        const double sd = ntot > 0 ? sqrt(ss / (double)ntot) : NAN;
        const double thr = mean + p.k_sigma * sd;
        // a float is above thr exactly if it is above the largest float not above thr
        const float thr_f = __double2float_rd(thr);
        auto above = [&](int64_t k) {
            const float v = sc[k];
            return isfinite(v) && v > thr_f;
        };
        // runs starting in this thread's chunk
        const int64_t chunk = (hi - lo + kPkThreads - 1) / kPkThreads;
        const int64_t a = lo + (int64_t)threadIdx.x * chunk, b = min(hi, a + chunk);
        int64_t i = a;
        if (i < b && i > 0 && above(i - 1))  // the run through a started in an earlier chunk
            while (i < len && above(i)) ++i;
        unsigned long long best = 0ull;
        int nq = 0;
        while (i < b) {
            if (!above(i)) {
                ++i;
                continue;
            }
            int64_t e = i, arg = i;
            while (e < len && above(e)) {
                if (sc[e] > sc[arg]) arg = e;
                ++e;
            }
            if (e - i >= p.min_width) {
                ++nq;
                const unsigned long long key = argmax_key(sc[arg], arg);
                best = key > best ? key : best;
                const int slot = atomicAdd(of(&c_n, 0), 1);
                if (slot < kPkCap) {
                    of(c_h, 0)[slot] = sc[arg];
                    of(c_i, 0)[slot] = (int)arg;
                    of(c_w, 0)[slot] = (int)(e - i);
                }
            }
            i = e;
        }
        nq = pk_block_sum(nq, red_i);
        best = pk_block_max(best, red_k);
        if (threadIdx.x == 0) {
            of(c_peaks, 0)[rank] = nq;
            of(c_best, 0)[rank] = best;
        }
        meet();  // every block's candidates are in the first one's list
        if (rank != 0) continue;  // (the next meeting is after the next star's first sums)
        int npk = 0;
        best = 0ull;
        for (int r = 0; r < C; ++r) {
            npk += c_peaks[r];
            best = c_best[r] > best ? c_best[r] : best;
        }
        const int ncand = min(c_n, kPkCap);
        // the highest max_peaks candidates, one block argmax each
        const int nlist = p.peaks ? min(p.max_peaks, ncand) : 0;
        for (int r = 0; r < nlist; ++r) {
            unsigned long long kbest = 0ull;
            int slot_best = -1;
            for (int q = threadIdx.x; q < ncand; q += kPkThreads) {
                if (c_w[q] < 0) continue;  // taken
                const unsigned long long key = argmax_key(c_h[q], c_i[q]);
                if (key > kbest) {
                    kbest = key;
                    slot_best = q;
                }
            }
            const unsigned long long kmax = pk_block_max(kbest, red_k);
            if (kbest == kmax && slot_best >= 0) {
                PeakDev &o = p.peaks[(size_t)s * p.max_peaks + r];
                o.index = c_i[slot_best];
                o.height = c_h[slot_best];
                o.width = c_w[slot_best];
                o.harmonic = 0;
                o.reserved = 0;
                c_w[slot_best] = -1;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            PeakSummaryDev &S = p.summary[s];
            S.mean = mean;
            S.sd = sd;
            S.sde = ntot > 0 ? (sd > 0.0 ? ((double)mx - mean) / sd : 0.0) : NAN;
            S.best_index = best ? key_index(best) : -1;
            S.best_score = best ? key_value(best) : NAN;
            S.n_peaks = npk;
            S.truncated = c_n > kPkCap ? 1 : 0;
            S.n_listed = nlist;
            if (p.peaks && nlist > 0) {
                const double Pb = p.periods[gb + p.peaks[(size_t)s * p.max_peaks].index];
                for (int r = 0; r < nlist; ++r) {
                    PeakDev &o = p.peaks[(size_t)s * p.max_peaks + r];
                    int h = 0;
                    if (r == 0) {
                        h = 1;
                    } else {
                        const double ratio = p.periods[gb + o.index] / Pb;
                        for (int m = 2; m <= 4 && h == 0; ++m) {
                            if (fabs(ratio - m) <= p.harm_tol * m) h = m;
                            else if (fabs(1.0 / ratio - m) <= p.harm_tol * m) h = -m;
                        }
                    }
                    o.harmonic = h;
                }
            }
        }
        __syncthreads();
    }
}

// Blocks per star: sixteen where the grids are long enough to give every thread of a cluster
// something (a cluster's meetings cost a few microseconds), else one. The GPU holds `clusters`
// of them at a time (a cluster keeps to one part of the chip); more stars take turns, and then a
// grid has to be longer by as much: 19 stars of 16,384 periods take 89 us in clusters and
// 46 us in a block each, 19 of 200,000 142 and 437 us.
constexpr int kPkCluster = 16;
constexpr int64_t kPkLong = 16384;

static cudaLaunchConfig_t pk_cluster_config(int nstars, cudaLaunchAttribute &at, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(nstars * kPkCluster));
    cfg.blockDim = dim3(kPkThreads);
    cfg.stream = st;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kPkCluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cfg;
}

int peaks_register()
{
    int n = 0;
    cudaError_t e = cudaFuncSetAttribute(peaks_kernel<kPkCluster>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) {
        cudaLaunchAttribute at{};
        const cudaLaunchConfig_t cfg = pk_cluster_config(1, at, nullptr);
        e = cudaOccupancyMaxActiveClusters(&n, peaks_kernel<kPkCluster>, &cfg);
    }
    if (e == cudaSuccess) return n;
    cudaGetLastError();
    return 0;
}

cudaError_t launch_peaks(const PeakParams &p, int num_sms, int clusters, cudaStream_t st)
{
    const int64_t turns = clusters > 0 ? (p.nstars + clusters - 1) / clusters : INT64_MAX / kPkLong;
    if (p.np / p.nstars >= kPkLong * turns) {
        cudaLaunchAttribute at{};
        const cudaLaunchConfig_t cfg = pk_cluster_config(p.nstars, at, st);
        return cudaLaunchKernelEx(&cfg, peaks_kernel<kPkCluster>, p);
    }
    const int grid = p.nstars < num_sms * 2 ? p.nstars : num_sms * 2;
    peaks_kernel<1><<<grid, kPkThreads, 0, st>>>(p);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ ROC

// Detection statistics of one detector over labelled scores (Sec. 3.2: ROC curves of stars
// scored by their best trial period). Every quantity is a count over pairs of scores, so it
// is exact and independent of the order of the atomics. A NaN score ranks below every
// number. Cost: n_neg^2 + n_pos * n_neg comparisons (10^8 for 10^4 of each).
constexpr int kRocThreads = 256;
constexpr int kRocTile = 2048;

__device__ __forceinline__ float roc_key(float v) { return v != v ? -INFINITY : v; }

__global__ void roc_init_kernel(RocParams p)
{
    const int t = threadIdx.x;
    if (t == 0) *p.u2 = 0ull;
    if (t < p.n_fpr) {
        p.tp[t] = 0ull;
        p.thr[t] = -INFINITY;  // the rule's value when k >= n_neg
    }
}

// thr[f] = the (k_f + 1)-th largest negative: negative j is it iff #{neg > neg_j} <= k_f <
// #{neg >= neg_j} (every such j holds the same value).
__global__ void __launch_bounds__(kRocThreads) roc_threshold_kernel(RocParams p)
{
    __shared__ float tile[kRocTile];
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const float v = j < p.n_neg ? roc_key(p.neg[j]) : 0.f;
    int64_t g = 0, e = 0;
    for (int64_t t0 = 0; t0 < p.n_neg; t0 += kRocTile) {
        const int nt = (int)min((int64_t)kRocTile, p.n_neg - t0);
        __syncthreads();
        for (int i = threadIdx.x; i < nt; i += blockDim.x) tile[i] = roc_key(p.neg[t0 + i]);
        __syncthreads();
        for (int i = 0; i < nt; ++i) {
            const float u = tile[i];
            g += u > v;
            e += u >= v;
        }
    }
    if (j < p.n_neg)
        for (int f = 0; f < p.n_fpr; ++f)
            if (g <= p.k[f] && p.k[f] < e) p.thr[f] = v;
}

__device__ __forceinline__ unsigned long long roc_block_sum(unsigned long long v, unsigned long long *red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    unsigned long long t = 0ull;
    if (threadIdx.x == 0)
        for (int w = 0; w < kRocThreads / 32; ++w) t += red[w];
    return t;
}

// u2 += 2 #{pos_i > neg_j} + #{pos_i == neg_j}; tp[f] += [pos_i > thr_f]
__global__ void __launch_bounds__(kRocThreads) roc_count_kernel(RocParams p)
{
    __shared__ float tile[kRocTile];
    __shared__ unsigned long long red[kRocThreads / 32];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = i < p.n_pos;
    const float v = live ? roc_key(p.pos[i]) : 0.f;
    unsigned long long c = 0ull;
    for (int64_t t0 = 0; t0 < p.n_neg; t0 += kRocTile) {
        const int nt = (int)min((int64_t)kRocTile, p.n_neg - t0);
        __syncthreads();
        for (int k = threadIdx.x; k < nt; k += blockDim.x) tile[k] = roc_key(p.neg[t0 + k]);
        __syncthreads();
        if (live)
            for (int k = 0; k < nt; ++k) {
                const float u = tile[k];
                c += (v > u ? 2ull : 0ull) + (v == u ? 1ull : 0ull);
            }
    }
    const unsigned long long s = roc_block_sum(c, red);
    if (threadIdx.x == 0 && s) atomicAdd(p.u2, s);
    for (int f = 0; f < p.n_fpr; ++f) {
        const unsigned long long d = roc_block_sum(live && v > p.thr[f] ? 1ull : 0ull, red);
        if (threadIdx.x == 0 && d) atomicAdd(&p.tp[f], d);
    }
}

cudaError_t launch_roc(const RocParams &p, int num_sms, cudaStream_t st)
{
    (void)num_sms;
    roc_init_kernel<<<1, 32, 0, st>>>(p);
    if (p.n_fpr > 0)
        roc_threshold_kernel<<<(int)((p.n_neg + kRocThreads - 1) / kRocThreads), kRocThreads, 0, st>>>(p);
    roc_count_kernel<<<(int)((p.n_pos + kRocThreads - 1) / kRocThreads), kRocThreads, 0, st>>>(p);
    return cudaGetLastError();
}

}  // namespace gpfc
