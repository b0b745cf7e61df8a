// fold_pack.cu -- the equal-width fold with one shared-memory reduction per update (sm_103a).
//
// Same results, bit for bit, as the reduction layout of fold.cu (kLayoutRed32): the flux in
// the same per-star fixed point, exact integer sums and counts, one rounding per bin. There an
// update is two 32-bit reductions (sum row, count row); here sum and count share one word:
//
//     word += 2^S + (xq + L),        |xq| <= L = floor((2^31 - 1) / min(chunk, n)),
//
// so a bin of c samples holds c 2^S + y with 0 <= y <= 2 L c. A group's words are emptied after
// a segment of tiles into L2: as they are, into a slot of the block's workspace (decoded and
// added up in the epilogue), where a star has at most four segments; else into 64-bit totals.
// A segment counts only if its words prove themselves: with c' and y' read from the stored word (mod 2^32),
//     every c' <= M, M the largest count with 2 L M < 2^S, and  sum of c' = samples folded.
// Then nothing wrapped (the sums of the true and the stored words differ by a multiple of 2^32
// and by less than 2^32, as 2 L n < 2^32 for a segment of n <= chunk samples), y <= 2 L c <=
// 2 L c' < 2^S, and so c' and y' are the true count and sum. A group that fails (a period so
// close to a multiple of the cadence that its samples pile up in a few bins) needs only its counts
// again: its words hold the sum of xq + c (2^S + L) mod 2^32, and |sum of xq| < 2^31 up to a chunk of
// samples. So its words are put aside, the segment's samples counted plainly, and both give the
// sum; from there on the group takes shorter segments, and in the end none: a blind group's words are
// put aside at the end of the star (or chunk) and its samples counted in a second turn of the tiles, all
// blind groups at once. A group predicted to fail starts with shorter segments, or blind. So a block
// folds no sample more than twice (plus one failed segment a group), and the groups that pass do so as
// ever.
//
// Below 256 bins, where the flux is not cut to the chunk's fixed point (layouts 1 and 2 sum FP32),
// the same scheme takes 31-bit flux (HILO): xq = hi 2^15 + lo, the word holds the count and the
// sum of lo, and a second word of the bin's record, 128 bytes on, the sum of hi. Sums are exact
// in units of 2^-30 max|x|, rounded once.
//
// Half the words also means half the shared memory: six groups of 32 periods share each
// sample read from the tile instead of three. A block is 16 warps; each takes every 16th
// 16-sample group of a tile and adds it to the bins of all period groups (lane l: period l of
// each), as in fold.cu.
//
// What bounds it: the integer multiplies of the phase (mad.hi 4.3 and mad.lo 2.0 cycles per
// warp instruction and scheduler; a reduction 4.0) and the moves the compiler puts on their
// pipe. A launch lasts as long as its slowest block. 30,000 periods of 65,000 samples into 256 bins,
// two words / one word, by where the periods lie: 0.5 to 100 days 1.14 / 0.75 ms, 0.2 to 1 day
// (the usual multiples of the cadence) 1.14 / 0.87, all within 10^-4 of 3, 7, 10 or 12.5 cadences
// 1.14 / 0.75..0.81 (2.4 where a failed tile was folded twice more).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "gpfc_common.cuh"
#include "gpfc_kernels.h"

namespace gpfc {

namespace {

constexpr int kPackWarps = 16;
constexpr int kPackThreads = 32 * kPackWarps;
constexpr int kPackTile = kMaxTile;        // 2048 samples
constexpr uint32_t kSlab = 65536;          // 256 bins: two period groups, 256-byte rows
constexpr uint32_t kSlabPhase = 0x9000;    // slabs start at this offset from a multiple of 64 KB
constexpr uint32_t kHdrBytes = 128 + 4 * kPackTile * 4 + 2 * (kPackTile / 16) * 4 + kPackMaxGroups * 32 * 4;

struct PackShared {
    uint64_t bars[2];
    int abort;
    uint32_t risk;    // predictor: OR over the block's periods, four bits a group
    uint32_t bad[2];  // groups that failed a check (of this and the next boundary, in turn)
    int blind_from[8];  // first tile that a blind group's words hold
    int pad[16];
};
static_assert(sizeof(PackShared) == 128, "header layout");

// Address of the records: 256 bins: the first address past the header that lies kSlabPhase past
// a multiple of 64 KB (below); else 128-byte aligned.
__host__ __device__ inline uint32_t pack_records_addr(uint32_t base, int nbins)
{
    const uint32_t end = base + kHdrBytes;
    if (nbins != 256) return (end + 127u) & ~127u;
    return ((end + (kSlab - kSlabPhase) + kSlab - 1u) & ~(kSlab - 1u)) - (kSlab - kSlabPhase);
}

__host__ __device__ inline uint32_t pack_records_bytes(int nbins, int groups)
{
    if (nbins < 256) return (uint32_t)groups * (uint32_t)nbins * 256u;
    return nbins == 256 ? (uint32_t)((groups + 1) / 2) * kSlab : (uint32_t)groups * (uint32_t)nbins * 128u;
}

// hi word of the 64-bit phase: umulhi(tl, Fl) + th Fl + tl Fh
__device__ __forceinline__ uint32_t phase_hi(uint32_t tl, uint32_t thF, uint32_t Fl, uint32_t Fh)
{
    uint32_t h;
    asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(h) : "r"(tl), "r"(Fl), "r"(tl * Fh + thF));
    return h;
}

// Shared address of a sample's bin word for one period (KIND 0: 256 bins, 1: a larger power of two;
// 2 and 3: below 256 bins, HILO, a power of two or any). With 256 bins the bin is the top
// byte of the phase and rows are 256 bytes, so one byte permutation builds the address: byte 0 =
// lane and group parity, byte 1 = bin, the rest the slab; the slab's distance from a multiple of
// 64 KB is the reduction's immediate offset.
template <int KIND>
__device__ __forceinline__ uint32_t word_addr(uint32_t hi, uint32_t tl, uint32_t Fl, uint32_t base, uint32_t nbins,
                                              int shift)
{
    if (KIND == 0) return __byte_perm(hi, base, 0x7634);
    if (KIND == 1) return base + ((hi >> shift) << 7);
    if (KIND == 2) return base + ((hi >> shift) << 8);
    const uint32_t lo = tl * Fl;
    const unsigned long long t = (unsigned long long)hi * nbins + (unsigned long long)__umulhi(lo, nbins);
    return base + ((uint32_t)(t >> 32) << 8);
}

template <int KIND>
__device__ __forceinline__ void word_add(uint32_t a, uint32_t v)
{
    if (KIND == 0) asm volatile("red.shared.add.u32 [%0+%2], %1;" ::"r"(a), "r"(v), "n"(kSlabPhase) : "memory");
    else asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

constexpr int kEpi = 8;  // bins of a row that the epilogue finishes at a time

__device__ __forceinline__ void st_row8(void *dst, const uint32_t *v)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                 "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

// A sample's increments: x as it is, or (HILO) a count and lo, and hi in the second word.
constexpr int kLoBits = 15;
template <int KIND>
__device__ __forceinline__ void sample_add(uint32_t a, uint32_t x, uint32_t one)
{
    if (KIND >= 2) {
        asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(a), "r"((x & ((1u << kLoBits) - 1u)) + one) : "memory");
        asm volatile("red.shared.add.u32 [%0+128], %1;" ::"r"(a), "r"((uint32_t)((int32_t)x >> kLoBits)) : "memory");
    } else {
        word_add<KIND>(a, x);
    }
}

struct PackHalf {
    uint4 a[2];  // tau low words of eight samples
    uint4 x[2];  // the packed increments, made by the prep pass
};

// samples 8 i .. 8 i + 7 of a tile
__device__ __forceinline__ void load_pack_half(uint32_t stl, uint32_t sxq, int i, PackHalf &H)
{
    const uint32_t o = 32u * (uint32_t)i;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        H.a[q] = lds_u32x4(stl + o + 16u * q);
        H.x[q] = lds_u32x4(sxq + o + 16u * q);
    }
}

}  // namespace

// Predictor of piled-up bins for a regular cadence: when the phase moves by r per cadence,
// samples k apart differ by k r mod 1; let that be d bins. The samples of one residue mod k
// then put min(seg / k, 1 / d) of a segment of seg samples into a bin they cross, and
// floor((k + seg d) / nbins) + 1 residues cross one. A group's segment length is at risk when a k up to
// seg's own reach passes 0.95 M that way. Only a guess (gaps, other cadences), and made only where at
// least half the steps are about the smallest one; the check after the segment decides.
constexpr int kPackLevels = 4;  // a group's segments: the block's (about 8 tiles), 4, 2 and 1 tiles, or
constexpr uint32_t kBlind = 31u;  // none: counted once more afterwards
constexpr int kPackSegTiles = 8;

template <int KIND, int G>
__global__ void __launch_bounds__(kPackThreads, 1) fold_pack_kernel(const FoldParams p)
{
    extern __shared__ __align__(128) uint8_t smem[];
    PackShared &sh = *reinterpret_cast<PackShared *>(smem);
    uint32_t *tl_buf = reinterpret_cast<uint32_t *>(smem + 128);
    uint32_t *xq_buf = tl_buf + 2 * kPackTile;
    uint32_t *thg_buf = xq_buf + 2 * kPackTile;
    uint32_t *cnt_sum = thg_buf + 2 * (kPackTile / 16);  // [G][32] counts of a segment
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nbins = p.nbins;
    constexpr int ppc = 32 * G;  // G = p.warps period groups
    if (KIND >= 2 && p.when == 1 && p.stats[0].wide) return;  // (the FP32 fold's)
    const uint32_t base = smem_u32(smem);
    const uint32_t rec = pack_records_addr(base, nbins);
    const uint32_t rec_bytes = pack_records_bytes(nbins, G);
    uint32_t dyn;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
    if (rec + rec_bytes > base + dyn) {  // (the launch sized the block for the device's window)
        report_error(p.status, kErrTimeout);
        return;
    }
    // row stride of a bin and start of period group j's words (lane's own)
    constexpr bool HILO = KIND >= 2;
    constexpr uint32_t row = KIND == 0 || HILO ? 256u : 128u;
    auto group_rec = [&](int j) {
        return (KIND == 0 ? rec + (uint32_t)(j >> 1) * kSlab + (uint32_t)(j & 1) * 128u
                          : rec + (uint32_t)j * (uint32_t)nbins * row) + 4u * (uint32_t)lane;
    };
    if (threadIdx.x == 0) {
        mbar_init(&sh.bars[0], 1);
        mbar_init(&sh.bars[1], 1);
        fence_mbar_init();
        sh.abort = 0;
    }
    __syncthreads();
    uint32_t consumed = 0u, issued = 0u;  // tiles, over the block's life (buffer = low bit)
    // this warp's share of the bins in flushes and epilogues, in eights where it can be
    int blo = warp * nbins / kPackWarps, bhi = (warp + 1) * nbins / kPackWarps;
    if ((nbins & 7) == 0) {
        blo = warp * (nbins / 8) / kPackWarps * 8;
        bhi = (warp + 1) * (nbins / 8) / kPackWarps * 8;
    }
    const bool vec_out = (nbins & 7) == 0 &&
                         ((reinterpret_cast<uintptr_t>(p.folded) | reinterpret_cast<uintptr_t>(p.sums) |
                           reinterpret_cast<uintptr_t>(p.counts)) & 31) == 0;
    // this block's workspace in L2, planes of [bin][32 G] words: two of 64-bit totals (count 2^40 +
    // biased sum up to 2^23 samples, else an int64 sum and, in the third plane, 32-bit counts),
    // then the slots, then one for words put aside
    const size_t plane = (size_t)nbins * ppc;
    constexpr int kPlanes = HILO ? kPackPlanesHilo : kPackPlanes;
    uint32_t *ws = reinterpret_cast<uint32_t *>(p.ws_sc) + (size_t)blockIdx.x * kPlanes * plane + lane;
    unsigned long long *ws_tot = reinterpret_cast<unsigned long long *>(ws - lane) + lane;
    uint32_t *ws_cnt = ws + 2 * plane, *ws_slot = ws + 3 * plane;
    uint32_t *ws_raw = ws + (size_t)(kPlanes - 1) * plane;  // words put aside

    int64_t task_end = p.ntasks;
    if (p.ntasks_dev) {
        const int64_t t = *p.ntasks_dev;
        task_end = t < task_end ? t : task_end;
    }
    for (int64_t task = p.task_begin + blockIdx.x; task < task_end; task += gridDim.x) {
        // the star of this task
        int s = 0;
        int64_t tbase = 0;
        if (p.task_off) {
            int lo = 0, hi = p.nstars - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (p.task_off[mid] <= task) lo = mid;
                else hi = mid - 1;
            }
            s = lo;
            tbase = p.task_off[s];
        }
        const int64_t lb = p.lc_off ? p.lc_off[s] : 0, le = p.lc_off ? p.lc_off[s + 1] : p.n;
        const int64_t gb = p.grid_off ? p.grid_off[s] : 0, ge = p.grid_off ? p.grid_off[s + 1] : p.np;
        // (more than 2^24 samples happens only for offsets the batch plan rejected)
        const int64_t nsamp = min(le - lb, (int64_t)1 << 24);
        const int64_t sbase = 256 * ((lb + 255) / 256 + s);
        const int64_t k0 = gb + (task - tbase) * ppc + lane;  // this lane's period of group 0
        // frequencies: warp j divides for period group j (FP64 division is slow: once per period,
        // not once per warp), through the words' memory
        uint2 *freq = reinterpret_cast<uint2 *>(smem + (rec - base));
        if (warp < G) {
            const int64_t k = k0 + 32 * warp;
            uint2 f = make_uint2(0u, 0xffffffffu);  // (no valid frequency reaches 2^63)
            if (k < ge) {
                const double P = p.periods[k];
                const double q = 1099511627776.0 / P;
                if (P > 0.0 && P < INFINITY && q < 9223372036854775808.0) {
                    const unsigned long long F = (unsigned long long)__double2ll_rn(q);
                    f = make_uint2((uint32_t)F, (uint32_t)(F >> 32));
                } else {
                    report_error(p.status, kErrRange);
                }
            }
            freq[threadIdx.x] = f;
        }
        __syncthreads();
        uint32_t Fl[G], Fh[G];
        uint32_t live = 0u;  // groups whose period of this lane is valid
#pragma unroll
        for (int j = 0; j < G; ++j) {
            Fl[j] = Fh[j] = 0u;
            const uint2 f = freq[32 * j + lane];
            if (f.y != 0xffffffffu) {
                Fl[j] = f.x;
                Fh[j] = f.y;
                live |= 1u << j;
            }
        }
        __syncthreads();
        // (HILO: lo < 2^15 whatever the star)
        const PackWord pw = HILO ? PackWord{0u, 256u, 23} : pack_word(nsamp, p.chunk);
        const bool wide = HILO || nsamp > ((int64_t)1 << 23);
        const unsigned long long bias = (1ull << 40) + pw.L;  // per count in a 64-bit total
        constexpr int tile = kPackTile;
        const int ntiles = (int)((nsamp + tile - 1) / tile);
        // (the plain sum of a blind group's samples fits 32 bits up to a chunk)
        const int span_tiles = nsamp <= (int64_t)p.chunk ? ntiles : p.chunk / tile;
        // The block's segments: of seg_tiles tiles, about kPackSegTiles but no more than a mean load of
        // about half M allows; into slots where a star of one chunk has at most kPackSegs of them.
        const int most = max(1, (int)fminf(0.55f * (float)pw.M * (float)nbins / (float)tile, 1e6f));
        int nsegs = max(1, (ntiles + kPackSegTiles - 1) / kPackSegTiles);
        if (nsegs > kPackSegs && nsamp <= (int64_t)p.chunk) nsegs = kPackSegs;
        nsegs = max(nsegs, (ntiles + most - 1) / most);
        const bool slots = nsamp <= (int64_t)p.chunk && nsegs <= kPackSegs;
        const int seg_tiles = max(1, (ntiles + nsegs - 1) / nsegs);

        // ---- each group's segment length: the longest whose predicted load stays below M
        if (threadIdx.x == 0) sh.risk = sh.bad[0] = sh.bad[1] = 0u;
        if (threadIdx.x < kPackMaxGroups * 32) cnt_sum[threadIdx.x] = 0u;
        for (uint32_t a = 16u * threadIdx.x; a < rec_bytes; a += 16u * kPackThreads)
            asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(rec + a), "r"(0u) : "memory");
        __syncthreads();
        {
            uint32_t risk = 0u;
            float seg[kPackLevels], top = 0.f;  // the longest length not ruled out
            int kmax[kPackLevels], kall = 0;
            const float lim = 0.95f * (float)pw.M, rbins = 1.f / (float)nbins;
#pragma unroll
            for (int v = 0; v < kPackLevels; ++v) {
                seg[v] = fminf((float)nsamp, (float)((v == 0 ? seg_tiles : min(seg_tiles, 8 >> v)) * tile));
                kmax[v] = 0;
                if (seg[v] * rbins > 0.8f * lim || lim < 4.f) risk |= 0x02108421u << v;  // (so lim > seg rbins below)
                else kmax[v] = (int)fminf(2.f * seg[v] / lim, 1024.f) + 1;
                kall = max(kall, kmax[v]);
                if (kmax[v] > 0) top = fmaxf(top, seg[v]);
            }
            // (of times without a regular cadence it would say nothing)
            const long long d0 = 2 * (int64_t)p.stats[s].nreg >= nsamp ? p.stats[s].dtau0 : 0;
#pragma unroll
            for (int j = 0; j < G; ++j) {
                if (((live >> j) & 1u) && d0 > 0) {
                    const unsigned long long F = ((unsigned long long)Fh[j] << 32) | Fl[j];
                    const uint32_t r = (uint32_t)(((unsigned long long)d0 * F) >> 32);
                    // the warps share the distances out
                    for (int k = 1 + warp; k <= kall; k += kPackWarps) {
                        const uint32_t ph = r * (uint32_t)k;
                        const float d = fmaxf((float)min(ph, 0u - ph) * (2.3283064365386963e-10f * (float)nbins), 1e-6f);
                        // (no level can be at risk beyond this distance: the longest, with 1 / d and
                        // without the rounding down)
                        if (d * (lim - top * rbins) > (float)k * rbins + 1.f) continue;
                        const float kr = __fdividef(1.f, (float)k), dr = __fdividef(1.f, d);
#pragma unroll
                        for (int v = 0; v < kPackLevels; ++v) {
                            const float res = __fadd_rd(fmaf(seg[v], d, (float)k) * rbins, 8388608.f) - 8388607.f;
                            if (k <= kmax[v] && fminf(seg[v] * kr, dr) * res > lim) risk |= 1u << (5 * j + v);
                        }
                    }
                }
            }
            risk = __reduce_or_sync(0xffffffffu, risk);
            if (lane == 0 && risk) atomicOr(&sh.risk, risk);
        }
        __syncthreads();
        // five bits a group: 0 (the block's segments), 4, 2 or 1 tiles, or blind
        uint32_t own = 0u;
#pragma unroll
        for (int j = 0; j < G; ++j) {
            const uint32_t risk = (sh.risk >> (5 * j)) & 15u;
            own |= (!(risk & 1u) ? 0u : (!(risk & 2u) ? 4u : (!(risk & 4u) ? 2u : (!(risk & 8u) ? 1u : kBlind)))) << (5 * j);
        }
        if (threadIdx.x < 8) sh.blind_from[threadIdx.x] = 0;
        auto len_of = [&](int j) { return (own >> (5 * j)) & 31u; };

        // each group's part of the address, kept in a register (formed again for every group of
        // samples it costs moves on the multiplies' pipe: 0.578 -> 0.555 ms for 152 blocks)
        uint32_t gaddr[G];
#pragma unroll
        for (int j = 0; j < G; ++j) {
            gaddr[j] = group_rec(j) - (KIND == 0 ? kSlabPhase : 0u);
            asm volatile("" : "+r"(gaddr[j]));
        }

        auto push = [&](int t) {
            if (threadIdx.x == 0) {
                const uint32_t b = issued & 1u;
                const int64_t i0 = (int64_t)t * tile;
                const int nv = (int)min((int64_t)tile, nsamp - i0);
                const uint32_t bytes = (uint32_t)(((nv + 3) & ~3) * 4);
                const uint32_t gbytes = (uint32_t)((((nv + 15) >> 4) * 4 + 15) & ~15);
                mbar_arrive_expect_tx(&sh.bars[b], 2u * bytes + gbytes);
                bulk_g2s(tl_buf + b * kPackTile, p.smp.tau_lo + sbase + i0, bytes, &sh.bars[b]);
                bulk_g2s(xq_buf + b * kPackTile, p.smp.xq + sbase + i0, bytes, &sh.bars[b]);
                bulk_g2s(thg_buf + b * (kPackTile / 16), p.smp.thg + (sbase + i0) / 16, gbytes, &sh.bars[b]);
            }
            ++issued;
        };

        // Every sample of tile t into the bins of all groups; or (count) a plain 1 into those of the
        // groups in mask. False (all threads) when a wait gave up.
        auto fold_tile = [&](int t, auto count, uint32_t mask) -> bool {
            constexpr bool COUNT = decltype(count)::value;
            const uint32_t b = consumed & 1u;
            const bool ok = mbar_wait_bounded(&sh.bars[b], (consumed >> 1) & 1u);
            ++consumed;
            if (!ok) {
                sh.abort = 1;
                report_error(p.status, kErrTimeout);
            } else {
                const int nv = (int)min((int64_t)tile, nsamp - (int64_t)t * tile);
                const int ng = nv >> 4;
                const uint32_t stl = smem_u32(tl_buf + b * kPackTile), sxq = smem_u32(xq_buf + b * kPackTile);
                const uint32_t sthg = smem_u32(thg_buf + b * (kPackTile / 16));
                const int32_t *gth = p.smp.tau_hi + sbase + (int64_t)t * tile;
                // one sample into every period group (mixed groups, tails)
                auto one = [&](int i, uint32_t th) {
                    const uint32_t tl = lds_u32(stl + 4u * i);
                    const uint32_t x = lds_u32(sxq + 4u * i);
#pragma unroll
                    for (int j = 0; j < G; ++j) {
                        if (COUNT && !((mask >> j) & 1u)) continue;
                        const uint32_t w = word_addr<KIND>(phase_hi(tl, th * Fl[j], Fl[j], Fh[j]), tl, Fl[j], gaddr[j],
                                                           (uint32_t)nbins, p.shift);
                        if (COUNT) word_add<KIND>(w, 1u);
                        else sample_add<KIND>(w, x, 1u << pw.S);
                    }
                };
                // a group whose samples differ in their high word (every ~256 days, or
                // unsorted times) reads each one's
                auto slow = [&](int g) {
#pragma unroll 2
                    for (int u = 0; u < 16; ++u) one(16 * g + u, (uint32_t)__ldg(gth + 16 * g + u));
                };
                {
                    // A 16-sample group into every period group as two halves, each loaded while
                    // the other is folded: eight samples at a time leave the registers that
                    // sixteen do not (those cost moves on the multiplies' own pipe).
                    auto half = [&](const PackHalf &H, uint32_t th) {
#pragma unroll
                        for (int j = 0; j < G; ++j) {
                            if (COUNT && !((mask >> j) & 1u)) continue;
                            const uint32_t thF = th * Fl[j];
                            uint32_t ad[8];
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const uint32_t tt[4] = {H.a[q].x, H.a[q].y, H.a[q].z, H.a[q].w};
#pragma unroll
                                for (int u = 0; u < 4; ++u)
                                    ad[4 * q + u] = word_addr<KIND>(phase_hi(tt[u], thF, Fl[j], Fh[j]), tt[u],
                                                                    Fl[j], gaddr[j], (uint32_t)nbins, p.shift);
                            }
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const uint32_t xx[4] = {H.x[q].x, H.x[q].y, H.x[q].z, H.x[q].w};
#pragma unroll
                                for (int u = 0; u < 4; ++u) {
                                    if (COUNT) word_add<KIND>(ad[4 * q + u], 1u);
                                    else sample_add<KIND>(ad[4 * q + u], xx[u], 1u << pw.S);
                                }
                            }
                        }
                    };
                    if (warp < ng) {
                        PackHalf A, B;
                        load_pack_half(stl, sxq, 2 * warp, A);
                        uint32_t th = lds_u32(sthg + 4u * (uint32_t)warp);
#pragma unroll 1
                        for (int g = warp; g < ng; g += kPackWarps) {
                            const int gn = min(g + kPackWarps, ng - 1);  // (past the end: loaded, not used)
                            load_pack_half(stl, sxq, 2 * g + 1, B);
                            const uint32_t thn = lds_u32(sthg + 4u * (uint32_t)gn);
                            if (__any_sync(0xffffffffu, th == 0x80000000u)) {  // (one value for the warp)
                                slow(g);
                                load_pack_half(stl, sxq, 2 * gn, A);
                            } else {
                                half(A, th);
                                load_pack_half(stl, sxq, 2 * gn, A);
                                half(B, th);
                            }
                            th = thn;
                        }
                    }
                }
                if (16 * ng + warp < nv) one(16 * ng + warp, (uint32_t)__ldg(gth + 16 * ng + warp));
            }
            __syncthreads();  // the tile is read and every reduction of it issued by all warps
            if (*reinterpret_cast<volatile int *>(&sh.abort)) {
                // let this block's copies in flight land before it leaves
                if (threadIdx.x == 0) {
                    if (!ok) mbar_wait_bounded(&sh.bars[b], ((consumed - 1u) >> 1) & 1u);
                    for (; consumed != issued; ++consumed)
                        mbar_wait_bounded(&sh.bars[consumed & 1u], (consumed >> 1) & 1u);
                }
                return false;
            }
            return true;
        };

        // The word (and HILO's second) of a segment that passed its check: sum of xq and count.
        using Sum = typename std::conditional<HILO, long long, int32_t>::type;
        const uint32_t ymask = (1u << pw.S) - 1u;
        auto decode = [&](uint32_t w, uint32_t w2, Sum &ds, uint32_t &dc) {
            dc = w >> pw.S;
            if constexpr (HILO) ds = (long long)(int32_t)w2 * (1 << kLoBits) + (long long)(w & ymask);
            else ds = (int32_t)((w & ymask) - pw.L * dc);
        };
        // Empty this warp's bins of group j into its totals (written, not added to, the first time):
        // words that passed; or, `raw` given, words that hold the counts beside the words before (mod
        // 2^32, w - count x increment is the sum: it fits 32 bits; HILO's sum of lo is below 2^32 and
        // its second word, from raw2 or as it is in shared memory, needs no count).
        auto flush = [&](int j, bool first, const uint32_t *raw, const uint32_t *raw2) {
            const uint32_t a = group_rec(j);
            for (int b0 = blo; b0 < bhi; b0 += 8) {
                const int nb = min(8, bhi - b0);
                unsigned long long tot[8];
                uint32_t cn[8], rw[8], rw2[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const size_t i = (size_t)(b0 + u) * ppc + 32 * j;
                    tot[u] = 0ull;
                    cn[u] = rw[u] = rw2[u] = 0u;
                    if (u < nb && !first) {
                        tot[u] = ws_tot[i];
                        if (wide) cn[u] = ws_cnt[i];
                    }
                    if (u < nb && raw) rw[u] = raw[i];
                    if (HILO && u < nb && raw2) rw2[u] = raw2[i];
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (u < nb) {
                        Sum ds;
                        uint32_t dc;
                        const uint32_t w = a + (uint32_t)(b0 + u) * row;
                        const uint32_t v = lds_u32(w), v2 = HILO ? (raw2 ? rw2[u] : lds_u32(w + 128u)) : 0u;
                        if (!raw) {
                            decode(v, v2, ds, dc);
                        } else {
                            dc = v;
                            if constexpr (HILO)
                                ds = (long long)(int32_t)v2 * (1 << kLoBits) + (long long)(rw[u] - (v << pw.S));
                            else ds = (int32_t)(rw[u] - v * pw.add());
                        }
                        sts_u32(w, 0u);
                        if (HILO) sts_u32(w + 128u, 0u);
                        tot[u] += (unsigned long long)(long long)ds + (wide ? 0ull : (unsigned long long)dc * bias);
                        ws_tot[(size_t)(b0 + u) * ppc + 32 * j] = tot[u];
                        if (wide) ws_cnt[(size_t)(b0 + u) * ppc + 32 * j] = cn[u] + dc;
                    }
                }
            }
        };
        // The words of group j (this warp's bins) put aside and cleared for the counts.
        auto put_aside = [&](int j) {
            const uint32_t a = group_rec(j);
            for (int b = blo; b < bhi; ++b) {
                ws_raw[(size_t)b * ppc + 32 * j] = lds_u32(a + (uint32_t)b * row);
                sts_u32(a + (uint32_t)b * row, 0u);
            }
        };
        // Group j's samples [i0, i1) of a failed segment (i0 is a multiple of 256) counted plainly, its words
        // being at raw (raw2), or put aside now; then into its totals. All threads together, a warp
        // sixteen samples at a time, half of them loaded while the other half is folded.
        auto redo = [&](int j, int64_t i0, int64_t i1, bool first, const uint32_t *raw, const uint32_t *raw2) {
            const uint32_t ab = group_rec(j) - (KIND == 0 ? kSlabPhase : 0u);
            uint32_t fl = 0u, fh = 0u;
#pragma unroll
            for (int q = 0; q < G; ++q)
                if (q == j) {
                    fl = Fl[q];
                    fh = Fh[q];
                }
            if (!raw) {
                put_aside(j);
                raw = ws_raw;
            }
            __syncthreads();
            const uint32_t *gtl = p.smp.tau_lo + sbase;
            const int32_t *gth = p.smp.tau_hi + sbase, *gtg = p.smp.thg + sbase / 16;
            auto one = [&](uint32_t tl, uint32_t thF) {
                word_add<KIND>(word_addr<KIND>(phase_hi(tl, thF, fl, fh), tl, fl, ab, (uint32_t)nbins, p.shift), 1u);
            };
            auto load = [&](int64_t h, uint4 (&A)[2]) {  // samples 8 h .. 8 h + 7 of the star
#pragma unroll
                for (int u = 0; u < 2; ++u) A[u] = __ldg(reinterpret_cast<const uint4 *>(gtl + 8 * h) + u);
            };
            auto half = [&](const uint4 (&A)[2], uint32_t thF) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    one(A[u].x, thF);
                    one(A[u].y, thF);
                    one(A[u].z, thF);
                    one(A[u].w, thF);
                }
            };
            const int64_t g1 = i1 >> 4;  // whole groups of sixteen
            int64_t g = (i0 >> 4) + warp;
            if (g < g1) {
                uint4 A[2], B[2];
                load(2 * g, A);
                uint32_t th = (uint32_t)__ldg(gtg + g);
#pragma unroll 1
                for (; g < g1; g += kPackWarps) {
                    const int64_t gn = min(g + kPackWarps, g1 - 1);  // (past the end: loaded, not used)
                    load(2 * g + 1, B);
                    const uint32_t thn = (uint32_t)__ldg(gtg + gn);
                    if (th == 0x80000000u) {  // (the group's samples differ in their high word)
#pragma unroll 1
                        for (int u = 0; u < 16; ++u) one(__ldg(gtl + 16 * g + u), (uint32_t)__ldg(gth + 16 * g + u) * fl);
                        load(2 * gn, A);
                    } else {
                        half(A, th * fl);
                        load(2 * gn, A);
                        half(B, th * fl);
                    }
                    th = thn;
                }
            }
            const int64_t i = 16 * g1 + warp;  // the star's last few
            if (i < i1) one(__ldg(gtl + i), (uint32_t)__ldg(gth + i) * fl);
            __syncthreads();
            flush(j, first, raw, raw2);
        };

        uint32_t have = 0u;   // groups whose totals hold something
        uint32_t turn = 0u;   // checks made
        uint32_t stored = 0u;  // kPackSegs - 1 bits a group: its slots that count
        int seg = 0;
        for (int t0 = 0; t0 < ntiles; t0 += span_tiles) {
            const int t1 = min(ntiles, t0 + span_tiles);
            push(t0);
            if (t0 + 1 < t1) push(t0 + 1);
            for (int t = t0, rt = 1; t < t1; ++t) {
                if (!fold_tile(t, std::false_type{}, 0u)) return;
                if (t + 2 < t1) push(t + 2);
                const bool last = t + 1 == ntiles, seg_end = t + 1 == t1 || rt == seg_tiles;
                uint32_t due = 0u;  // groups whose segment ends here
#pragma unroll
                for (int j = 0; j < G; ++j) {
                    const int len = (int)len_of(j);
                    if (len != (int)kBlind && (seg_end || (len && rt % len == 0))) due |= 1u << j;
                }
                if (due) {
                    const bool to_slot = slots && seg_end && !last;
                    uint32_t *slot = ws_slot + (size_t)(HILO ? 2 * seg : seg) * plane;
                    auto first_tile = [&](int j) {  // of group j's segment
                        const int len = (int)len_of(j);
                        return t + 1 - rt + (len ? (rt - 1) / len * len : 0);
                    };
                    // the check: every count at most M, and all samples counted; on the way the words
                    // of a group that keeps to the block's segments go to their slot
                    uint32_t bad = 0u;
#pragma unroll 1
                    for (int j = 0; j < G; ++j) {
                        if (!((due >> j) & 1u)) continue;
                        const uint32_t a = group_rec(j);
                        uint32_t sum = 0u, big = 0u;
                        const bool store = to_slot && !len_of(j);
                        uint32_t *w = slot + 32 * j;
#pragma unroll 4
                        for (int b = blo; b < bhi; ++b) {
                            const uint32_t v = lds_u32(a + (uint32_t)b * row), c = v >> pw.S;
                            if (store) {
                                w[(size_t)b * ppc] = v;
                                sts_u32(a + (uint32_t)b * row, 0u);
                                if (HILO) {
                                    w[plane + (size_t)b * ppc] = lds_u32(a + (uint32_t)b * row + 128u);
                                    sts_u32(a + (uint32_t)b * row + 128u, 0u);
                                }
                            }
                            sum += c;
                            big = max(big, c);
                        }
                        atomicAdd(&cnt_sum[32 * j + lane], sum);
                        if (big > pw.M && ((live >> j) & 1u)) bad |= 1u << j;
                    }
                    __syncthreads();
                    if (warp < G && ((due >> warp) & 1u)) {
                        const int64_t n = min(nsamp, (int64_t)(t + 1) * tile) - (int64_t)first_tile(warp) * tile;
                        if (cnt_sum[threadIdx.x] != (uint32_t)n && ((live >> warp) & 1u)) bad |= 1u << warp;
                        cnt_sum[threadIdx.x] = 0u;
                    }
                    bad = __reduce_or_sync(0xffffffffu, bad);
                    if (lane == 0 && bad) atomicOr(&sh.bad[turn & 1u], bad);
                    if (threadIdx.x == 0) sh.bad[(turn + 1u) & 1u] = 0u;
                    __syncthreads();
                    bad = sh.bad[turn & 1u];
                    ++turn;
#pragma unroll 1
                    for (int j = 0; j < G; ++j) {
                        if (!((due >> j) & 1u)) continue;
                        const bool first = !((have >> j) & 1u);
                        const uint32_t len = len_of(j);
                        if ((bad >> j) & 1u) {
                            const bool stored_now = to_slot && !len;
                            redo(j, (int64_t)first_tile(j) * tile, min(nsamp, (int64_t)(t + 1) * tile), first,
                                 stored_now ? slot : nullptr, stored_now ? slot + plane : nullptr);
                            have |= 1u << j;
                            // what piled its samples up does so again: shorter segments from here on (a
                            // boundary of the present length is one of the new length too), then none
                            const uint32_t now =
                                len ? len : (seg_tiles > 4 ? 8u : (seg_tiles > 2 ? 4u : (uint32_t)seg_tiles));
                            const uint32_t cut = now > 1u ? now >> 1 : kBlind;
                            own = (own & ~(31u << (5 * j))) | (cut << (5 * j));
                            if (threadIdx.x == 0) sh.blind_from[j] = t + 1;
                        } else if (to_slot && !len) {
                            stored |= 1u << (seg + (kPackSegs - 1) * j);
                        } else if (!last) {
                            flush(j, first, nullptr, nullptr);
                            have |= 1u << j;
                        }
                    }
                    __syncthreads();  // emptied before the next tile's reductions, or the epilogue
                }
                if (seg_end) {
                    rt = 1;
                    ++seg;
                } else {
                    ++rt;
                }
            }
            // blind groups: their words put aside, and their samples since then counted, all at once
            uint32_t blind = 0u;
            int from = t1;
#pragma unroll
            for (int j = 0; j < G; ++j) {
                if (len_of(j) == kBlind && sh.blind_from[j] < t1) {
                    blind |= 1u << j;
                    from = min(from, sh.blind_from[j]);
                }
            }
            if (blind) {
#pragma unroll 1
                for (int j = 0; j < G; ++j)
                    if ((blind >> j) & 1u) put_aside(j);
                __syncthreads();
                push(from);
                if (from + 1 < t1) push(from + 1);
                for (int t = from; t < t1; ++t) {
                    uint32_t mask = 0u;
#pragma unroll
                    for (int j = 0; j < G; ++j)
                        if (((blind >> j) & 1u) && sh.blind_from[j] <= t) mask |= 1u << j;
                    if (!fold_tile(t, std::true_type{}, mask)) return;
                    if (t + 2 < t1) push(t + 2);
                }
#pragma unroll 1
                for (int j = 0; j < G; ++j)
                    if ((blind >> j) & 1u) {
                        flush(j, !((have >> j) & 1u), ws_raw, nullptr);
                        have |= 1u << j;
                        if (threadIdx.x == 0) sh.blind_from[j] = t1;
                    }
                __syncthreads();
            }
        }

        // ---- epilogue: the last segment's words and the totals, straight into the output rows
        const double qscale = ldexp(1.0, -p.stats[s].qexp);
        const int qexp = -ilogb(qscale);
        const float qscale_f = (qexp >= -100 && qexp <= 100) ? __int_as_float((127 - qexp) << 23) : 0.f;
        const int conv = qscale_f == 0.f ? 2 : (!HILO && nsamp <= (int64_t)p.chunk ? 0 : 1);
        const float fh = p.stats[s].f_hi, fl = p.stats[s].f_lo;
#pragma unroll 1
        for (int j = 0; j < G; ++j) {
            const uint32_t a = group_rec(j);
            const int64_t k = k0 + 32 * j;
            const bool kvalid = k < ge;
            const int64_t orow = p.slot_k ? (task - p.task_begin) * ppc + 32 * j + lane : k;
            if (p.slot_k && warp == 0) p.slot_k[orow] = kvalid ? k : -1;
            const bool write = kvalid || p.slot_k;
            const uint32_t mine = stored >> ((kPackSegs - 1) * j);
            const bool totals = (have >> j) & 1u;
            const size_t o = (size_t)orow * nbins;
            for (int b0 = blo; b0 < bhi; b0 += kEpi) {
                Sum ds[kEpi];
                uint32_t c[kEpi];
                float S[kEpi];
#pragma unroll
                for (int u = 0; u < kEpi; ++u) {
                    c[u] = 0u;
                    ds[u] = 0;
                    const uint32_t w = a + (uint32_t)(b0 + u) * row;
                    if (b0 + u < bhi) decode(lds_u32(w), HILO ? lds_u32(w + 128u) : 0u, ds[u], c[u]);
                }
                if (slots) {
                    // (a star of at most one chunk: without HILO its bin sums are 32-bit integers)
                    constexpr int W = HILO ? 2 : 1;
                    uint32_t w[kPackSegs - 1][W][kEpi];
#pragma unroll
                    for (int q = 0; q < kPackSegs - 1; ++q)
#pragma unroll
                        for (int h = 0; h < W; ++h)
#pragma unroll
                            for (int u = 0; u < kEpi; ++u)
                                w[q][h][u] = ((mine >> q) & 1u) && b0 + u < bhi
                                                 ? ws_slot[(size_t)(W * q + h) * plane + (size_t)(b0 + u) * ppc + 32 * j]
                                                 : 0u;
#pragma unroll
                    for (int q = 0; q < kPackSegs - 1; ++q)
#pragma unroll
                        for (int u = 0; u < kEpi; ++u) {
                            Sum es;
                            uint32_t ec;
                            decode(w[q][0][u], w[q][W - 1][u], es, ec);
                            ds[u] += es;
                            c[u] += ec;
                        }
                }
#pragma unroll
                for (int u = 0; u < kEpi; ++u) {
                    long long S64 = ds[u];
                    if (totals && b0 + u < bhi) {
                        const size_t i = (size_t)(b0 + u) * ppc + 32 * j;
                        unsigned long long tot = ws_tot[i] + (unsigned long long)S64;
                        if (wide) {
                            c[u] += ws_cnt[i];
                        } else {
                            tot += (unsigned long long)c[u] * bias;
                            c[u] = (uint32_t)(tot >> 40);
                            tot -= (unsigned long long)c[u] * bias;
                        }
                        S64 = (long long)tot;
                    }
                    if (conv == 0) S[u] = __int2float_rn((int)S64) * qscale_f;
                    else if (conv == 1) S[u] = __ll2float_rn(S64) * qscale_f;
                    else S[u] = (float)((double)S64 * qscale);
                }
                if (!write) continue;
                float m[kEpi];
#pragma unroll
                for (int u = 0; u < kEpi; ++u) {
                    if (!kvalid) c[u] = 0u;
                    if (!c[u]) S[u] = 0.f;
                    if (p.folded) m[u] = c[u] ? fh + (fl + S[u] / (float)c[u]) : __int_as_float(0x7fc00000);
                }
                if (vec_out) {  // (a whole 32-byte sector per lane and store)
                    if (p.folded) st_row8(p.folded + o + b0, reinterpret_cast<const uint32_t *>(m));
                    if (p.sums) st_row8(p.sums + o + b0, reinterpret_cast<const uint32_t *>(S));
                    if (p.counts) st_row8(p.counts + o + b0, c);
                } else {
#pragma unroll
                    for (int u = 0; u < kEpi; ++u)
                        if (b0 + u < bhi) {
                            if (p.folded) p.folded[o + b0 + u] = m[u];
                            if (p.sums) p.sums[o + b0 + u] = S[u];
                            if (p.counts) p.counts[o + b0 + u] = (int)c[u];
                        }
                }
            }
        }
        __syncthreads();  // the words are read before the next task clears them
    }
    if (p.slot_k) {
        // slots of tasks in this launch's range that lie past the device task count
        const int64_t t0 = task_end > p.task_begin ? task_end : p.task_begin;
        for (int64_t task = t0 + blockIdx.x; task < p.ntasks && (int)threadIdx.x < ppc; task += gridDim.x)
            p.slot_k[(task - p.task_begin) * ppc + threadIdx.x] = -1;
    }
}

static size_t fold_pack_smem(int nbins, int groups, uint32_t window)
{
    return pack_records_addr(window, nbins) - window + pack_records_bytes(nbins, groups);
}

int fold_pack_groups(int nbins, uint32_t window)
{
    if (nbins > 256 && nbins != 512) return 0;
    int g = kPackMaxGroups;
    while (g > 0 && fold_pack_smem(nbins, g, window) > kSmemLimit) --g;
    return fold_pack_allowed(nbins, g);
}

// f(kernel) for the instance of these bins and groups (each kind with the groups it can hold;
// HILO with all but 5)
template <int KIND, int G, class F>
static cudaError_t with_groups(int groups, F f)
{
    if constexpr (G < 1) return cudaErrorInvalidValue;
    else if (groups == G) return f(fold_pack_kernel<KIND, G>);
    else return with_groups<KIND, (KIND >= 2 && G == 6 ? 4 : G - 1)>(groups, f);
}
template <class F>
static cudaError_t with_kernel(int nbins, int shift, int groups, F f)
{
    if (nbins < 256)
        return shift >= 0 ? with_groups<2, kPackMaxGroups>(groups, f) : with_groups<3, kPackMaxGroups>(groups, f);
    if (nbins == 256) return with_groups<0, kPackMaxGroups>(groups, f);
    if (nbins == 512) return with_groups<1, 3>(groups, f);  // 64 KB a group
    return cudaErrorInvalidValue;
}

// (5 has no HILO instance: a grid of that few periods a multiprocessor takes 4)
int fold_pack_allowed(int nbins, int groups) { return nbins < 256 && groups == 5 ? 4 : groups; }

int fold_pack_register()
{
    auto attr = [](auto kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
    };
    cudaError_t e = cudaSuccess;
    for (int g = 1; g <= kPackMaxGroups && e == cudaSuccess; ++g) {
        e = with_kernel(256, 24, g, attr);
        if (e == cudaSuccess && g <= 3) e = with_kernel(512, 23, g, attr);
        if (e == cudaSuccess && fold_pack_allowed(64, g) == g) e = with_kernel(64, 26, g, attr);
        if (e == cudaSuccess && fold_pack_allowed(64, g) == g) e = with_kernel(100, -1, g, attr);
    }
    return (int)e;
}

cudaError_t launch_fold_pack(const FoldParams &p, uint32_t window, int grid, cudaStream_t st)
{
    const size_t smem = fold_pack_smem(p.nbins, p.warps, window);
    if (p.warps < 1 || p.warps > kPackMaxGroups || smem > kSmemLimit || p.chunk != kPackChunk) return cudaErrorInvalidValue;
    return with_kernel(p.nbins, p.shift, p.warps, [&](auto kernel) {
        kernel<<<grid, kPackThreads, smem, st>>>(p);
        return cudaGetLastError();
    });
}

}  // namespace gpfc
