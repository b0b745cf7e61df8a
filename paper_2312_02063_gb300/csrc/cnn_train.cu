// cnn_train.cu -- backward pass, loss and Adam update of the CNN scorer (sm_103a).
//
// The forward pass for training is the tensor-core forward of cnn.cu run with its
// activation saves switched on (FP32 pre-activations, pooled outputs, the fc1 operand
// tiles and fc1's FP32 pre-activations), so the backward takes the ReLU and max-pool
// decisions the forward took. The backward pass:
//   fc2/fc1 head (per profile, CUDA cores);
//   dW(fc1) = dZ1^T h3 and dh3 = dZ1 W1 as BF16 tensor-core GEMMs (tcgemm.cu);
//   ReLU + max-pool backward (the gradient goes to the first maximum of each pair);
//   conv3 and conv2: weight gradients dW[co][ci,tap] = sum over (profile, position) of
//   da[co][l] h[ci][l + tap - 2] and input gradients dh[(profile, position)][ci] = sum over
//   (co, tap) of da[co][m - tap + 2] W[co][ci][tap] (circular), as BF16 tensor-core GEMMs
//   on operands packed from the saved activations (im2col in the operand layout);
//   conv1's 80 weights and every bias by CUDA-core reductions.
// GEMM operands are BF16 (round to nearest even), accumulation FP32. Every gradient is
// reduced deterministically: split-K partials and per-block partials are added in a fixed
// order. Loss: binary cross-entropy with logits (mean). Adam (Kingma & Ba) updates FP32
// master weights in place.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cuda_bf16.h>

#include "gpfc_cnn.h"
#include "gpfc_common.cuh"
#include "gpfc_tcgemm.h"

namespace gpfc {

__device__ __forceinline__ float bf2f(uint16_t b) { return __bfloat162float(__ushort_as_bfloat16(b)); }
__device__ __forceinline__ float rbf(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// ------------------------------------------------------------------ loss

// loss partials per block and dlogit = (sigmoid(z) - y) / n
__global__ void bce_kernel(const float *z, const float *y, int64_t n, float *dlogit, double *part)
{
    __shared__ double red[8];
    double acc = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float zi = z[i], yi = y[i];
        acc += (double)(fmaxf(zi, 0.f) - zi * yi + log1pf(expf(-fabsf(zi))));
        if (dlogit) dlogit[i] = (1.f / (1.f + expf(-zi)) - yi) / (float)n;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

__global__ void bce_finish_kernel(const double *part, int nblk, int64_t n, float *loss)
{
    if (threadIdx.x != 0) return;
    double t = 0.0;
    for (int b = 0; b < nblk; ++b) t += part[b];
    *loss = (float)(t / (double)n);
}

// ------------------------------------------------------------------ head: fc2 and fc1's ReLU

// dZ1[k][j] = [z1 > 0] dz_k wf2[j]; partials of dwf2, dbf1 (256 each) and dbf2 (1)
__global__ void __launch_bounds__(256) head_bwd_kernel(const float *z1, const float *dlogit, const float *wf2,
                                                       int64_t B, float *dZ1, float *part)
{
    const int j = threadIdx.x;
    const float w = rbf(wf2[j]);
    float gw = 0.f, gb = 0.f, gb2 = 0.f;
    for (int64_t k = blockIdx.x; k < B; k += gridDim.x) {
        const float dz = dlogit[k];
        const float z = z1[k * 256 + j];
        gw += dz * fmaxf(z, 0.f);
        const float d = z > 0.f ? dz * w : 0.f;
        dZ1[k * 256 + j] = d;
        gb += d;
        gb2 += dz;
    }
    float *pp = part + (size_t)blockIdx.x * 513;
    pp[j] = gw;
    pp[256 + j] = gb;
    if (j == 0) pp[512] = gb2;
}

// device fc1 feature fd = position * 64 + channel <-> PyTorch feature channel * 32 + position
__host__ __device__ __forceinline__ int pt_feature(int fd) { return (fd & 63) * 32 + (fd >> 6); }

struct LoadH3 {  // B(k = profile, n = fd) from the fc1 operand tiles: high + low BF16 terms
    const uint8_t *h3t;
    __device__ float operator()(int k, int fd) const
    {
        const int mt = k >> 7, r = k & 127, kc = fd >> 6, kk = fd & 63;
        const size_t off = ((size_t)mt * kH3Chunks + kc) * (128 * 64 * 2) +
                           (size_t)((r >> 3) * 1024 + (kk >> 3) * 128 + (r & 7) * 16 + (kk & 7) * 2);
        const size_t lo = (size_t)32 * (128 * 64 * 2);  // the low terms' chunk kc + 32
        return bf2f(*reinterpret_cast<const uint16_t *>(h3t + off)) +
               bf2f(*reinterpret_cast<const uint16_t *>(h3t + off + lo));
    }
};
// ------------------------------------------------------------------ GEMM operand loaders
// (element (row, k) of a packed operand; the packer rounds to BF16)

struct LdDZ1T {  // dW(fc1): A(j, profile)
    const float *dZ1;
    __device__ float operator()(uint32_t j, uint32_t k) const { return dZ1[(size_t)k * 256 + j]; }
};
struct LdH3T {  // dW(fc1): B(feature fd, profile) = h3 (high + low terms)
    const uint8_t *h3t;
    __device__ float operator()(uint32_t fd, uint32_t k) const { return LoadH3{h3t}((int)k, (int)fd); }
};
struct LdDZ1 {  // dh3: A(profile, j)
    const float *dZ1;
    __device__ float operator()(uint32_t k, uint32_t j) const { return dZ1[(size_t)k * 256 + j]; }
};
struct LdW1T {  // dh3: B(fd, j) = fc1.w[j][pt_feature(fd)]
    const float *w;
    __device__ float operator()(uint32_t fd, uint32_t j) const { return w[j * 2048 + pt_feature((int)fd)]; }
};
template <int COUT, int L>
struct LdDa {  // conv weight gradient: A(co, (profile b, position l))
    const float *da;
    __device__ float operator()(uint32_t co, uint32_t k) const { return da[((size_t)(k / L) * COUT + co) * L + (k % L)]; }
};
template <int CIN, int L>
struct LdHim {  // conv weight gradient: B((ci, tap), (b, l)) = h[b][ci][(l + tap - 2) mod L]
    const uint16_t *h;
    __device__ float operator()(uint32_t n, uint32_t k) const
    {
        const int ci = (int)(n / 5), tap = (int)(n % 5), l = (int)(k % L);
        return bf2f(h[((size_t)(k / L) * CIN + ci) * L + ((l + tap - 2 + L) % L)]);
    }
};
template <int COUT, int L>
struct LdDaShift {  // conv input gradient: A((b, m), (co, tap)) = da[b][co][(m - tap + 2) mod L]
    const float *da;
    __device__ float operator()(uint32_t r, uint32_t k) const
    {
        const int m = (int)(r % L), co = (int)(k / 5), tap = (int)(k % 5);
        return da[((size_t)(r / L) * COUT + co) * L + ((m - tap + 2 + L) % L)];
    }
};
template <int CIN>
struct LdWT {  // conv input gradient: B(ci, (co, tap)) = W[co][ci][tap]
    const float *W;
    __device__ float operator()(uint32_t ci, uint32_t k) const { return W[((k / 5) * CIN + ci) * 5 + (k % 5)]; }
};

// ------------------------------------------------------------------ ReLU + max-pool backward

// One profile at a time per block. da[k][c][2l+s] = g[k][l][c] if element 2l+s was the (first)
// maximum of relu(a) over the pair and a > 0 there; else 0. g is a GEMM's result, position-major
// (the device feature order for dh3): it goes through shared memory, a's and da's four positions
// a thread straight. The bias gradient is summed on the way, in a thread's registers across the
// block's profiles (its channels do not change), so da is not read again for it; and the first
// layer's weight gradient
//   dW[c][t] += sum_l da[c][l] x[(l + t - 2) mod L]
// too (CONV1), whose da is then never stored. Partials per block: [C] or, CONV1, [C][5], [C].
// Bound by memory: 4,096 profiles move 168 MB a layer (CONV1 105 MB).
template <int C, int L, bool CONV1>
__global__ void __launch_bounds__(256, 3) poolrelu_bwd_kernel(const float *a, const float *g, const float *x,
                                                              float *da, int64_t B, float *part)
{
    static_assert(C * L == 4096 && L % 4 == 0, "four float4 a thread");
    constexpr int LP = L / 2, GS = C + 1;  // row stride in shared memory: no bank conflicts along l
    constexpr int T = L / 4;               // threads of a channel
    __shared__ float gs[LP * GS];
    __shared__ float xs[CONV1 ? L : 1];
    __shared__ float red[CONV1 ? 8 * 4 * 6 : 1];
    const int t = threadIdx.x;
    float accb[4] = {0.f, 0.f, 0.f, 0.f};
    float accw[4][5];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 5; ++q) accw[i][q] = 0.f;
    for (int64_t k = blockIdx.x; k < B; k += gridDim.x) {
        const float4 *ak = reinterpret_cast<const float4 *>(a + k * 4096);
        const float4 *gk = reinterpret_cast<const float4 *>(g + k * 2048);
        float4 v[4], w[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) w[i] = gk[t + 256 * i];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = ak[t + 256 * i];
        __syncthreads();  // the profile before has been read
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int e = 4 * (t + 256 * i), lp = e / C, c = e % C;
            float *d = gs + lp * GS + c;
            d[0] = w[i].x;
            d[1] = w[i].y;
            d[2] = w[i].z;
            d[3] = w[i].w;
        }
        if (CONV1) xs[t] = x[k * L + t];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = t + 256 * i, c = e / T, l = 4 * (e % T);
            const float g0 = gs[(l / 2) * GS + c], g1 = gs[(l / 2 + 1) * GS + c];
            const bool s0 = fmaxf(v[i].y, 0.f) > fmaxf(v[i].x, 0.f), s1 = fmaxf(v[i].w, 0.f) > fmaxf(v[i].z, 0.f);
            float4 d;
            d.x = (!s0 && v[i].x > 0.f) ? g0 : 0.f;
            d.y = (s0 && v[i].y > 0.f) ? g0 : 0.f;
            d.z = (!s1 && v[i].z > 0.f) ? g1 : 0.f;
            d.w = (s1 && v[i].w > 0.f) ? g1 : 0.f;
            accb[i] += (d.x + d.y) + (d.z + d.w);
            if (CONV1) {
                float xx[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) xx[q] = xs[(l + q - 2) & (L - 1)];
#pragma unroll
                for (int q = 0; q < 5; ++q)
                    accw[i][q] +=
                        fmaf(d.x, xx[q], d.y * xx[q + 1]) + fmaf(d.z, xx[q + 2], d.w * xx[q + 3]);
            } else {
                reinterpret_cast<float4 *>(da + k * 4096)[e] = d;
            }
        }
    }
    // a channel's threads are T consecutive ones
    constexpr int TW = T < 32 ? T : 32;
    auto fold = [&](float s) {
#pragma unroll
        for (int o = TW / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    };
    if (CONV1) {  // two warps a channel
        static_assert(!CONV1 || T == 64, "two warps a channel");
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const float s = fold(q < 5 ? accw[i][q < 5 ? q : 0] : accb[i]);
                if ((t & 31) == 0) red[((t >> 5) * 4 + i) * 6 + q] = s;
            }
        __syncthreads();
        if (t < C * 6) {
            const int c = t / 6, q = t % 6, wp = 2 * (c & 3), i = c >> 2;
            const float s = red[(wp * 4 + i) * 6 + q] + red[((wp + 1) * 4 + i) * 6 + q];
            part[(size_t)blockIdx.x * (C * 6) + (q < 5 ? c * 5 + q : C * 5 + c)] = s;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float s = fold(accb[i]);
            if (t % TW == 0) part[(size_t)blockIdx.x * C + (t + 256 * i) / T] = s;
        }
    }
}

// out[i] = sum_b part[b][i] for i < n: a warp per output, its lanes the blocks in a fixed order
// (one thread per output waits out 304 dependent FP64 additions, 30 us); the row's outputs lie in
// up to three arrays of n0, n1 and n - n0 - n1.
__global__ void __launch_bounds__(256) reduce_parts_kernel(const float *part, int nblk, int n, float *out0, int n0,
                                                           float *out1, int n1, float *out2)
{
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= n) return;
    double s = 0.0;
    for (int b = threadIdx.x & 31; b < nblk; b += 32) s += (double)part[(size_t)b * n + i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x & 31) return;
    if (i < n0) out0[i] = (float)s;
    else if (i < n0 + n1) out1[i - n0] = (float)s;
    else out2[i - n0 - n1] = (float)s;
}

static void reduce_parts(const float *part, int nblk, float *out0, int n0, float *out1, int n1, float *out2, int n2,
                         cudaStream_t st)
{
    const int n = n0 + n1 + n2;
    reduce_parts_kernel<<<(n + 7) / 8, 256, 0, st>>>(part, nblk, n, out0, n0, out1, n1, out2);
}

// ------------------------------------------------------------------ Adam

__global__ void adam_kernel(float *p, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2,
                            float eps, float c1, float c2)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float mh = mi / c1, vh = vi / c2;
        p[i] -= lr * mh / (sqrtf(vh) + eps);
    }
}

// ------------------------------------------------------------------ host launches

size_t cnn_saved_bytes(int64_t B)
{
    return CnnSaved::layout(B).total;
}

CnnSaved CnnSaved::layout(int64_t B)
{
    CnnSaved s{};
    size_t o = 0;
    auto take = [&](size_t bytes) {
        o = (o + 255) & ~(size_t)255;
        const size_t r = o;
        o += bytes;
        return r;
    };
    s.x = take((size_t)B * 256 * 4);
    s.a1 = take((size_t)B * 16 * 256 * 4);
    s.h1 = take((size_t)B * 16 * 128 * 2);
    s.a2 = take((size_t)B * 32 * 128 * 4);
    s.h2 = take((size_t)B * 32 * 64 * 2);
    s.a3 = take((size_t)B * 64 * 64 * 4);
    s.h3t = take(cnn_h3t_bytes(B));
    s.z1 = take((size_t)B * 256 * 4);
    s.total = (o + 255) & ~(size_t)255;
    return s;
}

// ------------------------------------------------------------------ backward launches

// out(m, n) = sum over splits s of part[s][m][n], stored by st(m, n, value). A block takes 32
// outputs, its eight warps every eighth split each, added up in a fixed order (a thread per output
// leaves all but 40 blocks' worth of the chip idle for 152 dependent FP64 additions: 130 us for
// conv3's 64 x 160).
template <class ST>
__global__ void __launch_bounds__(256) reduce_splits_kernel(const float *part, int splits, int64_t rows, int cols,
                                                            ST st)
{
    __shared__ double red[8][32];
    const int64_t total = rows * cols;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t e0 = (int64_t)blockIdx.x * 32; e0 < total; e0 += (int64_t)gridDim.x * 32) {
        const int64_t e = e0 + lane;
        double v = 0.0;
        if (e < total)
            for (int s = w; s < splits; s += 8) v += (double)part[(size_t)s * total + e];
        red[w][lane] = v;
        __syncthreads();
        if (w == 0 && e < total) {
#pragma unroll
            for (int q = 1; q < 8; ++q) v += red[q][lane];
            st(e / cols, e % cols, (float)v);
        }
        __syncthreads();
    }
}
struct StWf1 {  // dW(fc1)[j][fd] -> PyTorch order
    float *g;
    __device__ void operator()(int64_t j, int64_t fd, float v) const { g[j * 2048 + pt_feature((int)fd)] = v; }
};
struct StRowMajor {
    float *g;
    int64_t ld;
    __device__ void operator()(int64_t r, int64_t c, float v) const { g[r * ld + c] = v; }
};
// The tensor-core GEMMs of one backward pass: (rows of A and of the output, rows of B = N,
// K, N tile, split-K count). Operands and partials share three workspace buffers.
struct BwdGemmShape {
    int64_t M, N, K;
    int bn, splits;
};

static BwdGemmShape bwd_shape(int which, int64_t B, int num_sms)
{
    BwdGemmShape s{};
    switch (which) {
    case 0: s = {256, 2048, B, 256, 1}; break;           // dW(fc1)
    case 1: s = {B, 2048, 256, 256, 1}; break;           // dh3
    case 2: s = {64, 160, B * 64, 160, 1}; break;        // dW(conv3)
    case 3: s = {B * 64, 32, 320, 32, 1}; break;         // dh2
    case 4: s = {32, 80, B * 128, 80, 1}; break;         // dW(conv2)
    default: s = {B * 128, 16, 160, 16, 1}; break;       // dh1
    }
    const int64_t mt = (s.M + 127) / 128, nt = (s.N + s.bn - 1) / s.bn, kch = (s.K + 63) / 64;
    if (mt * nt < num_sms) s.splits = (int)std::min<int64_t>(kch, (num_sms + mt * nt - 1) / (mt * nt));
    return s;
}

static void bwd_ws_sizes(int64_t B, int num_sms, size_t &a, size_t &b, size_t &part)
{
    a = b = part = 0;
    for (int w = 0; w < 6; ++w) {
        const BwdGemmShape s = bwd_shape(w, B, num_sms);
        a = std::max(a, packed_bytes(s.M, 128, s.K));
        b = std::max(b, packed_bytes(s.N, s.bn, s.K));
        part = std::max(part, (size_t)s.splits * (size_t)s.M * (size_t)((s.N + s.bn - 1) / s.bn * s.bn) * 4);
    }
}

size_t cnn_backward_ws_bytes(int64_t B, int nblk, int num_sms)
{
    size_t o = 0;
    auto take = [&](size_t bytes) { o = ((o + 255) & ~(size_t)255) + bytes; };
    take((size_t)B * 256 * 4);         // dZ1
    take((size_t)B * 2048 * 4);        // dH3, then dh2 and dh1
    take((size_t)B * 64 * 64 * 4);     // da3, then da2
    take((size_t)nblk * (16 * 5 + 16) * 4);  // conv1 weight/bias partials
    take((size_t)nblk * 64 * 4);       // bias partials
    take((size_t)nblk * 513 * 4);      // head partials
    size_t a, b, part;
    bwd_ws_sizes(B, num_sms, a, b, part);
    take(a);
    take(b);
    take(part);
    return o + 256;
}

// Pack A and B of GEMM `which`, run it and hand its partials to `store`; or, where `whole` is
// given and the GEMM's K is not split, leave them where they are: *whole is the row-major result
// (else it is what `store` wrote).
template <class LA, class LB, class ST>
static cudaError_t bwd_gemm(int which, int64_t B, int num_sms, LA la, LB lb, ST store, const float **whole,
                            uint8_t *pa, uint8_t *pb, float *part, cudaStream_t st)
{
    const BwdGemmShape s = bwd_shape(which, B, num_sms);
    const int64_t kch = (s.K + 63) / 64;
    const int64_t ga = std::min<int64_t>(65535, (s.M + 127) / 128 * kch);
    const int64_t gb = std::min<int64_t>(65535, (s.N + s.bn - 1) / s.bn * kch);
    pack_tiles_kernel<<<(int)ga, 256, 0, st>>>(s.M, 128, s.K, la, pa);
    pack_tiles_kernel<<<(int)gb, 256, 0, st>>>(s.N, s.bn, s.K, lb, pb);
    TcGemm g{};
    g.A = pa;
    g.B = pb;
    g.mtiles = (s.M + 127) / 128;
    g.ntiles = (int)((s.N + s.bn - 1) / s.bn);
    g.kchunks = (int)kch;
    g.bn = s.bn;
    g.splits = s.splits;
    g.rows_out = s.M;
    g.ldp = (int64_t)g.ntiles * s.bn;
    g.part = part;
    cudaError_t e = launch_tcgemm(g, num_sms, st);
    if (e != cudaSuccess) return e;
    if (whole && s.splits == 1) {
        *whole = part;
        return cudaSuccess;
    }
    const int64_t total = s.M * g.ldp;
    reduce_splits_kernel<<<(int)std::min<int64_t>(8192, (total + 31) / 32), 256, 0, st>>>(part, s.splits, s.M,
                                                                                            (int)g.ldp, store);
    return cudaGetLastError();
}

cudaError_t launch_cnn_backward(const CnnSrc &w, const uint8_t *saved, int64_t B, const float *dlogit,
                                const CnnGrads &g, void *ws, int nblk, int num_sms, cudaStream_t st)
{
    const CnnSaved S = CnnSaved::layout(B);
    uint8_t *base = static_cast<uint8_t *>(ws);
    size_t o = 0;
    auto take = [&](size_t bytes) {
        o = (o + 255) & ~(size_t)255;
        uint8_t *p = base + o;
        o += bytes;
        return p;
    };
    float *dZ1 = reinterpret_cast<float *>(take((size_t)B * 256 * 4));
    float *dh = reinterpret_cast<float *>(take((size_t)B * 2048 * 4));
    float *da = reinterpret_cast<float *>(take((size_t)B * 64 * 64 * 4));
    float *cpart = reinterpret_cast<float *>(take((size_t)nblk * (16 * 5 + 16) * 4));
    float *bpart = reinterpret_cast<float *>(take((size_t)nblk * 64 * 4));
    float *hpart = reinterpret_cast<float *>(take((size_t)nblk * 513 * 4));
    size_t sa, sb, sp;
    bwd_ws_sizes(B, num_sms, sa, sb, sp);
    uint8_t *pa = take(sa);
    uint8_t *pb = take(sb);
    float *gpart = reinterpret_cast<float *>(take(sp));
    const int sms = num_sms;

    const float *z1 = reinterpret_cast<const float *>(saved + S.z1);
    head_bwd_kernel<<<nblk, 256, 0, st>>>(z1, dlogit, w.wf2, B, dZ1, hpart);
    reduce_parts(hpart, nblk, g.wf2, 256, g.bf1, 256, g.bf2, 1, st);
    // dW(fc1)[256][2048] = dZ1^T h3; dh3[B][2048] = dZ1 W1
    const float *gp = dh;  // a GEMM's result for the layer below
    cudaError_t e = bwd_gemm(0, B, sms, LdDZ1T{dZ1}, LdH3T{saved + S.h3t}, StWf1{g.wf1}, nullptr, pa, pb, gpart, st);
    if (e == cudaSuccess)
        e = bwd_gemm(1, B, sms, LdDZ1{dZ1}, LdW1T{w.wf1}, StRowMajor{dh, 2048}, &gp, pa, pb, gpart, st);
    if (e != cudaSuccess) return e;
    // conv3: da3 and bias, dW[64][160] and dh2
    poolrelu_bwd_kernel<64, 64, false>
        <<<nblk, 256, 0, st>>>(reinterpret_cast<const float *>(saved + S.a3), gp, nullptr, da, B, bpart);
    reduce_parts(bpart, nblk, g.b3, 64, nullptr, 0, nullptr, 0, st);
    e = bwd_gemm(2, B, sms, LdDa<64, 64>{da}, LdHim<32, 64>{reinterpret_cast<const uint16_t *>(saved + S.h2)},
                 StRowMajor{g.w3, 160}, nullptr, pa, pb, gpart, st);
    gp = dh;
    if (e == cudaSuccess)
        e = bwd_gemm(3, B, sms, LdDaShift<64, 64>{da}, LdWT<32>{w.w3}, StRowMajor{dh, 32}, &gp, pa, pb, gpart, st);
    if (e != cudaSuccess) return e;
    // conv2: da2 and bias, dW[32][80] and dh1
    poolrelu_bwd_kernel<32, 128, false>
        <<<nblk, 256, 0, st>>>(reinterpret_cast<const float *>(saved + S.a2), gp, nullptr, da, B, bpart);
    reduce_parts(bpart, nblk, g.b2, 32, nullptr, 0, nullptr, 0, st);
    e = bwd_gemm(4, B, sms, LdDa<32, 128>{da}, LdHim<16, 128>{reinterpret_cast<const uint16_t *>(saved + S.h1)},
                 StRowMajor{g.w2, 80}, nullptr, pa, pb, gpart, st);
    gp = dh;
    if (e == cudaSuccess)
        e = bwd_gemm(5, B, sms, LdDaShift<32, 128>{da}, LdWT<16>{w.w2}, StRowMajor{dh, 16}, &gp, pa, pb, gpart, st);
    if (e != cudaSuccess) return e;
    // conv1 (16 x 5 weights) on CUDA cores
    poolrelu_bwd_kernel<16, 256, true>
        <<<nblk, 256, 0, st>>>(reinterpret_cast<const float *>(saved + S.a1), gp,
                               reinterpret_cast<const float *>(saved + S.x), nullptr, B, cpart);
    reduce_parts(cpart, nblk, g.w1, 80, g.b1, 16, nullptr, 0, st);
    return cudaGetLastError();
}

cudaError_t launch_bce(const float *z, const float *y, int64_t n, float *dlogit, float *loss, void *ws, cudaStream_t st)
{
    const int nblk = (int)std::min<int64_t>(256, (n + 255) / 256);
    double *part = static_cast<double *>(ws);
    bce_kernel<<<nblk, 256, 0, st>>>(z, y, n, dlogit, part);
    if (loss) bce_finish_kernel<<<1, 32, 0, st>>>(part, nblk, n, loss);
    return cudaGetLastError();
}

cudaError_t launch_adam(float *p, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2,
                        float eps, float c1, float c2, cudaStream_t st)
{
    const int grid = (int)std::min<int64_t>(1024, (n + 255) / 256);
    adam_kernel<<<grid, 256, 0, st>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

}  // namespace gpfc
