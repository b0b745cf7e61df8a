// gpfc_tcgemm.h -- the BF16 tensor-core GEMM of the CNN backward pass (tcgemm.cu) and the
// CUDA-core kernel that packs its operands.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace gpfc {

// part[s][m][n] = sum over split s's K chunks of A[m][k] B[n][k], m < rows_out, n < ntiles bn.
struct TcGemm {
    const uint8_t *A;  // [mtiles][kchunks] tiles of 128 x 64 BF16 (16 KB)
    const uint8_t *B;  // [ntiles][kchunks] tiles of bn x 64 BF16
    int64_t mtiles;
    int ntiles, kchunks, bn, splits;
    int64_t rows_out;  // rows of the output (<= 128 mtiles)
    float *part;       // [splits][rows_out][ldp] FP32
    int64_t ldp;       // = ntiles * bn
    uint32_t *status;
};

cudaError_t launch_tcgemm(const TcGemm &g, int num_sms, cudaStream_t st);

// Bytes of a packed operand of `rows` rows (padded to whole tiles of tile_rows) and K
// (padded to whole chunks of 64).
inline size_t packed_bytes(int64_t rows, int tile_rows, int64_t K)
{
    return (size_t)((rows + tile_rows - 1) / tile_rows) * (size_t)((K + 63) / 64) * (size_t)tile_rows * 128;
}

// Pack element (r, k) = ld(r, k) (zero outside rows x K) as BF16 (round to nearest even)
// into tiles [r / tile_rows][k / 64] of the K-major no-swizzle operand layout: row r's
// eight K values k..k+7 form one 16-byte core-matrix row.
//
// Bound by the bytes written and read. A block takes a tile at a time and its threads the
// 16-byte core rows in the tile's own order, so a warp stores 512 contiguous bytes and reads
// 8 rows x 4 K groups: neighbouring rows or K values of the source share 32-byte sectors
// whichever way round it lies. (One thread per K group along a row instead stores 16 bytes to
// every 128 and divides 64-bit indices: the im2col of 4,096 x 128 positions x 160 took 219 us.)
// Rows and K values are 32-bit: at most 128 positions of 2^22 profiles.
template <class LD>
__global__ void __launch_bounds__(256) pack_tiles_kernel(int64_t rows, int tile_rows, int64_t K, LD ld,
                                                         uint8_t *tiles)
{
    const int64_t kch = (K + 63) / 64;
    const int64_t ntiles = (rows + tile_rows - 1) / tile_rows * kch;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const uint32_t r0 = (uint32_t)(t / kch * tile_rows), kc = (uint32_t)(t % kch);
        uint4 *tile = reinterpret_cast<uint4 *>(tiles + (size_t)t * tile_rows * 128);
#pragma unroll 2
        for (int e = threadIdx.x; e < tile_rows * 8; e += 256) {
            const uint32_t r = r0 + (uint32_t)((e >> 6) * 8 + (e & 7)), k0 = kc * 64u + (uint32_t)((e >> 3) & 7) * 8u;
            float v[8];
#pragma unroll
            for (uint32_t h = 0; h < 8; ++h) v[h] = r < rows && k0 + h < K ? ld(r, k0 + h) : 0.f;
            uint32_t w[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * h], v[2 * h + 1]);
                w[h] = *reinterpret_cast<const uint32_t *>(&b);
            }
            tile[e] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

}  // namespace gpfc
