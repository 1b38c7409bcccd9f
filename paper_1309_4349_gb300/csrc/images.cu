// images.cu -- snapshot images of the lattice and their fraction of first
// neighbours, computed on the device (section "Image analysis": each site a white
// (A) or black (B) pixel, the image sloped to keep the triangular geometry and
// scaled down with supersampling to gray levels; the fraction of first neighbours
// of a gray image compares a randomly chosen neighbour pixel within a gray-level
// threshold delta_col).
//
// Geometry: site (x, y) covers u in [2x + y, 2x + y + 2) half-sites and v in
// [y, y+1) rows; the image is U = 2 Lx + Ly - 1 half-sites wide.  Output pixel
// (i, j) of a W x H image averages an S x S grid of samples at
// u = (2(iS + a) + 1) U / (2WS), v = (2(jS + b) + 1) Ly / (2HS), evaluated in
// integers so that the image is exact: row y = floor(v), site x = floor((u - y)/2),
// inside iff 0 <= x < Lx.  A pixel belongs to the lattice iff at least half its
// samples are inside; its gray level is round(255 n_A / n_in), halves up.
//
// The image estimator: every lattice pixel p = jW + i takes one of its eight
// neighbours, direction floor(w * 8 / 2^32) of (1,0), (1,1), (0,1), (-1,1), (-1,0),
// (-1,-1), (0,-1), (1,-1), w = word (p mod 4) of Philox(seed, {p div 4, 0xFFFFFFFC,
// m_lo, m_hi}); it is similar iff that neighbour is a lattice pixel whose gray
// level differs by at most delta.
#include "klmc_internal.h"
#include "philox.cuh"

namespace klmc {
namespace {

constexpr int kImgBlock = 256;

__device__ __forceinline__ uint32_t lattice_site(const void *lat, int packing, int pitch, int x, int y)
{
    if (packing == kPackBit) return (((const uint32_t *)lat)[(size_t)y * pitch + (x >> 5)] >> (x & 31)) & 1u;
    return ((const uint8_t *)lat)[(size_t)y * pitch + x] ? 1u : 0u;
}

constexpr int kSnapRows = 8;  // most image rows of a CTA

// The column of a sample n of WS across, in half-sites: floor(u).  Site x of row y covers
// half-sites 2x + y and 2x + y + 1, so the sample's site is (column - y) >> 1.
__device__ __forceinline__ int sample_column(long long n, long long U, long long WS)
{
    const unsigned long long num = (unsigned long long)((2 * n + 1) * U), den = (unsigned long long)(2 * WS);
    return (int)((num | den) >> 32 ? num / den : (uint32_t)num / (uint32_t)den);
}

// A thread takes one image column of R <= kSnapRows rows: its samples' columns are found once
// (a division each), the rows of the lattice that the CTA's image rows sample once per CTA.
// Bound: a load, a shift and a few operations per sample.  ST: samples per pixel side, known
// at compile time, or 0.  A 6143 x 3547 image of 8192^2 at 4 x 4 samples took 1158 us with two
// 64-bit divisions per sample, 191 us so.
template <int ST>
__global__ void __launch_bounds__(kImgBlock)
snapshot_kernel(const void *lat, int packing, int pitch, int Lx, int Ly, int W, int H, int S_, int R, uint8_t *image,
                uint8_t *mask)
{
    const int S = ST > 0 ? ST : S_;
    __shared__ int rows[kSnapRows * 64];
    const long long U = 2ll * Lx + Ly - 1;
    const int strips = (H + R - 1) / R, cols = (W + kImgBlock - 1) / kImgBlock;
    for (long long blk = blockIdx.x; blk < (long long)strips * cols; blk += gridDim.x) {
        const int strip = (int)(blk / cols);
        const int i = (int)(blk - (long long)strip * cols) * kImgBlock + (int)threadIdx.x;
        const int j0 = strip * R, nj = min(R, H - j0);
        __syncthreads();
        for (int k = threadIdx.x; k < nj * S; k += kImgBlock)
            rows[k] = sample_column((long long)j0 * S + k, Ly, (long long)H * S);  // floor(v) likewise
        __syncthreads();
        if (i >= W) continue;
        if (ST > 0) {
            int h[ST > 0 ? ST : 1];
#pragma unroll
            for (int a = 0; a < ST; ++a) h[a] = sample_column((long long)i * ST + a, U, (long long)W * ST);
            for (int jj = 0; jj < nj; ++jj) {
                int n_in = 0, n_A = 0;
#pragma unroll
                for (int b = 0; b < ST; ++b) {
                    const int y = rows[jj * ST + b];
                    const int x0 = (h[0] - y) >> 1, xe = (h[ST - 1] - y) >> 1;
                    if (packing == kPackBit && x0 >= 0 && xe < Lx && xe - x0 < 32) {
                        // all inside and within one 32-site window
                        const uint32_t *const row = (const uint32_t *)lat + (size_t)y * pitch;
                        const int w = x0 >> 5;
                        const uint32_t win = __funnelshift_r(row[w], row[min(w + 1, pitch - 1)], x0 & 31);
                        n_in += ST;
#pragma unroll
                        for (int a = 0; a < ST; ++a) n_A += (int)((win >> (((h[a] - y) >> 1) - x0)) & 1u);
                        continue;
                    }
#pragma unroll
                    for (int a = 0; a < ST; ++a) {
                        const int x = (h[a] - y) >> 1;
                        if ((unsigned)x < (unsigned)Lx) {
                            n_in += 1;
                            n_A += (int)lattice_site(lat, packing, pitch, x, y);
                        }
                    }
                }
                const size_t p = (size_t)(j0 + jj) * W + i;
                mask[p] = (uint8_t)(2 * n_in >= ST * ST);
                image[p] = n_in > 0 ? (uint8_t)((unsigned)(510 * n_A + n_in) / (unsigned)(2 * n_in)) : (uint8_t)0;
            }
        } else {
            int n_in[kSnapRows], n_A[kSnapRows];
#pragma unroll
            for (int jj = 0; jj < kSnapRows; ++jj) n_in[jj] = n_A[jj] = 0;
            for (int a = 0; a < S; ++a) {
                const int h = sample_column((long long)i * S + a, U, (long long)W * S);
#pragma unroll
                for (int jj = 0; jj < kSnapRows; ++jj) {
                    if (jj >= nj) break;
                    for (int b = 0; b < S; ++b) {
                        const int y = rows[jj * S + b], x = (h - y) >> 1;
                        if ((unsigned)x < (unsigned)Lx) {
                            n_in[jj] += 1;
                            n_A[jj] += (int)lattice_site(lat, packing, pitch, x, y);
                        }
                    }
                }
            }
#pragma unroll
            for (int jj = 0; jj < kSnapRows; ++jj) {
                if (jj >= nj) break;
                const size_t p = (size_t)(j0 + jj) * W + i;
                mask[p] = (uint8_t)(2 * n_in[jj] >= S * S);
                image[p] = n_in[jj] > 0 ? (uint8_t)((unsigned)(510 * n_A[jj] + n_in[jj]) / (unsigned)(2 * n_in[jj]))
                                        : (uint8_t)0;
            }
        }
    }
}

// Offsets of the eight directions, plus one, two bits each (a table in constant memory
// would be read once per distinct direction of a warp).
__device__ __forceinline__ int moore_i(int k) { return (int)((0x901Au >> (2 * k)) & 3u) - 1; }
__device__ __forceinline__ int moore_j(int k) { return (int)((0x01A9u >> (2 * k)) & 3u) - 1; }

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

__global__ void image_ffn_kernel(const uint8_t *image, const uint8_t *mask, int W, int H, int delta, uint32_t k0,
                                 uint32_t k1, unsigned long long m, long long *out)
{
    __shared__ long long red[2][kImgBlock / 32];
    const long long P = (long long)W * H;
    const long long G = (P + 3) / 4;
    const bool vec = ((((uintptr_t)image) | ((uintptr_t)mask)) & 3u) == 0u;
    int similar = 0, pixels = 0;  // fewer than 2^31 pixels
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < G;
         q += (long long)gridDim.x * blockDim.x) {
        // four pixels' levels and membership at a time where the buffers allow it
        uint32_t px = 0u, in = 0u;
        if (vec && 4 * q + 4 <= P) {
            px = ((const uint32_t *)image)[q];
            in = ((const uint32_t *)mask)[q];
        } else {
            for (int r = 0; r < 4 && 4 * q + r < P; ++r) {
                px |= (uint32_t)image[4 * q + r] << (8 * r);
                in |= (uint32_t)mask[4 * q + r] << (8 * r);
            }
        }
        if (in == 0u) continue;
        const Philox4 pw = philox4((uint32_t)q, 0xFFFFFFFCu, (uint32_t)m, (uint32_t)(m >> 32), k0, k1);
        const uint32_t *w = pw.v;
        const int j0 = (int)((uint32_t)(4 * q) / (uint32_t)W), i0 = (int)((uint32_t)(4 * q) - (uint32_t)j0 * (uint32_t)W);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = i0 + r < W ? i0 + r : (i0 + r) % W, j = i0 + r < W ? j0 : j0 + (i0 + r) / W;
            if (((in >> (8 * r)) & 0xFFu) == 0u) continue;
            pixels += 1;
            const int k = (int)(w[r] >> 29);
            const int a = i + moore_i(k), b = j + moore_j(k);
            if (a < 0 || a >= W || b < 0 || b >= H) continue;
            const long long qq = (long long)b * W + a;
            if (!mask[qq]) continue;
            const int d = (int)((px >> (8 * r)) & 0xFFu) - (int)image[qq];
            similar += (d <= delta && -d <= delta) ? 1 : 0;
        }
    }
    const long long s1 = warp_sum((long long)similar), s2 = warp_sum((long long)pixels);
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = s1;
        red[1][threadIdx.x >> 5] = s2;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        long long sum = 0;
        for (int w = 0; w < kImgBlock / 32; ++w) sum += red[threadIdx.x][w];
        if (sum) atomicAdd((unsigned long long *)out + threadIdx.x, (unsigned long long)sum);
    }
}

int img_grid(long long work)
{
    long long g = (work + kImgBlock - 1) / kImgBlock;
    if (g < 1) g = 1;
    if (g > 152 * 16) g = 152 * 16;
    return (int)g;
}

}  // namespace

cudaError_t launch_snapshot(const void *lat, int packing, int pitch, int Lx, int Ly, int W, int H, int S,
                            uint8_t *image, uint8_t *mask, cudaStream_t stream)
{
    // Small images take fewer rows per CTA, so that the chip is in use: 64 x 64 at 7 x 7 samples of
    // 8192^2 37 us with 8 rows, 8.6 with one; 300 x 300 at 5 x 5 of 300^2 19 and 8.7.
    const long long cols = (W + kImgBlock - 1) / kImgBlock;
    int R = kSnapRows;
    while (R > 1 && (H + R - 1) / R * cols < 152 * 4) R /= 2;
    const long long strips = (H + R - 1) / R;
    const int g = (int)(strips * cols < 152 * 64 ? strips * cols : 152 * 64);
    auto kernel = S == 1 ? snapshot_kernel<1>
                : (S == 2 ? snapshot_kernel<2> : (S == 3 ? snapshot_kernel<3> : (S == 4 ? snapshot_kernel<4>
                                                                                           : snapshot_kernel<0>)));
    kernel<<<g, kImgBlock, 0, stream>>>(lat, packing, pitch, Lx, Ly, W, H, S, R, image, mask);
    return cudaGetLastError();
}

cudaError_t launch_image_ffn(const uint8_t *image, const uint8_t *mask, int W, int H, int delta, uint32_t key0,
                             uint32_t key1, long long sample, long long *out2, cudaStream_t stream)
{
    cudaError_t e = cudaMemsetAsync(out2, 0, 2 * sizeof(long long), stream);
    if (e != cudaSuccess) return e;
    image_ffn_kernel<<<img_grid(((long long)W * H + 3) / 4), kImgBlock, 0, stream>>>(
        image, mask, W, H, delta, key0, key1, (unsigned long long)sample, out2);
    return cudaGetLastError();
}

}  // namespace klmc
