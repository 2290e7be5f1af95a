// Ingest transpose: time-major 8-bit samples [N][C] (the order of PSRFITS
// files and of Alg. 2's numpts x numchan input matrix, Sec. 2.3) into the
// channel-major [C][N] layout the dedispersion kernels read.  HBM-bound: one
// read and one write per byte.  Rows of the output that are 16-byte aligned take
// ingest_transpose16_kernel, whatever the input's alignment; others a kernel of
// 64 x 64 byte tiles with 4-byte or byte accesses.
#include "gsp_internal.cuh"

namespace {

constexpr int kTile = 64;
__global__ void __launch_bounds__(256) ingest_transpose_kernel(const uint8_t *__restrict__ in,
                                                               int64_t in_stride, int64_t N, int C,
                                                               uint8_t *__restrict__ out,
                                                               int64_t out_stride, bool words) {
    __shared__ uint8_t tile[kTile][kTile + 4];
    const int64_t t0 = (int64_t)blockIdx.x * kTile;   // time
    const int c0 = blockIdx.y * kTile;                // channel
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;  // 16 x 16 threads
    // load: rows are times, 4 channels per thread
    for (int r = ty; r < kTile; r += 16) {
        const int64_t t = t0 + r;
        const int c = c0 + 4 * tx;
        uint32_t v = 0;
        if (t < N) {
            const uint8_t *src = in + t * in_stride + c;
            if (words && c + 3 < C) {
                v = __ldg(reinterpret_cast<const uint32_t *>(src));
            } else {
                for (int k = 0; k < 4; k++)
                    if (c + k < C) v |= (uint32_t)__ldg(src + k) << (8 * k);
            }
        }
        tile[r][4 * tx + 0] = (uint8_t)v;
        tile[r][4 * tx + 1] = (uint8_t)(v >> 8);
        tile[r][4 * tx + 2] = (uint8_t)(v >> 16);
        tile[r][4 * tx + 3] = (uint8_t)(v >> 24);
    }
    __syncthreads();
    // store: rows are channels, 4 times per thread
    for (int r = ty; r < kTile; r += 16) {
        const int c = c0 + r;
        if (c >= C) continue;
        const int64_t t = t0 + 4 * tx;
        const uint32_t v = (uint32_t)tile[4 * tx + 0][r] | ((uint32_t)tile[4 * tx + 1][r] << 8) |
                           ((uint32_t)tile[4 * tx + 2][r] << 16) |
                           ((uint32_t)tile[4 * tx + 3][r] << 24);
        uint8_t *dst = out + (int64_t)c * out_stride + t;
        if (words && t + 3 < N) {
            *reinterpret_cast<uint32_t *>(dst) = v;
        } else {
            for (int k = 0; k < 4; k++)
                if (t + k < N) dst[k] = (uint8_t)(v >> (8 * k));
        }
    }
}

// The same with 16-byte stores (output pointer and stride 16-byte aligned) on 256
// (time) x 64 (channel) tiles.  Thread (r, q) loads bytes
// [16q, 16q + 16) of time rows 4r .. 4r + 3 and transposes their 4 x 4 byte blocks in
// registers (8 byte permutes per 16 bytes): 16 words of four samples, one per
// channel, into the shared tile [channel][time].  Each half warp then reads 256
// samples of a channel as 16-byte words and stores them, 256 contiguous bytes.
// The tile's word column is XORed with 8 times the channel group, which keeps both
// sides free of bank conflicts.  About 1.1 instructions per byte (four when each
// byte was gathered from shared memory on its own).  4096 x 262144 samples: 466 -> 349 us
// with nothing of them in L2, 320 with the order of tiles below (6.7 TB/s of the 6.8 measured).
// Edge tiles fall back to byte accesses.
// kVec: the input pointer and stride are 16-byte aligned too, and a thread's 16 bytes
// are one load.  Otherwise they are five aligned words shifted into place, where those
// words lie inside the matrix, or bytes (706 x 110948 samples with rows of 710 bytes:
// 95 us in the kernel of byte accesses above, 44 here; 4099-byte rows of 4096 channels,
// 262144 samples: 1060, 470).
//
// A tile is 64 channels wide, half of a 128-byte line of the input.  Tiles are
// therefore visited in groups of kGroup channel tiles side by side before the next
// time tile: with all time tiles of one channel tile first, every line comes from
// memory in two halves at different times (4096 x 2^20 samples, one / two / four /
// eight / all side by side: 2076 / 1377 / 1368 / 1376 / 1377 us; output rows of 2^20 + 16
// bytes: 2151 / 1491 / 1490 / 1508 / 1548).  Not so in the kernel above, whose stores of
// 64 bytes are the half lines (4096 x 262144, output rows of 262148 bytes: 734 us in
// time order, 830 in groups).
constexpr int kTileT16 = 256;
constexpr unsigned kGroup = 4;

// Tile of this CTA: grid (time tiles, channel tiles), renumbered within each kGroup
// rows of the grid.  32 bits hold the number: more than 2^30 time tiles and more than
// one channel tile would be over 2^42 bytes.
__device__ __forceinline__ void tile_of(unsigned *tt, unsigned *ct) {
    const unsigned c0 = blockIdx.y / kGroup * kGroup, g = min(kGroup, gridDim.y - c0);
    const unsigned k = (blockIdx.y - c0) * gridDim.x + blockIdx.x;
    *tt = k / g;
    *ct = c0 + k % g;
}

// 16 bytes at src from aligned words; false where one would reach outside [lo, hi).
__device__ __forceinline__ bool load16_shifted(const uint8_t *src, const uint8_t *lo,
                                               const uint8_t *hi, uint32_t (&v)[4]) {
    const unsigned sh = (unsigned)((uintptr_t)src & 3);
    const uint8_t *a = src - sh;
    if (a < lo || a + (sh ? 20 : 16) > hi) return false;
    uint32_t w[5];
#pragma unroll
    for (int k = 0; k < 4; k++) w[k] = __ldg(reinterpret_cast<const uint32_t *>(a) + k);
    w[4] = sh ? __ldg(reinterpret_cast<const uint32_t *>(a) + 4) : 0u;
#pragma unroll
    for (int k = 0; k < 4; k++) v[k] = __funnelshift_r(w[k], w[k + 1], 8 * sh);
    return true;
}

template <bool kVec>
__global__ void __launch_bounds__(256) ingest_transpose16_kernel(const uint8_t *__restrict__ in,
                                                                 int64_t in_stride, int64_t N,
                                                                 int C, uint8_t *__restrict__ out,
                                                                 int64_t out_stride) {
    __shared__ __align__(16) uint32_t tile[kTile][kTileT16 / 4];
    unsigned tt, ct;
    tile_of(&tt, &ct);
    const int64_t t0 = (int64_t)tt * kTileT16;
    const int c0 = (int)ct * kTile;
    {
        const int q = threadIdx.x & 3, r = threadIdx.x >> 2;
        const int c = c0 + 16 * q;
        uint32_t v[4][4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int64_t t = t0 + 4 * r + i;
            const uint8_t *src = in + t * in_stride + c;
            v[i][0] = v[i][1] = v[i][2] = v[i][3] = 0u;
            if (t < N) {
                bool done = false;
                if (c + 15 < C) {
                    if (kVec) {
                        const uint4 x = __ldcs(reinterpret_cast<const uint4 *>(src));
                        v[i][0] = x.x;
                        v[i][1] = x.y;
                        v[i][2] = x.z;
                        v[i][3] = x.w;
                        done = true;
                    } else {
                        done = load16_shifted(src, in, in + (N - 1) * in_stride + C, v[i]);
                    }
                }
                if (!done) {
#pragma unroll
                    for (int k = 0; k < 16; k++)
                        if (c + k < C) v[i][k >> 2] |= (uint32_t)__ldg(src + k) << (8 * (k & 3));
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint32_t lo01 = __byte_perm(v[0][k], v[1][k], 0x5140), lo23 = __byte_perm(v[2][k], v[3][k], 0x5140);
            const uint32_t hi01 = __byte_perm(v[0][k], v[1][k], 0x7362), hi23 = __byte_perm(v[2][k], v[3][k], 0x7362);
            const int col = r ^ (8 * q);
            tile[16 * q + 4 * k + 0][col] = __byte_perm(lo01, lo23, 0x5410);
            tile[16 * q + 4 * k + 1][col] = __byte_perm(lo01, lo23, 0x7632);
            tile[16 * q + 4 * k + 2][col] = __byte_perm(hi01, hi23, 0x5410);
            tile[16 * q + 4 * k + 3][col] = __byte_perm(hi01, hi23, 0x7632);
        }
    }
    __syncthreads();
    const int m = threadIdx.x & 15;        // 16-sample group inside the tile
    const int64_t t = t0 + 16 * m;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const int cl = (threadIdx.x >> 4) + 16 * j;  // channel inside the tile
        const int c = c0 + cl;
        if (c >= C) continue;
        const uint4 w = *reinterpret_cast<const uint4 *>(&tile[cl][(4 * m) ^ (8 * (cl >> 4))]);
        uint8_t *dst = out + (int64_t)c * out_stride + t;
        if (t + 15 < N) {
            __stcs(reinterpret_cast<uint4 *>(dst), w);
        } else {
            const uint32_t b[4] = {w.x, w.y, w.z, w.w};
            for (int k = 0; k < 16; k++)
                if (t + k < N) dst[k] = (uint8_t)(b[k >> 2] >> (8 * (k & 3)));
        }
    }
}

}  // namespace

extern "C" gsp_status gsp_ingest_transpose(const uint8_t *d_in, int64_t n_samp, int32_t nchan,
                                           int64_t in_stride, uint8_t *d_out, int64_t out_stride,
                                           void *stream) {
    if (!d_in || !d_out || n_samp < 0 || nchan <= 0 || in_stride < nchan || out_stride < n_samp)
        return GSP_ERR_INVALID_ARG;
    if (n_samp == 0) return GSP_OK;
    const int64_t tiles_t = (n_samp + kTile - 1) / kTile;
    const int tiles_c = (nchan + kTile - 1) / kTile;
    if (tiles_c > 65535 || tiles_t > 0x7fffffffll) return GSP_ERR_INVALID_ARG;
    const bool words = ((((uintptr_t)d_in | (uintptr_t)d_out) & 3) == 0) && (in_stride % 4 == 0) &&
                       (out_stride % 4 == 0);
    dim3 grid((unsigned)tiles_t, (unsigned)tiles_c);
    const bool out16 = ((uintptr_t)d_out & 15) == 0 && out_stride % 16 == 0;
    const bool in16 = ((uintptr_t)d_in & 15) == 0 && in_stride % 16 == 0;
    dim3 grid16((unsigned)((n_samp + kTileT16 - 1) / kTileT16), (unsigned)tiles_c);
    if (out16 && in16)
        ingest_transpose16_kernel<true><<<grid16, 256, 0, (cudaStream_t)stream>>>(
            d_in, in_stride, n_samp, nchan, d_out, out_stride);
    else if (out16)
        ingest_transpose16_kernel<false><<<grid16, 256, 0, (cudaStream_t)stream>>>(
            d_in, in_stride, n_samp, nchan, d_out, out_stride);
    else
        ingest_transpose_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(d_in, in_stride, n_samp,
                                                                        nchan, d_out, out_stride,
                                                                        words);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        gsp::record_error(e, "ingest transpose launch");
        return GSP_ERR_CUDA;
    }
    return GSP_OK;
}
