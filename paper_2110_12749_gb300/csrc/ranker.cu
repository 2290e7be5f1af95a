// Candidate ranker: a small CNN over 64 x 64 DM-time snippets of the
// single-pulse candidates, trained and run on the GPU (the project's own
// design for the candidate-ranking step the paper motivates, Sec. 1-2: it
// ranks the plain threshold output, never replaces it).
//
// Network: three conv 3x3 (pad 1) + bias + ReLU + 2x2 max-pool layers
// (1 -> 8 -> 16 -> 32 channels, 64x64 -> 8x8), fc 2048 -> 96 + ReLU, fc 96 -> 2.
// Activations are NHWC.  Each conv layer is one kernel with its bias, ReLU and
// pool: layer 0 (one input channel, K = 9) on the CUDA cores, layers 1 and 2 as
// implicit GEMMs on the tcgen05 tensor cores (BF16 operands, FP32 accumulation in
// tensor memory) that gather their taps straight from the activations; the same
// kernels run a training pass and then also keep the ReLU outputs and the pool's
// argmaxes.  Back-propagation: input gradients of layers 1 and 2 by the same implicit
// GEMM with mirrored taps; conv weight gradients on the CUDA cores from the pooled
// gradients (one nonzero per pooling window); both products of fc 2048 -> 96 by the
// tcgen05 GEMM (tc_gemm.cu).  The 96 -> 2 layer, the loss, the pool's way back,
// bias gradients and Adam are elementwise kernels in FP32.  Every operand of a
// product is rounded to bf16 (nearest even), at the same points as the CPU oracle.
// A training step at 256 snippets takes 230 us (im2col matrices, their transposes
// and GEMMs for every product: 860 us).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "dd_tiled.cuh"
#include "gsp_internal.cuh"
#include "tc_gemm.cuh"

namespace {

using bf16 = __nv_bfloat16;

constexpr int kS = 64;          // snippet side
constexpr int kFc = 2048;       // 32 x 8 x 8 features
constexpr int kHid = 96;        // hidden units of fc1 (202,786 parameters in all)
constexpr int kFc1Split = 8;    // most K chunks of fc1 (K = 2048: 32 steps of 64)
constexpr int kLayers = 3;
// per conv layer: input channels, output channels, input side
__host__ __device__ constexpr int cin_of(int l) { return l == 0 ? 1 : (l == 1 ? 8 : 16); }
__host__ __device__ constexpr int cout_of(int l) { return l == 0 ? 8 : (l == 1 ? 16 : 32); }
__host__ __device__ constexpr int side_of(int l) { return l == 0 ? 64 : (l == 1 ? 32 : 16); }

__host__ __device__ constexpr int round8(int v) { return (v + 7) & ~7; }
__host__ __device__ constexpr int kdim(int l) { return 9 * cin_of(l); }         // im2col K
__host__ __device__ constexpr int kpad(int l) { return round8(kdim(l)); }
constexpr int kSms = 152;      // SMs of a GB300: loops over the grid are sized for them
constexpr int kGradRows = 16;  // rows of the input-gradient weights (at least Cin of layers 1, 2)

// Parameter offsets in the flat FP32 vector (order w1 b1 w2 b2 w3 b3 w4 b4 w5 b5,
// each in the oracle's layout: conv w[co][ci][ky][kx], fc w[out][in]).
struct Offsets {
    int64_t w[5], b[5], total;
};
constexpr int kWsize[5] = {8 * 1 * 9, 16 * 8 * 9, 32 * 16 * 9, kHid * kFc, 2 * kHid};
constexpr int kBsize[5] = {8, 16, 32, kHid, 2};
Offsets offsets() {
    Offsets o{};
    int64_t p = 0;
    for (int i = 0; i < 5; i++) {
        o.w[i] = p;
        p += kWsize[i];
        o.b[i] = p;
        p += kBsize[i];
    }
    o.total = p;
    return o;
}

// ------------------------------------------------------------- elementwise

// fma(a, b.x, c.x), fma(a, b.y, c.y) as one packed instruction (two IEEE
// single-precision FMAs, the same results as two fmaf): half the issue slots
__device__ __forceinline__ float2 fma_pair(float a, float2 b, float2 c) {
    uint64_t av, bv, cv, d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(av) : "f"(a));
    asm("mov.b64 %0, {%1, %2};" : "=l"(bv) : "f"(b.x), "f"(b.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(cv) : "f"(c.x), "f"(c.y));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(av), "l"(bv), "l"(cv));
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(d));
    return r;
}

// Layer 0: conv 3x3 (1 -> 8, pad 1) + bias + ReLU + 2x2 max-pool straight from
// the FP32 snippets, on the CUDA cores: with one input channel the product has
// K = 9, too short for the tensor pipe to pay for its staging.  Rounding points:
// inputs and weights in bf16, the nine products and the bias summed in FP32, the
// pooled maximum rounded to bf16.  One thread per pair of horizontally adjacent
// pooled pixels reads its 4 x 6 input patch; per channel pair it loads the nine
// weights once and computes the 2 x 4 conv outputs (channels 2p and 2p + 1 share
// each packed FMA), then writes the two pixels' 8 bf16 results as two 16-byte
// stores (NHWC).  For inference; a training pass, which keeps the pre-pool values, runs
// conv0_train_tc_kernel.
__global__ void __launch_bounds__(256) conv0_pool_kernel(const float *__restrict__ x, int B,
                                                         const bf16 *__restrict__ W0,
                                                         const float *__restrict__ b0,
                                                         bf16 *__restrict__ a0) {
    constexpr int C = 8, KP = kpad(0), H = kS, H2 = kS / 2, HP = H2 / 2;
    __shared__ float2 sw[C / 2][9];  // channels 2p and 2p + 1 side by side
    __shared__ float2 sb[C / 2];
    for (int i = threadIdx.x; i < C * 9; i += blockDim.x) {
        const float w = __bfloat162float(W0[(i / 9) * KP + i % 9]);
        if ((i / 9) & 1) sw[i / 18][i % 9].y = w;
        else sw[i / 18][i % 9].x = w;
    }
    for (int i = threadIdx.x; i < C; i += blockDim.x) {
        if (i & 1) sb[i / 2].y = b0[i];
        else sb[i / 2].x = b0[i];
    }
    __syncthreads();
    const int64_t total = (int64_t)B * H2 * HP;  // pixel pairs
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = q / (H2 * HP);
        const int rem = (int)(q - b * H2 * HP);
        const int y2 = rem / HP, x2 = 2 * (rem - (rem / HP) * HP);  // first pooled column
        const float *img = x + b * H * H;
        float v[4][6];
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int yy = 2 * y2 - 1 + r;
#pragma unroll
            for (int c = 0; c < 6; c++) {
                const int xx = 2 * x2 - 1 + c;
                const bool in = yy >= 0 && yy < H && xx >= 0 && xx < H;
                v[r][c] = in ? __bfloat162float(__float2bfloat16_rn(__ldg(img + yy * H + xx)))
                             : 0.0f;
            }
        }
        __align__(16) bf16 out[2][C];
#pragma unroll
        for (int cp = 0; cp < C / 2; cp++) {  // channels 2 cp and 2 cp + 1 together
            float2 w[9];
#pragma unroll
            for (int k = 0; k < 9; k++) w[k] = sw[cp][k];
            const float2 bias = sb[cp];
#pragma unroll
            for (int px = 0; px < 2; px++) {
                float m0 = 0.0f, m1 = 0.0f;  // ReLU outputs are >= 0
#pragma unroll
                for (int dy = 0; dy < 2; dy++)
#pragma unroll
                    for (int dx = 0; dx < 2; dx++) {
                        float2 z = make_float2(0.0f, 0.0f);
#pragma unroll
                        for (int ky = 0; ky < 3; ky++)
#pragma unroll
                            for (int kx = 0; kx < 3; kx++)
                                z = fma_pair(v[dy + ky][2 * px + dx + kx], w[ky * 3 + kx], z);
                        m0 = fmaxf(m0, z.x + bias.x);
                        m1 = fmaxf(m1, z.y + bias.y);
                    }
                out[px][2 * cp] = __float2bfloat16_rn(m0);
                out[px][2 * cp + 1] = __float2bfloat16_rn(m1);
            }
        }
        const int64_t pix = (b * H2 + y2) * H2 + x2;
        *reinterpret_cast<uint4 *>(a0 + pix * C) = *reinterpret_cast<const uint4 *>(out[0]);
        *reinterpret_cast<uint4 *>(a0 + (pix + 1) * C) = *reinterpret_cast<const uint4 *>(out[1]);
    }
}

// Back through the pool and the ReLU: g[b][y][x][c] = ga[b][y/2][x/2][c] if (y, x)
// is the window's argmax and its pooled value a > 0, else 0, as bf16 [P][C]
// (P = B*H*H pixels); adds FP32 per-channel sums into db.  One thread per pooled
// pixel and 8 channels: it reads the gradient, argmax and pooled value once
// and writes the window's four pixels, 16 bytes each.  (A thread per pre-pool
// element that also scattered a transpose took 65 us per layer at 256 snippets.)
template <int C>
__global__ void __launch_bounds__(256) pool_back_kernel(const float *__restrict__ ga,
                                                        const uint8_t *__restrict__ idx,
                                                        const bf16 *__restrict__ a, int B, int H,
                                                        bf16 *__restrict__ g, float *__restrict__ db) {
    constexpr int G = C / 8;  // channel groups; 256 and the grid's stride are multiples of it
    __shared__ float sdb[C];
    for (int c = threadIdx.x; c < C; c += blockDim.x) sdb[c] = 0.0f;
    __syncthreads();
    const int H2 = H / 2;
    const int64_t total = (int64_t)B * H2 * H2 * G;
    float sum[8];
#pragma unroll
    for (int e = 0; e < 8; e++) sum[e] = 0.0f;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = i / G;
        const int c8 = (int)(i - q * G);
        const int64_t b = q / (H2 * H2);
        const int rem = (int)(q - b * H2 * H2);
        const int y2 = rem / H2, x2 = rem - (rem / H2) * H2;
        const float4 f0 = __ldg(reinterpret_cast<const float4 *>(ga + q * C) + 2 * c8);
        const float4 f1 = __ldg(reinterpret_cast<const float4 *>(ga + q * C) + 2 * c8 + 1);
        const uint2 k = __ldg(reinterpret_cast<const uint2 *>(idx + q * C) + c8);
        const uint4 av = __ldg(reinterpret_cast<const uint4 *>(a + q * C) + c8);
        const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
        const uint32_t ab[4] = {av.x, av.y, av.z, av.w};
        __align__(16) bf16 o[4][8];
#pragma unroll
        for (int e = 0; e < 8; e++) {
            // pooled values are >= 0: positive when any of their bits are set
            const bool pos = ((ab[e >> 1] >> (16 * (e & 1))) & 0x7fffu) != 0u;
            const float v = pos ? f[e] : 0.0f;
            const uint32_t at = ((e < 4 ? k.x : k.y) >> (8 * (e & 3))) & 0xffu;
            sum[e] += v;
            const bf16 w = __float2bfloat16_rn(v), zero = __float2bfloat16_rn(0.0f);
#pragma unroll
            for (int p = 0; p < 4; p++) o[p][e] = at == (uint32_t)p ? w : zero;
        }
#pragma unroll
        for (int p = 0; p < 4; p++)
            *reinterpret_cast<uint4 *>(g + ((b * H + 2 * y2 + p / 2) * H + 2 * x2 + p % 2) * C + 8 * c8) =
                *reinterpret_cast<const uint4 *>(o[p]);
    }
#pragma unroll
    for (int e = 0; e < 8; e++) {
        // lanes of the same channel group are G apart
        for (int o = 16; o >= G; o >>= 1) sum[e] += __shfl_xor_sync(0xffffffffu, sum[e], o);
        if ((threadIdx.x & 31) < G) atomicAdd(&sdb[8 * (threadIdx.x & (G - 1)) + e], sum[e]);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < C; c += blockDim.x)
        if (sdb[c] != 0.0f) atomicAdd(&db[c], sdb[c]);
}

// Weight gradient of a conv layer, dw[co][ci][ky][kx] += sum over the pixels of
// gz[p][co] * act[p + (ky - 1, kx - 1)][ci], from the pooled gradient: a pooling
// window has one nonzero gz per channel, at its argmax, so a quarter of the
// products of the dense sum do.  A CTA stages a strip of its image's activation (bf16 with
// a zero border; layer 0: the FP32 snippet rounded here) and its windows' bf16
// gradients; a thread owns output channel co and CP input channels and
// keeps their 9 CP sums in registers over all its windows.  Operands in bf16,
// exact products, FP32 sums, added atomically at the end.  Bound by the shared loads
// (one per tap and window).  Replaces an im2col, two transposes and a split-K
// GEMM whose 128-row tiles held 8 to 32 rows of work.
template <typename T, int CIN, int COUT, int SIDE>
__global__ void __launch_bounds__(256) conv_dw_kernel(const T *__restrict__ act, int B,
                                                      const float *__restrict__ ga,
                                                      const uint8_t *__restrict__ idx,
                                                      const bf16 *__restrict__ a,
                                                      float *__restrict__ dw) {
    constexpr int CP = CIN == 1 ? 1 : 2;               // input channels per thread
    constexpr int kOwn = COUT * (CIN / CP);            // threads that cover the weights
    constexpr int kSets = 256 / kOwn;                  // sets of them, sharing the windows
    static_assert(256 % kOwn == 0, "whole sets");
    constexpr int kStrips = SIDE / 16;                 // strips of 16 image rows per image
    constexpr int kRows = 18, kPitch = SIDE + 2;       // a strip with its border
    constexpr int PW = SIDE / 2, kWin = 8 * PW;        // pooling windows per strip
    __shared__ __align__(16) bf16 sa[kRows * kPitch * CIN + 8];
    __shared__ float sg[kWin * COUT];
    const int tid = threadIdx.x, set = tid / kOwn, own = tid % kOwn;
    const int co = own / (CIN / CP), cp = own % (CIN / CP);
    float acc[9][CP];
#pragma unroll
    for (int t = 0; t < 9; t++)
#pragma unroll
        for (int e = 0; e < CP; e++) acc[t][e] = 0.0f;
    for (int64_t u = blockIdx.x; u < (int64_t)B * kStrips; u += gridDim.x) {
        const int64_t b = u / kStrips;
        const int y0 = (int)(u - b * kStrips) * 16;  // first image row of the strip
        __syncthreads();
        for (int i = tid; i < kRows * kPitch; i += 256) {
            const int r = i / kPitch, c = i - r * kPitch;
            const int yy = y0 + r - 1, xx = c - 1;
            const bool in = yy >= 0 && yy < SIDE && xx >= 0 && xx < SIDE;
            const T *src = act + ((b * SIDE + (in ? yy : 0)) * SIDE + (in ? xx : 0)) * CIN;
            if constexpr (CIN % 8 == 0) {
#pragma unroll
                for (int c8 = 0; c8 < CIN / 8; c8++) {
                    uint4 v = make_uint4(0u, 0u, 0u, 0u);
                    if (in) v = __ldg(reinterpret_cast<const uint4 *>(src) + c8);
                    *reinterpret_cast<uint4 *>(&sa[i * CIN + 8 * c8]) = v;
                }
            } else {
                sa[i] = __float2bfloat16_rn(in ? (float)__ldg(src) : 0.0f);
            }
        }
        // the windows' gradients, their argmax in the two lowest bits (the values are
        // bf16: those bits are free in FP32)
        const int64_t q0 = (b * PW + y0 / 2) * PW;
        for (int i = tid; i < kWin * COUT; i += 256) {
            const int64_t o = q0 * COUT + i;
            const bool pos = __bfloat162float(a[o]) > 0.0f;
            const float v = __bfloat162float(__float2bfloat16_rn(pos ? __ldg(ga + o) : 0.0f));
            sg[i] = __uint_as_float(__float_as_uint(v) | (uint32_t)(idx[o] & 3u));
        }
        __syncthreads();
        for (int w = set; w < kWin; w += kSets) {
            const uint32_t bits = __float_as_uint(sg[w * COUT + co]);
            if ((bits & 0x7ffffff0u) == 0u) continue;
            const float gv = __uint_as_float(bits & ~3u);
            const int wy = w / PW, wx = w % PW;
            const int base = ((2 * wy + (int)((bits >> 1) & 1u)) * kPitch + 2 * wx + (int)(bits & 1u)) * CIN +
                             cp * CP;
#pragma unroll
            for (int t = 0; t < 9; t++) {
                const bf16 *p = &sa[base + ((t / 3) * kPitch + t % 3) * CIN];
                if constexpr (CP == 2) {
                    const uint32_t v = *reinterpret_cast<const uint32_t *>(p);
                    acc[t][0] = fmaf(gv, __uint_as_float(v << 16), acc[t][0]);
                    acc[t][CP - 1] = fmaf(gv, __uint_as_float(v & 0xffff0000u), acc[t][CP - 1]);
                } else {
                    acc[t][0] = fmaf(gv, __bfloat162float(*p), acc[t][0]);
                }
            }
        }
    }
    // the sets' sums, then one atomic per weight and CTA
    __shared__ float red[COUT * CIN * 9];
    for (int i = tid; i < COUT * CIN * 9; i += 256) red[i] = 0.0f;
    __syncthreads();
    {
#pragma unroll
        for (int t = 0; t < 9; t++)
#pragma unroll
            for (int e = 0; e < CP; e++) atomicAdd(&red[(co * CIN + cp * CP + e) * 9 + t], acc[t][e]);
    }
    __syncthreads();
    for (int i = tid; i < COUT * CIN * 9; i += 256) atomicAdd(&dw[i], red[i]);
}

// bf16 transpose: out[c][r] = in[r][c] for r < R, c < Cc (32 x 32 tiles).
__global__ void transpose_kernel(const bf16 *__restrict__ in, int64_t ldi, int64_t R, int Cc,
                                 bf16 *__restrict__ out, int64_t ldo) {
    __shared__ bf16 t[32][33];
    const int64_t r0 = (int64_t)blockIdx.x * 32;
    const int c0 = blockIdx.y * 32;
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const int64_t r = r0 + k;
        const int c = c0 + threadIdx.x;
        t[k][threadIdx.x] = (r < R && c < Cc) ? in[r * ldi + c] : __float2bfloat16_rn(0.0f);
    }
    __syncthreads();
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const int c = c0 + k;
        const int64_t r = r0 + threadIdx.x;
        if (c < Cc && r < R) out[(int64_t)c * ldo + r] = t[threadIdx.x][k];
    }
}

// fc 96 -> 2 (CUDA cores): z5[b][o] = sum_k a4[b][k] * bf16(w5[o][k]) + b5[o].
__global__ void fc2_kernel(const bf16 *__restrict__ a4, const float *__restrict__ w5,
                           const float *__restrict__ b5, int B, float *__restrict__ z5) {
    gsp::wait_prior_grid();  // a4 comes from the kernel launched just before
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B * 2) return;
    const int b = i / 2, o = i % 2;
    float s = 0.0f;
    for (int k = 0; k < kHid; k++)
        s = fmaf((float)a4[b * kHid + k], __bfloat162float(__float2bfloat16_rn(w5[o * kHid + k])), s);
    z5[i] = s + b5[o];
}

// Mean softmax cross-entropy and its gradient g5 = (softmax - onehot) / B, one
// block; loss_out (optional) receives the mean loss.
__global__ void loss_kernel(const float *__restrict__ z5, const int32_t *__restrict__ y, int B,
                            float *__restrict__ g5, float *__restrict__ loss_out) {
    __shared__ float red[256];
    float acc = 0.0f;
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
        const float z0 = z5[2 * b], z1 = z5[2 * b + 1];
        const float m = fmaxf(z0, z1);
        const float e0 = expf(z0 - m), e1 = expf(z1 - m);
        const float s = e0 + e1;
        const int lab = y[b] ? 1 : 0;
        acc += -logf((lab ? e1 : e0) / s);
        g5[2 * b] = (e0 / s - (lab == 0 ? 1.0f : 0.0f)) / (float)B;
        g5[2 * b + 1] = (e1 / s - (lab == 1 ? 1.0f : 0.0f)) / (float)B;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0 && loss_out) *loss_out = red[0] / (float)B;
}

// Back through fc 96 -> 2 and the ReLU of fc1 (CUDA cores):
//   dw5[o][k] += sum_b bf16(g5[b][o]) * a4[b][k],  db5[o] += sum_b g5[b][o]
//   g4[b][k]  = (sum_o bf16(g5[b][o]) * bf16(w5[o][k])) * [z4[b][k] > 0]
// g4 is written as bf16 [B][96] and transposed [96][ldT]; db4 += FP32 sums.  The
// blocks take the snippets in turn and add their sums atomically (one block summing
// dw5 over the whole batch took 39 us at 256 snippets).
__global__ void fc2_back_kernel(const float *__restrict__ g5, const bf16 *__restrict__ a4,
                                const float *__restrict__ w5, const float *__restrict__ z4,
                                int B, float *__restrict__ dw5, float *__restrict__ db5,
                                bf16 *__restrict__ g4, bf16 *__restrict__ g4T, int64_t ldT,
                                float *__restrict__ db4) {
    const int k = threadIdx.x;  // kHid threads: one hidden unit each
    const float w0 = __bfloat162float(__float2bfloat16_rn(w5[k]));
    const float w1 = __bfloat162float(__float2bfloat16_rn(w5[kHid + k]));
    float s0 = 0.0f, s1 = 0.0f, t0 = 0.0f, t1 = 0.0f, dsum = 0.0f;
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        const float2 g = __ldg(reinterpret_cast<const float2 *>(g5) + b);
        const float h0 = __bfloat162float(__float2bfloat16_rn(g.x));
        const float h1 = __bfloat162float(__float2bfloat16_rn(g.y));
        const float act = (float)a4[b * kHid + k];
        s0 = fmaf(h0, act, s0);
        s1 = fmaf(h1, act, s1);
        t0 += g.x;
        t1 += g.y;
        const float v = z4[b * kHid + k] > 0.0f ? h0 * w0 + h1 * w1 : 0.0f;
        g4[b * kHid + k] = __float2bfloat16_rn(v);
        g4T[(int64_t)k * ldT + b] = __float2bfloat16_rn(v);
        dsum += v;
    }
    atomicAdd(&dw5[k], s0);
    atomicAdd(&dw5[kHid + k], s1);
    atomicAdd(&db4[k], dsum);
    if (k == 0) {
        atomicAdd(&db5[0], t0);
        atomicAdd(&db5[1], t1);
    }
}

// Adam on the flat FP32 parameter vector (step number t >= 1).
__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g,
                            float *__restrict__ m, float *__restrict__ v, int64_t n, float lr,
                            float b1, float b2, float eps, float c1, float c2) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// bf16 copies of the weights: conv W[co][(ky*3+kx)*Cin + ci] (padded to Kp) from
// w[co][ci][ky][kx]; for the input gradients of layers 1 and 2 the product's other side,
// WG[ci][(ky*3+kx)*Cout + co] (16 rows, zero past Cin); and the fc1 weight W4
// [96][2048] with its transpose W4T [2048][96].
__global__ void pack_kernel(const float *__restrict__ params, int64_t w1, int64_t w2, int64_t w3,
                            int64_t w4, bf16 *__restrict__ W0, bf16 *__restrict__ W1,
                            bf16 *__restrict__ W2, bf16 *__restrict__ WG1, bf16 *__restrict__ WG2,
                            bf16 *__restrict__ W4, bf16 *__restrict__ W4T) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < (int64_t)kHid * kFc) {
        const bf16 v = __float2bfloat16_rn(params[w4 + i]);
        W4[i] = v;
        W4T[(i % kFc) * kHid + i / kFc] = v;
    }
    const int64_t woff[3] = {w1, w2, w3};
    bf16 *Wd[3] = {W0, W1, W2};
    bf16 *WGd[3] = {nullptr, WG1, WG2};
#pragma unroll
    for (int l = 0; l < kLayers; l++) {
        const int Cin = cin_of(l), Cout = cout_of(l), Kp = kpad(l);
        if (i < (int64_t)Cout * Kp) {
            const int co = (int)(i / Kp), k = (int)(i % Kp);
            float v = 0.0f;
            if (k < 9 * Cin) {
                const int tap = k / Cin, ci = k % Cin;
                v = params[woff[l] + ((int64_t)co * Cin + ci) * 9 + tap];
            }
            Wd[l][i] = __float2bfloat16_rn(v);
        }
        if (l > 0 && i < (int64_t)kGradRows * 9 * Cout) {
            const int ci = (int)(i / (9 * Cout)), k = (int)(i % (9 * Cout));
            const int tap = k / Cout, co = k % Cout;
            WGd[l][i] = __float2bfloat16_rn(ci < Cin ? params[woff[l] + ((int64_t)co * Cin + ci) * 9 + tap] : 0.0f);
        }
    }
}

}  // namespace

namespace {

// fc1's epilogue after a split-K product: z4 = ReLU(sum over the S partial
// products, in chunk order, + bias) and a4 = bf16(z4).  One thread per output.
__global__ void fc1_finish_kernel(const float *__restrict__ part, int S, int64_t zstride, int B,
                                  const float *__restrict__ bias, float *__restrict__ z4,
                                  bf16 *__restrict__ a4) {
    gsp::wait_prior_grid();  // part comes from the kernel launched just before
    const int64_t total = (int64_t)B * kHid;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        float acc = part[i];
        for (int z = 1; z < S; z++) acc += part[(int64_t)z * zstride + i];
        const float v = fmaxf(acc + bias[i % kHid], 0.0f);
        z4[i] = v;
        a4[i] = __float2bfloat16_rn(v);
    }
}

// ------------------------------------------- fused conv layers for inference

namespace tc = gsp::tc;
namespace ptx = gsp::ptx;

constexpr long long kConvBudget = 2000000000ll;  // ~1 s of SM clock per wait

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
                 "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Layers 1 and 2 of an inference pass: conv 3x3 (CIN -> COUT, pad 1) as an
// implicit GEMM on the tcgen05 tensor cores, + bias + ReLU + 2x2 max-pool in
// the epilogue, from the bf16 NHWC activation act [B][SIDE][SIDE][CIN] to the
// pooled bf16 NHWC output out [B][SIDE/2][SIDE/2][COUT].  The products and
// their rounding points are those of the im2col + GEMM + pool path (the same
// K order and K = 16 steps, FP32 accumulation in tensor memory, bias after
// the accumulation, the pooled maximum rounded to bf16).
//
// Persistent CTAs of 4 warps stride over 128-pixel M tiles (a tile is 128 /
// SIDE whole image rows, so every 2x2 pooling window lies inside it).  Each
// thread gathers the 9 taps of its pixel straight from act with 16-byte
// cp.async copies (zero-filled outside the image) into the K-major
// core-matrix layout; the weights are staged once per CTA.  One A buffer and
// one accumulator per CTA, so that many CTAs fit an SM.  Per tile: wait for
// the gather, MMAs, wait for them; then the next tile's gather runs under
// this tile's epilogue, which pools mostly in registers:
//  * SIDE 16: a tile is 8 image rows, warp w holding rows 2w and 2w + 1
//    (lane l: row 2w + l / 16, column l % 16), so each pooling window lies in
//    one warp: two shuffles (partners l ^ 1 and l ^ 16).
//  * SIDE 32: a tile is 4 image rows, warp w holding row w: a shuffle pools
//    column pairs (l ^ 1), and warps 1 and 3 hand their row maxima to warps 0
//    and 2 through a 2 KB shared buffer.
// Every wait is bounded; on a timeout the kernel sets *err, waits (bounded)
// for its MMAs in flight and releases its tensor memory.
//
// kMode: kInfer as above; kTrain also stores the ReLU outputs z (FP32
// [B][SIDE][SIDE][COUT]) and the pool's argmax idx (first maximum in (0,0),
// (0,1), (1,0), (1,1) order); kGrad is the input gradient of such a layer: act
// is the gradient of its pre-activations, the taps are mirrored, each tap's product
// has its own accumulator (16 columns) and the nine are added in tap order, and the sums
// are stored as FP32 z_out [B][SIDE][SIDE][nz] (nz <= 16 channels) without bias, ReLU
// and pool.
enum ConvMode { kInfer, kTrain, kGrad };

// Tensor-memory columns of a CTA (a power of two, at least 32).
__host__ __device__ constexpr uint32_t conv_tmem_cols(int cout, ConvMode mode) {
    return mode == kGrad ? 256u : (cout < 32 ? 32u : (uint32_t)cout);
}

template <int CIN, int COUT, int SIDE, ConvMode kMode>
__global__ void __launch_bounds__(128) conv_pool_solo_tc_kernel(const bf16 *__restrict__ act,
                                                                int B, const bf16 *__restrict__ W,
                                                                const float *__restrict__ bias,
                                                                bf16 *__restrict__ out,
                                                                float *__restrict__ z_out,
                                                                uint8_t *__restrict__ idx, int nz,
                                                                int *err) {
    constexpr int PW = SIDE / 2;
    static_assert(CIN % 8 == 0 && COUT % 16 == 0 && COUT <= 32, "shapes of layers 1 and 2");
    static_assert(SIDE == 16 || SIDE == 32, "16 x 16 or 32 x 32 images");
    constexpr int K = 9 * CIN;
    constexpr int NK16 = (K + 15) / 16;
    constexpr int KC = K / 8;
    constexpr int KCS = NK16 * 2;
    constexpr uint32_t SBO = KCS * 128;
    constexpr int A_BYTES = 128 * KCS * 16;
    constexpr uint32_t kCols = conv_tmem_cols(COUT, kMode);
    constexpr uint32_t kIdesc = tc::idesc_bf16(128, COUT);
    constexpr int kTapSteps = kMode == kGrad ? CIN / 16 : NK16;  // K = 16 steps per accumulator
    static_assert(kMode != kGrad || (COUT == 16 && CIN % 16 == 0), "one 16-column accumulator per tap");
    constexpr int KP = (K + 7) & ~7;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *sA = smem, *sB = smem + A_BYTES;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sB + COUT * KCS * 16);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar + 1);
    __shared__ float sbias[COUT];
    __shared__ __align__(16) float sx[SIDE == 32 ? 2 : 1][16][16];  // SIDE 32: odd rows' maxima
    __shared__ uint32_t sk[SIDE == 32 ? 2 : 1][16];                 // and which column has them (training)

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t ntiles = (int64_t)B * SIDE * SIDE / 128;
    const int64_t my = blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    if (warp == 0) tc::tmem_alloc(tc::smem_u32(tmem_slot), kCols);
    if (tid == 0) tc::mbar_init1(tc::smem_u32(bar));
    for (int i = tid; i < COUT; i += 128) sbias[i] = kMode == kGrad ? 0.0f : bias[i];
    for (int idx = tid; idx < COUT * KCS; idx += 128) {
        const int n = idx % COUT, q = idx / COUT;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (q < KC) v = __ldg(reinterpret_cast<const uint4 *>(W + (int64_t)n * KP) + q);
        *reinterpret_cast<uint4 *>(sB + (n >> 3) * SBO + q * 128 + (n & 7) * 16) = v;
    }
    for (int idx = tid; idx < 128 * (KCS - KC); idx += 128) {
        const int r = idx & 127, q = KC + (idx >> 7);
        *reinterpret_cast<uint4 *>(sA + (r >> 3) * SBO + q * 128 + (r & 7) * 16) =
            make_uint4(0u, 0u, 0u, 0u);
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tmem_slot;
    gsp::wait_prior_grid();  // act comes from the kernel launched just before
    const uint32_t a_addr = tc::smem_u32(sA), b_addr = tc::smem_u32(sB);
    const uint32_t bar0 = tc::smem_u32(bar);

    auto gather = [&](int64_t tile) {
        const int64_t p = tile * 128 + tid;
        const int rem = (int)(p & (SIDE * SIDE - 1));
        const int y = rem / SIDE, x = rem % SIDE;
        const bf16 *base = act + p * CIN;
        const uint32_t dst = a_addr + (tid >> 3) * SBO + (tid & 7) * 16;
#pragma unroll
        for (int tap = 0; tap < 9; tap++) {
            const int dy = kMode == kGrad ? 1 - tap / 3 : tap / 3 - 1;
            const int dx = kMode == kGrad ? 1 - tap % 3 : tap % 3 - 1;
            const bool in = (unsigned)(y + dy) < (unsigned)SIDE && (unsigned)(x + dx) < (unsigned)SIDE;
            const bf16 *src = in ? base + (dy * SIDE + dx) * CIN : act;
#pragma unroll
            for (int j = 0; j < CIN / 8; j++)
                cp_async16(dst + (tap * (CIN / 8) + j) * 128, src + (in ? j * 8 : 0), in ? 16u : 0u);
        }
    };
    // bias + ReLU, 2x2 max, bf16 stores by the lane of each window's first pixel
    auto epilogue = [&](int64_t tile) {
        const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16);
        const int64_t m0 = tile * 128;
        const int64_t b = m0 / (SIDE * SIDE);
        const int y0 = (int)(m0 - b * SIDE * SIDE) / SIDE;  // the tile's first image row
        const int py = SIDE == 16 ? y0 / 2 + warp : y0 / 2 + (warp >> 1);  // pooled row
        const int px = SIDE == 16 ? (lane & 15) >> 1 : lane >> 1;
        bf16 *dst = out + ((b * PW + py) * PW + px) * COUT;
        const bool writer = SIDE == 16 ? (lane & 17) == 0 : ((lane & 1) == 0 && (warp & 1) == 0);
        if constexpr (kMode == kGrad) {
            float v[16];
            tc::tmem_ld16(taddr, v);
#pragma unroll
            for (int t = 1; t < 9; t++) {
                float w[16];
                tc::tmem_ld16(taddr + (uint32_t)(t * COUT), w);
#pragma unroll
                for (int c = 0; c < 16; c++) v[c] += w[c];
            }
            float4 *o = reinterpret_cast<float4 *>(z_out + (m0 + tid) * nz);
#pragma unroll
            for (int c = 0; c < 16; c += 4)
                if (c < nz) o[c / 4] = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
        } else {
#pragma unroll
        for (int c0 = 0; c0 < COUT; c0 += 16) {
            float v[16];
            tc::tmem_ld16(taddr + (uint32_t)c0, v);
            float z[16];
            uint32_t k1 = 0, k2 = 0;  // bit c: the window's maximum is in its second column / row
#pragma unroll
            for (int c = 0; c < 16; c++) z[c] = fmaxf(v[c] + sbias[c0 + c], 0.0f);
            if constexpr (kMode == kTrain) {
                float4 *o = reinterpret_cast<float4 *>(z_out + (m0 + tid) * COUT + c0);
#pragma unroll
                for (int c = 0; c < 16; c += 4) o[c / 4] = make_float4(z[c], z[c + 1], z[c + 2], z[c + 3]);
            }
#pragma unroll
            for (int c = 0; c < 16; c++) {
                const float r = __shfl_xor_sync(0xffffffffu, z[c], 1);
                if (kMode == kTrain) k1 |= (r > z[c] ? 1u : 0u) << c;  // of even columns' lanes
                z[c] = fmaxf(z[c], r);
            }
            if (SIDE == 16) {
                const uint32_t kb = kMode == kTrain ? __shfl_xor_sync(0xffffffffu, k1, 16) : 0u;
#pragma unroll
                for (int c = 0; c < 16; c++) {
                    const float r = __shfl_xor_sync(0xffffffffu, z[c], 16);
                    if (kMode == kTrain) k2 |= (r > z[c] ? 1u : 0u) << c;
                    z[c] = fmaxf(z[c], r);
                }
                k1 = (k1 & ~k2) | (kb & k2);
            }
            if (SIDE == 32) {
                // the odd row of each row pair hands its column-pair maxima over
                if ((warp & 1) && (lane & 1) == 0) {
#pragma unroll
                    for (int c = 0; c < 16; c += 4)
                        *reinterpret_cast<float4 *>(&sx[warp >> 1][lane >> 1][c]) =
                            make_float4(z[c], z[c + 1], z[c + 2], z[c + 3]);
                    if (kMode == kTrain) sk[warp >> 1][lane >> 1] = k1;
                }
                __syncthreads();
                if (writer) {
                    const uint32_t kb = kMode == kTrain ? sk[warp >> 1][lane >> 1] : 0u;
#pragma unroll
                    for (int c = 0; c < 16; c += 4) {
                        const float4 q = *reinterpret_cast<const float4 *>(&sx[warp >> 1][lane >> 1][c]);
                        if (kMode == kTrain)
                            k2 |= ((q.x > z[c] ? 1u : 0u) | (q.y > z[c + 1] ? 2u : 0u) |
                                   (q.z > z[c + 2] ? 4u : 0u) | (q.w > z[c + 3] ? 8u : 0u)) << c;
                        z[c] = fmaxf(z[c], q.x);
                        z[c + 1] = fmaxf(z[c + 1], q.y);
                        z[c + 2] = fmaxf(z[c + 2], q.z);
                        z[c + 3] = fmaxf(z[c + 3], q.w);
                    }
                    k1 = (k1 & ~k2) | (kb & k2);
                }
                __syncthreads();  // sx is rewritten by the next column block or tile
            }
            if (writer) {
                __align__(16) bf16 o[16];
#pragma unroll
                for (int c = 0; c < 16; c++) o[c] = __float2bfloat16_rn(z[c]);
                *reinterpret_cast<uint4 *>(dst + c0) = *reinterpret_cast<const uint4 *>(o);
                *reinterpret_cast<uint4 *>(dst + c0 + 8) = *reinterpret_cast<const uint4 *>(o + 8);
                if constexpr (kMode == kTrain) {
                    uint32_t kk[4];
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        kk[j] = 0;
#pragma unroll
                        for (int e = 0; e < 4; e++)
                            kk[j] |= (((k1 >> (4 * j + e)) & 1u) | (((k2 >> (4 * j + e)) & 1u) << 1)) << (8 * e);
                    }
                    *reinterpret_cast<uint4 *>(idx + ((b * PW + py) * PW + px) * COUT + c0) =
                        make_uint4(kk[0], kk[1], kk[2], kk[3]);
                }
            }
        }
        }
    };

    uint32_t ph = 0u;
    bool pend = false, ok = true;
    if (my > 0) {
        gather(blockIdx.x);
        cp_async_commit();
    }
    for (int64_t k = 0; k < my; k++) {
        const int64_t tile = blockIdx.x + k * gridDim.x;
        cp_async_wait<0>();
        tc::fence_proxy_async();  // this thread's copies -> tensor-core reads
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if (tid == 0) {
#pragma unroll
            for (int kk = 0; kk < NK16; kk++) {
                const uint64_t ad = tc::smem_desc(a_addr + kk * 256, 128, SBO);
                const uint64_t bd = tc::smem_desc(b_addr + kk * 256, 128, SBO);
                tc::mma_bf16(tmem + (uint32_t)(kk / kTapSteps * COUT), ad, bd, kIdesc,
                             kk % kTapSteps > 0 ? 1u : 0u);
            }
            tc::mma_commit(bar0);
        }
        pend = true;
        const bool done = tc::mbar_wait_bounded(bar0, ph, kConvBudget);
        if (!__syncthreads_and(done)) {
            ok = false;
            break;
        }
        ph ^= 1u;
        pend = false;
        tc::fence_after();
        if (k + 1 < my) {  // the MMAs are done with A: refill it under the epilogue
            gather(tile + gridDim.x);
            cp_async_commit();
        }
        epilogue(tile);
    }
    cp_async_wait<0>();
    if (!ok) {
        if (tid == 0) atomicExch(err, 1);
        if (pend) (void)tc::mbar_wait_bounded(bar0, ph, kConvBudget);
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, kCols);
}

// Layer 0 of a training pass: conv 3x3 (1 -> 8, pad 1) + bias + ReLU + 2x2 max-pool
// from the FP32 snippets, keeping the ReLU outputs z (FP32 [B][64][64][8]) and the
// pool's argmax.  One K = 16 MMA per 128-pixel tile (two image rows; the nine taps
// and seven zeros, eight channels and eight zeros), so that z has the tensor
// cores' summation order; the tile's rows are built by the threads, one pixel each.
// Bound by the 33 MB of z per 256 snippets; small CTAs, 16 per SM, hide the chain of
// gather, MMA and epilogue.
__global__ void __launch_bounds__(128) conv0_train_tc_kernel(const float *__restrict__ x, int B,
                                                             const bf16 *__restrict__ W0,
                                                             const float *__restrict__ b0,
                                                             bf16 *__restrict__ a0,
                                                             float *__restrict__ z_out,
                                                             uint8_t *__restrict__ idx, int *err) {
    constexpr int C = 8;
    constexpr uint32_t SBO = 256, kIdesc = tc::idesc_bf16(128, 16);
    __shared__ __align__(1024) uint8_t sA[128 * 32];
    __shared__ __align__(128) uint8_t sB[16 * 32];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tmem_slot;
    __shared__ float sbias[C];
    __shared__ __align__(16) float sx[2][16][C];  // odd rows' column-pair maxima
    __shared__ uint32_t sk[2][16];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) tc::tmem_alloc(tc::smem_u32(&tmem_slot), 32);
    if (tid == 0) tc::mbar_init1(tc::smem_u32(&bar));
    if (tid < C) sbias[tid] = b0[tid];
    if (tid < 32) {  // weights: row n < 8, half q of K
        const int n = tid & 15, q = tid >> 4;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (n < C) v = __ldg(reinterpret_cast<const uint4 *>(W0 + n * kpad(0)) + q);
        *reinterpret_cast<uint4 *>(sB + (n >> 3) * SBO + q * 128 + (n & 7) * 16) = v;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_slot, bar0 = tc::smem_u32(&bar);
    const uint64_t ad = tc::smem_desc(tc::smem_u32(sA), 128, SBO), bd = tc::smem_desc(tc::smem_u32(sB), 128, SBO);
    const int64_t ntiles = (int64_t)B * kS * kS / 128;
    uint32_t ph = 0;
    bool ok = true, pend = false;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t b = tile / (kS * kS / 128);
        const int y0 = 2 * (int)(tile - b * (kS * kS / 128));
        const int y = y0 + (warp >> 1), xc = (warp & 1) * 32 + lane;
        const float *img = x + b * kS * kS;
        __align__(16) bf16 row[16];
#pragma unroll
        for (int t = 0; t < 16; t++) row[t] = __float2bfloat16_rn(0.0f);
#pragma unroll
        for (int t = 0; t < 9; t++) {
            const int yy = y + t / 3 - 1, xx = xc + t % 3 - 1;
            if ((unsigned)yy < (unsigned)kS && (unsigned)xx < (unsigned)kS)
                row[t] = __float2bfloat16_rn(__ldg(img + yy * kS + xx));
        }
        uint8_t *dst = sA + (tid >> 3) * SBO + (tid & 7) * 16;
        *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(row);
        *reinterpret_cast<uint4 *>(dst + 128) = *reinterpret_cast<const uint4 *>(row + 8);
        tc::fence_proxy_async();
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if (tid == 0) {
            tc::mma_bf16(tmem, ad, bd, kIdesc, 0u);
            tc::mma_commit(bar0);
        }
        pend = true;
        const bool done = tc::mbar_wait_bounded(bar0, ph, kConvBudget);
        if (!__syncthreads_and(done)) {
            ok = false;
            break;
        }
        ph ^= 1u;
        pend = false;
        tc::fence_after();
        float v[16], z[C];
        tc::tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16), v);
        uint32_t k1 = 0, k2 = 0;
#pragma unroll
        for (int c = 0; c < C; c++) z[c] = fmaxf(v[c] + sbias[c], 0.0f);
        float4 *o = reinterpret_cast<float4 *>(z_out + ((b * kS + y) * kS + xc) * C);
        o[0] = make_float4(z[0], z[1], z[2], z[3]);
        o[1] = make_float4(z[4], z[5], z[6], z[7]);
#pragma unroll
        for (int c = 0; c < C; c++) {
            const float r = __shfl_xor_sync(0xffffffffu, z[c], 1);
            k1 |= (r > z[c] ? 1u : 0u) << c;
            z[c] = fmaxf(z[c], r);
        }
        if (warp >= 2 && (lane & 1) == 0) {
            float4 *q = reinterpret_cast<float4 *>(sx[warp & 1][lane >> 1]);
            q[0] = make_float4(z[0], z[1], z[2], z[3]);
            q[1] = make_float4(z[4], z[5], z[6], z[7]);
            sk[warp & 1][lane >> 1] = k1;
        }
        __syncthreads();
        if (warp < 2 && (lane & 1) == 0) {
            const float *q = sx[warp][lane >> 1];
            const uint32_t kb = sk[warp][lane >> 1];
            __align__(16) bf16 h[C];
            uint32_t kk[2] = {0u, 0u};
#pragma unroll
            for (int c = 0; c < C; c++) {
                const bool low = q[c] > z[c];
                h[c] = __float2bfloat16_rn(fmaxf(z[c], q[c]));
                k2 = low ? 2u + ((kb >> c) & 1u) : ((k1 >> c) & 1u);
                kk[c >> 2] |= k2 << (8 * (c & 3));
            }
            const int64_t pix = (b * (kS / 2) + y0 / 2) * (kS / 2) + (xc >> 1);
            *reinterpret_cast<uint4 *>(a0 + pix * C) = *reinterpret_cast<const uint4 *>(h);
            *reinterpret_cast<uint2 *>(idx + pix * C) = make_uint2(kk[0], kk[1]);
        }
        // sA and the accumulator are rewritten after the next tile's barriers, sx after its
        // first one
    }
    if (!ok) {
        if (tid == 0) atomicExch(err, 1);
        if (pend) (void)tc::mbar_wait_bounded(bar0, ph, kConvBudget);
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 32);
}

template <int CIN, int COUT>
constexpr int conv_pool_solo_smem() {
    return 128 * ((9 * CIN + 15) / 16) * 2 * 16 + COUT * ((9 * CIN + 15) / 16) * 2 * 16 + 8 + 16;
}

}  // namespace

struct gsp_ranker_s {
    int max_batch = 0;
    Offsets off{};
    float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
    int64_t step = 0;
    // packed bf16 weights
    bf16 *W[kLayers] = {}, *WG[kLayers] = {}, *W4 = nullptr, *W4T = nullptr;
    // activations
    bf16 *a[kLayers] = {};
    float *z[kLayers] = {};
    uint8_t *idx[kLayers] = {};
    float *z4 = nullptr, *z5 = nullptr, *g5 = nullptr, *ga3 = nullptr, *loss = nullptr;
    bf16 *a4 = nullptr, *g4 = nullptr, *g4T = nullptr, *a3T = nullptr;
    // backward scratch
    bf16 *gz[kLayers] = {};
    float *ga[kLayers] = {};    // gradient w.r.t. the pooled output of layer l
    float *fc1_part = nullptr;  // [kFc1Split][max_batch][kHid] partial products of fc1
    int *err = nullptr;
    std::vector<void *> allocs;
    int32_t launches = 0;
    int32_t last_n = 0;      // snippets of the last pass
    int last_pass = 0;       // 0 none, 1 inference (gsp_ranker_forward), 2 training step
};

namespace {

template <typename T>
bool ralloc(gsp_ranker_s *r, T **p, size_t n) {
    if (cudaMalloc((void **)p, std::max<size_t>(n, 1) * sizeof(T)) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    r->allocs.push_back(*p);
    return true;
}

void free_ranker(gsp_ranker_s *r) {
    if (!r) return;
    for (void *p : r->allocs) cudaFree(p);
    delete r;
}

int blocks_for(int64_t n, int threads = 256) {
    return (int)std::min<int64_t>((n + threads - 1) / threads, kSms * 16);
}

#define RK_LAUNCH(...)                                \
    do {                                              \
        __VA_ARGS__;                                  \
        cudaError_t e_ = cudaGetLastError();          \
        if (e_ != cudaSuccess) return e_;             \
        r->launches++;                                \
    } while (0)

cudaError_t pack(gsp_ranker_s *r, cudaStream_t s) {
    RK_LAUNCH((pack_kernel<<<blocks_for((int64_t)kHid * kFc), 256, 0, s>>>(
        r->params, r->off.w[0], r->off.w[1], r->off.w[2], r->off.w[3], r->W[0], r->W[1], r->W[2],
        r->WG[1], r->WG[2], r->W4, r->W4T)));
    return cudaSuccess;
}

cudaError_t gemm(gsp_ranker_s *r, const bf16 *A, int64_t lda, const bf16 *B, int64_t ldb, float *C,
                 int64_t ldc, bf16 *Cb, int64_t ldcb, int M, int N, int K, const float *bias,
                 bool relu, int splitk, cudaStream_t s) {
    cudaError_t e = gsp::launch_gemm_bf16(A, lda, B, ldb, C, ldc, Cb, ldcb, M, N, K, bias, relu,
                                          splitk, r->err, s);
    if (e == cudaSuccess) r->launches++;
    return e;
}

// CTAs per SM of a fused conv kernel from its resources: shared memory (stages +
// static + the per-CTA reservation), registers, threads, and at most 512
// tensor-memory columns per SM (cols per CTA).  The runtime's occupancy query
// answers one CTA per SM for these kernels whatever their shared memory, while
// several do run side by side (four CTAs per SM run layer 1 2.3x faster than
// one), so the count is computed here.  Also raises the kernel's dynamic
// shared-memory limit on the current device and asks for the largest
// shared-memory carveout (every launch calls that too: attributes are per device).
template <typename Kern>
cudaError_t conv_ctas_per_sm(Kern kern, int smem, int cols, int *out) {
    cudaError_t e = gsp::ensure_kernel_smem(reinterpret_cast<const void *>(kern), smem, true);
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kern);
    int dev = 0, smem_sm = 0, resv = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&resv, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (e != cudaSuccess) return e;
    const int by_smem = smem_sm / (smem + (int)fa.sharedSizeBytes + resv);
    const int by_regs = 65536 / (128 * std::max(fa.numRegs, 1));
    const int by_tmem = 512 / std::max(32, cols);
    *out = std::max(1, std::min(std::min(by_smem, by_regs), std::min(by_tmem, 16)));
    return cudaSuccess;
}

template <int CIN, int COUT, int SIDE, ConvMode kMode>
cudaError_t launch_conv(gsp_ranker_s *r, const bf16 *act, int n, const bf16 *W, const float *bias,
                        bf16 *out, float *z, uint8_t *idx, int nz, cudaStream_t s) {
    constexpr int smem = conv_pool_solo_smem<CIN, COUT>();
    auto kern = conv_pool_solo_tc_kernel<CIN, COUT, SIDE, kMode>;
    static int blocks_per_sm = 0;
    if (blocks_per_sm == 0) {
        cudaError_t e = conv_ctas_per_sm(kern, smem, (int)conv_tmem_cols(COUT, kMode), &blocks_per_sm);
        if (e != cudaSuccess) return e;
    } else {
        cudaError_t e = gsp::ensure_kernel_smem(reinterpret_cast<const void *>(kern), smem, true);
        if (e != cudaSuccess) return e;
    }
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int64_t ntiles = (int64_t)n * SIDE * SIDE / 128;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ntiles, (int64_t)sms * blocks_per_sm));
    // a programmatic dependent of the kernel before it (it waits in wait_prior_grid)
    e = gsp::launch_dependent(kern, dim3(grid), dim3(128), (size_t)smem, s, act, n, W, bias, out, z, idx,
                              nz, r->err);
    if (e != cudaSuccess) return e;
    r->launches++;
    return cudaSuccess;
}

// Forward pass of n snippets (FP32 [n][64][64]); logits into r->z5.  Each conv
// layer is one fused conv + bias + ReLU + pool kernel; in a training pass they
// also keep the ReLU outputs and the pool argmaxes.
cudaError_t forward(gsp_ranker_s *r, const float *x, int n, bool train, cudaStream_t s) {
    const int grid0 = blocks_for((int64_t)n * kS * kS / 8);
    const float *const b1 = r->params + r->off.b[1], *const b2 = r->params + r->off.b[2];
    cudaError_t e;
    if (train) {
        RK_LAUNCH((conv0_train_tc_kernel<<<(int)std::min<int64_t>((int64_t)n * kS * kS / 128, kSms * 16), 128, 0,
                                           s>>>(x, n, r->W[0], r->params + r->off.b[0], r->a[0], r->z[0],
                                                r->idx[0], r->err)));
        e = launch_conv<8, 16, 32, kTrain>(r, r->a[0], n, r->W[1], b1, r->a[1], r->z[1], r->idx[1], 0, s);
        if (e == cudaSuccess)
            e = launch_conv<16, 32, 16, kTrain>(r, r->a[1], n, r->W[2], b2, r->a[2], r->z[2], r->idx[2], 0, s);
    } else {
        RK_LAUNCH((conv0_pool_kernel<<<grid0, 256, 0, s>>>(x, n, r->W[0], r->params + r->off.b[0], r->a[0])));
        e = launch_conv<8, 16, 32, kInfer>(r, r->a[0], n, r->W[1], b1, r->a[1], nullptr, nullptr, 0, s);
        if (e == cudaSuccess)
            e = launch_conv<16, 32, 16, kInfer>(r, r->a[1], n, r->W[2], b2, r->a[2], nullptr, nullptr, 0, s);
    }
    if (e != cudaSuccess) return e;
    // fc1 (K = 2048) as a deterministic split-K product: enough K chunks for a
    // CTA per SM even at one column block, at least four 64-wide steps each;
    // the chunks' partial products are summed in order by fc1_finish_kernel
    int dev = 0, nsm = kSms;
    if (cudaGetDevice(&dev) == cudaSuccess)
        (void)cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int mt = (n + 127) / 128;
    const int want = std::max(1, std::min(kFc1Split, std::min(kFc / (4 * 64), nsm / mt)));
    const int64_t zs = (int64_t)r->max_batch * kHid;
    int used = 1;
    // each kernel after the first is launched as a
    // programmatic dependent of the one before (its blocks are scheduled while
    // that kernel drains and wait for its output in wait_prior_grid)
    e = gsp::launch_gemm_bf16(r->a[2], kFc, r->W4, kFc, r->fc1_part, kHid, nullptr, 0, n, kHid, kFc,
                              nullptr, false, want, r->err, s, zs, &used, true);
    if (e != cudaSuccess) return e;
    r->launches++;
    e = gsp::launch_dependent(fc1_finish_kernel, dim3(blocks_for((int64_t)n * kHid)), dim3(256), 0, s,
                              (const float *)r->fc1_part, used, zs, n,
                              (const float *)(r->params + r->off.b[3]), r->z4, r->a4);
    if (e == cudaSuccess)
        e = gsp::launch_dependent(fc2_kernel, dim3((2 * n + 127) / 128), dim3(128), 0, s,
                                  (const bf16 *)r->a4, (const float *)(r->params + r->off.w[4]),
                                  (const float *)(r->params + r->off.b[4]), n, r->z5);
    if (e != cudaSuccess) return e;
    r->launches += 2;
    return cudaSuccess;
}

// Loss, gradients (into r->grads, the oracle's layout) and one Adam step.
cudaError_t backward(gsp_ranker_s *r, const float *x, const int32_t *labels, int n, float lr,
                     cudaStream_t s) {
    const int n8 = round8(n);
    cudaError_t e = cudaMemsetAsync(r->grads, 0, (size_t)r->off.total * sizeof(float), s);
    if (n8 != n) {  // the padding columns of the transposed operands
        if (e == cudaSuccess) e = cudaMemsetAsync(r->g4T, 0, (size_t)kHid * n8 * sizeof(bf16), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(r->a3T, 0, (size_t)kFc * n8 * sizeof(bf16), s);
    }
    if (e != cudaSuccess) return e;
    float *const gr = r->grads;
    const Offsets &o = r->off;
    RK_LAUNCH((loss_kernel<<<1, 256, 0, s>>>(r->z5, labels, n, r->g5, r->loss)));
    RK_LAUNCH((fc2_back_kernel<<<std::min((n + 3) / 4, kSms), kHid, 0, s>>>(
        r->g5, r->a4, r->params + o.w[4], r->z4, n, gr + o.w[4], gr + o.b[4], r->g4, r->g4T, n8,
        gr + o.b[3])));
    {
        dim3 grid((unsigned)((n + 31) / 32), (unsigned)(kFc / 32));
        RK_LAUNCH((transpose_kernel<<<grid, dim3(32, 8), 0, s>>>(r->a[2], kFc, n, kFc, r->a3T, n8)));
    }
    e = gemm(r, r->g4T, n8, r->a3T, n8, gr + o.w[3], kFc, nullptr, 0, kHid, kFc, n8, nullptr, false, 1, s);
    if (e == cudaSuccess)
        e = gemm(r, r->g4, kHid, r->W4T, kHid, r->ga[2], kFc, nullptr, 0, n, kFc, kHid, nullptr,
                 false, 1, s);
    if (e != cudaSuccess) return e;
    // per layer: back through pool and ReLU, weight gradient, input gradient
    RK_LAUNCH((pool_back_kernel<32><<<blocks_for((int64_t)n * 8 * 8 * 4), 256, 0, s>>>(
        r->ga[2], r->idx[2], r->a[2], n, 16, r->gz[2], gr + o.b[2])));
    e = launch_conv<32, kGradRows, 16, kGrad>(r, r->gz[2], n, r->WG[2], nullptr, nullptr, r->ga[1], nullptr, 16, s);
    if (e != cudaSuccess) return e;
    RK_LAUNCH((conv_dw_kernel<bf16, 16, 32, 16><<<std::min(n, 6 * kSms), 256, 0, s>>>(
        r->a[1], n, r->ga[2], r->idx[2], r->a[2], gr + o.w[2])));
    RK_LAUNCH((pool_back_kernel<16><<<blocks_for((int64_t)n * 16 * 16 * 2), 256, 0, s>>>(
        r->ga[1], r->idx[1], r->a[1], n, 32, r->gz[1], gr + o.b[1])));
    e = launch_conv<16, kGradRows, 32, kGrad>(r, r->gz[1], n, r->WG[1], nullptr, nullptr, r->ga[0], nullptr, 8, s);
    if (e != cudaSuccess) return e;
    RK_LAUNCH((conv_dw_kernel<bf16, 8, 16, 32><<<std::min(2 * n, 6 * kSms), 256, 0, s>>>(
        r->a[0], n, r->ga[1], r->idx[1], r->a[1], gr + o.w[1])));
    RK_LAUNCH((pool_back_kernel<8><<<blocks_for((int64_t)n * 32 * 32), 256, 0, s>>>(
        r->ga[0], r->idx[0], r->a[0], n, 64, r->gz[0], gr + o.b[0])));
    RK_LAUNCH((conv_dw_kernel<float, 1, 8, 64><<<std::min(4 * n, 6 * kSms), 256, 0, s>>>(
        x, n, r->ga[0], r->idx[0], r->a[0], gr + o.w[0])));
    r->step++;
    const double c1 = 1.0 - std::pow(0.9, (double)r->step);
    const double c2 = 1.0 - std::pow(0.999, (double)r->step);
    RK_LAUNCH((adam_kernel<<<blocks_for(r->off.total), 256, 0, s>>>(
        r->params, r->grads, r->m, r->v, r->off.total, lr, 0.9f, 0.999f, 1e-8f, (float)c1,
        (float)c2)));
    return pack(r, s);
}

gsp_status status_of(cudaError_t e, const char *what) {
    if (e == cudaSuccess) return GSP_OK;
    gsp::record_error(e, what);
    return e == cudaErrorInvalidValue ? GSP_ERR_INVALID_ARG : GSP_ERR_CUDA;
}

// Snippet of candidate blockIdx.x: out[i][j] = sum over the samples s of time
// bin j (f = max(1, w / 4) samples, bins centred on t + w / 2) of the
// normalised series of row dm - 32 + i, ((D - m) - (c0 + beta j)) / sigma_ref
// (0 in bad blocks, rows with sigma_ref = 0, outside the rows or past Ls),
// divided by sqrt(f).  A bin is summed as exact integer runs inside one search
// block, with the block's trend applied in closed form.
//
// A row of the snippet reads 64 f consecutive samples of D.  The CTA streams
// them through a shared-memory ring of two halves with 1-D bulk copies (one
// per row, 16-byte aligned span [t_al, t_end) around the row's 64 f samples,
// completion counted on the half's mbarrier): thread 0 fills half (b & 1) with
// the S rows of batch b while the warps sum batch b - 1 from the other half,
// S = the rows of this candidate's span that fit a half.  The warps share the
// batch's 2 S half-rows of 32 bins; lane l sums one bin (f is odd except for
// f = 2, so the lanes' strided reads hit distinct banks).  A candidate whose span
// leaves [0, stride) of its rows, or a series that is not 16-byte aligned,
// reads D directly instead (same sums).  Every wait is bounded; a wait that
// gives up sets *err, waits (bounded) for the copies it issued and leaves.
// Bytes per half of the ring: a sweep of 8 to 48 KB halves (and of 128- and
// 256-thread CTAs) over a searched beam's 130k candidates put 24 KB halves and
// 256 threads first, at 4.6 TB/s of snippet reads (three CTAs per SM).
constexpr int kSnipHalf = 24 * 1024;
constexpr long long kSnipBudget = 2000000000ll;

// One run's term of a bin, ((sd - n m) - (n c0 + beta sj)) / sigma_ref, from
// dev = sd - n m (exact; sd the run's sum) and sj = the sum of its in-block
// sample indices, rounded step by step (no contraction into FMAs), so that
// both snippet paths give the same float.
__device__ __forceinline__ float run_term(float dev, int n, int64_t sj, const gsp::BlockParam &q,
                                          float inv) {
    const float t = __fadd_rn(__fmul_rn((float)n, q.c0), __fmul_rn(q.beta, (float)sj));
    return __fmul_rn(__fsub_rn(dev, t), inv);
}

// Positions inside a candidate's rows are int32 offsets from T0 = b0 * B, the
// start of the first search block its bins touch (b0 = max(tlo, 0) / B); a
// block index bi is then relative to b0.  bsh = log2(B) when B is a power of
// two, else -1.
__device__ __forceinline__ int rel_block(int r, int B, int bsh) {
    return bsh >= 0 ? (r >> bsh) : r / B;
}

// Bin [r0, r1) of one row (relative positions, clipped to the searched
// span); src[off + r] is the sample at relative position r and brow[bi] the
// parameters of relative block bi.  At most two runs (f <= B), each summed
// exactly in Acc: int32 (wrapping, exact) when f times the largest D stays
// below 2^31, else int64.
template <typename Acc>
__device__ __forceinline__ float snippet_bin(const int32_t *src, int off, int r0, int r1, int B,
                                             int bsh, const gsp::BlockParam *brow, float inv) {
    float v = 0.0f;
    int s0 = r0;
    while (s0 < r1) {
        const int bi = rel_block(s0, B, bsh), bs = bi * B;
        const int e = min(r1, bs + B);
        const int n = e - s0;
        const gsp::BlockParam q = brow[bi];
        if (q.good) {
            const int32_t *p = src + off + s0;
            Acc sd = 0;  // exact
#pragma unroll 4
            for (int k = 0; k < n; k++) sd += p[k];
            const int64_t sj = (int64_t)n * (s0 - bs) + (int64_t)n * (n - 1) / 2;
            const float dev =
                sizeof(Acc) == 4
                    ? (float)(int32_t)((uint32_t)sd - (uint32_t)n * (uint32_t)q.m)
                    : (float)((int64_t)sd - (int64_t)n * q.m);
            v = __fadd_rn(v, run_term(dev, n, sj, q, inv));
        }
        s0 = e;
    }
    return v;
}

template <int HALF>
__global__ void __launch_bounds__(256) snippet_kernel(
    const int32_t *__restrict__ D, int64_t stride, int ndm, int64_t Ls, int B,
    const gsp::BlockParam *__restrict__ bp, int64_t nb_max, const float *__restrict__ sinv,
    const gsp_cand *__restrict__ cands, const int32_t *__restrict__ order, int64_t dmax,
    float *__restrict__ out, int *err) {
    extern __shared__ __align__(128) int32_t ring[];  // 2 * HALF bytes
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ float s_inv[kS];
    const int64_t ck = order ? order[blockIdx.x] : blockIdx.x;  // this CTA's candidate
    const gsp_cand c = cands[ck];
    const int f = max(1, c.width / 4);
    const int64_t tlo = c.t + c.width / 2 - (int64_t)(kS / 2) * f;  // first sample of bin 0
    const float rs = 1.0f / sqrtf((float)f);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nwarps = (int)(blockDim.x >> 5);
    float *o = out + ck * kS * kS;
    // the 16-byte aligned span of every row: samples [t_al, t_end)
    const int64_t t_al = tlo >= 0 ? (tlo & ~(int64_t)3) : -((-tlo + 3) & ~(int64_t)3);
    const int64_t t_end = (tlo + (int64_t)kS * f + 3) & ~(int64_t)3;
    const int64_t rowb64 = (t_end - t_al) * 4;
    const bool bulk = ((reinterpret_cast<uintptr_t>(D) & 15u) == 0) && (stride % 4 == 0) &&
                      t_al >= 0 && t_end <= stride && rowb64 <= HALF;
    const uint32_t rowb = bulk ? (uint32_t)rowb64 : 0u;
    const int S = bulk ? min(kS, (int)(HALF / rowb)) : kS;  // rows per batch
    const int nbatch = (kS + S - 1) / S;
    const int64_t b0 = max(tlo, (int64_t)0) / B;           // first search block of the span
    const int64_t T0 = b0 * B;
    const int alo = (int)(tlo - T0);                       // bin 0 relative to T0
    const int lrel = (int)min(Ls - T0, (int64_t)1 << 30);  // end of the searched span
    const int bsh = (B & (B - 1)) == 0 ? __ffs(B) - 1 : -1;
    const bool narrow = (int64_t)f * dmax < 2147483648ll;  // int32 run sums are exact
    for (int i = tid; i < kS; i += blockDim.x) {
        const int r = c.dm_idx - kS / 2 + i;
        s_inv[i] = (r >= 0 && r < ndm) ? sinv[r] : 0.0f;
    }
    const uint32_t ring0 = ptx::smem_addr(ring);
    const uint32_t bar0 = ptx::smem_addr(&bar[0]);
    if (tid == 0) {
        ptx::mbar_init(bar0, 1);
        ptx::mbar_init(bar0 + 8, 1);
        ptx::fence_barrier_init();
    }
    __syncthreads();
    // thread 0: the copies of batch b into half b & 1 (rows with sigma_ref = 0
    // are not copied); returns the bytes expected on the half's barrier
    auto issue = [&](int b) {
        const int r0 = b * S, n = min(S, kS - r0);
        uint32_t bytes = 0;
        for (int k = 0; k < n; k++) bytes += s_inv[r0 + k] != 0.0f ? rowb : 0u;
        const uint32_t hb = bar0 + 8u * (uint32_t)(b & 1);
        ptx::mbar_arrive_expect_tx(hb, bytes);
        for (int k = 0; k < n; k++) {
            if (s_inv[r0 + k] == 0.0f) continue;
            const int r = c.dm_idx - kS / 2 + r0 + k;
            ptx::bulk_g2s(ring0 + (uint32_t)(b & 1) * HALF + (uint32_t)k * rowb,
                          D + (int64_t)r * stride + t_al, rowb, hb);
        }
    };
    if (bulk && tid == 0) {
        issue(0);
        if (nbatch > 1) issue(1);
    }
    bool ok = true;
    int waited = 0;  // batches whose copies are known to have landed
    for (int b = 0; b < nbatch; b++) {
        const int r0 = b * S, n = min(S, kS - r0);
        if (bulk) {
            const bool done = ptx::mbar_wait(bar0 + 8u * (uint32_t)(b & 1), (uint32_t)((b >> 1) & 1),
                                             kSnipBudget);
            if (!__syncthreads_and(done)) {
                ok = false;
                break;
            }
            waited = b + 1;
        }
        const int32_t *half = ring + (size_t)(b & 1) * (HALF / 4);
        // 2 n half-rows of 32 bins over the warps: warp task wt is row wt / 2,
        // bins 32 (wt % 2) + lane
        for (int wt = warp; wt < 2 * n; wt += nwarps) {
            const int k = wt >> 1, i = r0 + k, j = 32 * (wt & 1) + lane;
            const float inv = s_inv[i];
            float v = 0.0f;
            if (inv != 0.0f) {  // warp-uniform
                const int r = c.dm_idx - kS / 2 + i;
                const gsp::BlockParam *brow = bp + (int64_t)r * nb_max + b0;
                // the ring row holds samples t_al.. (T0 - t_al <= 3); D's row from T0
                const int32_t *src = bulk ? half + (size_t)k * (rowb / 4) : D + (int64_t)r * stride + T0;
                const int off = bulk ? (int)(T0 - t_al) : 0;
                const int r0 = max(alo + j * f, 0), r1 = min(alo + (j + 1) * f, lrel);
                v = narrow ? snippet_bin<int32_t>(src, off, r0, r1, B, bsh, brow, inv)
                           : snippet_bin<int64_t>(src, off, r0, r1, B, bsh, brow, inv);
            }
            o[i * kS + j] = v * rs;
        }
        if (bulk && b + 2 < nbatch) {
            __syncthreads();  // every warp is done with half b & 1
            if (tid == 0) issue(b + 2);
        }
    }
    if (!ok) {
        if (tid == 0) atomicExch(err, 1);
        // the copies of the (at most two) batches issued but not waited for
        for (int b = waited; b < min(nbatch, waited + 2); b++)
            (void)ptx::mbar_wait(bar0 + 8u * (uint32_t)(b & 1), (uint32_t)((b >> 1) & 1), kSnipBudget);
    }
}

// 1 / sigma_ref of every row in FP32 (0 where sigma_ref = 0), once per
// snippet call: FP64 division is slow on this GPU, so the snippet CTAs read
// these instead of dividing per row.
__global__ void inv_sigma_kernel(const double *__restrict__ sref, int ndm, float *__restrict__ sinv) {
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < ndm; r += gridDim.x * blockDim.x)
        sinv[r] = sref[r] > 0.0 ? (float)(1.0 / sref[r]) : 0.0f;
}

// The order in which the snippet CTAs take the candidates: by time bucket
// (t >> shift), a counting sort.  Candidates close in time share the samples
// of their rows' windows, so CTAs that run together then find them in L2
// whatever the caller's order (gsp_candidates sorts by DM first).  Each CTA
// still writes its own candidate's snippet, so the output does not depend on
// the order within a bucket (which the atomics leave open).
__global__ void time_bucket_count_kernel(const gsp_cand *__restrict__ cands, int n, int shift,
                                         int nbk, uint32_t *__restrict__ hist) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int64_t bk = min(max(cands[k].t >> shift, (int64_t)0), (int64_t)nbk - 1);
        atomicAdd(hist + bk, 1u);
    }
}

// hist[0 .. nbk) -> exclusive prefix (one CTA of 1024 threads; nbk <= 1024)
__global__ void __launch_bounds__(1024) time_bucket_scan_kernel(uint32_t *__restrict__ hist,
                                                                int nbk) {
    __shared__ uint32_t wsum[32];
    const int i = threadIdx.x, lane = i & 31, warp = i >> 5;
    const uint32_t v = i < nbk ? hist[i] : 0u;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    uint32_t off = 0;
    for (int w = 0; w < warp; w++) off += wsum[w];
    if (i < nbk) hist[i] = off + x - v;
}

__global__ void time_bucket_scatter_kernel(const gsp_cand *__restrict__ cands, int n, int shift,
                                           int nbk, uint32_t *__restrict__ next,
                                           int32_t *__restrict__ order) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int64_t bk = min(max(cands[k].t >> shift, (int64_t)0), (int64_t)nbk - 1);
        order[atomicAdd(next + bk, 1u)] = k;
    }
}

// Block-local inclusive prefix sums of a series, for snippets of wide bins:
// P[r][b B + k] = sum of D[r][b B .. b B + k] (mod 2^32) for every search block
// b < nb of every row.  A run of samples inside one block then sums to the
// difference of two entries, exact whenever the run's true sum lies within
// int32 (at most f samples of at most nchan * 255 each).  One CTA per (row,
// block) job, grid-stride; each warp scans 128 consecutive samples of a
// 1024-sample chunk with shuffles, the warps' totals are combined through
// shared memory, and a carry runs across the chunks of a block.
__global__ void __launch_bounds__(256) block_prefix_kernel(const int32_t *__restrict__ D,
                                                           int64_t stride, int ndm, int64_t nb,
                                                           int B, int32_t *__restrict__ P,
                                                           int64_t pstride) {
    __shared__ uint32_t wsum[8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int64_t job = blockIdx.x; job < (int64_t)ndm * nb; job += gridDim.x) {
        const int64_t r = job / nb, b = job - r * nb;
        const int32_t *src = D + r * stride + b * B;
        int32_t *dst = P + r * pstride + b * B;
        uint32_t carry = 0;  // sum of the block's samples before this chunk
        for (int c0 = 0; c0 < B; c0 += 1024) {
            uint32_t v[4], run = 0;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const int idx = c0 + warp * 128 + k * 32 + lane;
                uint32_t x = idx < B ? (uint32_t)__ldg(src + idx) : 0u;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                v[k] = x + run;
                run += __shfl_sync(0xffffffffu, x, 31);
            }
            if (lane == 0) wsum[warp] = run;
            __syncthreads();
            uint32_t off = carry, tot = 0;
#pragma unroll
            for (int w = 0; w < 8; w++) {
                off += w < warp ? wsum[w] : 0u;
                tot += wsum[w];
            }
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const int idx = c0 + warp * 128 + k * 32 + lane;
                if (idx < B) dst[idx] = (int32_t)(v[k] + off);
            }
            carry += tot;
            __syncthreads();  // wsum is rewritten by the next chunk
        }
    }
}

// Bin [r0, r1) of one row (relative positions as in snippet_bin) from the
// block-local prefix sums, pc[r] the entry at relative position r: at most two
// runs (f <= B), the second one starting a block; the three prefix entries are
// loaded before any is used.  Run sums are differences mod 2^32, exact since
// they lie within int32; the same run_term arithmetic as snippet_bin, so the
// same float.
__device__ __forceinline__ float snippet_bin_prefix(const int32_t *__restrict__ pc, int r0, int r1,
                                                    int B, int bsh, const gsp::BlockParam *brow,
                                                    float inv) {
    if (r0 >= r1) return 0.0f;
    const int bi = rel_block(r0, B, bsh), bs = bi * B, be = bs + B;
    const bool split = r1 > be;
    const int e1 = split ? be : r1;
    const uint32_t p_lo = r0 > bs ? (uint32_t)__ldg(pc + r0 - 1) : 0u;
    const uint32_t p_hi = (uint32_t)__ldg(pc + e1 - 1);
    const uint32_t p_2 = split ? (uint32_t)__ldg(pc + r1 - 1) : 0u;
    float v = 0.0f;
    {
        const int n = e1 - r0;
        const gsp::BlockParam q = brow[bi];
        if (q.good) {
            const float dev = (float)(int32_t)(p_hi - p_lo - (uint32_t)n * (uint32_t)q.m);
            const int64_t sj = (int64_t)n * (r0 - bs) + (int64_t)n * (n - 1) / 2;
            v = __fadd_rn(v, run_term(dev, n, sj, q, inv));
        }
    }
    if (split) {  // [be, r1) at the start of block bi + 1
        const int n = r1 - be;
        const gsp::BlockParam q = brow[bi + 1];
        if (q.good) {
            const float dev = (float)(int32_t)(p_2 - (uint32_t)n * (uint32_t)q.m);
            const int64_t sj = (int64_t)n * (n - 1) / 2;
            v = __fadd_rn(v, run_term(dev, n, sj, q, inv));
        }
    }
    return v;
}

// Snippets from the block-local prefix sums P of the series D (see
// snippet_kernel for the definition): two to three 4-byte loads per bin instead
// of f.  CTA per candidate; warp w builds rows w, w + 8, ..., lane l bins l and
// l + 32.  A candidate whose bins could span more than two blocks (f > B) or
// whose run sums could leave int32 sums its bins from D directly.
__global__ void __launch_bounds__(256) snippet_prefix_kernel(
    const int32_t *__restrict__ P, int64_t pstride, const int32_t *__restrict__ D, int64_t stride,
    int ndm, int64_t Ls, int B, const gsp::BlockParam *__restrict__ bp, int64_t nb_max,
    const float *__restrict__ sinv, const gsp_cand *__restrict__ cands,
    const int32_t *__restrict__ order, int64_t dmax, float *__restrict__ out) {
    const int64_t ck = order ? order[blockIdx.x] : blockIdx.x;  // this CTA's candidate
    const gsp_cand c = cands[ck];
    const int f = max(1, c.width / 4);
    const bool via_prefix = f <= B && (int64_t)f * dmax < 2147483648ll;
    const int64_t tlo = c.t + c.width / 2 - (int64_t)(kS / 2) * f;  // first sample of bin 0
    const int64_t b0 = max(tlo, (int64_t)0) / B, T0 = b0 * B;
    const int alo = (int)(tlo - T0);
    const int lrel = (int)min(Ls - T0, (int64_t)1 << 30);
    const int bsh = (B & (B - 1)) == 0 ? __ffs(B) - 1 : -1;
    const float rs = 1.0f / sqrtf((float)f);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = (int)(blockDim.x >> 5);
    float *o = out + ck * kS * kS;
    const int ra0 = max(alo + lane * f, 0), ra1 = min(alo + (lane + 1) * f, lrel);
    const int rb0 = max(alo + (32 + lane) * f, 0), rb1 = min(alo + (33 + lane) * f, lrel);
    for (int i = warp; i < kS; i += nwarps) {
        const int r = c.dm_idx - kS / 2 + i;
        const float inv = (r >= 0 && r < ndm) ? sinv[r] : 0.0f;
        float v0 = 0.0f, v1 = 0.0f;
        if (inv != 0.0f) {  // warp-uniform
            const gsp::BlockParam *brow = bp + (int64_t)r * nb_max + b0;
            if (via_prefix) {
                const int32_t *pc = P + (int64_t)r * pstride + T0;
                v0 = snippet_bin_prefix(pc, ra0, ra1, B, bsh, brow, inv);
                v1 = snippet_bin_prefix(pc, rb0, rb1, B, bsh, brow, inv);
            } else {
                const int32_t *dc = D + (int64_t)r * stride + T0;
                v0 = snippet_bin<int64_t>(dc, 0, ra0, ra1, B, bsh, brow, inv);
                v1 = snippet_bin<int64_t>(dc, 0, rb0, rb1, B, bsh, brow, inv);
            }
        }
        o[i * kS + lane] = v0 * rs;
        o[i * kS + 32 + lane] = v1 * rs;
    }
}

}  // namespace

extern "C" {

gsp_status gsp_ranker_snippets(gsp_plan_t p, const int32_t *d_D, int64_t stride,
                               const gsp_cand *d_cands, int32_t n, float *d_out, void *stream) {
    if (!p || !d_D || !d_cands || !d_out || n < 0) return GSP_ERR_INVALID_ARG;
    if (!p->have_search) return GSP_ERR_STATE;
    if (n == 0) return GSP_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const int B = p->desc.block_len;
    const int64_t Ls = p->last_nb * B;
    const int64_t dmax = (int64_t)p->desc.nchan * 255;
    // prefix sums pay off once the candidates' direct reads (64 x 64 f samples
    // each; f is taken as 4 here, the narrowest bins that fill a 16-byte
    // chunk) exceed building them (one read and one write of the series)
    const bool big = (int64_t)n * kS * kS * 4 >= 2 * (int64_t)p->desc.ndm * Ls;
    const bool use_prefix = Ls > 0 && (p->snippet_path == 2 || (p->snippet_path == 0 && big));
    // CTAs take the candidates in time order (buckets of 2^shift samples, at
    // most 1024 buckets over the series)
    int shift = 12;
    while (shift < 40 && (std::max<int64_t>(Ls, 1) >> shift) >= 1024) shift++;
    const int nbk = (int)std::min<int64_t>(1024, (std::max<int64_t>(Ls, 1) >> shift) + 1);
    if ((size_t)n > p->d_order_elems) {
        cudaFree(p->d_order);
        p->d_order = nullptr;
        p->d_order_elems = 0;
        if (cudaMalloc((void **)&p->d_order, (size_t)n * sizeof(int32_t)) != cudaSuccess) {
            (void)cudaGetLastError();
            return GSP_ERR_OOM;
        }
        p->d_order_elems = (size_t)n;
    }
    if (!p->d_order_hist &&
        cudaMalloc((void **)&p->d_order_hist, 1024 * sizeof(uint32_t)) != cudaSuccess) {
        (void)cudaGetLastError();
        p->d_order_hist = nullptr;
        return GSP_ERR_OOM;
    }
    if (!p->d_sinv &&
        cudaMalloc((void **)&p->d_sinv, (size_t)p->desc.ndm * sizeof(float)) != cudaSuccess) {
        (void)cudaGetLastError();
        p->d_sinv = nullptr;
        return GSP_ERR_OOM;
    }
    {
        const int g = (int)std::min<int64_t>(((int64_t)n + 255) / 256, (int64_t)p->num_sms * 4);
        cudaError_t e = cudaMemsetAsync(p->d_order_hist, 0, (size_t)nbk * sizeof(uint32_t), s);
        if (e == cudaSuccess) {
            time_bucket_count_kernel<<<g, 256, 0, s>>>(d_cands, n, shift, nbk, p->d_order_hist);
            time_bucket_scan_kernel<<<1, 1024, 0, s>>>(p->d_order_hist, nbk);
            time_bucket_scatter_kernel<<<g, 256, 0, s>>>(d_cands, n, shift, nbk, p->d_order_hist,
                                                         p->d_order);
            inv_sigma_kernel<<<(p->desc.ndm + 255) / 256, 256, 0, s>>>(p->d_sref, p->desc.ndm,
                                                                     p->d_sinv);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return status_of(e, "snippet order launch");
    }
    if (use_prefix) {
        const int64_t pstride = (Ls + 3) & ~(int64_t)3;
        const size_t need = (size_t)p->desc.ndm * (size_t)pstride;
        if (need > p->d_prefix_elems) {
            cudaFree(p->d_prefix);
            p->d_prefix = nullptr;
            p->d_prefix_elems = 0;
            p->prefix_seq = 0;
            if (cudaMalloc((void **)&p->d_prefix, need * sizeof(int32_t)) != cudaSuccess) {
                (void)cudaGetLastError();
                return GSP_ERR_OOM;
            }
            p->d_prefix_elems = need;
        }
        if (p->prefix_seq != p->search_seq || p->prefix_src != d_D || p->prefix_src_stride != stride ||
            p->prefix_stride != pstride) {
            const int64_t jobs = (int64_t)p->desc.ndm * p->last_nb;
            const int grid = (int)std::min<int64_t>(jobs, (int64_t)p->num_sms * 8);
            block_prefix_kernel<<<grid, 256, 0, s>>>(d_D, stride, p->desc.ndm, p->last_nb, B,
                                                      p->d_prefix, pstride);
            cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return status_of(e, "prefix launch");
            p->prefix_seq = p->search_seq;
            p->prefix_src = d_D;
            p->prefix_src_stride = stride;
            p->prefix_stride = pstride;
        }
        snippet_prefix_kernel<<<n, 256, 0, s>>>(p->d_prefix, pstride, d_D, stride, p->desc.ndm, Ls,
                                                B, p->d_bparam, p->nb_max, p->d_sinv, d_cands,
                                                p->d_order, dmax, d_out);
        return status_of(cudaGetLastError(), "snippet launch");
    }
    {
        cudaError_t e = gsp::ensure_kernel_smem(
            reinterpret_cast<const void *>(snippet_kernel<kSnipHalf>), 2 * kSnipHalf, true);
        if (e != cudaSuccess) return status_of(e, "snippet attributes");
    }
    snippet_kernel<kSnipHalf><<<n, 256, 2 * kSnipHalf, s>>>(
        d_D, stride, p->desc.ndm, Ls, B, p->d_bparam, p->nb_max, p->d_sinv, d_cands, p->d_order,
        dmax, d_out, p->d_err);
    return status_of(cudaGetLastError(), "snippet launch");
}

int64_t gsp_ranker_num_params(void) { return offsets().total; }

gsp_status gsp_ranker_create(gsp_ranker_t *out, int32_t max_batch, uint64_t seed) {
    if (!out || max_batch < 1 || max_batch > 4096) return GSP_ERR_INVALID_ARG;
    *out = nullptr;
    gsp_ranker_s *r = new (std::nothrow) gsp_ranker_s();
    if (!r) return GSP_ERR_OOM;
    r->max_batch = max_batch;
    r->off = offsets();
    const int Bm = max_batch, B8 = round8(Bm);
    const int64_t T = r->off.total;
    bool ok = ralloc(r, &r->params, T) && ralloc(r, &r->grads, T) && ralloc(r, &r->m, T) &&
              ralloc(r, &r->v, T) && ralloc(r, &r->W4, (size_t)kHid * kFc) &&
              ralloc(r, &r->W4T, (size_t)kHid * kFc) && ralloc(r, &r->z4, (size_t)Bm * kHid) &&
              ralloc(r, &r->a4, (size_t)Bm * kHid) && ralloc(r, &r->z5, (size_t)Bm * 2) &&
              ralloc(r, &r->g5, (size_t)Bm * 2) && ralloc(r, &r->g4, (size_t)Bm * kHid) &&
              ralloc(r, &r->g4T, (size_t)kHid * B8) && ralloc(r, &r->a3T, (size_t)kFc * B8) &&
              ralloc(r, &r->loss, 1) && ralloc(r, &r->err, 1);
    for (int l = 0; ok && l < kLayers; l++) {
        const int H = side_of(l), Cout = cout_of(l), Kp = kpad(l);
        const int64_t P = (int64_t)Bm * H * H;
        ok = ralloc(r, &r->W[l], (size_t)Cout * Kp) && ralloc(r, &r->WG[l], (size_t)kGradRows * 9 * Cout) &&
             ralloc(r, &r->z[l], (size_t)P * Cout) && ralloc(r, &r->a[l], (size_t)P / 4 * Cout) &&
             ralloc(r, &r->idx[l], (size_t)P / 4 * Cout) && ralloc(r, &r->gz[l], (size_t)P * Cout) &&
             ralloc(r, &r->ga[l], (size_t)P / 4 * Cout);
    }
    ok = ok && ralloc(r, &r->fc1_part, (size_t)kFc1Split * Bm * kHid);
    if (!ok) {
        free_ranker(r);
        return GSP_ERR_OOM;
    }
    // He-uniform weights, zero biases, from a 64-bit LCG (host)
    std::vector<float> h((size_t)T, 0.0f);
    uint64_t st = seed * 6364136223846793005ull + 1442695040888963407ull;
    for (int i = 0; i < 5; i++) {
        const int fan_in = i < 3 ? 9 * cin_of(i) : (i == 3 ? kFc : kHid);
        const double lim = std::sqrt(6.0 / fan_in);
        for (int64_t j = 0; j < kWsize[i]; j++) {
            st = st * 6364136223846793005ull + 1442695040888963407ull;
            const double u = (double)(st >> 11) * (1.0 / 9007199254740992.0);
            h[(size_t)(r->off.w[i] + j)] = (float)((2.0 * u - 1.0) * lim);
        }
    }
    cudaError_t e = cudaMemcpy(r->params, h.data(), (size_t)T * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(r->m, 0, (size_t)T * 4);
    if (e == cudaSuccess) e = cudaMemset(r->v, 0, (size_t)T * 4);
    if (e == cudaSuccess) e = cudaMemset(r->err, 0, sizeof(int));
    if (e == cudaSuccess) e = pack(r, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        gsp::record_error(e, "ranker init");
        free_ranker(r);
        return GSP_ERR_CUDA;
    }
    *out = r;
    return GSP_OK;
}

gsp_status gsp_ranker_destroy(gsp_ranker_t r) {
    if (!r) return GSP_ERR_INVALID_ARG;
    cudaError_t e = cudaDeviceSynchronize();
    free_ranker(r);
    return e == cudaSuccess ? GSP_OK : GSP_ERR_CUDA;
}

gsp_status gsp_ranker_set_params(gsp_ranker_t r, const float *host_params) {
    if (!r || !host_params) return GSP_ERR_INVALID_ARG;
    cudaError_t e = cudaMemcpy(r->params, host_params, (size_t)r->off.total * 4,
                               cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(r->m, 0, (size_t)r->off.total * 4);
    if (e == cudaSuccess) e = cudaMemset(r->v, 0, (size_t)r->off.total * 4);
    if (e == cudaSuccess) e = pack(r, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    r->step = 0;
    return status_of(e, "ranker set params");
}

gsp_status gsp_ranker_get_params(gsp_ranker_t r, float *host_params, float *host_grads) {
    if (!r) return GSP_ERR_INVALID_ARG;
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess && host_params)
        e = cudaMemcpy(host_params, r->params, (size_t)r->off.total * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && host_grads)
        e = cudaMemcpy(host_grads, r->grads, (size_t)r->off.total * 4, cudaMemcpyDeviceToHost);
    return status_of(e, "ranker get params");
}

gsp_status gsp_ranker_forward(gsp_ranker_t r, const float *d_x, int32_t n, float *d_logits,
                              void *stream) {
    if (!r || !d_x || n < 1 || n > r->max_batch) return GSP_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    r->launches = 0;
    cudaError_t e = forward(r, d_x, n, false, s);
    r->last_n = n;
    r->last_pass = 1;
    if (e == cudaSuccess && d_logits)
        e = cudaMemcpyAsync(d_logits, r->z5, (size_t)n * 2 * 4, cudaMemcpyDeviceToDevice, s);
    return status_of(e, "ranker forward");
}

gsp_status gsp_ranker_train_step(gsp_ranker_t r, const float *d_x, const int32_t *d_labels,
                                 int32_t n, float lr, float *d_loss, void *stream) {
    if (!r || !d_x || !d_labels || n < 1 || n > r->max_batch || !(lr >= 0.0f))
        return GSP_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    r->launches = 0;
    cudaError_t e = forward(r, d_x, n, true, s);
    if (e == cudaSuccess) e = backward(r, d_x, d_labels, n, lr, s);
    r->last_n = n;
    r->last_pass = 2;
    if (e == cudaSuccess && d_loss)
        e = cudaMemcpyAsync(d_loss, r->loss, sizeof(float), cudaMemcpyDeviceToDevice, s);
    return status_of(e, "ranker train step");
}

gsp_status gsp_ranker_finish(gsp_ranker_t r, void *stream) {
    if (!r) return GSP_ERR_INVALID_ARG;
    cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
    int flag = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&flag, r->err, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return status_of(e, "ranker finish");
    if (flag) {
        cudaMemset(r->err, 0, sizeof(int));
        return GSP_ERR_TIMEOUT;
    }
    return GSP_OK;
}

int32_t gsp_ranker_launches(gsp_ranker_t r) { return r ? r->launches : -1; }

gsp_status gsp_ranker_tensor(gsp_ranker_t r, const char *name, void *host_out, int64_t cap_bytes,
                             int64_t *bytes) {
    if (!r || !name || !bytes || cap_bytes < 0) return GSP_ERR_INVALID_ARG;
    if (r->last_pass == 0) return GSP_ERR_STATE;
    const int64_t n = r->last_n;
    const void *src = nullptr;
    int64_t size = 0;
    bool train_only = false;
    const std::string nm(name);
    for (int l = 0; l < kLayers && !src; l++) {
        const int64_t H = side_of(l), H2 = H / 2, C = cout_of(l);
        const std::string d = std::to_string(l);
        if (nm == "a" + d) { src = r->a[l]; size = n * H2 * H2 * C * 2; }
        else if (nm == "z" + d) { src = r->z[l]; size = n * H * H * C * 4; train_only = true; }
        else if (nm == "idx" + d) { src = r->idx[l]; size = n * H2 * H2 * C; train_only = true; }
        else if (nm == "ga" + d) { src = r->ga[l]; size = n * H2 * H2 * C * 4; train_only = true; }
        else if (nm == "gz" + d) { src = r->gz[l]; size = n * H * H * C * 2; train_only = true; }
    }
    if (!src) {
        if (nm == "z4") { src = r->z4; size = n * kHid * 4; }
        else if (nm == "a4") { src = r->a4; size = n * kHid * 2; }
        else if (nm == "z5") { src = r->z5; size = n * 2 * 4; }
        else if (nm == "g5") { src = r->g5; size = n * 2 * 4; train_only = true; }
        else if (nm == "g4") { src = r->g4; size = n * kHid * 2; train_only = true; }
        else return GSP_ERR_INVALID_ARG;
    }
    if (train_only && r->last_pass != 2) return GSP_ERR_STATE;
    *bytes = size;
    if (!host_out || cap_bytes < size) return GSP_ERR_CAPACITY;
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(host_out, src, (size_t)size, cudaMemcpyDeviceToHost);
    return status_of(e, "ranker tensor");
}

}  // extern "C"
