// Brute-force dedispersion on the tensor cores (tcgen05), exact.
//
//   D[dm][t] = sum_c X[c][t + delay[dm][c]]
//
// The shift of every (DM, channel) is done by a matrix product with a 0/1
// matrix.  An MMA of one channel has
//   rows    (i, tau): DM i of a block of 16, output phase tau of 8 (M = 128),
//   columns u:        groups of 8 consecutive samples (N <= 256),
//   K       s:        16 consecutive samples,
//   A[(i, tau)][s] = 1 where s = tau + shift_i (0 <= shift_i <= 8), else 0,
//   B[s][u]        = X[c][s_c + 8 u + s],
// so that row (i, tau), column u receives X[c][s_c + v + shift_i], v = 8u + tau.
// B is a Hankel matrix: in the K-major core-matrix layout (8 rows of 16 bytes)
// with 8 samples of 2 bytes per row, row u + 1 starts 16 bytes after row u and
// the second half of K 16 bytes after the first, so one copy of the channel's
// samples in shared memory, read through overlapping core matrices (leading
// offset 16, stride offset 128 bytes), is the whole operand.  A sample b is
// stored as the 16-bit integer b, which as an f16 is the subnormal b 2^-24: the
// products and their FP32 sums (below 2^24 units of 2^-24) are exact.  A lives in
// tensor memory (8 columns per channel), D in the other 256 columns for the
// whole channel loop.
//
// Frames.  The 16 delays of a channel differ by more than 8 samples over a
// band, so the rows of D are kept displaced: column position v of DM i holds
// output sample t = v - R_i.  R_i is constant over a frame (a run of channels in
// order of increasing delay) in which delay_i - R_i varies by at most 8 over
// the block; between frames row group i is moved right by e_i = 0..16 samples
// inside tensor memory (a lane rotation within the 8 phases and a move by up
// to two columns).  A frame is centred on a channel ahead of its first one, so it
// spans twice the 8 samples: 22 frames for the 4096 channels at a DM step of 0.5,
// 1000-1500 MHz, 36 at 0.8.
//
// Bound.  Per channel and block an MMA issues 128 x N x 16 products for 128 N
// useful additions and takes N / 2 clocks of the tensor pipe (measured: 120 at N = 240,
// 136 at N = 256): 256 additions per clock and SM, against 86 of the shared-load bound
// kernel in dedisperse.cu.  The same 16 x N samples are copied, widened
// and read from shared memory: 2 (copy) + 3 + 4 (widen) + 8 (operand) bytes per
// 8 samples x 128-byte clock, which nearly fills the shared-memory port too.
#include <algorithm>
#include <cstring>

#include "dd_mma.cuh"
#include "dd_tiled.cuh"
#include "gsp_internal.cuh"
#include "tc_gemm.cuh"

namespace gsp {
namespace {

constexpr int kKdm = 16;               // DM trials per block
constexpr int kChunk = 8;              // channels per pipeline slot
constexpr int kSlots = 4;              // pipeline slots (raw bytes, widened samples, A)
constexpr int kCols = 256;             // columns of D (samples / 8)
constexpr int kRawPitch = 8 * kCols + 32;        // bytes of a channel's window
constexpr int kWidePitch = (kCols + 1) * 16;     // bytes of its widened samples
constexpr int kRawSlot = kChunk * kRawPitch;
constexpr int kWideSlot = kChunk * kWidePitch;
// Warps by role (the first two roles: one quarter of the tensor-memory lanes each).
constexpr int kAWarp = 4;              // 4: write A (warps 0-3 move the rows of D and store it)
constexpr int kWideWarp = 8;           // 11: widen the channels in turn (16.1 ms on a
                                       // 131072-sample chunk; 8: 16.6, 10: 16.5, 12: 17.0)
constexpr int kWideWarps = 11;
static_assert(kWideWarps <= 2 * kChunk, "a widening warp leaves out one chunk at most");
constexpr int kMmaWarp = kWideWarp + kWideWarps;  // issue the products (one lane)
constexpr int kCopyWarp = kMmaWarp + 1;           // 2: copy the channels' windows of the chunks in turn
constexpr int kCopyWarps = 2;
constexpr int kThreads = 32 * (kCopyWarp + kCopyWarps);
constexpr int kMaxShift = 8;           // shift_i of a channel: 0..8
constexpr int kMaxMove = 16;           // e_i of a frame boundary: 0..16
constexpr uint32_t kTmemA = kCols;     // first tensor-memory column of A
constexpr int kSmem = kSlots * (kRawSlot + kWideSlot) + 256;

struct MmaBeam {
    const uint8_t *x;
    int64_t x_stride, n_in, n_out;
    const int32_t *base;     // [nblk][nchan] window start of each position, relative to t0
    const uint8_t *shift;    // [nblk][nchunk][16][8] shift_i
    const MmaFrame *frames;  // all blocks' frames
    const int32_t *foff;     // [nblk + 1] first frame of each block
    const int32_t *crmax;    // [nblk][nchunk] largest R_i of the chunk's frames
    const int32_t *rlast;    // [nblk][16] R_i of the last frame
    int32_t *out;
    int64_t out_stride;
    unsigned long long *bsum;
    int64_t nb_max, Ls, ntiles, item0;
    int ndm, nblk, grp, B, T, rev;
    int add;  // add to the series that is there (the other channels' sums)
};

struct MmaArgs {
    MmaBeam beam[kMmaMaxBeams];
    int nbeams, nchan;
    int *err;
    int64_t items;
    long long budget;
    int starve;
};

// Columns of the products of a frame whose largest R is rmax (a multiple of 16).
__device__ __forceinline__ int frame_cols(int T, int rmax) { return ((T + rmax + 127) >> 7) << 4; }

__device__ __forceinline__ void mma_decode(const MmaArgs &a, int64_t item, int *bi, int64_t *tile,
                                           int *blk) {
    int b = 0;
    while (b + 1 < a.nbeams && item >= a.beam[b + 1].item0) b++;
    const MmaBeam &bt = a.beam[b];
    const int64_t idx = item - bt.item0;
    const int64_t nfull = bt.nblk / bt.grp;
    const int64_t per_group = bt.ntiles * bt.grp;
    if (idx < nfull * per_group) {
        const int64_t g = idx / per_group, r = idx - g * per_group;
        *tile = r / bt.grp;
        *blk = (int)(g * bt.grp + (r - *tile * bt.grp));
    } else {
        const int64_t rem = bt.nblk - nfull * bt.grp;
        const int64_t r = idx - nfull * per_group;
        *tile = r / rem;
        *blk = (int)(nfull * bt.grp + (r - *tile * rem));
    }
    *bi = b;
}

// D (+)= A B with A (f16) in tensor memory, B through a shared-memory descriptor.
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint32_t blo, uint32_t bhi,
                                       uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 b;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 b, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %4, p;\n\t}"
        ::"r"(d), "r"(a), "r"(blo), "r"(bhi), "r"(idesc), "r"(accumulate)
        : "memory");
}

#define GSP_R16(r, o)                                                                          \
    "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), \
        "=r"(r[o + 6]), "=r"(r[o + 7]), "=r"(r[o + 8]), "=r"(r[o + 9]), "=r"(r[o + 10]),        \
        "=r"(r[o + 11]), "=r"(r[o + 12]), "=r"(r[o + 13]), "=r"(r[o + 14]), "=r"(r[o + 15])
#define GSP_I16(r, o)                                                                        \
    "r"(r[o]), "r"(r[o + 1]), "r"(r[o + 2]), "r"(r[o + 3]), "r"(r[o + 4]), "r"(r[o + 5]),     \
        "r"(r[o + 6]), "r"(r[o + 7]), "r"(r[o + 8]), "r"(r[o + 9]), "r"(r[o + 10]),           \
        "r"(r[o + 11]), "r"(r[o + 12]), "r"(r[o + 13]), "r"(r[o + 14]), "r"(r[o + 15])

__device__ __forceinline__ void tmem_store16(uint32_t addr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};"
        ::GSP_I16(r, 0), "r"(addr)
        : "memory");
}
// 16 columns of this thread's lane; the values are there after tmem_wait_ld16.
__device__ __forceinline__ void tmem_load16_async(uint32_t addr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : GSP_R16(r, 0)
        : "r"(addr)
        : "memory");
}
#define GSP_RW16(r)                                                                            \
    "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),         \
        "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), \
        "+r"(r[14]), "+r"(r[15])
__device__ __forceinline__ void tmem_wait_ld16(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : GSP_RW16(r)::"memory");
}
__device__ __forceinline__ void tmem_wait_st() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Widen n groups of 8 samples of a channel: lane l takes groups l, l + 32, ...
// src: this lane's first aligned word (kOdd: at 4 modulo 8), bs: the first
// sample's bit in it.  All loads of up to 8 groups are issued before their use.
template <bool kOdd>
__device__ __forceinline__ void widen_channel(uint32_t src, uint32_t dst, uint32_t bs, int n, int lane) {
    for (int j0 = 0; 32 * j0 < n; j0 += 8) {
        uint32_t x0[8], x1[8], x2[8];
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const uint32_t p = src + 256u * (uint32_t)(j0 + j);
            if (32 * (j0 + j) + lane < n) {
                const uint2 y = ptx::lds64(kOdd ? p + 4u : p);
                const uint32_t z = ptx::lds32(kOdd ? p : p + 8u);
                x0[j] = kOdd ? z : y.x;
                x1[j] = kOdd ? y.x : y.y;
                x2[j] = kOdd ? y.y : z;
            } else {
                x0[j] = x1[j] = x2[j] = 0u;
            }
        }
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const uint32_t lo = __funnelshift_r(x0[j], x1[j], bs), hi = __funnelshift_r(x1[j], x2[j], bs);
            const uint32_t v[4] = {__byte_perm(lo, 0, 0x4140), __byte_perm(lo, 0, 0x4342),
                                   __byte_perm(hi, 0, 0x4140), __byte_perm(hi, 0, 0x4342)};
            if (32 * (j0 + j) + lane < n) ptx::sts128(dst + 512u * (uint32_t)(j0 + j), v);
        }
    }
}

// One work item per (beam, time tile, DM block); persistent CTAs, one per SM, stride over them,
// their pipelines running on across items.  Warps:
//   0-3   move the rows of D between frames, store D;
//   4-7   write A of each chunk;
//   8-18  widen the channels in turn;
//   19    issues the MMAs (one lane);
//   20-21 copy the channels' windows of every other chunk each (1-D bulk copies).
// Every wait is bounded: a warp whose wait gives up reports it and leaves its
// loop; the MMA lane and the copying warp then wait for what they have in flight, and
// tensor memory is freed after all warps have met.  (Where the wait for the row moves gives up,
// the MMA lane first runs to the end of the item, waiting for and freeing its chunks but
// issuing no more products: every way straight out of that loop made the compiler's
// code for it slower, 16.08 -> 16.22 ms on a 131072-sample chunk.)
__global__ void __launch_bounds__(kThreads, 1) dd_mma_kernel(const __grid_constant__ MmaArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    uint8_t *raw = smem;                                 // [kSlots][kChunk][kRawPitch]
    uint8_t *wide = smem + kSlots * kRawSlot;            // [kSlots][kChunk][kWidePitch]
    uint64_t *bars = reinterpret_cast<uint64_t *>(wide + kSlots * kWideSlot);
    const uint32_t raw0 = ptx::smem_addr(raw), wide0 = ptx::smem_addr(wide);
    const uint32_t bar0 = ptx::smem_addr(bars);
    auto raw_full = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    auto raw_empty = [&](int i) { return bar0 + 8u * (uint32_t)(kSlots + i); };
    auto slot_full = [&](int i) { return bar0 + 8u * (uint32_t)(2 * kSlots + i); };
    auto slot_empty = [&](int i) { return bar0 + 8u * (uint32_t)(3 * kSlots + i); };
    const uint32_t frame_done = bar0 + 8u * (4 * kSlots), rows_moved = frame_done + 8u;
    const uint32_t drained = frame_done + 16u;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 4 * kSlots + 3);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int C = a.nchan, nchunk = (C + kChunk - 1) / kChunk;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kSlots; i++) {
            ptx::mbar_init(raw_full(i), 1);
            ptx::mbar_init(raw_empty(i), kChunk);
            ptx::mbar_init(slot_full(i), kChunk + 4);  // the widening warps and the writers of A
            ptx::mbar_init(slot_empty(i), 1);
        }
        ptx::mbar_init(frame_done, 1);
        ptx::mbar_init(rows_moved, 4);
        ptx::mbar_init(drained, 1);
        ptx::fence_barrier_init();
    }
    if (warp == 0) tc::tmem_alloc(tc::smem_u32(tmem_slot), 512);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;
    uint32_t g = 0;   // chunks so far (across items): slot g % kSlots, round g / kSlots
    uint32_t ev = 0;  // frame boundaries and item ends so far
    uint32_t last = 0;  // copying warps: one past their last chunk

    if (warp < kAWarp) {
        // ------------------------------------------- row moves, epilogue
        const uint32_t tq = tmem + ((uint32_t)(warp * 32) << 16);
        const int tau = lane & 7, dmi = warp * 4 + (lane >> 3);
        for (int64_t item = blockIdx.x; item < a.items && ok; item += gridDim.x) {
            int bi, blk;
            int64_t tile;
            mma_decode(a, item, &bi, &tile, &blk);
            const MmaBeam &bt = a.beam[bi];
            const int64_t t0 = tile * bt.T;
            const MmaFrame *fr = bt.frames + bt.foff[blk];
            const int nfr = bt.foff[blk + 1] - bt.foff[blk];
            if (bt.add) {
                // the series that the item adds to, towards L2: the epilogue waits for a
                // round trip per 16 columns
                const int d = blk * kKdm + dmi;
                const int n = d < bt.ndm ? (int)min((int64_t)bt.T, bt.n_out - t0) : 0;
                const int32_t *o = bt.out + (int64_t)min(d, bt.ndm - 1) * bt.out_stride + t0;
                for (int j = 32 * tau; j < n; j += 256) asm volatile("prefetch.global.L2 [%0];" ::"l"(o + j));
            }
            for (int f = 1; f < nfr; f++) {
                // the frame's record, loaded ahead of its boundary
                const int ne = (int)__ldg(&fr[f].e[dmi]), nrmax = __ldg(&fr[f].rmax);
                // the products of the frame are complete: move the rows
                if (!__all_sync(0xffffffffu, ptx::mbar_wait(frame_done, ev & 1u, a.budget))) {
                    ok = false;
                    break;
                }
                ev++;
                tc::fence_after();
                const int ncols = frame_cols(bt.T, nrmax);
                const int src = (lane & 24) | ((tau - ne) & 7);
                const int kc = (ne + 7 - tau) >> 3;  // columns moved: 0, 1 or 2
                // masks, not selects: nvcc turns selects on kc into divergent branches
                // (1000 clocks per 16 columns against 130)
                const uint32_t k0 = kc == 0 ? ~0u : 0u, k1 = kc == 1 ? ~0u : 0u, k2 = ~(k0 | k1);
                uint32_t c1 = 0u, c2 = 0u;          // columns c0 - 1 and c0 - 2 after the rotation
                uint32_t va[16], vb[16];
                // 16 columns at a time, the next ones being loaded (columns past ncols are
                // loaded but not used)
                auto move16 = [&](uint32_t (&v)[16], int c0) {
                    uint32_t n[16];
#pragma unroll
                    for (int i = 0; i < 16; i++) v[i] = __shfl_sync(0xffffffffu, v[i], src);
#pragma unroll
                    for (int i = 0; i < 16; i++) {
                        const uint32_t m1 = i >= 1 ? v[i >= 1 ? i - 1 : 0] : c1;
                        const uint32_t m2 = i >= 2 ? v[i >= 2 ? i - 2 : 0] : (i == 1 ? c1 : c2);
                        n[i] = (v[i] & k0) | (m1 & k1) | (m2 & k2);
                    }
                    tmem_store16(tq + (uint32_t)c0, n);
                    c1 = v[15];
                    c2 = v[14];
                };
                tmem_load16_async(tq, va);
                for (int c0 = 0; c0 < ncols; c0 += 32) {
                    tmem_wait_ld16(va);
                    tmem_load16_async(tq + (uint32_t)c0 + 16u, vb);
                    move16(va, c0);
                    tmem_wait_ld16(vb);
                    if (c0 + 32 < ncols) tmem_load16_async(tq + (uint32_t)c0 + 32u, va);
                    if (c0 + 16 < ncols) move16(vb, c0 + 16);
                }
                tmem_wait_st();
                tc::fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(rows_moved);
            }
            if (!ok) break;
            if (!__all_sync(0xffffffffu, ptx::mbar_wait(frame_done, ev & 1u, a.budget))) {
                ok = false;
                break;
            }
            ev++;
            tc::fence_after();
            // store the tile: lane (i, tau), column u holds sample t = 8u + tau - R_i
            const int d = blk * kKdm + dmi;
            const int R = bt.rlast[(int64_t)blk * kKdm + dmi];
            const int tlim = d < bt.ndm ? (int)min((int64_t)bt.T, bt.n_out - t0) : 0;  // stored samples
            int32_t *orow = bt.out + (int64_t)min(d, bt.ndm - 1) * bt.out_stride + t0;
            const bool sums = bt.bsum != nullptr && d < bt.ndm;
            const int64_t kb = t0 / bt.B;               // first search block of the tile
            int blk_e = (int)((kb + 1) * bt.B - t0);    // end of the current block (tile time)
            // samples of the tile that lie in search blocks
            const int slim = sums ? max(0, (int)min((int64_t)tlim, bt.Ls - t0)) : 0;
            unsigned long long *q = sums ? bt.bsum + ((int64_t)d * bt.nb_max + kb) * 3 : nullptr;
            unsigned long long s0 = 0, s1 = 0, s2 = 0;  // of the current block: sum x, sum j x, sum x^2
            auto flush = [&]() {
                if (slim > 0 && blk_e - bt.B < slim) {
                    atomicAdd(q, s0);
                    atomicAdd(q + 1, s1);
                    atomicAdd(q + 2, s2);
                    q += 3;
                }
                s0 = s1 = s2 = 0;
                blk_e += bt.B;
            };
            const int ncols = frame_cols(bt.T, nfr > 0 ? fr[nfr - 1].rmax : 0);
            uint32_t va[16], vb[16];
            // 16 columns at a time: the sums run in 32 bits inside them (x < 2^24,
            // sum i x < 2^31), unless a lane comes to a search block's end there
            const bool add = bt.add != 0;  // another kernel has left the other channels' sums
            auto store16 = [&](const uint32_t (&v)[16], int c0) {
                const int tf = 8 * c0 + tau - R;  // the lane's first sample
                int32_t x[16];
#pragma unroll
                for (int i = 0; i < 16; i++) x[i] = (int32_t)(__uint_as_float(v[i]) * 16777216.0f);
                if (add) {
                    int32_t o[16];
#pragma unroll
                    for (int i = 0; i < 16; i++)
                        o[i] = (unsigned)(tf + 8 * i) < (unsigned)tlim ? __ldcs(orow + tf + 8 * i) : 0;
#pragma unroll
                    for (int i = 0; i < 16; i++) x[i] += o[i];
                }
#pragma unroll
                for (int i = 0; i < 16; i++) {
                    const int t = tf + 8 * i;
                    if ((unsigned)t < (unsigned)tlim) __stcs(orow + t, x[i]);
                    x[i] = (unsigned)t < (unsigned)slim ? x[i] : 0;
                }
                if (!__any_sync(0xffffffffu, sums && tf + 120 >= blk_e)) {
                    uint32_t b0 = 0, b1 = 0;
#pragma unroll
                    for (int i = 0; i < 16; i++) {
                        b0 += (uint32_t)x[i];
                        b1 += (uint32_t)i * (uint32_t)x[i];
                        s2 += (unsigned long long)((long long)x[i] * x[i]);
                    }
                    s0 += b0;
                    s1 += (unsigned long long)((long long)(tf - blk_e + bt.B) * (long long)b0) +
                          8ull * (unsigned long long)b1;
                } else {
#pragma unroll
                    for (int i = 0; i < 16; i++) {
                        const int t = tf + 8 * i;
                        if (t >= blk_e) flush();
                        s0 += (unsigned long long)x[i];
                        s1 += (unsigned long long)((long long)(t - blk_e + bt.B) * x[i]);
                        s2 += (unsigned long long)((long long)x[i] * x[i]);
                    }
                    __syncwarp();
                }
            };
            tmem_load16_async(tq, va);
            for (int c0 = 0; c0 < ncols; c0 += 32) {
                tmem_wait_ld16(va);
                tmem_load16_async(tq + (uint32_t)c0 + 16u, vb);
                store16(va, c0);
                tmem_wait_ld16(vb);
                if (c0 + 32 < ncols) tmem_load16_async(tq + (uint32_t)c0 + 32u, va);
                if (c0 + 16 < ncols) store16(vb, c0 + 16);
            }
            if (sums) flush();
            __syncwarp();
            tc::fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(rows_moved);
        }
    } else if (warp < kWideWarp) {
        // ------------------------------------------------------- A
        const int q = warp - kAWarp;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + kTmemA;
        const int tau = lane & 7, dmi = q * 4 + (lane >> 3);
        for (int64_t item = blockIdx.x; item < a.items && ok; item += gridDim.x) {
            int bi, blk;
            int64_t tile;
            mma_decode(a, item, &bi, &tile, &blk);
            const uint2 *sh = reinterpret_cast<const uint2 *>(a.beam[bi].shift) +
                              (int64_t)blk * nchunk * kKdm + dmi;
            uint2 nsh = __ldg(sh);
            for (int ch = 0; ch < nchunk; ch++, g++) {
                const int slot = (int)(g % kSlots);
                const uint2 csh = nsh;
                if (ch + 1 < nchunk) nsh = __ldg(sh + (int64_t)(ch + 1) * kKdm);
                if (!__all_sync(0xffffffffu, ptx::mbar_wait(slot_empty(slot), ((g / kSlots) & 1u) ^ 1u,
                                                            a.budget))) {
                    ok = false;
                    break;
                }
                tc::fence_after();
#pragma unroll
                for (int h = 0; h < kChunk / 2; h++) {
                    uint32_t r[16];
#pragma unroll
                    for (int j = 0; j < 2; j++) {
                        const int k = 2 * h + j;
                        const uint32_t w = k < 4 ? csh.x : csh.y;
                        const uint32_t s = (uint32_t)tau + ((w >> (8 * (k & 3))) & 0xffu);
                        const uint32_t one = (s & 1u) ? 0x3C000000u : 0x00003C00u;
#pragma unroll
                        for (int i = 0; i < 8; i++) r[8 * j + i] = (s >> 1) == (uint32_t)i ? one : 0u;
                    }
                    tmem_store16(tq + (uint32_t)(slot * kChunk * 8 + h * 16), r);
                }
                tmem_wait_st();
                tc::fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(slot_full(slot));
            }
        }
    } else if (warp < kMmaWarp) {
        // ------------------------------------------------------- widening
        // channels (8 nchunk per item, the last ones of an item may be none) go to the
        // warps in turn, counted over the CTA's items: c0 is the first of this item
        uint32_t c0 = 0;
        for (int64_t item = blockIdx.x; item < a.items && ok; item += gridDim.x) {
            int bi, blk;
            int64_t tile;
            mma_decode(a, item, &bi, &tile, &blk);
            const MmaBeam &bt = a.beam[bi];
            const uint32_t t0lo = (uint32_t)(tile * bt.T);
            const int32_t *base = bt.base + (int64_t)blk * C;
            const int32_t *crmax = bt.crmax + (int64_t)blk * nchunk;
            int pos = (warp - kWideWarp + kWideWarps - (int)(c0 % kWideWarps)) % kWideWarps;
            int nbase = pos < C ? __ldg(base + pos) : 0;
            int nrm = pos < nchunk * kChunk ? __ldg(crmax + pos / kChunk) : 0;
            for (; pos < nchunk * kChunk; pos += kWideWarps) {
                const int k = pos % kChunk;
                const uint32_t gc = g + (uint32_t)(pos / kChunk);
                const int slot = (int)(gc % kSlots);
                const uint32_t par = (gc / kSlots) & 1u;
                const uint32_t off = (t0lo + (uint32_t)nbase) & 15u;  // first sample's byte in the window
                const int n = frame_cols(bt.T, nrm) + 1;              // groups of 8 samples
                const int np = pos + kWideWarps;
                if (np < nchunk * kChunk) {
                    nbase = np < C ? __ldg(base + np) : 0;
                    nrm = __ldg(crmax + np / kChunk);
                }
                // in this order: a warp that had no channel of this slot's last chunk may come
                // here before that chunk's copy has landed, and the parity of raw_full would
                // then read as complete a round early.  The slot's products of that chunk are
                // done only after its copy has been read, so raw_full has moved on by then.  (A
                // warp leaves out one chunk at most, so slot_empty is never two rounds behind.)
                const bool landed = ptx::mbar_wait(slot_empty(slot), par ^ 1u, a.budget) &&
                                    ptx::mbar_wait(raw_full(slot), par, a.budget);
                if (!__all_sync(0xffffffffu, landed)) {
                    ok = false;
                    break;
                }
                if (pos < C) {
                    // 8 samples per lane and step: three aligned words, two funnel shifts to
                    // the first sample's byte, four byte permutes, one 16-byte store
                    const uint32_t src = raw0 + (uint32_t)(slot * kRawSlot + k * kRawPitch) +
                                         (off & ~3u) + 8u * lane;
                    const uint32_t dst = wide0 + (uint32_t)(slot * kWideSlot + k * kWidePitch) + 16u * lane;
                    const uint32_t bs = 8u * (off & 3u);
                    if (off & 4u) widen_channel<true>(src, dst, bs, n, lane);
                    else widen_channel<false>(src, dst, bs, n, lane);
                }
                tc::fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                    ptx::mbar_arrive(slot_full(slot));
                    ptx::mbar_arrive(raw_empty(slot));
                }
            }
            g += (uint32_t)nchunk;
            c0 += (uint32_t)(nchunk * kChunk);
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------- MMA issue
        if (lane == 0) {
            constexpr uint32_t kIdesc = (1u << 4) | ((128u >> 4) << 24);  // f16 x f16 -> f32, M = 128
            // descriptor of B: overlapping core matrices, 16 bytes between the halves of K
            // and 128 between 8-row groups (only the start address varies)
            const uint64_t desc_w = tc::smem_desc(wide0, 16, 128);
            const uint32_t dlo0 = (uint32_t)desc_w, dhi = (uint32_t)(desc_w >> 32);
            int slot = 0;
            uint32_t par = 0;
            bool ready = false;  // this chunk's slot is known to be full
            for (int64_t item = blockIdx.x; item < a.items && ok; item += gridDim.x) {
                int bi, blk;
                int64_t tile;
                mma_decode(a, item, &bi, &tile, &blk);
                const MmaBeam &bt = a.beam[bi];
                const MmaFrame *fr = bt.frames + bt.foff[blk];
                const int nfr = bt.foff[blk + 1] - bt.foff[blk];
                auto shape = [&](int rmax) {
                    return kIdesc | ((uint32_t)(frame_cols(bt.T, rmax) >> 3) << 17);
                };
                // the next frame's record is loaded ahead of its boundary
                int f = 1, next = nfr > 1 ? __ldg(&fr[1].pos) : INT32_MAX;
                int nrmax = nfr > 1 ? __ldg(&fr[1].rmax) : 0;
                uint32_t idesc = shape(__ldg(&fr[0].rmax));
                for (int pos = 0; pos < C; pos += kChunk) {
                    if (!ready && !ptx::mbar_wait(slot_full(slot), par, a.budget)) {
                        ok = false;
                        break;
                    }
                    ready = false;
                    tc::fence_after();
                    const uint32_t acol = tmem + kTmemA + (uint32_t)(slot * kChunk * 8);
                    const uint32_t dlo = dlo0 + (uint32_t)(slot * (kWideSlot / 16));
                    const uint32_t empty = slot_empty(slot);
                    if (++slot == kSlots) {
                        slot = 0;
                        par ^= 1u;
                    }
                    // straight-line issue of a whole chunk (a loop with the frame test costs its
                    // single lane 230 clocks per product, twice the product's own time); the
                    // next chunk's barrier is tested while the queue is full
                    if (pos + kChunk <= C && next >= pos + kChunk) {
                        mma_ts(tmem, acol, dlo, dhi, idesc, pos > 0 ? 1u : 0u);
#pragma unroll
                        for (int k = 1; k < kChunk; k++) {
                            mma_ts(tmem, acol + (uint32_t)(k * 8), dlo + (uint32_t)(k * (kWidePitch / 16)),
                                   dhi, idesc, 1u);
                            if (k == kChunk / 2) ready = ptx::mbar_try_wait(slot_full(slot), par);
                        }
                        tc::mma_commit(empty);
                        continue;
                    }
                    const int n = min(kChunk, C - pos);
                    for (int k = 0; k < n && ok; k++) {
                        while (next == pos + k) {
                            tc::mma_commit(frame_done);
                            if (!ptx::mbar_wait(rows_moved, ev & 1u, a.budget)) {
                                ok = false;
                                break;
                            }
                            ev++;
                            tc::fence_after();
                            idesc = shape(nrmax);
                            f++;
                            next = f < nfr ? __ldg(&fr[f].pos) : INT32_MAX;
                            nrmax = f < nfr ? __ldg(&fr[f].rmax) : 0;
                        }
                        if (!ok) break;
                        mma_ts(tmem, acol + (uint32_t)(k * 8), dlo + (uint32_t)(k * (kWidePitch / 16)), dhi,
                               idesc, (pos | k) != 0 ? 1u : 0u);
                    }
                    tc::mma_commit(empty);
                }
                if (!ok) break;
                tc::mma_commit(frame_done);
                if (!ptx::mbar_wait(rows_moved, ev & 1u, a.budget)) {
                    ok = false;
                    break;
                }
                ev++;
                tc::fence_after();
            }
            if (!ok) {  // nothing of this CTA's may be running when tensor memory is freed
                tc::mma_commit(drained);
                (void)ptx::mbar_wait(drained, 0u, kWaitLimit);
            }
        }
        ok = __all_sync(0xffffffffu, ok);
    } else if (!a.starve) {
        // ------------------------------------------------------- copies
        const int grp = warp - kCopyWarp;
        for (int64_t item = blockIdx.x; item < a.items && ok; item += gridDim.x) {
            int bi, blk;
            int64_t tile;
            mma_decode(a, item, &bi, &tile, &blk);
            const MmaBeam &bt = a.beam[bi];
            const int T = bt.T;
            // t0 is a multiple of 16; positions below 64 bits are relative to a window (a delay
            // may be up to 2^31 - 1)
            const int64_t t0 = tile * T, left = bt.n_in - t0;
            const int before = (int)min(t0, (int64_t)4096);  // input before the tile, if little
            const int32_t *base = bt.base + (int64_t)blk * C;
            const int32_t *crmax = bt.crmax + (int64_t)blk * nchunk;
            const int k = lane;  // channel of the chunk (lanes 0..7)
            int ch = (grp + kCopyWarps - (int)(g % kCopyWarps)) % kCopyWarps;
            const int64_t step = (bt.rev ? -1 : 1) * bt.x_stride;
            const uint8_t *row = bt.x + t0 + (bt.rev ? (int64_t)(C - 1) * bt.x_stride : 0) +
                                 step * (ch * kChunk + k);
            int nbase = k < kChunk && ch * kChunk + k < C ? __ldg(base + ch * kChunk + k) : 0;
            int nrm = ch < nchunk ? __ldg(crmax + ch) : 0;
            for (; ch < nchunk; ch += kCopyWarps, row += step * (kCopyWarps * kChunk)) {
                const uint32_t gc = g + (uint32_t)ch;
                const int slot = (int)(gc % kSlots);
                const int pos = ch * kChunk + k;
                const bool in = k < kChunk && pos < C;
                const int off = nbase & 15, w0 = nbase - off;  // the window starts 16-byte aligned
                const int need = 8 * (frame_cols(T, nrm) + 1);  // samples from it
                if (ch + kCopyWarps < nchunk) {
                    const int np = pos + kCopyWarps * kChunk;
                    nbase = k < kChunk && np < C ? __ldg(base + np) : 0;
                    nrm = __ldg(crmax + ch + kCopyWarps);
                }
                // bytes [lo, hi) of the window, whole 16-byte pieces up to hi16; the samples before
                // the input (only columns of t < 0 take them) and past its end are left as they are
                const int hi = (int)min(left - w0, (int64_t)((off + need + 15) & ~15)), hi16 = hi & ~15;
                const int lo = w0 < 0 ? max(-w0 - before, 0) : 0;
                const uint32_t bytes = in && hi16 > lo ? (uint32_t)(hi16 - lo) : 0u;
                const uint32_t tot = __reduce_add_sync(0xffffffffu, bytes);
                if (!__all_sync(0xffffffffu, ptx::mbar_wait(raw_empty(slot), ((gc / kSlots) & 1u) ^ 1u,
                                                            a.budget))) {
                    ok = false;
                    break;
                }
                const uint32_t dst = (uint32_t)(slot * kRawSlot + k * kRawPitch);
                if (in && hi > hi16)  // the last bytes of the input
                    for (int i = max(lo, hi16); i < hi; i++) raw[dst + (uint32_t)i] = row[(int64_t)w0 + i];
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_expect_tx(raw_full(slot), tot);
                __syncwarp();
                if (bytes > 0)
                    ptx::bulk_g2s(raw0 + dst + (uint32_t)lo, row + ((int64_t)w0 + lo), bytes, raw_full(slot));
                last = gc + 1u;
            }
            g += (uint32_t)nchunk;
        }
        // never leave with copies in flight (the last phases this warp began)
        for (uint32_t i = last > (uint32_t)kSlots ? last - kSlots : 0u; i < last; i++)
            if (i % kCopyWarps == (last - 1u) % kCopyWarps &&
                !__all_sync(0xffffffffu, ptx::mbar_wait(raw_full((int)(i % kSlots)), (i / kSlots) & 1u,
                                                        kWaitLimit))) {
                ok = false;
                break;
            }
    }
    if (!ok && lane == 0) atomicExch(a.err, 1);
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

}  // namespace

namespace {

struct Range {
    int lo, hi;
};

// The range of x[i] - y[i] over a block.
Range range_of(const int32_t *x, const int32_t *y) {
    int32_t lo = INT32_MAX, hi = INT32_MIN;
    for (int i = 0; i < kKdm; i++) {
        const int32_t v = x[i] - y[i];
        lo = std::min(lo, v);
        hi = std::max(hi, v);
    }
    return Range{lo, hi};
}

// Delays of block b by position, the 16 trials side by side (loops over them vectorise).
void block_delays(const int32_t *delays, int ndm, int C, bool rev, int npos, int b, int32_t *dl) {
    for (int i = 0; i < kKdm; i++) {
        const int32_t *row = delays + (size_t)std::min(ndm - 1, b * kKdm + i) * C;
        int32_t *d = dl + i;
        if (rev)
            for (int pos = 0; pos < npos; pos++) d[(size_t)pos * kKdm] = row[C - 1 - pos];
        else
            for (int pos = 0; pos < npos; pos++) d[(size_t)pos * kKdm] = row[pos];
    }
}

// The frames of one block, each followed by visit(position, smallest delay - R) for its
// positions; R is left at the last frame's.  false if a row moves further than a tile.
template <typename Visit>
bool block_frames(const int32_t *dl, int npos, int32_t (&R)[kKdm], std::vector<MmaFrame> *frames,
                  Visit visit) {
    for (int i = 0; i < kKdm; i++) R[i] = 0;
    bool first = true;
    int rmax = 0;
    for (int p0 = 0; p0 < npos;) {
        // centre the frame on the furthest channel whose delays differ from those of
        // p0 by amounts within 8 samples of each other, with moves of at most 16
        const int32_t *d0 = dl + (size_t)p0 * kKdm;
        int best = p0;
        for (int pos = p0; pos < npos; pos++) {
            const int32_t *d = dl + (size_t)pos * kKdm;
            const Range dv = range_of(d, d0), ev = range_of(d, R);
            if (dv.hi - dv.lo > kMaxShift || (!first && ev.hi - ev.lo > kMaxMove)) break;
            best = pos;
        }
        const int32_t *ref = dl + (size_t)best * kKdm;
        for (bool more = true; more;) {
            const int elo = range_of(ref, R).lo;
            MmaFrame fr;
            fr.pos = p0;
            more = false;
            rmax = 0;
            for (int i = 0; i < kKdm; i++) {
                int e = ref[i] - R[i] - elo;
                if (!first && e > kMaxMove) {  // a steep step: several moves
                    e = kMaxMove;
                    more = true;
                }
                fr.e[i] = first ? 0 : (uint8_t)e;
                R[i] += e;
                rmax = std::max(rmax, (int)R[i]);
            }
            fr.rmax = rmax;
            if (rmax > 8 * kCols) return false;
            frames->push_back(fr);
            first = false;
        }
        int pos = p0;
        for (; pos < npos; pos++) {
            const Range v = range_of(dl + (size_t)pos * kKdm, R);
            if (v.hi - v.lo > kMaxShift) break;
            visit(pos, v.lo, rmax);
        }
        p0 = pos;
    }
    return true;
}

}  // namespace

bool mma_plan_tables(const int32_t *delays, int ndm, int C, bool rev, int npos, MmaTables *t) {
    const int nblk = (ndm + kKdm - 1) / kKdm, nchunk = (npos + kChunk - 1) / kChunk;
    t->base.assign((size_t)nblk * npos, 0);
    t->shift.assign((size_t)nblk * nchunk * kKdm * kChunk, 0);
    t->crmax.assign((size_t)nblk * nchunk, 0);
    t->rlast.assign((size_t)nblk * kKdm, 0);
    t->foff.assign(1, 0);
    t->frames.clear();
    t->rmax = 0;
    t->mean_cols_r = 0.0;
    // the blocks are independent; their frames are put together at the end
    std::vector<std::vector<MmaFrame>> fr((size_t)nblk);
    std::vector<double> sum_r((size_t)nblk, 0.0);
    std::atomic<bool> fits{true};
    const bool ran = parallel_ranges(nblk, std::max(1, 30000 / (npos * kKdm)), [&](int64_t b0, int64_t b1) {
        std::vector<int32_t> dl((size_t)npos * kKdm);
        for (int64_t b = b0; b < b1 && fits; b++) {
            block_delays(delays, ndm, C, rev, npos, (int)b, dl.data());
            int32_t R[kKdm];
            if (!block_frames(dl.data(), npos, R, &fr[b], [&](int pos, int lo, int rmax) {
                    const int32_t *d = dl.data() + (size_t)pos * kKdm;
                    t->base[(size_t)b * npos + pos] = lo;
                    uint8_t *sh = t->shift.data() + ((size_t)b * nchunk + pos / kChunk) * kKdm * kChunk +
                                  pos % kChunk;
                    for (int i = 0; i < kKdm; i++) sh[i * kChunk] = (uint8_t)(d[i] - R[i] - lo);
                    int32_t &cr = t->crmax[(size_t)b * nchunk + pos / kChunk];
                    cr = std::max(cr, rmax);
                    sum_r[b] += rmax;
                }))
                fits = false;
            for (int i = 0; i < kKdm; i++) t->rlast[(size_t)b * kKdm + i] = R[i];
        }
    });
    if (!ran || !fits) return false;
    for (int b = 0; b < nblk; b++) {
        t->frames.insert(t->frames.end(), fr[b].begin(), fr[b].end());
        t->foff.push_back((int32_t)t->frames.size());
        t->mean_cols_r += sum_r[b];
    }
    for (int32_t r : t->rlast) t->rmax = std::max(t->rmax, (int)r);
    t->mean_cols_r /= (double)nblk * npos;
    return true;
}

int mma_split(const int32_t *delays, int ndm, int C, bool rev, int step, double other_rate,
              double other_fixed) {
    const int nblk = (ndm + kKdm - 1) / kKdm;
    // the last block but one (complete, and as steep as any on a uniform grid)
    std::vector<int32_t> dl((size_t)C * kKdm);
    block_delays(delays, ndm, C, rev, C, std::max(0, nblk - 2), dl.data());
    std::vector<MmaFrame> frames;
    int32_t R[kKdm];
    int reach = 0;  // positions whose rows stay within a tile
    (void)block_frames(dl.data(), C, R, &frames, [&](int pos, int, int) { reach = pos + 1; });
    // clocks per sample of 16 trials: at least a twentieth less
    double best = 0.95 * 16.0 * (C / other_rate + other_fixed);
    int npos = 0;
    size_t f = 0;
    double sum_r = 0.0;
    int at = 0;
    // the rest's rows start or end at the split, depending on the order: whole steps of them
    // before it, or whole steps of positions
    for (int n = rev && C % step ? C % step : step; n < std::min(C, reach + 1); n += step) {
        const int rest = C - n;
        for (; at < n; at++) {
            while (f < frames.size() && frames[f].pos <= at) f++;
            sum_r += frames[f - 1].rmax;
        }
        MmaShape m;
        m.rmax = frames[f - 1].rmax + frames[f - 1].rmax / 8;  // other blocks may drift a little further
        m.mean_r = sum_r / n;
        m.frames_per_block = (double)f;
        const int T = mma_tile_len(m.rmax);
        if (T < 512 || n < 256) continue;
        const double c = mma_item_clocks(m, n, T, true) / T + 16.0 * (rest / other_rate + other_fixed);
        if (c < best) {
            best = c;
            npos = n;
        }
    }
    return npos;
}

int mma_tile_len(int rmax) { return std::max(0, (8 * kCols - rmax) & ~15); }

// Measured on GB300: 165 clocks per channel at T + R = 1840 samples (the product, N = 240,
// takes 120; the rest is the shared-memory port's, see above) and not under 152 for a
// shorter tile, 5,500 per frame boundary (drain, move, restart), 14,000 per item for its
// start and epilogue, 8 per sample for reading the series that it adds to (17 without the
// lines fetched ahead: 842 channels, 2062 trials 2046 us, 1956 with).  Within 4% of 23 out of
// 26 launches of 74 to 4096 channels, 6 and 12% high at 74 channels and 5% at 664; the choice
// by it was within 2% of the fastest kernel but at 74 channels (3 and 7%, between two
// byte variants).  The same without the floor and with 4,000 per boundary was up to 40% low,
// and took grids of step 0.75 at 1000-1300 channels (2.50 ms) from the byte kernel (2.23).
double mma_item_clocks(const MmaShape &m, int nchan, int T, bool add) {
    return nchan * std::max(152.0, 0.67 * ((T + m.mean_r) / 8.0 + 8.0) + 4.0) +
           m.frames_per_block * (14.0 * T / 8.0 + 2900.0) + 14000.0 + (add ? 8.0 * T : 0.0);
}

double mma_launch_clocks(const MmaShape &m, int nchan, int ndm, int64_t n_out, int num_sms, bool add,
                         int *tile) {
    const int nblk = (ndm + kKdm - 1) / kKdm, tmax = mma_tile_len(m.rmax);
    *tile = 0;
    if (tmax < 16) return 1e30;
    // the longest tile, or the shorter one whose waves of work items take least
    const int64_t lo = (n_out + tmax - 1) / tmax;
    double best = 0.0;
    for (int64_t k = lo; k == lo || (k <= 4 * lo && k <= lo + 64); k++) {
        const int T = std::min(tmax, (int)(((n_out + k - 1) / k + 15) & ~(int64_t)15));
        if (T < 256 && k > lo) break;
        const int64_t items = (n_out + T - 1) / T * nblk;
        const double c = (double)((items + num_sms - 1) / num_sms) * mma_item_clocks(m, nchan, T, add);
        if (*tile == 0 || c < best) {
            best = c;
            *tile = T;
        }
    }
    return best + kLaunchClocks;
}

cudaError_t launch_dedisperse_mma(const BeamLaunch *beams, int nbeams, bool add, int num_sms, int *err,
                                  cudaStream_t s, int32_t *nlaunch) {
    if (nbeams < 1 || nbeams > kMmaMaxBeams) return cudaErrorInvalidValue;
    cudaError_t e = ensure_kernel_smem(reinterpret_cast<const void *>(dd_mma_kernel), kSmem);
    if (e != cudaSuccess) return e;
    MmaArgs a;
    std::memset(&a, 0, sizeof(a));
    a.nchan = beams[0].plan->mma.shape.npos;
    int64_t items = 0;
    for (int b = 0; b < nbeams; b++) {
        const BeamLaunch &in = beams[b];
        const gsp_plan_s *p = in.plan;
        if (p->mma.shape.npos != a.nchan || !p->mma.d_frames) return cudaErrorInvalidValue;
        MmaBeam &bt = a.beam[b];
        bt.rev = p->desc.freq_descending ? 0 : 1;
        // the first npos positions: the last npos rows, or the first ones
        bt.x = in.x + (bt.rev ? (int64_t)(p->desc.nchan - a.nchan) * in.x_stride : 0);
        bt.x_stride = in.x_stride;
        bt.add = add ? 1 : 0;
        bt.n_in = in.n_in;
        bt.n_out = in.n_out;
        bt.base = p->mma.d_base;
        bt.shift = p->mma.d_shift;
        bt.frames = p->mma.d_frames;
        bt.foff = p->mma.d_foff;
        bt.crmax = p->mma.d_crmax;
        bt.rlast = p->mma.d_rlast;
        bt.out = in.out;
        bt.out_stride = in.out_stride;
        bt.bsum = in.bsum;
        bt.nb_max = p->nb_max;
        bt.B = p->desc.block_len;
        bt.Ls = (in.n_out / bt.B) * bt.B;
        bt.ndm = p->desc.ndm;
        bt.nblk = (p->desc.ndm + kKdm - 1) / kKdm;
        bt.grp = p->geom.grp[kdm_index(kKdm)];
        if (in.bsum && (bt.B < kMmaMinBlock || bt.B > kMmaMaxBlock)) return cudaErrorInvalidValue;
        // the longest tiles for a batch, those of the best wave count for one beam
        const int tmax = mma_tile_len(p->mma.shape.rmax);
        if (tmax < 16) return cudaErrorInvalidValue;
        const int64_t nt = (in.n_out + tmax - 1) / tmax;
        bt.T = std::min(tmax, (int)(((in.n_out + nt - 1) / nt + 15) & ~(int64_t)15));
        if (nbeams == 1)
            (void)mma_launch_clocks(p->mma.shape, a.nchan, p->desc.ndm, in.n_out, num_sms, add, &bt.T);
        bt.ntiles = (in.n_out + bt.T - 1) / bt.T;
        bt.item0 = items;
        items += bt.ntiles * bt.nblk;
    }
    a.nbeams = nbeams;
    a.err = err;
    a.items = items;
    a.budget = beams[0].plan->wait_budget;
    a.starve = beams[0].plan->wait_starve;
    const int64_t grid = std::min<int64_t>(items, num_sms);
    if (grid < 1) return cudaErrorInvalidConfiguration;
    dd_mma_kernel<<<(unsigned)grid, kThreads, kSmem, s>>>(a);
    *nlaunch += 1;
    return cudaGetLastError();
}

}  // namespace gsp
