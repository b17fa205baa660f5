// Dense large kernel (ESC paper, Section 3.2: LK in R^{KxKx16x16}; Eq. 4 line 3 with that LK) on the FP32 pipe, for fp32
// tensors in either layout and for the bf16 ones that the tensor-core kernels do not take:
//
//   out[b,n,y,x] = sum_{k,i,j} w_dense[n,k,i,j] x[b,k,y+i-P,x+j-P] + sum_{i,j} dk[b,n,i,j] x[b,n,y+i-1,x+j-1] (+ bias[b,n])
//
// Bound: FP32 FMA pipe (16 * 16 * K * K multiply-adds per pixel against 128 bytes of attention channels).  fp32 products
// have no exact form on the tensor cores, so the arithmetic stays fp32 and the point is to keep the pipe busy: a thread owns
// 8 pixels of a row x 8 output channels, as 32 pairs of neighbouring channels for the packed multiply-add (two per
// instruction: with scalar ones the kernel was a tenth slower).  The staged inputs are doubled (x, x), so that a 16-byte
// read is two ready operands.  Per (input channel, kernel row), K = 13: ten reads of inputs, two reads of weights per tap
// that all lanes share, 416 packed multiply-adds (832 issue cycles) -- 36 reads beside them.  Lane order: eight consecutive
// lanes are 2 positions of 8 pixels x 4 rows, and the row pitch is 4 mod 16 words, so that the 16-byte reads of a phase
// fall in distinct banks.
//
// A block of 128 threads (four warps: the two halves of the output channels x two groups of four rows) computes a tile of
// 64 x 8 pixels, one input channel at a time: halo tile and that channel's K x K x 16 weights, tap-major, fetched with
// cp.async into a second buffer while the previous channel is multiplied (bf16 values are converted, so they are loaded and
// stored).  The input channels may be split over a cluster of 2, 4 or 8 blocks, whose accumulators are added
// through distributed shared memory in rank order: small maps then fill the chip (64x64 pixels are 8 tiles) and large ones
// balance better over it; `choose_split` has the rule.  dk is merged into the weights of its channel; the
// kernel rows that carry it (the middle three) come last, so the kernel before this one (which writes dk) is waited for
// only after the first channel's other rows.
// Measured: 640x360 fp32 NCHW, whole forward 7,330 us (one thread per output) -> 402 us, 0.67 of the FP32 pipe's 268 us; 16
// patches of 64x64 131 us.  What is left beside the 832 issue cycles of a row: the packed multiply-add's three 64-bit operands
// and the reads' write-back share the register file (the order of the products and the number of resident warps change 3 % each).
#pragma once
#include "common.cuh"
#include "stencil_generic.cuh"
#include "conv_fuse.cuh"
#include <cooperative_groups.h>
#include <algorithm>

namespace esc { namespace dense32 {

constexpr int CA = 16, TX = 64, TY = 8, PX = 8, NH = 8, kThreads = 128, kWPitch = 20;   // 20: taps fall in eight bank groups while staging
constexpr int kAcc = PX * NH;

template <int K> struct Geo {
    static constexpr int Rows = TY + K - 1;
    static constexpr int Cols = TX + K - 1;
    static constexpr int Pitch = (2 * Cols + 11) / 16 * 16 + 4;       // words per staged row of doubled values: 4 mod 16
    static constexpr int kTile = Rows * Pitch;
    static constexpr int kStage = kTile + K * K * kWPitch;
    static constexpr int kRed = kAcc * kThreads;                      // the accumulators of a block, for the cluster's sum
    static constexpr size_t smem_bytes(int split) { return sizeof(float) * (size_t)(split > 1 && kRed > 2 * kStage ? kRed : 2 * kStage); }
    static_assert(Pitch >= 2 * Cols && Pitch % 16 == 4 && kTile % 4 == 0 && Cols <= 96, "16-byte rows, distinct banks; staging");
};

__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

template <typename T, int LAYOUT, int K>
__global__ void __launch_bounds__(kThreads, 4)
stencil_dense_fp32(const T* __restrict__ x, T* __restrict__ out, int C, int H, int W, const T* __restrict__ w_dense,
                   const float* __restrict__ dk, const float* __restrict__ bias, int tiles_x, int tiles_y, int split, const CopyJob job)
{
    namespace cg = cooperative_groups;
    using G = Geo<K>;
    constexpr int P = (K - 1) / 2, Pitch = G::Pitch;
    extern __shared__ __align__(16) float sm[];
    // two buffers of [tile: Rows x Pitch | weights: K*K taps x kWPitch, 16 output channels each]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, half = warp & 1;
    if (job.blocks != 0 && blockIdx.x >= job.first_block) {              // whole clusters of copy blocks
        run_copy_job(job, blockIdx.x - job.first_block, tid, kThreads);
        return;
    }
    unsigned u = blockIdx.x;
    const int rank = (int)(u % (unsigned)split); u /= (unsigned)split;
    const int tx = (int)(u % (unsigned)tiles_x); u /= (unsigned)tiles_x;
    const int ty = (int)(u % (unsigned)tiles_y);
    const int b = (int)(u / (unsigned)tiles_y);
    const int xpos = (lane & 1) + 2 * (lane >> 3), row = ((lane >> 1) & 3) + 4 * (warp >> 1);
    const int x0 = tx * TX - P, y0 = ty * TY - P;

    unsigned long long acc2[PX][NH / 2];                  // output channels 2q, 2q + 1 of this half
#pragma unroll
    for (int p = 0; p < PX; ++p)
#pragma unroll
        for (int q = 0; q < NH / 2; ++q) acc2[p][q] = 0ull;

    auto stage = [&](int k, float* buf) {                 // a warp takes every fourth halo row and four output channels' taps
#pragma unroll 1
        for (int r = warp; r < G::Rows; r += 4) {
            const int yy = y0 + r;
            const bool rv = yy >= 0 && yy < H;
            float* dst = buf + r * Pitch + 2 * lane;
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                const int xx = x0 + lane + 32 * u;
                const bool v = rv && xx >= 0 && xx < W;
                if (32 * u + lane < G::Cols) {
                    const T* src = x + (v ? elem_index<LAYOUT>(b, k, yy, xx, C, H, W) : 0);
                    if constexpr (sizeof(T) == 4) {
                        const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + 64 * u);
                        fuse::cp_async4(d, src, v);
                        fuse::cp_async4(d + 4, src, v);
                    } else {
                        const float f = v ? Elem<T>::to_f32(*src) : 0.f;
                        *reinterpret_cast<float2*>(dst + 64 * u) = make_float2(f, f);
                    }
                }
            }
        }
        float* wm = buf + G::kTile;
#pragma unroll 1
        for (int n = warp; n < CA; n += 4) {
            const T* wk = w_dense + ((size_t)n * CA + k) * K * K;
#pragma unroll
            for (int u = 0; u < (K * K + 31) / 32; ++u) {
                const int t = lane + 32 * u;
                if (t < K * K) {
                    if constexpr (sizeof(T) == 4) fuse::cp_async4((uint32_t)__cvta_generic_to_shared(wm + t * kWPitch + n), wk + t, true);
                    else wm[t * kWPitch + n] = Elem<T>::to_f32(wk[t]);
                }
            }
        }
        fuse::cp_async_commit();
    };
    const int per = CA / split;
    stage(rank * per, sm);
    for (int s = 0; s < per; ++s) {
        const int k = rank * per + s;
        float* tile = sm + (s & 1) * G::kStage;
        float* wm = tile + G::kTile;
        if (s + 1 < per) stage(k + 1, sm + ((s + 1) & 1) * G::kStage);
        else fuse::cp_async_commit();
        fuse::cp_async_wait<1>();
        __syncthreads();                                  // this channel is there for every warp
#pragma unroll 1
        for (int ii = 0; ii < K; ++ii) {
            if (ii == K - 3) {                            // the middle rows: merge dk first (Eq. 5 for the diagonal channel)
                if (s == 0) pdl_wait_primary();
                if (tid < 9) wm[((P - 1 + tid / 3) * K + P - 1 + tid % 3) * kWPitch + k] += __ldcg(dk + ((size_t)b * CA + k) * 9 + tid);
                __syncthreads();
            }
            const int i = ii < P - 1 ? ii : ii < K - 3 ? ii + 3 : ii - (K - 3) + P - 1;
            unsigned long long in[PX + K - 1];            // (x, x)
            const ulonglong2* xr = reinterpret_cast<const ulonglong2*>(tile + (row + i) * Pitch + 2 * xpos * PX);
#pragma unroll
            for (int v = 0; v < (PX + K - 1) / 2; ++v) {
                const ulonglong2 q = xr[v];
                in[2 * v] = q.x; in[2 * v + 1] = q.y;
            }
            const ulonglong2* wr = reinterpret_cast<const ulonglong2*>(wm + i * K * kWPitch + half * NH);
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const ulonglong2 w0 = wr[j * (kWPitch / 4)], w1 = wr[j * (kWPitch / 4) + 1];
                const unsigned long long w[NH / 2] = {w0.x, w0.y, w1.x, w1.y};
#pragma unroll
                for (int q = 0; q < NH / 2; ++q)
#pragma unroll
                    for (int p = 0; p < PX; ++p) {        // back and forth: each product shares an operand with the one before
                        const int pp = (q & 1) ? PX - 1 - p : p;
                        fma2(acc2[pp][q], w[q], in[pp + j]);
                    }
            }
        }
        __syncthreads();                                  // this buffer may be refilled
    }
    float acc[PX][NH];
#pragma unroll
    for (int p = 0; p < PX; ++p)
#pragma unroll
        for (int q = 0; q < NH / 2; ++q) {
            acc[p][2 * q] = __uint_as_float((unsigned)acc2[p][q]);
            acc[p][2 * q + 1] = __uint_as_float((unsigned)(acc2[p][q] >> 32));
        }

    const int oy = ty * TY + row, ox = tx * TX + xpos * PX;
    if (split == 1) {
        if (oy >= H) return;
        float c0[NH];
#pragma unroll
        for (int n = 0; n < NH; ++n) c0[n] = bias ? bias[(size_t)b * CA + half * NH + n] : 0.f;
#pragma unroll
        for (int p = 0; p < PX; ++p)
            if (ox + p < W) {
#pragma unroll
                for (int n = 0; n < NH; ++n)
                    out[elem_index<LAYOUT>(b, half * NH + n, oy, ox + p, C, H, W)] = Elem<T>::from_f32(acc[p][n] + c0[n]);
            }
        return;
    }
    // Add the cluster's accumulators: every block parks its own in shared memory, and each sums a share of them over the
    // ranks in order.  A share is whole channels (NCHW) or whole pixels (NHWC), so that what is written is contiguous.
    cg::cluster_group cluster = cg::this_cluster();
#pragma unroll
    for (int p = 0; p < PX; ++p)
#pragma unroll
        for (int n = 0; n < NH; ++n) sm[(LAYOUT == kNCHW ? n * PX + p : p * NH + n) * kThreads + tid] = acc[p][n];
    cluster.sync();
    const int share = kAcc / split;
    for (int v0 = rank * share; v0 < (rank + 1) * share; v0 += 8) {
        float t[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) t[q] = 0.f;
        for (int r = 0; r < split; ++r) {
            const float* src = cluster.map_shared_rank(sm, r) + v0 * kThreads + tid;
#pragma unroll
            for (int q = 0; q < 8; ++q) t[q] += src[q * kThreads];
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int n = half * NH + (LAYOUT == kNCHW ? v0 / PX : q), p = LAYOUT == kNCHW ? q : v0 / NH;
            if (oy < H && ox + p < W)
                out[elem_index<LAYOUT>(b, n, oy, ox + p, C, H, W)] = Elem<T>::from_f32(t[q] + (bias ? bias[(size_t)b * CA + n] : 0.f));
        }
    }
    cluster.sync();                                       // nobody leaves while its accumulators are being read
}

// Blocks of a cluster (1, 2, 4, 8) that share a tile's sixteen input channels.  The blocks of an SM take turns on its four
// schedulers (a block is a warp on each), so the launch takes about (blocks per SM, rounded up) times a block's 16 / split
// channels plus the exchange -- and a quarter more where one block has an SM to itself (18.8 k cycles per channel, 17.2 k
// side by side with another, 15 k with four).  Measured, fp32 NCHW, K = 13, whole forward, split 1 / 2 / 4 / 8: 64x64 153 / 81 /
// 44 / 26 us; 320x180 274 / 141 / 135 / 119; 427x240 274 / 202 / 198 / 198; 640x360 518 / 439 / 413 / 422.
inline int choose_split(long long tiles, int sms) {
    int best = 1;
    double best_cost = 1e30;
    for (int split = 1; split <= 8; split *= 2) {
        const double per_sm = (double)((tiles * split + sms - 1) / sms);
        const double cost = per_sm * (16.0 / split + 0.3) * (1.0 + 0.25 / std::min(per_sm, 4.0));
        if (cost < best_cost * 0.99) { best_cost = cost; best = split; }
    }
    return best;
}

}}  // namespace esc::dense32
