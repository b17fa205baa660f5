// Backward pass of the module's closing 1x1 convolution (ESC paper, Eq. 4 line 4, with the block's residual, Eq. 3
// line 3):  out = W_fuse cat + b_fuse + residual  per pixel.  With go = dL/dout:
//
//   g_cat[c]  = sum_n W_fuse[n,c] go[n]          per pixel
//   g_W[n,c]  = sum_pixels go[n] cat[c]
//   g_b[n]    = sum_pixels go[n]
//   (the residual's gradient is go itself)
//
// bf16, C in {32, 48, 64}: all three in ONE pass over go and cat on the tensor cores (below).  Elsewhere: conv_fuse_fp32 with
// the transposed matrix and wgrad_fp32 (conv_fuse_fp32.cuh).  Blocks write their sums of g_W and g_b once; `sum_wgrad` adds
// them in block order.
#pragma once
#include "common.cuh"
#include "stencil_toeplitz.cuh"
#include "conv_fuse.cuh"
#include "conv_fuse_fp32.cuh"

namespace esc { namespace fuse { namespace bwd {

constexpr int kThreads = 256;
inline bool supported(int C) { return f32::supported(C); }

// ---- bf16 on the tensor cores --------------------------------------------------------------------------------------------
// A block takes a run of pixels (passes of 256), 128 at a time through three buffers filled with cp.async, two of them in flight.
// g_W = go^T [C x pixels] . cat [pixels x C] is one matrix product with the pixels as the contraction axis (bf16 products are
// exact in fp32, the accumulation is fp32): warp w owns pixels 16 w .. 16 w + 15 of every piece and the whole C x C accumulator
// (C = 64: 128 registers), (C/16) x (C/8) mma.sync.m16n8k16 per piece plus C/16 with a B operand of ones for g_b.  g_cat of the
// same 16 pixels is go times W, whose fragments come from shared memory; it is written over the warp's own go values and
// stored from there.  At the end the warps put their accumulators side by side into shared memory and the block adds
// them per element in warp order.
// Bound: HBM -- go and cat read, g_cat written, 6 C bytes per pixel (2 KFLOP at C = 64 each way).  64 patches of 64x64, C = 64:
// 19.5 us for the sums, 2.8 for a transposed copy of W and 15.2 for g_cat as kernels of their own (134 MB); one pass of 101 MB
// now, 15 us less of the whole backward pass; its floor at the copy bandwidth is 15.6 us.
// Rows of a staged piece: pixels of C channels (NHWC) or channels of 128 pixels (NCHW, H W a multiple of 8 so that eight
// consecutive pixels of the flat list lie in one image), 16 bytes longer than that, so that the eight rows of an ldmatrix fall
// into different banks; what is transposed for one layout is not for the other.
namespace mma {
using tma::toep::ldsm_x4; using tma::toep::ldsm_x4_trans; using tma::toep::mma_bf16;
constexpr int kPiece = 128;                                        // pixels per buffer: 16 per warp
constexpr int kStages = 3;

template <int LAYOUT, int C> struct MGeom {
    static constexpr int PITCH = LAYOUT == kNHWC ? C * 2 + 16 : kPiece * 2 + 16;   // bytes per staged row
    static constexpr int TILE = (LAYOUT == kNHWC ? kPiece : C) * PITCH;            // one tensor, one buffer
    static constexpr int WPITCH = C * 2 + 16, WBYTES = C * WPITCH;                 // W as it is: rows n, columns c
    static constexpr size_t kStageBytes = (size_t)kStages * 2 * TILE + WBYTES;
    static constexpr size_t kSumBytes = (size_t)(kThreads / 32) * (C * C + C) * sizeof(float);   // every warp's sums side by side
    static constexpr size_t kSmemBytes = kStageBytes > kSumBytes ? kStageBytes : kSumBytes;
    static_assert(kSmemBytes <= 227 * 1024, "shared memory");
};

template <int LAYOUT, int C>
__global__ void __launch_bounds__(kThreads, 1)
fuse_backward_bf16(const __nv_bfloat16* __restrict__ cat, const __nv_bfloat16* __restrict__ go, const __nv_bfloat16* __restrict__ w,
                   __nv_bfloat16* __restrict__ g_cat, long long HW, long long pixels, int passes,
                   float* __restrict__ part)                       // [gridDim.x][C * C + C]
{
    using G = MGeom<LAYOUT, C>;
    constexpr int MT = C / 16, NT = C / 8, CH = C / 8;              // m tiles, n tiles, 16-byte pieces of a pixel's channels
    constexpr bool kNh = LAYOUT == kNHWC;
    extern __shared__ __align__(128) unsigned char smb[];
    pdl_launch_dependents();                                        // sum_wgrad may be scheduled; it waits for this grid's end
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int mi = lane >> 3, mr = lane & 7;
    const uint32_t sm0 = tma::smem_u32(smb), wsm = sm0 + (uint32_t)(kStages * 2 * G::TILE);
    // ldmatrix lane addresses inside a tile.  Sums: (channels 0-7 | 8-15 of a group) x (pixels 0-7 | 8-15 of the warp's 16).
    const uint32_t lane_sum = kNh ? (uint32_t)((16 * warp + 8 * (mi >> 1) + mr) * G::PITCH + (mi & 1) * 16)
                                  : (uint32_t)((8 * (mi & 1) + mr) * G::PITCH + (16 * warp + 8 * (mi >> 1)) * 2);
    // go as the other product's operand: NHWC as A (pixels 0-7 | 8-15 x channels 0-7 | 8-15), NCHW as B (channels x pixels)
    const uint32_t lane_go = kNh ? (uint32_t)((16 * warp + 8 * (mi & 1) + mr) * G::PITCH + (mi >> 1) * 16)
                                 : (uint32_t)((8 * (mi & 1) + mr) * G::PITCH + (16 * warp + 8 * (mi >> 1)) * 2);
    // W [n][c], always transposed: NHWC as B (k = n halves, then the next eight columns c), NCHW as A (rows c, k = n)
    const uint32_t lane_w = wsm + (kNh ? (uint32_t)((8 * (mi & 1) + mr) * G::WPITCH + (mi >> 1) * 16)
                                       : (uint32_t)((8 * (mi >> 1) + mr) * G::WPITCH + (mi & 1) * 16));
    for (int e = tid; e < C * CH; e += kThreads)
        cp_async16(wsm + (uint32_t)((e / CH) * G::WPITCH + (e % CH) * 16), w + (size_t)e * 8, true);
    float acc[MT][NT][4], accb[MT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m) {
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[m][n][v] = 0.f;
#pragma unroll
        for (int v = 0; v < 4; ++v) accb[m][v] = 0.f;
    }
    const long long first = (long long)blockIdx.x * passes * kThreads;             // the block's run of pixels
    const long long last = first + (long long)passes * kThreads < pixels ? first + (long long)passes * kThreads : pixels;
    const int pieces = first < last ? (int)((last - first + kPiece - 1) / kPiece) : 0;
    auto stage = [&](int s) {
        const long long p0 = first + (long long)s * kPiece;
        const uint32_t gbuf = sm0 + (uint32_t)((s % kStages) * 2 * G::TILE), cbuf = gbuf + G::TILE;
        if (kNh) {
#pragma unroll
            for (int u = 0; u < kPiece * CH / kThreads; ++u) {
                const int e = tid + u * kThreads, r = e / CH, q = e % CH;
                const long long px = p0 + r;
                const bool valid = px < last;
                const size_t src = (size_t)(valid ? px : first) * C + q * 8;
                cp_async16(gbuf + (uint32_t)(r * G::PITCH + q * 16), go + src, valid);
                cp_async16(cbuf + (uint32_t)(r * G::PITCH + q * 16), cat + src, valid);
            }
        } else {
            const int q = tid % (kPiece / 8);                      // a thread keeps its eight pixels
            const long long px = p0 + q * 8;
            const bool valid = px < last;                          // eight pixels never straddle `last` or an image
            const long long b = valid ? px / HW : 0;
            const size_t src0 = (size_t)b * C * HW + (valid ? px - b * HW : 0);
#pragma unroll
            for (int u = 0; u < C * (kPiece / 8) / kThreads; ++u) {
                const int c = tid / (kPiece / 8) + u * (kThreads / (kPiece / 8));
                const size_t src = src0 + (size_t)c * HW;
                cp_async16(gbuf + (uint32_t)(c * G::PITCH + q * 16), go + src, valid);
                cp_async16(cbuf + (uint32_t)(c * G::PITCH + q * 16), cat + src, valid);
            }
        }
        cp_async_commit();
    };
    static_assert(kPiece * CH % kThreads == 0, "pieces per thread");
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) {
        if (s < pieces) stage(s);
        else cp_async_commit();
    }
    for (int s = 0; s < pieces; ++s) {
        cp_async_wait<kStages - 2>();
        __syncthreads();                                          // piece s is there for every warp, and piece s - 1 is done with
        if (s + kStages - 1 < pieces) stage(s + kStages - 1);
        else cp_async_commit();
        const uint32_t gtile = sm0 + (uint32_t)((s % kStages) * 2 * G::TILE), gbuf = gtile + lane_sum, cbuf = gbuf + G::TILE;
        uint32_t a[MT][4];
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            if (kNh) ldsm_x4_trans(gbuf + (uint32_t)(m * 32), a[m]);
            else ldsm_x4(gbuf + (uint32_t)(m * 16 * G::PITCH), a[m]);
            mma_bf16(accb[m], a[m][0], a[m][1], a[m][2], a[m][3], 0x3F803F80u, 0x3F803F80u);   // times ones: the sum over pixels
        }
#pragma unroll
        for (int n2 = 0; n2 < MT; ++n2) {
            uint32_t b[4];                                        // cat, same arrangement: channel group n2
            if (kNh) ldsm_x4_trans(cbuf + (uint32_t)(n2 * 32), b);
            else ldsm_x4(cbuf + (uint32_t)(n2 * 16 * G::PITCH), b);
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                mma_bf16(acc[m][2 * n2], a[m][0], a[m][1], a[m][2], a[m][3], b[0], b[2]);
                mma_bf16(acc[m][2 * n2 + 1], a[m][0], a[m][1], a[m][2], a[m][3], b[1], b[3]);
            }
        }
        // ---- g_cat of the warp's 16 pixels ----------------------------------------------------------------------------
        float d[MT][2][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int v = 0; v < 4; ++v) d[m][h][v] = 0.f;
#pragma unroll
        for (int ks = 0; ks < MT; ++ks) {
            uint32_t x[4];
            if (kNh) ldsm_x4(gtile + lane_go + (uint32_t)(ks * 32), x);
            else ldsm_x4_trans(gtile + lane_go + (uint32_t)(ks * 16 * G::PITCH), x);
#pragma unroll
            for (int m = 0; m < MT; ++m) {                        // 16 channels c
                uint32_t y[4];
                ldsm_x4_trans(lane_w + (uint32_t)(ks * 16 * G::WPITCH + m * 32), y);
                if (kNh) {
                    mma_bf16(d[m][0], x[0], x[1], x[2], x[3], y[0], y[1]);
                    mma_bf16(d[m][1], x[0], x[1], x[2], x[3], y[2], y[3]);
                } else {
                    mma_bf16(d[m][0], y[0], y[1], y[2], y[3], x[0], x[1]);
                    mma_bf16(d[m][1], y[0], y[1], y[2], y[3], x[2], x[3]);
                }
            }
        }
        __syncwarp();                                             // the warp alone reads its 16 pixels of go
        unsigned char* gsm = smb + (s % kStages) * 2 * G::TILE;
        const int g = lane >> 2, t = lane & 3;
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const __nv_bfloat162 h2 = __floats2bfloat162_rn(d[m][h][2 * v], d[m][h][2 * v + 1]);
                    // NHWC: pixel g + 8 v, channels 16 m + 8 h + 2t, + 1; NCHW: channel 16 m + g + 8 v, pixels 8 h + 2t, + 1
                    const int at = kNh ? (16 * warp + g + 8 * v) * G::PITCH + (16 * m + 8 * h + 2 * t) * 2
                                       : (16 * m + g + 8 * v) * G::PITCH + (16 * warp + 8 * h + 2 * t) * 2;
                    *reinterpret_cast<uint32_t*>(gsm + at) = *reinterpret_cast<const uint32_t*>(&h2);
                }
        __syncwarp();
        const long long p0 = first + (long long)s * kPiece + 16 * warp;
        if (kNh) {
#pragma unroll
            for (int u = 0; u < 16 * CH / 32; ++u) {              // the warp's 16 pixels are 32 C contiguous bytes
                const int e = lane + 32 * u, r = e / CH, q = e % CH;
                if (p0 + r < last)
                    *(reinterpret_cast<uint4*>(g_cat + (size_t)(p0 + r) * C) + q) = *reinterpret_cast<const uint4*>(gsm + (16 * warp + r) * G::PITCH + q * 16);
            }
        } else {
            const long long px = p0 + 8 * (lane & 1);             // two pieces of eight pixels per channel
            if (px < last) {
                const long long b = px / HW;
                const size_t dst = (size_t)b * C * HW + (size_t)(px - b * HW);
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    const int c = 16 * m + (lane >> 1);
                    *reinterpret_cast<uint4*>(g_cat + dst + (size_t)c * HW) = *reinterpret_cast<const uint4*>(gsm + c * G::PITCH + (16 * warp + 8 * (lane & 1)) * 2);
                }
            }
        }
    }
    if (!part) return;
    cp_async_wait<0>();
    __syncthreads();
    // acc[m][n]: [0], [1] = go channel 16 m + g, cat channels 8 n + 2t, + 1; [2], [3] = go channel + 8.
    // Every warp puts its sums into a region of its own; then they are added per element in warp order.
    constexpr int kPart = C * C + C;
    float* sum = reinterpret_cast<float*>(smb) + warp * kPart;
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int m = 0; m < MT; ++m) {
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int v = 0; v < 4; v += 2)
                *reinterpret_cast<float2*>(sum + (16 * m + g + 8 * (v >> 1)) * C + 8 * n + 2 * t) = make_float2(acc[m][n][v], acc[m][n][v + 1]);
        if (t == 0) {                                             // every column of accb holds the same sum: take column 0
            sum[C * C + 16 * m + g] = accb[m][0];
            sum[C * C + 16 * m + g + 8] = accb[m][2];
        }
    }
    __syncthreads();
    const float* all = reinterpret_cast<const float*>(smb);
    float* out = part + (size_t)blockIdx.x * kPart;
    for (int e = tid; e < kPart; e += kThreads) {
        float v = all[e];
#pragma unroll
        for (int k = 1; k < kThreads / 32; ++k) v += all[k * kPart + e];
        out[e] = v;
    }
}

// bf16 with aligned tensors: NHWC, or NCHW planes of whole 16-byte pieces
inline bool applies(int C, long long HW, int dtype, int layout, const void* w) {
    return dtype == 1 /*bf16*/ && (C == 32 || C == 48 || C == 64) && (layout == kNHWC || HW % 8 == 0) &&
           (reinterpret_cast<uintptr_t>(w) & 15u) == 0;
}
}  // namespace mma

// g_W [C*C] and g_b [C]: the lanes of a warp take 32 consecutive sums, the 32 warps every 32nd block each (in order), then the warps
// are added in order.  A chain of latencies: with eight warps a thread added up to 32 blocks one round trip after the other, 6.6 us for
// 256 blocks at C = 64; 4.0 us now, and scheduled while the kernel in front of it drains.
constexpr int kSumWarps = 32;
__global__ void __launch_bounds__(kSumWarps * 32)
sum_wgrad(const float* __restrict__ part, int C, int blocks, float* __restrict__ g_w, float* __restrict__ g_b)
{
    __shared__ float acc[kSumWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, e = blockIdx.x * 32 + lane, n = C * C + C;
    pdl_wait_primary();
    float s = 0.f;
    if (e < n) {
#pragma unroll 8
        for (int k = warp; k < blocks; k += kSumWarps) s += __ldcg(part + (size_t)k * n + e);
    }
    acc[warp][lane] = s;
    __syncthreads();
    if (warp != 0 || e >= n) return;
#pragma unroll
    for (int k = 1; k < kSumWarps; ++k) s += acc[k][lane];
    if (e < C * C) { if (g_w) g_w[e] = s; }
    else if (g_b) g_b[e - C * C] = s;
}

}}}  // namespace esc::fuse::bwd
