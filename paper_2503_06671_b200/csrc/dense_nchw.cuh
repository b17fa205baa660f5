// The dense large kernel's tensor-core kernels want a pixel's 16 attention channels side by side (32 bytes: the K axis of an
// operand).  For bf16 NCHW tensors `pack16` writes those channels once as [B][H][W][16] and copies the identity planes on the
// way; the stencil kernel then reads the packed map and writes NCHW itself.
// Bound: HBM, 64 bytes per pixel for the packing.  A thread takes a pixel: sixteen 2-byte reads, each 64 contiguous bytes over
// the warp, and 32 bytes written.  With it the dense form runs on tcgen05 on NCHW tensors too; the rule between that and the
// FP32-pipe kernel, which needs no packing, stands at `nchw_wants_packing`.
#pragma once
#include "common.cuh"
#include "stencil_generic.cuh"

namespace esc { namespace dense16 {

constexpr int CA = 16, kThreads = 256;

__global__ void __launch_bounds__(kThreads)
pack16(const __nv_bfloat16* __restrict__ x, __nv_bfloat16* __restrict__ packed, int C, long long HW, long long pixels, unsigned blocks,
       const CopyJob job)
{
    if (blockIdx.x >= blocks) {
        run_copy_job(job, blockIdx.x - blocks, threadIdx.x, kThreads);
        return;
    }
    const long long step = (long long)blocks * kThreads;
    for (long long px = (long long)blockIdx.x * kThreads + threadIdx.x; px < pixels; px += step) {
        const long long b = px / HW;
        const unsigned short* src = reinterpret_cast<const unsigned short*>(x) + (size_t)b * C * HW + (px - b * HW);
        unsigned v[CA];
#pragma unroll
        for (int c = 0; c < CA; ++c) v[c] = __ldg(src + (size_t)c * HW);
        uint4* dst = reinterpret_cast<uint4*>(packed + (size_t)px * CA);
        dst[0] = make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16), v[6] | (v[7] << 16));
        dst[1] = make_uint4(v[8] | (v[9] << 16), v[10] | (v[11] << 16), v[12] | (v[13] << 16), v[14] | (v[15] << 16));
    }
}

constexpr int kMaxK = 13;                           // the tcgen05 kernel's
inline size_t packed_bytes(int B, int Ca, long long HW, int K) { return Ca == CA && K <= kMaxK ? (size_t)B * HW * CA * 2 : 0; }

// bf16 NCHW, K <= 13: tcgen05 behind a packing pass from so many pixels on that it is the faster way.  Measured, forward, K = 13,
// FP32 pipe / packed: 64x64 30.5 / 27 us, 90x90 45.6 / 26.7, 427x240 213 / 29.4, 640x360 430 / 39; 48x48 (K = 9) 22.9 / 25.
// Backward, the old kernels / packed: 17 x (96x96) 759 / 129 us, 640x360 1,530 / 156.
constexpr long long kPackPixels = 4096;
inline bool nchw_wants_packing(int B, int Ca, int H, int W, int K, int dtype, int layout) {
    return dtype == 1 /*bf16*/ && layout == kNCHW && Ca == CA && K <= kMaxK && (long long)B * H * W >= kPackPixels;
}

}}  // namespace esc::dense16
