// Guarded generic stencils for any odd K <= 17, any shape, either layout or element type
// (ESC paper, Section 3.3, Eq. 4 lines 3-4): a halo tile is staged in shared memory as fp32 with zeros outside the image, the
// per-image merged kernel ZP(dk) + LK^s (Eq. 5) sits beside it, and the taps are accumulated in fp32.
#pragma once
#include "common.cuh"

namespace esc {

// One staged input value of attention channel c: the feature itself, or -- in the decomposed form of
// Eq. 5, (F_att * LK^c) * (ZP(DK) + LK^s) -- the point-wise mix sum_k w_point[c][k] * x[k] of the
// pixel's C_a attention channels (fp32, channel order).  Outside the image both are zero.
template <typename T, int LAYOUT>
__device__ __forceinline__ float staged_value(const T* __restrict__ x, const T* __restrict__ w_point, int b, int c,
                                              int y, int xx, int C, int Ca, int H, int W) {
    if (y < 0 || y >= H || xx < 0 || xx >= W) return 0.f;
    if (w_point == nullptr) return Elem<T>::to_f32(x[elem_index<LAYOUT>(b, c, y, xx, C, H, W)]);
    float v = 0.f;
    for (int k = 0; k < Ca; ++k)
        v = fmaf(Elem<T>::to_f32(w_point[(size_t)c * Ca + k]), Elem<T>::to_f32(x[elem_index<LAYOUT>(b, k, y, xx, C, H, W)]), v);
    return v;
}

// The identity channels (Concat of Eq. 4 line 4) as a strided 2-D copy -- `rows` rows of `row_units` units of
// `unit_bytes` bytes, `stride_units` apart, starting `offset_units` into both tensors -- done by the last
// `blocks` blocks (from `first_block` on) of the same launch that computes the attention channels, so that
// the copy, bound by HBM, runs beside the tail of the arithmetic instead of in a launch of its own after it
// (measured: better than putting the copy blocks first).  blocks == 0: nothing to copy.
struct CopyJob {
    const void* src;
    void* dst;
    long long rows, row_units, stride_units, offset_units;
    int unit_bytes;
    unsigned first_block, blocks;
};

template <typename U>
__device__ __forceinline__ void copy_job_units(const CopyJob& j, unsigned rank, unsigned tid, unsigned nthreads) {
    const U* __restrict__ src = static_cast<const U*>(j.src);
    U* __restrict__ dst = static_cast<U*>(j.dst);
    const long long total = j.rows * j.row_units, step = (long long)j.blocks * nthreads;
    for (long long i = (long long)rank * nthreads + tid; i < total; i += step) {
        const long long r = i / j.row_units, q = i - r * j.row_units;
        const long long e = r * j.stride_units + j.offset_units + q;
        dst[e] = src[e];
    }
}
__device__ __forceinline__ void run_copy_job(const CopyJob& j, unsigned rank, unsigned tid, unsigned nthreads) {
    if (j.unit_bytes == 16) copy_job_units<uint4>(j, rank, tid, nthreads);
    else if (j.unit_bytes == 4) copy_job_units<uint32_t>(j, rank, tid, nthreads);
    else copy_job_units<uint16_t>(j, rank, tid, nthreads);
}

// Register-tiled variant: a patch of outputs per thread.  The loop runs over the input rows that a patch touches: a row costs a few
// 16-byte reads and is used by up to OY output rows, each with its kernel row (broadcast 16-byte reads).  It serves the fp32 cases
// and the bf16 ones that no tensor-core or TMA kernel takes.  Built for every odd kernel size KT (one in the middle of a larger one's
// zeros would multiply inputs outside its window, and make NaN of the non-finite ones).  A thread per output in a loop over the taps
// took 48 us where this takes 21 (174x131 fp32, K = 17, whole forward).
// Two geometries: 64 x 32 tiles with 2 x 8 patches, and 32 x 32 tiles with 2 x 4 patches for launches that would otherwise leave most
// SMs with one block or none (a 64x64 fp32 map: 15 us as 16 tiles of 64 x 64, 6 us as 64 of the smallest).  PER_SM blocks an SM: 8
// (64 registers a thread) where there are as many, 6 (80 registers, fewer instructions) where there are not: 640x360 fp32, whole
// forward, 68.4 us with 8, 83.0 with 6 and 74.6 with the 64 x 64 tiles that large maps used to get; 320x180 22.9 and 20.8.
// CB channels per block, 128 threads each.  One on NCHW tensors, whose rows are contiguous.  Four where that makes a thread's
// load 16 bytes of a pixel instead of 4 (NHWC; the results go back through shared memory to leave the same way), and with the
// point-wise mix, whose inputs -- all C_a channels of the pixel -- are then read for four outputs instead of one.  Measured,
// one against four channels, fp32, whole forward: 320x180 NHWC 36 -> 24 us, 640x360 NHWC 111 -> 77; with the mix 135 -> 30 and
// 400 -> 90 (NCHW 44 -> 27 and 138 -> 89).
template <int TX_, int TY_, int OX_, int OY_>
struct RtGeom {
    static constexpr int TX = TX_, TY = TY_, OX = OX_, OY = OY_;
    static constexpr int Threads = (TX / OX) * (TY / OY);       // per channel: 128
    static_assert(OX % 4 == 0 && Threads == 128, "geometry");
};
using RtSmall = RtGeom<64, 32, 8, 2>;
using RtTiny = RtGeom<32, 32, 4, 2>;
template <class G, int KT, int CB>
struct RtLayout {
    static constexpr int Pitch = (G::TX + KT + 2) / 4 * 4, Rows = G::TY + KT - 1; // floats per staged row, a multiple of 4; staged rows
    static constexpr int WRow = (KT + 3) / 4 * 4;                                 // taps per kernel row, padded
    static constexpr int Threads = CB * G::Threads;
    static constexpr int Floats = CB * (Rows * Pitch + KT * WRow);
    static_assert(KT % 2 == 1 && G::TX * G::TY <= Rows * Pitch, "the results fit in the tile's place");
    static int bytes(int Ca, bool mix) { return (Floats + (mix ? CB * Ca : 0)) * 4; }
};

template <typename T> struct Vec4;                                                 // four neighbouring channels of a pixel
template <> struct Vec4<float> {
    using type = float4;
    __device__ static void get(const float4& q, float (&f)[4]) { f[0] = q.x; f[1] = q.y; f[2] = q.z; f[3] = q.w; }
    __device__ static float4 put(const float (&f)[4]) { return make_float4(f[0], f[1], f[2], f[3]); }
};
template <> struct Vec4<__nv_bfloat16> {
    using type = uint2;
    __device__ static void get(const uint2& q, float (&f)[4]) {
        f[0] = __uint_as_float(q.x << 16); f[1] = __uint_as_float(q.x & 0xffff0000u);
        f[2] = __uint_as_float(q.y << 16); f[3] = __uint_as_float(q.y & 0xffff0000u);
    }
    __device__ static uint2 put(const float (&f)[4]) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(f[0], f[1]), b = __floats2bfloat162_rn(f[2], f[3]);
        return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    }
};

template <typename T, int LAYOUT, int KT, class G, int CB, int PER_SM>
__global__ void __launch_bounds__(CB * 128, PER_SM)
stencil_regtile(const T* __restrict__ x, T* __restrict__ out, int C, int Ca, int H, int W,
                const T* __restrict__ w_large, const T* __restrict__ w_point, const float* __restrict__ dk,
                int tiles_x, int tiles_y, const CopyJob job, const float* __restrict__ bias)
{
    using L = RtLayout<G, KT, CB>;
    constexpr int TX = G::TX, TY = G::TY, OX = G::OX, OY = G::OY, Pitch = L::Pitch, Rows = L::Rows, Threads = L::Threads, WRow = L::WRow;
    constexpr int P = (KT - 1) / 2, Plane = Rows * Pitch;
    extern __shared__ __align__(16) float rt_smem[];
    float* tiles = rt_smem;                            // [CB][Rows][Pitch], zeros outside the image
    float* wms = rt_smem + CB * Plane;                 // [CB][KT][WRow]: merged kernel
    float* wps = wms + CB * KT * WRow;                 // [Ca][CB]: point-wise filter, if there is one
    if (job.blocks != 0 && blockIdx.x >= job.first_block) {
        run_copy_job(job, blockIdx.x - job.first_block, threadIdx.x, Threads);
        return;
    }

    long long bid = blockIdx.x;
    const int tx = (int)(bid % tiles_x); bid /= tiles_x;
    const int ty = (int)(bid % tiles_y); bid /= tiles_y;
    const int c0 = (int)(bid % (Ca / CB)) * CB;
    const int b = (int)(bid / (Ca / CB));
    const int tid = threadIdx.x;
    const int y0 = ty * TY - P, x0 = tx * TX - P;

    if (CB > 1 && w_point != nullptr) {
        for (int t = tid; t < CB * Ca; t += Threads) wps[t] = Elem<T>::to_f32(w_point[(size_t)(c0 + t % CB) * Ca + t / CB]);
        __syncthreads();
    }
    // several loads of a thread are in flight before the first is stored: the staging is a chain of round trips otherwise
    constexpr int U = CB == 1 ? 8 : 4;
    for (int t0 = tid; t0 < Plane; t0 += U * Threads) {
        float v[U][CB];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int t = t0 + u * Threads, r = t / Pitch, q = t % Pitch, y = y0 + r, xx = x0 + q;
#pragma unroll
            for (int i = 0; i < CB; ++i) v[u][i] = 0.f;
            if constexpr (CB == 1) {
                if (t < Plane) v[u][0] = staged_value<T, LAYOUT>(x, w_point, b, c0, y, xx, C, Ca, H, W);
            } else if (t < Plane && (unsigned)y < (unsigned)H && (unsigned)xx < (unsigned)W) {
                using V4 = typename Vec4<T>::type;
                if (w_point == nullptr) {
                    if constexpr (LAYOUT == kNHWC) Vec4<T>::get(__ldg(reinterpret_cast<const V4*>(x + elem_index<LAYOUT>(b, c0, y, xx, C, H, W))), v[u]);
                    else
#pragma unroll
                        for (int i = 0; i < CB; ++i) v[u][i] = Elem<T>::to_f32(x[elem_index<LAYOUT>(b, c0 + i, y, xx, C, H, W)]);
                } else {                               // fp32, channel order
                    for (int k = 0; k < Ca; k += 4) {
                        float f[4];
                        if constexpr (LAYOUT == kNHWC) Vec4<T>::get(__ldg(reinterpret_cast<const V4*>(x + elem_index<LAYOUT>(b, k, y, xx, C, H, W))), f);
                        else
#pragma unroll
                            for (int i = 0; i < 4; ++i) f[i] = Elem<T>::to_f32(x[elem_index<LAYOUT>(b, k + i, y, xx, C, H, W)]);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float4 w = *reinterpret_cast<const float4*>(wps + (k + j) * CB);
                            v[u][0] = fmaf(w.x, f[j], v[u][0]); v[u][1] = fmaf(w.y, f[j], v[u][1]);
                            v[u][2] = fmaf(w.z, f[j], v[u][2]); v[u][3] = fmaf(w.w, f[j], v[u][3]);
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int t = t0 + u * Threads;
            if (t < Plane)
#pragma unroll
                for (int i = 0; i < CB; ++i) tiles[i * Plane + t] = v[u][i];
        }
    }
    for (int t = tid; t < CB * KT * WRow; t += Threads) {
        const int i = t / WRow % KT, j = t % WRow;
        wms[t] = j < KT ? Elem<T>::to_f32(w_large[((size_t)(c0 + t / (KT * WRow)) * KT + i) * KT + j]) : 0.f;
    }
    __syncthreads();

    const int cb = CB == 1 ? 0 : tid / 128, ti = CB == 1 ? tid : tid % 128, c = c0 + cb;
    const float* tile = tiles + cb * Plane;
    float* wm = wms + cb * (KT * WRow);
    const int lx = ti % (TX / OX), ly = ti / (TX / OX);
    float acc[OY][OX];
#pragma unroll
    for (int a = 0; a < OY; ++a)
#pragma unroll
        for (int o = 0; o < OX; ++o) acc[a][o] = 0.f;
    // The input rows that meet the dk-carrying kernel rows (P - 1 .. P + 1) of some output row come last: dk, which the kernel
    // before this one writes beside it, is asked for only then.  (Merged before the first row it was waited for with nothing
    // done: 320x180 fp32, whole forward, 24.9 -> 20.8 us.)
    constexpr int kRows = OY + KT - 1, kLate = P - 1, kLateRows = OY + 2;
#pragma unroll 1
    for (int rr = 0; rr < kRows; ++rr) {
        if (rr == kRows - kLateRows) {
            pdl_wait_primary();
            if (ti < 9) wm[(P - 1 + ti / 3) * WRow + P - 1 + ti % 3] += __ldcg(dk + ((size_t)b * Ca + c) * 9 + ti);
            __syncthreads();
        }
        const int r = rr < kLate ? rr : rr < kRows - kLateRows ? rr + kLateRows : rr - (kRows - kLateRows) + kLate;   // input row of the patch window
        constexpr int kIn = (OX + KT + 2) / 4 * 4;         // OX + KT - 1 of them are used
        float in[kIn];
        const float4* trow = reinterpret_cast<const float4*>(tile + (ly * OY + r) * Pitch + lx * OX);
#pragma unroll
        for (int v = 0; v < kIn / 4; ++v) {
            const float4 q = trow[v];
            in[4 * v] = q.x; in[4 * v + 1] = q.y; in[4 * v + 2] = q.z; in[4 * v + 3] = q.w;
        }
#pragma unroll
        for (int a = 0; a < OY; ++a) {
            const int i = r - a;                           // kernel row that maps input row r to output row a
            if (i >= 0 && i < KT) {
                float w[WRow];
                const float4* wrow = reinterpret_cast<const float4*>(wm + i * WRow);
#pragma unroll
                for (int v = 0; v < WRow / 4; ++v) {
                    const float4 q = wrow[v];
                    w[4 * v] = q.x; w[4 * v + 1] = q.y; w[4 * v + 2] = q.z; w[4 * v + 3] = q.w;
                }
#pragma unroll
                for (int j = 0; j < KT; ++j)
#pragma unroll
                    for (int o = 0; o < OX; ++o) acc[a][o] = fmaf(w[j], in[o + j], acc[a][o]);
            }
        }
    }
    const float acc0 = bias ? __ldcg(bias + (size_t)b * Ca + c) : 0.f;   // the backward pass adds a constant per (image, channel)
#pragma unroll
    for (int a = 0; a < OY; ++a)
#pragma unroll
        for (int o = 0; o < OX; ++o) acc[a][o] += acc0;
    if constexpr (CB > 1 && LAYOUT == kNHWC) {
        __syncthreads();                                   // every thread is done with the tiles
        float* res = tiles + cb * Plane;                   // [TY][TX] of this channel
#pragma unroll
        for (int a = 0; a < OY; ++a)
#pragma unroll
            for (int o = 0; o < OX; o += 4)
                *reinterpret_cast<float4*>(res + (ly * OY + a) * TX + lx * OX + o) = make_float4(acc[a][o], acc[a][o + 1], acc[a][o + 2], acc[a][o + 3]);
        __syncthreads();
        for (int t = tid; t < TX * TY; t += Threads) {
            const int oy = ty * TY + t / TX, ox = tx * TX + t % TX;
            if (oy >= H || ox >= W) continue;
            const float f[4] = {tiles[t], tiles[Plane + t], tiles[2 * Plane + t], tiles[3 * Plane + t]};
            *reinterpret_cast<typename Vec4<T>::type*>(out + elem_index<LAYOUT>(b, c0, oy, ox, C, H, W)) = Vec4<T>::put(f);
        }
    } else {
        const int ox0 = tx * TX + lx * OX;
#pragma unroll
        for (int a = 0; a < OY; ++a) {
            const int oy = ty * TY + ly * OY + a;
            if (oy < H) {
#pragma unroll
                for (int o = 0; o < OX; ++o)
                    if (ox0 + o < W) out[elem_index<LAYOUT>(b, c, oy, ox0 + o, C, H, W)] = Elem<T>::from_f32(acc[a][o]);
            }
        }
    }
}

// Copy of the channels that the module leaves untouched (Concat of Eq. 4 line 4), written as a
// strided 2-D copy: `rows` rows of `row_units` units, `stride_units` apart, starting
// `offset_units` into both tensors.  U is the widest unit all three quantities divide into.
template <typename U>
__global__ void __launch_bounds__(256)
copy_through(const U* __restrict__ src, U* __restrict__ dst, long long rows, long long row_units,
             long long stride_units, long long offset_units)
{
    const long long total = rows * row_units;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += step) {
        const long long r = i / row_units, q = i - r * row_units;
        const long long e = r * stride_units + offset_units + q;
        dst[e] = src[e];
    }
}

}  // namespace esc
