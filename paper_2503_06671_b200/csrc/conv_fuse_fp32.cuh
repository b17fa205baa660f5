// The closing 1x1 convolution (ESC paper, Eq. 4 line 4, with the residual of Eq. 3 line 3) and its weight gradient on the FP32
// pipe, for C in {16, 32, 48, 64}: fp32 tensors in either layout, and the bf16 ones that the tensor-core kernels do not take.
//
// conv_fuse_fp32:  out[n] = b[n] + sum_k W[n][k] cat[k] (+ residual[n]) per pixel, or with kTrans W[k][n] -- the backward
// pass's g_cat, from the same matrix (no transposed copy).  cat is (att | idt) as in the tensor-core kernels: channels below
// Ca from one tensor, the rest from the other.  A warp owns 128 pixels x 16 output channels, a lane 2 x 4 pixels x 8
// channels as 32 packed pairs of neighbouring pixels; W lies in shared memory doubled (w, w), input channel by input
// channel, so that six 16-byte reads feed 32 packed multiply-adds (64 issue cycles) per input channel.  Tiles of 128 pixels
// are staged channel by channel (a channel's pixels contiguous: conflict-free reads); three blocks per SM cover each other's
// staging.  Bound: HBM for large maps (2 - 3 maps of C * 4 bytes per pixel against C * C multiply-adds: 16.7 MFMA per MB),
// latency for small ones.  8 x (64x64) fp32 NCHW, C = 64, cold: 495 us as one thread per output out of a pixel-major tile
// (32-way bank conflicts) -> 15.5 us (25 MB: 4 us at the copy bandwidth).
//
// wgrad_fp32:  g_W[n][c] = sum_px go[n] cat[c],  g_b[n] = sum_px go[n].  Both tensors are staged pixel by pixel, go doubled; a
// thread owns 8 x 8 pairs of channels as 32 packed multiply-adds per pixel against six 16-byte reads; the block's pixels are
// dealt to as many slices of (C / 8)^2 threads as fit 256 (C = 64: four), whose sums are added in slice order at the end, and
// the blocks' by sum_wgrad.  The old kernel (4x4 register tiles, eight reads per 64 scalar multiply-adds, half the SMs idle at
// 32,768 pixels) took 72 us on the same batch, this one 18.
#pragma once
#include "common.cuh"
#include "conv_fuse.cuh"

namespace esc { namespace fuse { namespace f32 {

using u64 = unsigned long long;
__device__ __forceinline__ void fma2(u64& acc, u64 a, u64 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b)); }
__device__ __forceinline__ u64 pack2(float lo, float hi) { return (u64)__float_as_uint(lo) | ((u64)__float_as_uint(hi) << 32); }
__device__ __forceinline__ float lo2(u64 v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi2(u64 v) { return __uint_as_float((unsigned)(v >> 32)); }

inline bool supported(int C) { return C == 16 || C == 32 || C == 48 || C == 64; }

constexpr int kTilePx = 128;
template <int C> struct CGeom {
    static constexpr int kThreads = 2 * C;                         // C / 16 warps
    static constexpr int WP = 2 * C + 4;                           // floats per input channel of doubled weights
    static constexpr size_t kSmemBytes = (size_t)(C * WP + C * kTilePx) * sizeof(float);
};

template <typename T>
struct Params {
    const T *att, *idt, *w, *bias, *residual;
    T* out;
    long long HW, pixels;            // pixels of one image, of all
    int B, Ca;
    int vec;                         // 16-byte pieces are aligned: HW a multiple of 4 (NCHW)
};

template <typename T, int LAYOUT, int C, bool kTrans>
__global__ void __launch_bounds__(CGeom<C>::kThreads, C == 64 ? 3 : 4)
conv_fuse_fp32(const Params<T> p)
{
    using G = CGeom<C>;
    constexpr int kThreads = G::kThreads;
    extern __shared__ __align__(16) float smf[];
    float* wsm = smf;                                              // [C input channels][WP]
    float* xs = smf + C * G::WP;                                   // [C][kTilePx]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pg = lane & 15, n0 = warp * 16 + (lane >> 4) * 8;    // this lane: pixels 4 pg .. + 3 and 64 + 4 pg .. + 3, channels n0 .. + 7
    for (int e = tid; e < C * C; e += kThreads) {
        const float v = Elem<T>::to_f32(p.w[e]);
        const int n = kTrans ? e % C : e / C, k = kTrans ? e / C : e % C;
        *reinterpret_cast<float2*>(wsm + k * G::WP + 2 * n) = make_float2(v, v);
    }
    float bs[8];
#pragma unroll
    for (int n = 0; n < 8; ++n) bs[n] = p.bias ? Elem<T>::to_f32(p.bias[n0 + n]) : 0.f;
    pdl_wait_primary();                                            // the tensors come from the kernel before this one
    pdl_launch_dependents();

    // NCHW: tiles of one image; NHWC: of the flat list of pixels
    const long long per_img = LAYOUT == kNCHW ? (p.HW + kTilePx - 1) / kTilePx : 0;
    const long long ntiles = LAYOUT == kNCHW ? per_img * p.B : (p.pixels + kTilePx - 1) / kTilePx;
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const long long b = LAYOUT == kNCHW ? tile / per_img : 0, q0 = (LAYOUT == kNCHW ? tile - b * per_img : tile) * kTilePx;
        const int left = (int)min((LAYOUT == kNCHW ? p.HW : p.pixels) - q0, (long long)kTilePx);
        const size_t base = LAYOUT == kNCHW ? (size_t)b * C * p.HW + q0 : (size_t)q0 * C;
        if (tile != blockIdx.x) __syncthreads();                   // the tile before this one is read
        if (LAYOUT == kNCHW && sizeof(T) == 4) {
            const uint32_t d = (uint32_t)__cvta_generic_to_shared(xs);
            if (p.vec) {
                for (int e = tid; e < C * (kTilePx / 4); e += kThreads) {
                    const int c = e / (kTilePx / 4), q = (e % (kTilePx / 4)) * 4;
                    const bool ok = q < left;
                    cp_async16(d + (uint32_t)(c * kTilePx + q) * 4, (c < p.Ca ? p.att : p.idt) + base + (size_t)c * p.HW + (ok ? q : 0), ok);
                }
            } else {
                for (int e = tid; e < C * kTilePx; e += kThreads) {
                    const int c = e / kTilePx, q = e % kTilePx;
                    const bool ok = q < left;
                    cp_async4(d + (uint32_t)(c * kTilePx + q) * 4, (c < p.Ca ? p.att : p.idt) + base + (size_t)c * p.HW + (ok ? q : 0), ok);
                }
            }
            cp_async_commit();
            cp_async_wait<0>();
        } else if (LAYOUT == kNCHW) {
#pragma unroll 8
            for (int e = tid; e < C * kTilePx; e += kThreads) {
                const int c = e / kTilePx, q = e % kTilePx;
                xs[e] = q < left ? Elem<T>::to_f32(((c < p.Ca ? p.att : p.idt) + base + (size_t)c * p.HW)[q]) : 0.f;
            }
        } else {
            constexpr int V = Elem<T>::kVec;                       // channels of a 16-byte piece; lanes take neighbouring pixels
#pragma unroll 4
            for (int e = tid; e < kTilePx * (C / V); e += kThreads) {
                const int q = e % kTilePx, c0 = (e / kTilePx) * V;
                float f[V];
                if (c0 + V <= p.Ca || c0 >= p.Ca) {
                    const T* src = c0 < p.Ca ? p.att : p.idt;
                    if (q < left) unpack16<T>(*reinterpret_cast<const uint4*>(src + base + (size_t)q * C + c0), f);
                    else {
#pragma unroll
                        for (int v = 0; v < V; ++v) f[v] = 0.f;
                    }
                } else {                                           // the piece holds channels of both tensors
#pragma unroll
                    for (int v = 0; v < V; ++v)
                        f[v] = q < left ? Elem<T>::to_f32((c0 + v < p.Ca ? p.att : p.idt)[base + (size_t)q * C + c0 + v]) : 0.f;
                }
#pragma unroll
                for (int v = 0; v < V; ++v) xs[(c0 + v) * kTilePx + q] = f[v];
            }
        }
        __syncthreads();

        u64 acc[8][4];                                             // [channel][pixel pair]
#pragma unroll
        for (int n = 0; n < 8; ++n)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[n][q] = pack2(bs[n], bs[n]);
#pragma unroll 2
        for (int k = 0; k < C; ++k) {
            const ulonglong2 xa = *reinterpret_cast<const ulonglong2*>(xs + k * kTilePx + 4 * pg);
            const ulonglong2 xb = *reinterpret_cast<const ulonglong2*>(xs + k * kTilePx + 64 + 4 * pg);
            const u64 xv[4] = {xa.x, xa.y, xb.x, xb.y};
            const ulonglong2* wr = reinterpret_cast<const ulonglong2*>(wsm + k * G::WP + 2 * n0);
#pragma unroll
            for (int n2 = 0; n2 < 4; ++n2) {
                const ulonglong2 w = wr[n2];
#pragma unroll
                for (int q = 0; q < 4; ++q) fma2(acc[2 * n2][q], w.x, xv[q]);
#pragma unroll
                for (int q = 3; q >= 0; --q) fma2(acc[2 * n2 + 1][q], w.y, xv[q]);
            }
        }

        if (LAYOUT == kNCHW) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int q = 64 * h + 4 * pg;
#pragma unroll
                for (int n = 0; n < 8; ++n) {
                    const size_t at = base + (size_t)(n0 + n) * p.HW + q;
                    float v[4] = {lo2(acc[n][2 * h]), hi2(acc[n][2 * h]), lo2(acc[n][2 * h + 1]), hi2(acc[n][2 * h + 1])};
                    if (sizeof(T) == 4 && p.vec) {                 // left is a multiple of 4
                        if (q < left) {
                            if (p.residual) {
                                const float4 r = *reinterpret_cast<const float4*>(p.residual + at);
                                v[0] += r.x; v[1] += r.y; v[2] += r.z; v[3] += r.w;
                            }
                            *reinterpret_cast<float4*>(p.out + at) = make_float4(v[0], v[1], v[2], v[3]);
                        }
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (q + u < left) {
                                if (p.residual) v[u] += Elem<T>::to_f32(p.residual[at + u]);
                                p.out[at + u] = Elem<T>::from_f32(v[u]);
                            }
                    }
                }
            }
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int px = 64 * (q >> 2) + 4 * pg + (q & 3);
                if (px < left) {
                    const size_t at = base + (size_t)px * C + n0;  // eight channels: one 32-byte (fp32) or 16-byte piece
                    float v[8];
#pragma unroll
                    for (int n = 0; n < 8; ++n) v[n] = (q & 1) ? hi2(acc[n][q >> 1]) : lo2(acc[n][q >> 1]);
                    if (p.residual) {
#pragma unroll
                        for (int n = 0; n < 8; ++n) v[n] += Elem<T>::to_f32(p.residual[at + n]);
                    }
                    if constexpr (sizeof(T) == 4) {
                        *reinterpret_cast<float4*>(p.out + at) = make_float4(v[0], v[1], v[2], v[3]);
                        *reinterpret_cast<float4*>(p.out + at + 4) = make_float4(v[4], v[5], v[6], v[7]);
                    } else {
                        uint32_t o[4];
#pragma unroll
                        for (int n = 0; n < 4; ++n) {
                            const __nv_bfloat162 h2 = __floats2bfloat162_rn(v[2 * n], v[2 * n + 1]);
                            o[n] = *reinterpret_cast<const uint32_t*>(&h2);
                        }
                        *reinterpret_cast<uint4*>(p.out + at) = make_uint4(o[0], o[1], o[2], o[3]);
                    }
                }
            }
        }
    }
}

// first: no kernel of the same call stands in front of this one.  Then w may come from the kernel that does, and this one, which reads
// w before it waits, must not start before that has finished.
template <typename T, int LAYOUT, int C, bool kTrans>
inline cudaError_t launch_c(const Params<T>& p, cudaStream_t st, bool first) {
    using G = CGeom<C>;
    auto* fn = conv_fuse_fp32<T, LAYOUT, C, kTrans>;
    static bool attr_set[tma::kMaxDevices] = {};
    const int dev = tma::current_device();
    if (dev < 0) return cudaErrorInvalidDevice;
    if (!attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::kSmemBytes);
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    const long long tiles = LAYOUT == kNCHW ? (p.HW + kTilePx - 1) / kTilePx * p.B : (p.pixels + kTilePx - 1) / kTilePx;
    const long long cap = (C == 64 ? 3LL : 4LL) * (tma::sm_count() > 0 ? tma::sm_count() : 148);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles < cap ? tiles : cap));
    cfg.blockDim = dim3(G::kThreads);
    cfg.dynamicSmemBytes = G::kSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];                                   // may stage its weights while the kernel before it drains
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = first ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, fn, p);
}
template <typename T, int LAYOUT, bool kTrans>
inline cudaError_t launch(int C, const Params<T>& p, cudaStream_t st, bool first) {
    switch (C) {
        case 16: return launch_c<T, LAYOUT, 16, kTrans>(p, st, first);
        case 32: return launch_c<T, LAYOUT, 32, kTrans>(p, st, first);
        case 48: return launch_c<T, LAYOUT, 48, kTrans>(p, st, first);
        case 64: return launch_c<T, LAYOUT, 64, kTrans>(p, st, first);
        default: return cudaErrorInvalidValue;
    }
}

// ---- weight gradient -----------------------------------------------------------------------------------------------------
constexpr int kWThreads = 256, kWPx = 64;                          // pixels per pass
template <int C> struct WGeom {
    static constexpr int G = C / 8, kSliceThreads = G * G, kSlices = kWThreads / kSliceThreads;
    static constexpr int GP = 2 * C + 4, XP = C + 4;               // floats per staged pixel: go doubled, cat
    static constexpr int kPart = C * C + C;
    static constexpr int kStage = kWPx * (GP + XP), kRed = kSlices * kPart;
    static constexpr size_t kSmemBytes = sizeof(float) * (size_t)(kStage > kRed ? kStage : kRed);
};

template <typename T, int LAYOUT, int C>
__global__ void __launch_bounds__(kWThreads, 2)
wgrad_fp32(const T* __restrict__ cat, const T* __restrict__ go, long long HW, long long pixels, int passes,
           float* __restrict__ part)                               // [gridDim.x][C * C + C]
{
    using W = WGeom<C>;
    extern __shared__ __align__(16) float smf[];
    float* gs = smf;                                               // [kWPx][GP]: (go, go)
    float* xs = smf + kWPx * W::GP;                                // [kWPx][XP]
    const int tid = threadIdx.x;
    const int slice = tid / W::kSliceThreads, st = tid % W::kSliceThreads, ng = st / W::G, cg = st % W::G;
    const bool active = slice < W::kSlices;
    // go channels 2 ng + {0, 1} + 2 G i and cat channels 4 cg .. + 3, C / 2 + 4 cg .. + 3: lanes read neighbouring 16 bytes
    u64 acc[8][4];                                                 // [go channel][cat pair]
#pragma unroll
    for (int n = 0; n < 8; ++n)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[n][q] = 0ull;
    // the sums of this row group's eight go channels are dealt to its threads: channel number cg, cg + G, ..
    constexpr int kGb = (8 + W::G - 1) / W::G;
    float gb[kGb];
#pragma unroll
    for (int u = 0; u < kGb; ++u) gb[u] = 0.f;
    for (int pass = 0; pass < passes; ++pass) {
        const long long px0 = ((long long)blockIdx.x * passes + pass) * kWPx;
        if (px0 >= pixels) break;
        if (pass) __syncthreads();
        const int left = (int)min(pixels - px0, (long long)kWPx);
        if (LAYOUT == kNCHW) {
            const int q = tid % kWPx;                              // a thread keeps its pixel: one division per pass
            const long long px = px0 + (q < left ? q : 0), b = px / HW;
            const size_t base = (size_t)b * C * HW + (size_t)(px - b * HW);
#pragma unroll 8
            for (int c = tid / kWPx; c < C; c += kWThreads / kWPx) {
                const float a = q < left ? Elem<T>::to_f32(go[base + (size_t)c * HW]) : 0.f;
                const float v = q < left ? Elem<T>::to_f32(cat[base + (size_t)c * HW]) : 0.f;
                *reinterpret_cast<float2*>(gs + q * W::GP + 2 * c) = make_float2(a, a);
                xs[q * W::XP + c] = v;
            }
        } else {
            constexpr int V = Elem<T>::kVec;
#pragma unroll 4
            for (int e = tid; e < kWPx * (C / V); e += kWThreads) {
                const int q = e / (C / V), c0 = (e % (C / V)) * V;
                float a[V], v[V];
                if (q < left) {
                    unpack16<T>(*reinterpret_cast<const uint4*>(go + (size_t)(px0 + q) * C + c0), a);
                    unpack16<T>(*reinterpret_cast<const uint4*>(cat + (size_t)(px0 + q) * C + c0), v);
                } else {
#pragma unroll
                    for (int i = 0; i < V; ++i) a[i] = v[i] = 0.f;
                }
#pragma unroll
                for (int i = 0; i < V; i += 2)
                    *reinterpret_cast<float4*>(gs + q * W::GP + 2 * (c0 + i)) = make_float4(a[i], a[i], a[i + 1], a[i + 1]);
#pragma unroll
                for (int i = 0; i < V; i += 4)
                    *reinterpret_cast<float4*>(xs + q * W::XP + c0 + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
            }
        }
        __syncthreads();
        if (active) {
#pragma unroll 2
            for (int q = slice; q < kWPx; q += W::kSlices) {
                const float* gp = gs + q * W::GP + 4 * ng;
                const ulonglong2 xa = *reinterpret_cast<const ulonglong2*>(xs + q * W::XP + 4 * cg);
                const ulonglong2 xb = *reinterpret_cast<const ulonglong2*>(xs + q * W::XP + C / 2 + 4 * cg);
                const u64 xv[4] = {xa.x, xa.y, xb.x, xb.y};
#pragma unroll
                for (int u = 0; u < kGb; ++u) {
                    const int n = cg + u * W::G;
                    if (n < 8) gb[u] += gp[2 * (n & 1) + 4 * W::G * (n >> 1)];
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(gp + 4 * W::G * i);
#pragma unroll
                    for (int u = 0; u < 4; ++u) fma2(acc[2 * i][u], g.x, xv[u]);
#pragma unroll
                    for (int u = 3; u >= 0; --u) fma2(acc[2 * i + 1][u], g.y, xv[u]);
                }
            }
        }
    }
    __syncthreads();
    if (active) {                                                  // every slice's sums side by side, then added in slice order
        float* red = smf + slice * W::kPart;
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            const int nn = 2 * ng + (n & 1) + 2 * W::G * (n >> 1);
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float4*>(red + nn * C + (C / 2) * h + 4 * cg) =
                    make_float4(lo2(acc[n][2 * h]), hi2(acc[n][2 * h]), lo2(acc[n][2 * h + 1]), hi2(acc[n][2 * h + 1]));
        }
#pragma unroll
        for (int u = 0; u < kGb; ++u) {
            const int n = cg + u * W::G;
            if (n < 8) red[C * C + 2 * ng + (n & 1) + 2 * W::G * (n >> 1)] = gb[u];
        }
    }
    __syncthreads();
    float* out = part + (size_t)blockIdx.x * W::kPart;
    for (int e = tid; e < W::kPart; e += kWThreads) {
        float s = smf[e];
        for (int k = 1; k < W::kSlices; ++k) s += smf[k * W::kPart + e];
        out[e] = s;
    }
}

}}}  // namespace esc::fuse::f32
