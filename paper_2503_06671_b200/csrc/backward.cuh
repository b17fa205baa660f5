// Backward pass of the ConvAttn forward (ESC paper, Section 3.3, Eq. 4, depth-wise LK; one-layer estimator, or the
// two-layer estimator of Eq. 4 line 2 at the end of this file), the chain rule written out.  With go = dL/dout and Wm[b,c] = LK[c] + ZP(dk[b,c]):
//
//   g_tap[b,c,i,j] = sum_{y,x} go[b,c,y,x] * x~[b,c,y+i-6,x+j-6]      per-image tap gradient  (kernel tap_grad)
//   g_lk = sum_b g_tap;   g_dk = central 3x3 of g_tap;   g_b = sum_b g_dk;   g_W[o,k] = sum_b g_dk[b,o] g[b,k]
//   g_g[b,k] = sum_o W[o,k] g_dk[b,o]                                          (estimator_image, estimator_weights)
//   g_x[b,c] = go[b,c] (*) flip(Wm[b,c]) + g_g[b,c] / (H W)   (c < C_a),   g_x[b,c] = go[b,c]  (c >= C_a)
//
// The last line is the forward stencil applied to go with both kernels rotated by 180 degrees and a
// per-(image, channel) constant added, so it runs on the forward kernels; `estimator_image` prepares the rotated
// kernels and the constants for it.  Every reduction is done in a fixed order: results are reproducible.
#pragma once
#include "common.cuh"
#include "stencil_generic.cuh"
#include "gap_dynkernel.cuh"

namespace esc { namespace bwd {

constexpr int K = 13, P = 6, TAPS = K * K;
constexpr int TX = 64, TY = 64;                           // tile of go per block
constexpr int XP = TX + K - 1;                            // 76 floats per staged x row (a multiple of 4)
constexpr int XR = TY + K - 1;                            // 76 staged x rows
constexpr int kThreads = 128;
constexpr int kSlot = 176;                                // floats per (image, channel, tile): 169 taps, sum of x, padding
static_assert(XP % 4 == 0 && TAPS + 1 <= kSlot, "layout");

// ---- kernel 1: per-tile partial tap gradients and partial sums of x ---------------------------------------
// Block = (image b, attention channel c, 64x64 tile), 128 threads or, with the kernel rows shared among them, four times 128.  The x halo tile (zeros outside the
// image) and the go tile (zeros outside) are staged in shared memory as fp32; a thread keeps its patch of 8 rows x 4 columns of go in
// registers (the eight lanes of a 16-byte read phase then sit side by side, free of bank conflicts) and, for every kernel row i, reads
// the eight x rows its patch meets (four 16-byte reads each) and forms the 13 partial sums of that row: 416 FMAs per 32 reads.  The 13
// sums are then added over the block in a fixed order: inside a warp by halving -- at each step a lane passes on the half of the values
// that it does not keep, 16 shuffles where a butterfly per value takes 65 --, then warps in order.
// Small launches share the kernel rows: one block of four warps an SM is a chain of latencies.  (The NHWC form below shares them among up
// to four blocks, `row_shares`, which each stage the tile; here that gave 16.7 us for 21.8.)  8 images of 64x64,
// 16 channels, fp32: 21.8 -> 12.5 us; whole backward of the module, NHWC, 93 -> 77 us, 40 of 48x48 173 -> 148 (NCHW 142 -> 131).
constexpr int kPY = 8, kPX = 4;                           // a thread's patch of go
// Sums of s[0 .. 15] over the warp: lane l holds that of value reduce_index(l).
__device__ __forceinline__ float reduce16(float (&s)[16], int lane) {
#pragma unroll
    for (int h = 8, m = 16; h >= 1; h >>= 1, m >>= 1) {
        const bool up = lane & m;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const float send = up ? s[k] : s[k + h], keep = up ? s[k + h] : s[k];
            s[k] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
    }
    return s[0] + __shfl_xor_sync(0xffffffffu, s[0], 1);
}
__device__ __forceinline__ int reduce_index(int lane) { return lane >> 1; }
// The 13 sums of kernel row i over a thread's patch g; xr: the patch's first x row and column for i = 0.
template <int PITCH>
__device__ __forceinline__ void row_sums(const float* xr, int i, const float (&g)[kPY][kPX], float (&s)[16]) {
#pragma unroll
    for (int j = 0; j < 16; ++j) s[j] = 0.f;
#pragma unroll
    for (int a = 0; a < kPY; ++a) {
        float in[kPX + K - 1];                            // x row a + i of the patch, 16 columns
        const float4* xv = reinterpret_cast<const float4*>(xr + (a + i) * PITCH);
#pragma unroll
        for (int v = 0; v < (kPX + K - 1) / 4; ++v) {
            const float4 q = xv[v];
            in[4 * v] = q.x; in[4 * v + 1] = q.y; in[4 * v + 2] = q.z; in[4 * v + 3] = q.w;
        }
#pragma unroll
        for (int j = 0; j < K; ++j)
#pragma unroll
            for (int o = 0; o < kPX; ++o) s[j] = fmaf(g[a][o], in[o + j], s[j]);
    }
}
// A thread's patch of go, and the sum of x over it.
template <int PITCH, int GPITCH>
__device__ __forceinline__ float load_patch(const float* xr, const float* gr, float (&g)[kPY][kPX]) {
    float sx = 0.f;
#pragma unroll
    for (int a = 0; a < kPY; ++a) {
        const float4 q = *reinterpret_cast<const float4*>(gr + a * GPITCH);
        g[a][0] = q.x; g[a][1] = q.y; g[a][2] = q.z; g[a][3] = q.w;
        const float4* xv = reinterpret_cast<const float4*>(xr + (a + P) * PITCH + P - 2);   // 16-byte aligned: P - 2 = 4
        const float4 u0 = xv[0], u1 = xv[1];              // the patch's own pixels are floats 2..5 of these
        sx += (u0.z + u0.w) + (u1.x + u1.y);
    }
    return sx;
}
// Blocks that share a tile's kernel rows: as many as it takes to have `per_sm` blocks on every SM, at most four.
inline int row_shares(long long blocks, int per_sm, int sms) {
    const long long n = ((long long)per_sm * sms) / (blocks > 0 ? blocks : 1);
    return n < 1 ? 1 : n > 4 ? 4 : (int)n;
}

template <typename T, int LAYOUT, int SHARES>
__global__ void __launch_bounds__(kThreads * SHARES)
tap_grad(const T* __restrict__ x, const T* __restrict__ go, int C, int Ca, int H, int W, int tiles_x, int tiles_y,
         int ia, int ib,                // the kernel rows wanted: all, or 5 to 7 where nobody asks for g_lk
         float* __restrict__ part)      // [B][Ca][tiles][kSlot]
{
    __shared__ __align__(16) float xt[XR * XP];
    __shared__ __align__(16) float gt[TY * TX];
    __shared__ float red[K][kThreads / 32][16];
    __shared__ float redx[kThreads / 32];

    long long bid = blockIdx.x;
    const int tiles = tiles_x * tiles_y;
    const int tile = (int)(bid % tiles); bid /= tiles;
    const int c = (int)(bid % Ca);
    const int b = (int)(bid / Ca);
    const int tx = tile % tiles_x, ty = tile / tiles_x;
    constexpr int N = kThreads * SHARES;
    const int all = threadIdx.x, tid = all % kThreads, share = all / kThreads, lane = tid & 31, warp = tid >> 5;
    const int y0 = ty * TY, x0 = tx * TX;
    const int i0 = ia + (ib - ia) * share / SHARES, i1 = ia + (ib - ia) * (share + 1) / SHARES;        // these 128 threads' kernel rows

    constexpr int U = 8;                                  // loads of a thread in flight
    for (int t0 = all; t0 < XR * XP; t0 += U * N) {
        float v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int t = t0 + u * N, r = t / XP, q = t % XP, y = y0 - P + r, xx = x0 - P + q;
            v[u] = (t < XR * XP && y >= 0 && y < H && xx >= 0 && xx < W) ? Elem<T>::to_f32(x[elem_index<LAYOUT>(b, c, y, xx, C, H, W)]) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (t0 + u * N < XR * XP) xt[t0 + u * N] = v[u];
    }
    for (int t0 = all; t0 < TY * TX; t0 += U * N) {
        float v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int t = t0 + u * N, y = y0 + t / TX, xx = x0 + t % TX;
            v[u] = (y < H && xx < W) ? Elem<T>::to_f32(go[elem_index<LAYOUT>(b, c, y, xx, C, H, W)]) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) gt[t0 + u * N] = v[u];
    }
    static_assert(TY * TX % (U * N) == 0 && (TX / kPX) * (TY / kPY) == kThreads, "whole rounds; one patch per thread");
    __syncthreads();

    const int lx = tid % (TX / kPX), ly = tid / (TX / kPX);
    const float* xr = xt + ly * kPY * XP + lx * kPX;
    float g[kPY][kPX];
    float sx = load_patch<XP, TX>(xr, gt + ly * kPY * TX + lx * kPX, g);      // sum of x over the patch (for the GAP of this image)
#pragma unroll 1
    for (int i = i0; i < i1; ++i) {
        float s[16];
        row_sums<XP>(xr, i, g, s);
        const float t = reduce16(s, lane);
        if ((lane & 1) == 0) red[i][warp][reduce_index(lane)] = t;
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) sx += __shfl_xor_sync(0xffffffffu, sx, o);
    if (lane == 0 && share == 0) redx[warp] = sx;
    __syncthreads();
    float* slot = part + (((size_t)b * Ca + c) * tiles + tile) * kSlot;
    for (int e = ia * K + all; e < ib * K; e += N) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) t += red[e / K][w][e % K];
        slot[e] = t;
    }
    if (all == 0) {
        float t = 0.f;
        for (int w = 0; w < kThreads / 32; ++w) t += redx[w];
        slot[TAPS] = t;
    }
}

// ---- kernel 1, NHWC form: eight channels per block -----------------------------------------------------------
// In NHWC a block per channel would fetch every pixel's line once per channel with 2-byte loads.  Here a block
// takes eight neighbouring channels (16 bytes of a bf16 pixel, 32 of an fp32 one) of a 32x32 tile: pixels are
// read with 16-byte loads and spread over eight planar fp32 tiles in shared memory; warp w then works on channel
// w on its own (8x4 patch of go per lane), so the sums of a row's 13 values stay inside the warp.
namespace n8 {
constexpr int TX = 32, TY = 32, CH = 8;
constexpr int XP = TX + K - 1, XR = TY + K - 1;          // 44 x 44 staged x per channel (44 is a multiple of 4)
constexpr int kThreads = CH * 32;                        // 256
constexpr size_t kSmemBytes = (size_t)CH * (XR * XP + TY * TX) * sizeof(float);   // 94,720
static_assert(XP % 4 == 0, "16-byte reads of staged rows");
}  // namespace n8

template <typename T>
__global__ void __launch_bounds__(n8::kThreads)
tap_grad_nhwc8(const T* __restrict__ x, const T* __restrict__ go, int C, int Ca, int H, int W, int tiles_x, int tiles_y,
               int ia, int ib, float* __restrict__ part)      // [B][Ca][tiles][kSlot]
{
    constexpr int TX = n8::TX, TY = n8::TY, CH = n8::CH, XP = n8::XP, XR = n8::XR, kThreads = n8::kThreads;
    constexpr int V = Elem<T>::kVec;                      // elements per 16-byte load: 8 (bf16) or 4 (fp32)
    extern __shared__ __align__(16) float sm[];
    float* xt = sm;                                       // [CH][XR*XP]
    float* gt = sm + CH * XR * XP;                        // [CH][TY*TX]

    long long bid = blockIdx.x;
    const int tiles = tiles_x * tiles_y, octets = Ca / CH;
    const int tile = (int)(bid % tiles); bid /= tiles;
    const int oct = (int)(bid % octets);
    const int b = (int)(bid / octets);
    const int tx = tile % tiles_x, ty = tile / tiles_x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int y0 = ty * TY, x0 = tx * TX;
    const T* xb = x + (size_t)b * H * W * C + oct * CH;
    const T* gb = go + (size_t)b * H * W * C + oct * CH;

    for (int t = tid; t < XR * XP * (CH / V); t += kThreads) {
        const int h = t % (CH / V), pix = t / (CH / V);   // which 16-byte piece of the pixel's eight channels
        const int r = pix / XP, q = pix % XP;
        const int y = y0 - P + r, xx = x0 - P + q;
        float f[V];
        if (y >= 0 && y < H && xx >= 0 && xx < W)
            unpack16<T>(__ldg(reinterpret_cast<const uint4*>(xb + ((size_t)y * W + xx) * C + h * V)), f);
        else {
#pragma unroll
            for (int v = 0; v < V; ++v) f[v] = 0.f;
        }
#pragma unroll
        for (int v = 0; v < V; ++v) xt[(h * V + v) * (XR * XP) + pix] = f[v];
    }
    for (int t = tid; t < TY * TX * (CH / V); t += kThreads) {
        const int h = t % (CH / V), pix = t / (CH / V);
        const int r = pix / TX, q = pix % TX;
        const int y = y0 + r, xx = x0 + q;
        float f[V];
        if (y < H && xx < W)
            unpack16<T>(__ldg(reinterpret_cast<const uint4*>(gb + ((size_t)y * W + xx) * C + h * V)), f);
        else {
#pragma unroll
            for (int v = 0; v < V; ++v) f[v] = 0.f;
        }
#pragma unroll
        for (int v = 0; v < V; ++v) gt[(h * V + v) * (TY * TX) + pix] = f[v];
    }
    __syncthreads();

    constexpr int TXP = TX / kPX;
    static_assert(TXP * (TY / kPY) == 32, "one warp covers a channel's tile");
    const int lx = lane % TXP, ly = lane / TXP;
    const float* xr = xt + warp * (XR * XP) + ly * kPY * XP + lx * kPX;       // this warp's channel
    float g[kPY][kPX];
    float sx = load_patch<XP, TX>(xr, gt + warp * (TY * TX) + ly * kPY * TX + lx * kPX, g);
    float* slot = part + (((size_t)b * Ca + oct * CH + warp) * tiles + tile) * kSlot;
    const int i0 = ia + (ib - ia) * (int)blockIdx.y / (int)gridDim.y, i1 = ia + (ib - ia) * ((int)blockIdx.y + 1) / (int)gridDim.y;   // this block's kernel rows
#pragma unroll 1
    for (int i = i0; i < i1; ++i) {
        float s[16];
        row_sums<XP>(xr, i, g, s);
        const float t = reduce16(s, lane);
        if ((lane & 1) == 0 && reduce_index(lane) < K) slot[i * K + reduce_index(lane)] = t;
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) sx += __shfl_xor_sync(0xffffffffu, sx, o);
    if (lane == 0 && blockIdx.y == 0) slot[TAPS] = sx;
}

// ---- kernel 2a: add the tiles of one (image, channel) in a fixed order -----------------------------------------
// Block = (image, channel); kSumGroups groups of 192 threads take every kSumGroups-th tile each (sixteen loads in
// flight, added in order), then the groups' sums are added in group order.  In the decomposed form the sums of x that came with the
// taps are those of the mixed features: the threads that have no tap add up the chunks' sums of x in their place.
constexpr int kSumGroups = 4, kSumThreads = 192 * kSumGroups;
__global__ void __launch_bounds__(kSumThreads)
sum_tiles(const float* __restrict__ part, int tiles, const float* __restrict__ xs_part, int chunks, int Ca,
          float* __restrict__ gtap)                              // gtap [B*Ca][kSlot]
{
    constexpr int kSpare = 192 - (TAPS + 1), kX = kSpare * kSumGroups;
    static_assert(kX > 64 && kX <= 96, "one warp adds the threads' sums of x");
    __shared__ float acc[kSumGroups][192], xacc[96];
    auto sum = [](const float* p, int n, size_t pitch, int first, int step) {      // p[first], p[first + step], ..: sixteen in flight
        float s = 0.f;
        for (int k0 = first; k0 < n; k0 += 16 * step) {
            float v[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) v[u] = k0 + u * step < n ? __ldcg(p + (size_t)(k0 + u * step) * pitch) : 0.f;
#pragma unroll
            for (int u = 0; u < 16; ++u) s += v[u];
        }
        return s;
    };
    const size_t bc = blockIdx.x;
    const int t = threadIdx.x % 192, grp = threadIdx.x / 192;
    pdl_launch_dependents();
    pdl_wait_primary();
    if (t <= TAPS) {
        acc[grp][t] = sum(part + bc * tiles * kSlot + t, tiles, kSlot, grp, kSumGroups);
    } else if (xs_part) {
        const int x = grp * kSpare + t - (TAPS + 1);
        xacc[x] = sum(xs_part + (bc / Ca) * chunks * Ca + bc % Ca, chunks, Ca, x, kX);
    }
    __syncthreads();
    if (grp == 0 && t <= TAPS) {
        float s = acc[0][t];
#pragma unroll
        for (int q = 1; q < kSumGroups; ++q) s += acc[q][t];
        if (t < TAPS || !xs_part) gtap[bc * kSlot + t] = s;
    }
    if (xs_part && grp == 1 && t < 32) {
        const float s = warp_sum(xacc[t] + xacc[t + 32] + (t + 64 < kX ? xacc[t + 64] : 0.f));
        if (t == 0) gtap[bc * kSlot + TAPS] = s;
    }
}

// ---- the estimator's part -----------------------------------------------------------------------------------------
// One linear layer (hidden == 0): g = pooled means, dk = b_last + W g;  g_W[o,k] = sum_b g_dk[b,o] g[b,k],  g_b = sum_b g_dk,
//   g_g[b,k] = sum_o W[o,k] g_dk[b,o].
// Two layers with the exact GELU between them, as Eq. 4 line 2 writes it:
//   t = W_down g + b_down,  a = phi(t),  dk = W_up a + b_up;   phi'(t) = Phi(t) + t n(t)
//   g_a[b,m] = sum_o W_up[o,m] g_dk[b,o],   g_t = g_a * phi'(t),   g_g[b,k] = sum_m W_down[m,k] g_t[b,m]
//   g_b_up = sum_b g_dk,  g_W_up[o,m] = sum_b g_dk[b,o] a[b,m],  g_b_down = sum_b g_t,  g_W_down[m,k] = sum_b g_t[b,m] g[b,k]
__device__ __forceinline__ float gelu_exact_prime(float t) {
    return 0.5f * erfcf(-0.70710678118654752f * t) + t * 0.3989422804014327f * expf(-0.5f * t * t);
}

// Tap gradients as [B*Ca][tiles][kSlot]: tiles == 1 is sum_tiles' result.  With few tiles the kernels below add them up
// themselves, which is a launch less (64 patches of 64x64: sum_tiles took 6.5 us).
constexpr int kDirectTiles = 16;
struct Taps {
    const float* p;
    int tiles;
    template <bool kAll>                                         // all loads in flight, not four
    __device__ __forceinline__ float get(size_t bc, int slot) const {
        const float* q = p + bc * tiles * kSlot + slot;
        float s = 0.f;
        if constexpr (kAll) {
            float v[kDirectTiles];
#pragma unroll
            for (int t = 0; t < kDirectTiles; ++t) v[t] = t < tiles ? __ldcg(q + (size_t)t * kSlot) : 0.f;
#pragma unroll
            for (int t = 0; t < kDirectTiles; ++t) s += v[t];
        } else {
#pragma unroll 4
            for (int t = 0; t < tiles; ++t) s += __ldcg(q + (size_t)t * kSlot);
        }
        return s;
    }
};
// Per-image values for the sums over images: g_dk [B][9 Ca], pooled means [B][Ca], activations and g_t [B][hidden].
struct ImageValues { float *gdk, *mean, *act, *gt; };

// kernel 2b.  An image is one block, or two where there are few images: its pooled means and g_dk, the estimator's forward values and the
// part of the chain that belongs to one image; dk (rotated) and the GAP-path constant go to the stencil pass that follows -- of two blocks
// the first writes dk and the second the constant.  The blocks behind them take g_lk = sum_b g_tap, 32 consecutive taps each (the
// lanes), images dealt to the eight warps and the warps added in order, the kFlipBlocks behind those the rotated LK, and where there are
// few images (kFew) the last ones the estimator's weight gradients, 256 elements each, from means and g_dk of their own.
// Bound: latency of a few dependent phases.  Every sum that is longer than a few terms is taken by a warp and nothing waits for sum_tiles
// where there are few tiles: 64 patches of 64x64 with two layers took 6.5 (sum_tiles) + 8.3 + 22 us cold, the last one a thread per
// output over 64 images; 8 + 4.6 us now, overlapping their neighbours.
constexpr int kFlipBlocks = 8, kEstThreads = 256, kEstMaxCa = 1024;
// Few images: two blocks an image, and blocks of weight gradients that work out means, g_dk and the hidden layer of all images for
// themselves instead of a launch behind this one.  Measured, whole backward pass, bf16 NHWC, as a launch of its own / here: one layer,
// 640x360 57.7 / 54.5 us, 4 x (96x96) 30.3 / 28.6, 8 x (64x64) 29.1 / 28.7, 16 x (64x64) 29.7 / 30.2; two layers, h = 8, 640x360
// 59.9 / 56.0, 2 x (96x96) 30.9 / 29.9, 4 x (64x64) 29.9 / 31.2, 8 x (64x64) 30.6 / 35.6.  Not where the means are sums over chunks
// (decomposed, up to 16 tiles an image), image after image, from three images on: 2 x (96x96) 43.0 / 42.2, 8 x (64x64) 42.8 / 45.3; nor
// in front of the dense form's stencil, which works ahead of dk and so hides the other launch: 64x64 42.6 / 43.4.
inline bool few_images(int B, int Ca, int hidden, bool dense, bool chunk_means) {
    return !dense && B <= kEstThreads / 32 && B * hidden <= 16 && (!chunk_means || B <= 2) && B * Ca <= kEstMaxCa;
}
struct EstimatorGrads { float *w_last, *b_last, *w_down, *b_down; };
template <typename T, bool kFew>
__global__ void __launch_bounds__(kEstThreads)
estimator_image(const Taps taps, const float* __restrict__ xs_part, int chunks, int B, int Ca, int hidden, int H, int W, int KK,
                const T* __restrict__ w_large, const T* __restrict__ w_down, const T* __restrict__ b_down,
                const T* __restrict__ w_last, const T* __restrict__ b_last, const ImageValues iv, float* __restrict__ dk_flip,
                float* __restrict__ bias, float* __restrict__ g_lk, T* __restrict__ w_flip, const EstimatorGrads eg)
{
    extern __shared__ float sm[];
    __shared__ float red[kEstThreads];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, ltaps = KK * KK;
    const int image_blocks = kFew ? 2 * B : B, lk_blocks = g_lk ? (Ca * ltaps + 31) / 32 : 0, flip_blocks = w_flip ? kFlipBlocks : 0;
    const int job = (int)blockIdx.x - image_blocks;
    // The stencil that follows few images gains nothing from an early start, its blocks only take the SMs' registers from these (640x360,
    // 105 blocks: 62.9 us for the whole pass with it, 56.9 without).
    if (!kFew) pdl_launch_dependents();
    pdl_wait_primary();
    if (job >= 0 && job < lk_blocks) {
        const int e = job * 32 + lane, off = (K - KK) / 2;       // a smaller large kernel sits in the middle of the 13 x 13 taps
        float s = 0.f;
        if (e < Ca * ltaps) {
            const int c = e / ltaps, t = (e % ltaps) / KK + off, u = (e % ltaps) % KK + off;
#pragma unroll 4
            for (int b = warp; b < B; b += kEstThreads / 32) s += taps.template get<kFew>((size_t)b * Ca + c, t * K + u);
        }
        red[tid] = s;
        __syncthreads();
        if (warp == 0 && e < Ca * ltaps) {
            for (int w = 1; w < kEstThreads / 32; ++w) s += red[w * 32 + lane];
            g_lk[e] = s;
        }
        return;
    }
    if (job >= lk_blocks && job < lk_blocks + flip_blocks) {
        for (int e = (job - lk_blocks) * kEstThreads + tid; e < Ca * ltaps; e += kFlipBlocks * kEstThreads)
            w_flip[(size_t)(e / ltaps) * ltaps + (ltaps - 1 - e % ltaps)] = w_large[e];
        return;
    }
    const float inv_hw = 1.0f / ((float)H * (float)W);
    // values of images b0 .. b0 + n - 1: pooled means gm [n][Ca], g_dk gd [n][9 Ca], activations aa and g_t gs [n][hidden]
    auto images = [&](int b0, int images_n, float* gm, float* gd, float* aa, float* gs) {
        const int n = kFew ? images_n : 1;
        if (xs_part) {
            // decomposed form: the taps saw the mixed features, the pooled means are those of x: chunks of pixels, dealt to groups of
            // Ca threads, the groups added in order
            const int ng = kEstThreads / Ca, k = tid % Ca, j = tid / Ca;
            for (int b = 0; b < n; ++b) {
                float s = 0.f;
                if (j < ng) {
#pragma unroll 8
                    for (int c = j; c < chunks; c += ng) s += __ldcg(xs_part + ((size_t)(b0 + b) * chunks + c) * Ca + k);
                }
                if (b) __syncthreads();
                red[tid] = s;
                __syncthreads();
                if (tid < Ca) {
                    for (int g = 1; g < ng; ++g) s += red[g * Ca + tid];
                    gm[b * Ca + tid] = s * inv_hw;
                }
            }
        } else {
            for (int k = tid; k < n * Ca; k += kEstThreads) gm[k] = taps.template get<kFew>((size_t)b0 * Ca + k, TAPS) * inv_hw;
        }
        for (int o = tid; o < n * 9 * Ca; o += kEstThreads) {     // o = c*9 + i*3 + j -> the middle 3x3 of the tap gradient
            const int c = o / 9, i = (o % 9) / 3, j = o % 3;
            const float v = taps.template get<kFew>((size_t)b0 * Ca + c, (i + P - 1) * K + (j + P - 1));
            gd[o] = v;
            if (!kFew) iv.gdk[(size_t)b0 * 9 * Ca + o] = v;       // iv: for estimator_weights
        }
        __syncthreads();
        if (!kFew)
            for (int k = tid; k < n * Ca; k += kEstThreads) iv.mean[(size_t)b0 * Ca + k] = gm[k];
        if (hidden > 0) {
            for (int bm = warp; bm < n * hidden; bm += kEstThreads / 32) {
                const int b = kFew ? bm / hidden : 0, m = bm - b * hidden;            // one image where not few
                float t = 0.f, g = 0.f;
                for (int k = lane; k < Ca; k += 32) t = fmaf(Elem<T>::to_f32(w_down[(size_t)m * Ca + k]), gm[b * Ca + k], t);
#pragma unroll 8
                for (int o = lane; o < 9 * Ca; o += 32) g = fmaf(Elem<T>::to_f32(w_last[(size_t)o * hidden + m]), gd[b * 9 * Ca + o], g);
                t = warp_sum(t) + Elem<T>::to_f32(b_down[m]);
                g = warp_sum(g) * gelu_exact_prime(t);
                if (lane == 0) {
                    aa[bm] = gelu_exact(t);
                    gs[bm] = g;
                    if (!kFew) { iv.act[(size_t)b0 * hidden + bm] = aa[bm]; iv.gt[(size_t)b0 * hidden + bm] = g; }
                }
            }
            __syncthreads();
        }
    };
    const int n_in = hidden > 0 ? hidden : Ca;
    if (kFew && job >= 0) {
        // weight gradients of few images: elements as in estimator_weights, images in order
        float *aa = sm, *gs = aa + B * hidden, *gm = gs + B * hidden, *gd = gm + B * Ca;
        const int n0 = 9 * Ca * n_in, n1 = n0 + 9 * Ca, n2 = n1 + hidden * Ca, n3 = n2 + hidden;
        const int e = (job - lk_blocks - flip_blocks) * kEstThreads + tid;
        images(0, B, gm, gd, aa, gs);
        const float *p = nullptr, *q = nullptr;
        int sp = 0, sq = 0;
        float* out = nullptr;
        if (e < n0) { p = gd + e / n_in; sp = 9 * Ca; q = (hidden > 0 ? aa : gm) + e % n_in; sq = n_in; out = eg.w_last ? eg.w_last + e : nullptr; }
        else if (e < n1) { p = gd + (e - n0); sp = 9 * Ca; out = eg.b_last ? eg.b_last + (e - n0) : nullptr; }
        else if (e < n2) { p = gs + (e - n1) / Ca; sp = hidden; q = gm + (e - n1) % Ca; sq = Ca; out = eg.w_down ? eg.w_down + (e - n1) : nullptr; }
        else if (e < n3) { p = gs + (e - n2); sp = hidden; out = eg.b_down ? eg.b_down + (e - n2) : nullptr; }
        if (!out) return;
        float s = 0.f;                                           // as estimator_weights adds up one image per warp: the same bits
        for (int b = 0; b < B; ++b) s = __fadd_rn(s, q ? __fmul_rn(p[b * sp], q[b * sq]) : p[b * sp]);
        *out = s;
        return;
    }
    const int b = kFew ? blockIdx.x / 2 : blockIdx.x, part = kFew ? 1 + (blockIdx.x & 1) : 3;     // bit 0: dk, bit 1: the constant
    float *aa = sm, *gs = aa + hidden;
    // in shared memory, or where they go anyway if C_a is too large for it
    float* gm = Ca <= kEstMaxCa ? gs + hidden : iv.mean + (size_t)b * Ca;
    float* gd = Ca <= kEstMaxCa ? gm + Ca : iv.gdk + (size_t)b * 9 * Ca;
    images(b, 1, gm, gd, aa, gs);
    if (part & 1) {
        const float* vin = hidden > 0 ? aa : gm;
        for (int o = tid; o < 9 * Ca; o += kEstThreads) {
            float s = Elem<T>::to_f32(b_last[o]);
#pragma unroll 8
            for (int m = 0; m < n_in; ++m) s = fmaf(Elem<T>::to_f32(w_last[(size_t)o * n_in + m]), vin[m], s);
            dk_flip[(size_t)b * Ca * 9 + (o / 9) * 9 + (8 - o % 9)] = s;
        }
    }
    if (part & 2) {
        // bias[b][k] = g_g[b][k] / (H W): a warp per element
        for (int k = warp; k < Ca; k += kEstThreads / 32) {
            float s = 0.f;
            if (hidden > 0) {
                for (int m = lane; m < hidden; m += 32) s = fmaf(Elem<T>::to_f32(w_down[(size_t)m * Ca + k]), gs[m], s);
            } else {
#pragma unroll 8
                for (int o = lane; o < 9 * Ca; o += 32) s = fmaf(Elem<T>::to_f32(w_last[(size_t)o * Ca + k]), gd[o], s);
            }
            s = warp_sum(s);
            if (lane == 0) bias[(size_t)b * Ca + k] = s * inv_hw;
        }
    }
}

// kernel 2c: the estimator's weight gradients, sums over images: 32 consecutive elements per block (the lanes), images dealt to
// the eight warps in order, the warps added in order.  Elements: g_W_last [9 Ca][n_in], g_b_last [9 Ca], then (two layers)
// g_W_down [hidden][Ca], g_b_down [hidden].
__global__ void __launch_bounds__(kEstThreads)
estimator_weights(const ImageValues iv, int B, int Ca, int hidden, float* __restrict__ g_wl, float* __restrict__ g_bl,
                  float* __restrict__ g_wd, float* __restrict__ g_bd)
{
    __shared__ float red[kEstThreads];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_in = hidden > 0 ? hidden : Ca, n0 = 9 * Ca * n_in, n1 = n0 + 9 * Ca, n2 = n1 + hidden * Ca, n3 = n2 + hidden;
    pdl_launch_dependents();
    pdl_wait_primary();
    const int e = blockIdx.x * 32 + lane;
    const float *p = nullptr, *q = nullptr;
    int sp = 0, sq = 0;
    float* out = nullptr;
    if (e < n0) { p = iv.gdk + e / n_in; sp = 9 * Ca; q = (hidden > 0 ? iv.act : iv.mean) + e % n_in; sq = n_in; out = g_wl ? g_wl + e : nullptr; }
    else if (e < n1) { p = iv.gdk + (e - n0); sp = 9 * Ca; out = g_bl ? g_bl + (e - n0) : nullptr; }
    else if (e < n2) { p = iv.gt + (e - n1) / Ca; sp = hidden; q = iv.mean + (e - n1) % Ca; sq = Ca; out = g_wd ? g_wd + (e - n1) : nullptr; }
    else if (e < n3) { p = iv.gt + (e - n2); sp = hidden; out = g_bd ? g_bd + (e - n2) : nullptr; }
    float s = 0.f;
    if (out) {
#pragma unroll 8
        for (int b = warp; b < B; b += kEstThreads / 32)
            s = fmaf(__ldcg(p + (size_t)b * sp), q ? __ldcg(q + (size_t)b * sq) : 1.0f, s);
    }
    red[threadIdx.x] = s;
    __syncthreads();
    if (warp != 0 || !out) return;
#pragma unroll
    for (int w = 1; w < kEstThreads / 32; ++w) s += red[w * 32 + lane];
    *out = s;
}

}}  // namespace esc::bwd
