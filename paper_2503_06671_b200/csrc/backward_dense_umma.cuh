// Gradient of the dense large kernel (ESC paper, Section 3.2, differentiated) on the fifth-generation tensor cores, for NHWC bf16
// tensors with 16 attention channels:
//
//   g_wd[n,k,i,j] = sum_{b,y,x} go[b,n,y,x] * x~[b,k,y+i-6,x+j-6]
//
// Formulation.  The pixels are the contraction axis.  For ONE staged input row and 16 of its pixels, one tcgen05.mma takes as
// A (M = 128) eight tap columns j x 16 input channels -- the same 16 pixels of x shifted by 0 .. 7 pixels -- and as B (N = 208)
// the 13 go rows that the input row meets (tap rows i) x 16 output channels:
//
//   D_h[(j, k)][(i, n)] += sum_px x[row][px + j][k] * go[row - i][px][n],     h = 0: j = 0 .. 7,  h = 1: j = 5 .. 12
//
// 13 x 13 of the 16 x 13 (j, i) pairs are useful (columns 5 .. 7 are formed twice), all 43,264 sums sit in 416 columns of tensor
// memory for the whole life of a block, and nothing is unfolded: both operands are MN-major views of pixel-major rows
// ([pixel][16 channels], 32 bytes, as TMA writes them with the 32-byte swizzle).  An MN-atom is 16 channels of eight pixels; the
// next atom of A lies one PIXEL (32 bytes) further on -- the tap shift --, the next atom of B one go ROW further on.  The swizzle
// is a function of the shared-memory address, so overlapping and shifted views are legal.  At the ends of a tile's rows the
// instruction takes only the go rows that exist (N = 16 .. 192).
//
// A block walks units (a strip of up to 64 columns x up to 32 go rows of one image, contiguous runs of them): warp 0 requests go
// rows (two tiles) and the rows + 12 input rows (a ring of eight groups) in turn, four rows per TMA load, so that the first
// instruction waits for eight rows and not for the tile; warp 1 issues; at the end warps 2-9 read the sums and write them
// once, 128 contiguous bytes per store instruction; `sum_dense_umma` adds the blocks in order.
// bf16 products are exact in fp32 and the accumulation is fp32, as in the warp-level kernel (backward_dense.cuh), whose
// mma.sync ceiling is 41 us for the 22.7 GFLOP of 64 patches of 64x64.
// Bound: an instruction of M = 128 takes 39 cycles at N = 16 and N / 2 from N = 128 on, whatever the operands' layout (measured
// on this formulation's descriptors): 28.5 k cycles for a unit of 32 rows x 64 columns (352 instructions).  64 patches of 64x64:
// 113 us (warp-level kernel) -> 30.6 us, of which 6 k cycles until the first rows have landed and 5.5 k for the sums' way out.
#pragma once
#include "backward_dense.cuh"
#include "stencil_dense_umma.cuh"

namespace esc { namespace bwd { namespace dense { namespace umma {

using tma::u64; using tma::smem_u32; using tma::mbar_init; using tma::mbar_expect_tx; using tma::mbar_wait; using tma::tma_load_4d;
using tma::mbar_arrive;
using tma::umma::mbar_wait_warp; using tma::umma::mma_f16; using tma::umma::mma_commit; using tma::umma::tc_fence_after; using tma::umma::tc_fence_before;
using tma::umma::tmem_ld16; using tma::umma::tmem_zero16; using tma::umma::tmem_wait_st;

constexpr int kMaxRows = 32, kMaxCols = 64;                        // go tile
constexpr int kGroup = 4, kRing = 8;                               // rows per TMA load; groups of input rows in the ring
constexpr int GO_BYTES = kMaxRows * kMaxCols * 32;
constexpr int XG_BYTES = kGroup * (kMaxCols + 16) * 32;
constexpr int kThreads = 320;
constexpr int kGoGroups = kMaxRows / kGroup;
constexpr int kBarOffset = 2 * GO_BYTES + kRing * XG_BYTES;
constexpr size_t kSmemBytes = kBarOffset + 512;
constexpr int kCols1 = K * CA;                                     // tensor-memory column of D_1
static_assert((2 * kRing + 2 * kGoGroups + 3) * 8 + 4 <= 512, "barriers fit");
static_assert(XG_BYTES % 1024 == 0 && kSmemBytes <= 227 * 1024 && 2 * kCols1 <= 512, "layout");

struct Params {
    int B, H, W;
    int strips, segs, strip_w, seg_rows;
    long long units;
    float* part;                     // [gridDim.x][13 column blocks: i = 12 - block][16 n][13 j][16 k]
    unsigned* ctrl;
};

// MN-major operand, 32-byte swizzle: atoms of 16 channels x 8 pixels (256 contiguous bytes); the next atom along M or N is `mn`
// bytes further on, the next eight pixels 256 bytes.
__device__ __forceinline__ unsigned long long desc_mn(uint32_t addr, uint32_t mn) {
    return (unsigned long long)((addr >> 4) & 0x3FFFu) | ((unsigned long long)((mn >> 4) & 0x3FFFu) << 16) |
           ((unsigned long long)(256u >> 4) << 32) | (1ull << 46) | (6ull << 61);
}
// D fp32, A and B bf16, both MN-major, M = 128, N = n
__device__ __forceinline__ uint32_t instr_desc_mn(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(n >> 3) << 17) | (8u << 24);
}

struct Tile { int b, x0, ya, rows; };
__device__ __forceinline__ Tile decode(long long uv, const Params& p) {
    unsigned u = (unsigned)uv;
    Tile t;
    const int seg = (int)(u % (unsigned)p.segs); u /= (unsigned)p.segs;
    t.x0 = (int)(u % (unsigned)p.strips) * p.strip_w;
    t.b = (int)(u / (unsigned)p.strips);
    t.ya = seg * p.seg_rows;
    t.rows = min(p.seg_rows, p.H - t.ya);
    return t;
}

__global__ void __launch_bounds__(kThreads, 1)
tap_grad_dense_umma(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_go, const Params p)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    u64* bars = reinterpret_cast<u64*>(smem + kBarOffset);
    const uint32_t xfull0 = smem_u32(bars), xfree0 = xfull0 + 8 * kRing, gfull0 = xfree0 + 8 * kRing,
                   gfree0 = gfull0 + 16 * kGoGroups, done = gfree0 + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kRing + 2 * kGoGroups + 3);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // warp: known to be uniform
    if (tid == 0) {
        for (int s = 0; s < kRing; ++s) { mbar_init(xfull0 + 8 * s, 1); mbar_init(xfree0 + 8 * s, 1); }
        for (int s = 0; s < 2 * kGoGroups; ++s) mbar_init(gfull0 + 8 * s, 1);
        for (int s = 0; s < 2; ++s) mbar_init(gfree0 + 8 * s, 1);
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    if (warp >= 2) {                                               // every instruction accumulates; warps 2-5 clear D_0, 6-9 D_1
        for (int s = 0; s < K; ++s) tmem_zero16(lane_base + (uint32_t)(((warp - 2) / 4 * K + s) * CA));
        tmem_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    const long long u0 = p.units * blockIdx.x / gridDim.x, u1 = p.units * (blockIdx.x + 1) / gridDim.x;
    const int spx = p.strip_w + 16;
    if (warp == 0) {
        if (lane == 0) {
            bool alive = true;
            unsigned xg = 0, it = 0;                               // groups of input rows and go tiles requested so far
            for (long long u = u0; u < u1 && alive; ++u, ++it) {
                const Tile t = decode(u, p);
                const int gb = (int)(it & 1);
                if (it >= 2) alive = mbar_wait(gfree0 + 8 * gb, ((it >> 1) - 1) & 1, p.ctrl, 0xE0000000u | it);
                if (!alive) break;
                const int go_bytes = kGroup * p.strip_w * 32, go_groups = (t.rows + kGroup - 1) / kGroup;
                const int groups = (t.rows + K - 1 + kGroup - 1) / kGroup;
                // every barrier of the go tile completes one phase per use of the tile, which is what the issuer's parity counts
                for (int g = go_groups; g < kGoGroups; ++g) mbar_arrive(gfull0 + 8 * (gb * kGoGroups + g));
                for (int g = 0; g < groups && alive; ++g, ++xg) {
                    if (g < go_groups) {
                        const uint32_t bar = gfull0 + 8 * (gb * kGoGroups + g);
                        mbar_expect_tx(bar, (unsigned)go_bytes);
                        tma_load_4d(smem_u32(smem) + (uint32_t)(gb * GO_BYTES + g * go_bytes), &map_go, bar, 0, t.x0, t.ya + g * kGroup, t.b);
                    }
                    const int slot = (int)(xg % kRing);
                    if (xg >= kRing) alive = mbar_wait(xfree0 + 8 * slot, (xg / kRing - 1) & 1, p.ctrl, 0xE1000000u | xg);
                    if (!alive) break;
                    mbar_expect_tx(xfull0 + 8 * slot, (unsigned)(kGroup * spx * 32));
                    tma_load_4d(smem_u32(smem) + (uint32_t)(2 * GO_BYTES + slot * XG_BYTES), &map_x, xfull0 + 8 * slot, 0, t.x0 - P,
                                t.ya - P + g * kGroup, t.b);
                }
            }
        }
    } else if (warp == 1) {
        bool alive = true;
        unsigned xg = 0, it = 0;
        for (long long u = u0; u < u1 && alive; ++u, ++it) {
            const Tile t = decode(u, p);
            const int gb = (int)(it & 1);
            const int n_in = t.rows + K - 1, steps = (min(p.strip_w, p.W - t.x0) + 15) / 16;
            const uint32_t go_a = smem_u32(smem) + (uint32_t)(gb * GO_BYTES);
            for (int n = 0; n < n_in; ++n) {
                const int slot = (int)(xg % kRing), in_group = n % kGroup;
                if (in_group == 0) {
                    if (n < t.rows) alive = mbar_wait_warp(gfull0 + 8 * (gb * kGoGroups + n / kGroup), (it >> 1) & 1, p.ctrl, 0xE2000000u | it);
                    if (alive) alive = mbar_wait_warp(xfull0 + 8 * slot, (xg / kRing) & 1, p.ctrl, 0xE3000000u | xg);
                    if (!alive) break;
                    tc_fence_after();
                }
                // input row n (image row ya - 6 + n) meets go rows r = n - i: column block 12 - i = 12 - n + r
                const int r_lo = max(0, n - (K - 1)), r_hi = min(t.rows - 1, n), cnt = r_hi - r_lo + 1;
                const uint32_t d0 = tmem + (uint32_t)((K - 1 - n + r_lo) * CA), idesc = instr_desc_mn(cnt * CA);
                unsigned long long db = desc_mn(go_a + (uint32_t)(r_lo * p.strip_w * 32), (uint32_t)(p.strip_w * 32));
                unsigned long long da = desc_mn(smem_u32(smem) + (uint32_t)(2 * GO_BYTES + slot * XG_BYTES + in_group * spx * 32), 32u);
                for (int s = 0; s < steps; ++s) {
                    mma_f16(d0, da, db, idesc);
                    mma_f16(d0 + (uint32_t)kCols1, da + 5 * 2, db, idesc);                 // five pixels of 32 bytes further on
                    da += 16 * 2; db += 16 * 2;
                }
                if (in_group == kGroup - 1 || n == n_in - 1) { mma_commit(xfree0 + 8 * slot); ++xg; }
            }
            mma_commit(gfree0 + 8 * gb);
        }
        mma_commit(done);                                          // arrives when every instruction above has finished
    } else {
        if (lane == 0) mbar_wait(done, 0, p.ctrl, 0xE4000000u);
        __syncwarp();
        tc_fence_after();
        const int m = (warp & 3) * 32 + lane, h = (warp - 2) / 4;  // lane of tensor memory: (tap column, input channel)
        const bool wr = h == 0 || m >= 3 * CA;                     // h = 1 holds columns 5 .. 12; 5 .. 7 are there already
        float* col = p.part + (size_t)blockIdx.x * kPartFloats + (h ? 5 * CA + m : m);
#pragma unroll 2
        for (int cb = 0; cb < K; ++cb) {
            uint32_t r[16];
            tmem_ld16(lane_base + (uint32_t)(h * kCols1 + cb * CA), r);
            if (wr) {
#pragma unroll
                for (int n = 0; n < 16; ++n) col[(cb * CA + n) * (K * CA)] = __uint_as_float(r[n]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// g_wd [CA][CA][KK][KK] = the middle KK x KK of the blocks' sums, blocks added in a fixed order: a warp's lanes take 32
// consecutive sums, the eight warps every eighth block each, then the warps are added in order.
constexpr int kSumWarps = 8;
__global__ void __launch_bounds__(kSumWarps * 32)
sum_dense_umma(const float* __restrict__ part, int blocks, int KK, float* __restrict__ g_wd)
{
    __shared__ float acc[kSumWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
    float s = 0.f;
    const float* q = part + e;
#pragma unroll 8
    for (int b = warp; b < blocks; b += kSumWarps) s += __ldcg(q + (size_t)b * kPartFloats);
    acc[warp][lane] = s;
    __syncthreads();
    if (warp != 0) return;
#pragma unroll
    for (int w = 1; w < kSumWarps; ++w) s += acc[w][lane];
    const int k = e % CA, j = (e / CA) % K, n = (e / (CA * K)) % CA, cb = e / (CA * K * CA), off = (K - KK) / 2;
    const int i = K - 1 - cb - off, jj = j - off;
    if (i >= 0 && i < KK && jj >= 0 && jj < KK) g_wd[((size_t)(n * CA + k) * KK + i) * KK + jj] = s;
}
static_assert(kPartFloats % 32 == 0, "whole warps of sums");

inline bool applies(int C, int Ca, int dtype, int layout, const void* x, const void* go) {
    return dtype == 1 /*bf16*/ && layout == kNHWC && Ca == CA && C % 8 == 0 && (reinterpret_cast<uintptr_t>(x) & 15u) == 0 &&
           (reinterpret_cast<uintptr_t>(go) & 15u) == 0;
}

// Strips of equal width (a multiple of 16, at most 64); rows per unit from {32, 24, 16, 8}: a unit costs its rows + 12 row-times
// (and about 6 more to fill the pipeline), so long units where there are enough of them, short ones where SMs would idle.
inline void plan(Params& p, int sms) {
    p.strips = (p.W + kMaxCols - 1) / kMaxCols;
    p.strip_w = ((p.W + p.strips - 1) / p.strips + 15) / 16 * 16;
    p.strips = (p.W + p.strip_w - 1) / p.strip_w;
    double best = 1e30;
    for (int rows = kMaxRows; rows >= 8; rows -= 8) {
        const int segs = (p.H + rows - 1) / rows, even = (p.H + segs - 1) / segs;
        const long long units = (long long)p.B * p.strips * segs, per = (units + sms - 1) / sms;
        const double cost = (double)per * (even + 12) + 6;
        if (cost < best * 0.98) { best = cost; p.seg_rows = even; p.segs = segs; p.units = units; }
    }
}

inline int try_launch(int B, int C, int Ca, int H, int W, int dtype, int layout, const void* x, const void* go, float* part,
                      int max_blocks, unsigned* ctrl, cudaStream_t st, int* blocks, int* launches, std::string* err) {
    if (!applies(C, Ca, dtype, layout, x, go)) return tma::kNotApplicable;
    Params p;
    p.B = B; p.H = H; p.W = W; p.part = part; p.ctrl = ctrl;
    plan(p, max_blocks);
    if (p.units > 0x7fffffffLL) return tma::kNotApplicable;
    tma::EncodeTiledFn fn = tma::encode_fn();
    if (!fn) return tma::kNotApplicable;
    CUtensorMap m_x, m_go;
    const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
    const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const cuuint32_t box_x[4] = {(cuuint32_t)CA, (cuuint32_t)(p.strip_w + 16), kGroup, 1};
    const cuuint32_t box_g[4] = {(cuuint32_t)CA, (cuuint32_t)p.strip_w, kGroup, 1};
    for (int q = 0; q < 2; ++q)
        if (fn(q ? &m_go : &m_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(q ? go : x), dims, strides, q ? box_g : box_x, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_64B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return tma::kNotApplicable;
    static bool attr_set[tma::kMaxDevices] = {};
    const int dev = tma::current_device();
    if (dev < 0) return tma::kNotApplicable;
    if (!attr_set[dev]) {
        if (cudaFuncSetAttribute(tap_grad_dense_umma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes) != cudaSuccess) {
            (void)cudaGetLastError();
            return tma::kNotApplicable;
        }
        attr_set[dev] = true;
    }
    *blocks = (int)(p.units < max_blocks ? p.units : max_blocks);
    tap_grad_dense_umma<<<(unsigned)*blocks, kThreads, kSmemBytes, st>>>(m_x, m_go, p);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        char buf[256];
        snprintf(buf, sizeof buf, "tap_grad_dense_umma launch: %s (%s)", cudaGetErrorName(e), cudaGetErrorString(e));
        *err = buf;
        return 7;  // ESC_ERR_CUDA
    }
    ++*launches;
    return 0;
}

}}}}  // namespace esc::bwd::dense::umma
