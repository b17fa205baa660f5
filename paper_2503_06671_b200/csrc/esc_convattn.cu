// C ABI of the ConvAttn forward library: argument checks, scratch layout, kernel selection and
// launches.  The arithmetic lives in the kernels (gap_dynkernel.cuh, stencil_generic.cuh,
// stencil_tma.cuh); nothing here touches tensor data on the host.
#include "../../include/esc_convattn.h"

#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <utility>

#include "common.cuh"
#include "gap_dynkernel.cuh"
#include "stencil_generic.cuh"
#include "stencil_tma.cuh"
#include "stencil_toeplitz.cuh"
#include "stencil_toeplitz_nchw.cuh"
#include "backward_toeplitz.cuh"
#include "backward_toeplitz_nchw.cuh"
#include "stencil_dense.cuh"
#include "stencil_dense_umma.cuh"
#include "stencil_dw_umma.cuh"
#include "stencil_dense_fp32.cuh"
#include "dense_nchw.cuh"
#include <type_traits>
#include "backward.cuh"
#include "backward_pw.cuh"
#include "backward_dense.cuh"
#include "backward_dense_umma.cuh"
#include "conv_fuse.cuh"
#include "conv_fuse_backward.cuh"

namespace {

thread_local std::string g_last_error;
thread_local int g_last_path = 0;
thread_local int g_last_tile_w = 0;
thread_local int g_tile_policy = 0;      // 0 = by cost, else the tile width to use
thread_local int g_engine_policy = 0;    // ESC_ENGINE_AUTO / _FP32 / _TENSOR for the depth-wise stencil
thread_local int g_last_launches = 0;
thread_local int g_dense_engine = 0;     // 0: tcgen05 kernel where it applies, 1: the mma.sync kernel
thread_local bool g_fuse_stage1 = true;  // tensor-core kernel: stage 1 inside it where every CTA has at most two units

int cuda_fail(cudaError_t e, const char* what) {
    char buf[320];
    snprintf(buf, sizeof buf, "%s: %s (%s)", what, cudaGetErrorName(e), cudaGetErrorString(e));
    g_last_error = buf;
    return ESC_ERR_CUDA;
}
#define ESC_CUDA(call)                                        \
    do {                                                      \
        cudaError_t e__ = (call);                             \
        if (e__ != cudaSuccess) return cuda_fail(e__, #call); \
    } while (0)

size_t elem_size(int dtype) { return dtype == ESC_BF16 ? 2 : 4; }

struct Problem {
    int B, C, Ca, H, W, K, dtype, layout;
    const void* w_point = nullptr;   // [Ca][Ca] point-wise filter LK^c of the decomposed form (Eq. 5), or none
    bool dense = false;              // w_large is the dense kernel [Ca][Ca][K][K] of Section 3.2
    const float* bias = nullptr;     // [B][Ca] constant per (image, channel) added to the attention outputs (backward pass)
    bool skip_copy = false;          // the identity channels are not written (the fused 1x1 convolution reads them from x)
    bool pack_room = false;          // the caller's workspace has room for the packed map(s)
    size_t es() const { return elem_size(dtype); }
    size_t elems() const { return (size_t)B * C * H * W; }
};

int check_shape(const Problem& p) {
    if (p.B <= 0 || p.C <= 0 || p.H <= 0 || p.W <= 0 || p.Ca <= 0 || p.Ca > p.C) return ESC_ERR_SHAPE;
    if (p.K < 3 || (p.K & 1) == 0) return ESC_ERR_SHAPE;   // the 3x3 dynamic kernel is folded into the K x K one
    if (p.K > ESC_MAX_K) return ESC_ERR_UNSUPPORTED;
    if (p.dtype != ESC_F32 && p.dtype != ESC_BF16) return ESC_ERR_UNSUPPORTED;
    if (p.layout != ESC_NCHW && p.layout != ESC_NHWC) return ESC_ERR_UNSUPPORTED;
    // every byte offset the kernels form must fit in 62 bits
    const long double n = (long double)p.B * p.C * p.H * p.W;
    if (n > 1.0e18L) return ESC_ERR_SHAPE;
    return ESC_OK;
}

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

int check_tensors(const Problem& p, const void* x, const void* out) {
    if (!x || !out) return ESC_ERR_NULL;
    if (!aligned(x, 16) || !aligned(out, 16)) return ESC_ERR_ALIGN;
    const uintptr_t xa = reinterpret_cast<uintptr_t>(x), oa = reinterpret_cast<uintptr_t>(out);
    const size_t bytes = p.elems() * p.es();
    if (xa < oa + bytes && oa < xa + bytes) return ESC_ERR_ALIAS;
    return ESC_OK;
}

// ---- workspace layout -------------------------------------------------------------------
//   [ctrl words: header + arrival counters + launch flags, see ctrl_images][pad to 256][dk: B*Ca*9 floats][pad]
//   [partials: B*S*Ca floats][pad][per-unit sums of the one-launch form: kMaxFusedUnits * SMs * 16 floats][pad]
//   [large kernel padded to 13 x 13, bf16]                        (the last two only where a tensor-core kernel can run: C_a % 16 == 0)
size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct Workspace {
    unsigned* ctrl;
    unsigned* arrivals;
    unsigned* flags;
    float* dk;
    float* partial;
    float* unit_sums;
    void* lk_pad;                    // [Ca][13][13] bf16: a smaller large kernel zero-padded for the tensor-core kernels
    void* packed;                    // C_a = 16: [B][H][W][16] bf16, the attention channels of an NCHW map for the dense form
};

bool is_large_map(int B, long long HW) { return (long double)B * HW >= 1.5e6L; }

// SM count of the current device; a B200's 148 where no device can be asked (size queries on a
// machine without a GPU).
int sms_or_nominal() {
    const int v = esc::tma::sm_count();
    return v > 0 ? v : 148;
}

// Grid of the GAP kernel.  Narrow: at most one block per SM, which is what fits beside a CTA of the
// FP32 stencil kernel (58 k registers).  Wide: three blocks per SM, for batches in front of the Toeplitz stencil kernels, whose
// CTAs need every image's dk early (measured on 64 patches
// of 64x64: 35.5 us per forward against 37.8; a single 640x360 map: 37.4 against 36.2, so single images
// keep the narrow grid).  Large: two blocks of 512 threads per SM, for maps so large that the stencil kernel takes many waves and
// the GAP kernel runs ahead of it rather than beside it.
// In front of the tcgen05 depth-wise kernel nothing runs beside it either (that kernel's CTA takes all registers of an SM): large,
// whatever K and B are, up to 64 attention channels.  Forward, us, narrow / wide / large: 1280x720, 32 of 64 channels 131 / 130 / 124; 900x500,
// 48 of 192 119 / 121 / 115; 64 x (96x96), 32 of 64, K = 9 109 / 105 / 103; 300 x (40x40) 108 / 90 / 91.  Beyond that many channels the
// estimators behind the pooling count for more, and the fewer slabs there are the sooner the first image's can start: 16 x (96x96), 128 of
// 256 172 / 243 / 277; 128 x (40x40), 96 of 128 134 / 185 / 189; 4 x (300x300), 128 262 / 305 / 303; 500x500, 128 of 256 223 / 232 / 220.
enum class GapGrid { Narrow, Wide, Large };
GapGrid gap_grid(int B, int Ca, long long HW, bool toeplitz, bool dw_umma) {
    if (is_large_map(B, HW) || (dw_umma && Ca <= 64)) return GapGrid::Large;
    return toeplitz && !dw_umma && B > 1 ? GapGrid::Wide : GapGrid::Narrow;
}

int slabs_for(int B, long long HW, bool wide) {
    // At most one work item per block over the whole batch, so that every block walks one item and no
    // image waits for a second round; at least 512 pixels per slab.
    const long long sms = sms_or_nominal();
    const long long target = wide ? 3 * sms : sms;
    long long s = target / B;
    const long long cap = (HW + 511) / 512;
    if (s > cap) s = cap;
    if (s > esc::kMaxSlabs) s = esc::kMaxSlabs;
    if (s < 1) s = 1;
    return (int)s;
}

// A buffer is zeroed once and then serves calls of any shape, in any order.  The arrival counters must be zero between calls, so
// nothing but counters may lie where another shape has them: they and the flags (whose value at rest does not matter) have a place
// for kCtrlImages images that no shape puts anything else on.  Beyond that many images the counters are cleared by every call.
constexpr int kCtrlImages = 640;
int ctrl_images(int B) { return B > kCtrlImages ? B : kCtrlImages; }

// Fills `w` for a workspace at `ws` (null: only the size is wanted) and returns the size that every call needs.  The packed map
// lies behind that: only the dense form on bf16 NCHW tensors has a use for it, and does without where there is no room.
size_t carve(void* ws, int B, int Ca, long long HW, Workspace& w) {
    char* base = static_cast<char*>(ws);
    const int n = ctrl_images(B);
    const bool tensor = Ca % esc::tma::CG == 0;
    size_t off = round_up((size_t)(esc::kCtrlHeaderWords + 2 * (size_t)n) * 4, 256);
    auto take = [&](size_t bytes) {
        char* p = base + off;
        off += round_up(bytes, 256);
        return p;
    };
    w.ctrl = reinterpret_cast<unsigned*>(base);
    w.arrivals = w.ctrl + esc::kCtrlHeaderWords;
    w.flags = w.arrivals + n;
    w.dk = reinterpret_cast<float*>(take((size_t)B * Ca * 9 * 4));
    w.partial = reinterpret_cast<float*>(take((size_t)B * slabs_for(B, HW, true) * Ca * 4));   // room for either grid policy
    w.unit_sums = reinterpret_cast<float*>(take(tensor ? (size_t)esc::tma::toep::kMaxFusedUnits * sms_or_nominal() * 16 * 4 : 0));
    w.lk_pad = take(tensor ? (size_t)Ca * 169 * 2 : 0);
    w.packed = base + off;
    return off;
}
Workspace carve(void* ws, int B, int Ca, long long HW) {
    Workspace w;
    carve(ws, B, Ca, HW, w);
    return w;
}
size_t workspace_bytes(int B, int Ca, long long HW) {
    Workspace w;
    return carve(nullptr, B, Ca, HW, w);
}
size_t workspace_bytes_packed(int B, int Ca, long long HW, int K) {
    return workspace_bytes(B, Ca, HW) + round_up(esc::dense16::packed_bytes(B, Ca, HW, K), 256);
}
// In front of a kernel that counts arrivals.
int clear_counters(const Workspace& w, int B, cudaStream_t st) {
    if (B > kCtrlImages) ESC_CUDA(cudaMemsetAsync(w.arrivals, 0, (size_t)B * sizeof(unsigned), st));
    return ESC_OK;
}

int check_workspace(const Problem& p, const void* ws, size_t bytes) {
    if (!ws || !aligned(ws, 256)) return ESC_ERR_WORKSPACE;
    if (bytes < workspace_bytes(p.B, p.Ca, (long long)p.H * p.W)) return ESC_ERR_WORKSPACE;
    return ESC_OK;
}

// ---- stage 1 ------------------------------------------------------------------------------
// The estimator's weights: one linear layer (hidden == 0: w_last [9*Ca][Ca]) or two layers with the
// GELU between them (w_down [hidden][Ca], b_down [hidden], w_last = w_up [9*Ca][hidden]).
struct Estimator {
    const void *w_last, *b_last, *w_down, *b_down;
    int hidden;
};

template <typename T, int LAYOUT, int kThreads>
int launch_gap_n(const Problem& p, const void* x, const Estimator& est, const Workspace& w, float* dk_out, cudaStream_t st, int S,
                 long long cap) {
    const long long items = (long long)p.B * S;
    const unsigned grid = (unsigned)(items < cap ? items : cap);
    const size_t scratch = (size_t)esc::gap_scratch_floats(LAYOUT, p.C, p.Ca, esc::Elem<T>::kVec, kThreads);
    const size_t smem = (scratch + p.Ca) * sizeof(float);
    if (smem > 48 * 1024) return ESC_ERR_UNSUPPORTED;
    // Same shared-memory carve-out as the stencil kernel: an SM changes its L1/shared split only
    // when idle, so with different preferences the two kernels could never share an SM.
    static bool carveout_set[esc::tma::kMaxDevices] = {};   // per device and per instantiation
    const int dev = esc::tma::current_device();
    if (dev < 0) return ESC_ERR_UNSUPPORTED;
    if (!carveout_set[dev]) {
        ESC_CUDA(cudaFuncSetAttribute(esc::gap_dynkernel<T, LAYOUT, kThreads>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                      cudaSharedmemCarveoutMaxShared));
        carveout_set[dev] = true;
    }
    esc::gap_dynkernel<T, LAYOUT, kThreads><<<grid, kThreads, smem, st>>>(
        static_cast<const T*>(x), p.B, p.C, p.Ca, p.H, p.W, S, static_cast<const T*>(est.w_last),
        static_cast<const T*>(est.b_last), static_cast<const T*>(est.w_down), static_cast<const T*>(est.b_down),
        est.hidden, w.partial, w.arrivals, dk_out);
    ESC_CUDA(cudaGetLastError());
    ++g_last_launches;
    return ESC_OK;
}
template <typename T, int LAYOUT>
int launch_gap_t(const Problem& p, const void* x, const Estimator& est,
                 const Workspace& w, float* dk_out, cudaStream_t st, GapGrid grid) {
    const long long HW = (long long)p.H * p.W, sms = sms_or_nominal();
    const bool wide = grid != GapGrid::Narrow;
    const int S = slabs_for(p.B, HW, wide);
    // Large maps: bound by DRAM and by how many bytes are in flight, so two blocks of 512 threads on each SM instead of three of 128,
    // as long as their scratch fits (C_a up to 720).  1920x1080 bf16 NHWC, 32 of 64 channels (265 MB of whole lines): 65 -> 58 us.
    const int smem_large = (esc::gap_scratch_floats(LAYOUT, p.C, p.Ca, esc::Elem<T>::kVec, esc::kGapThreadsLarge) + p.Ca) * 4;
    if (grid == GapGrid::Large && smem_large <= 48 * 1024) {
        const long long s2 = 2 * sms / p.B < 1 ? 1 : 2 * sms / p.B;
        return launch_gap_n<T, LAYOUT, esc::kGapThreadsLarge>(p, x, est, w, dk_out, st, S < s2 ? S : (int)s2, 2 * sms);
    }
    return launch_gap_n<T, LAYOUT, esc::kGapThreads>(p, x, est, w, dk_out, st, S, wide ? 3 * sms : sms);
}

int launch_gap(const Problem& p, const void* x, const Estimator& est,
               const Workspace& w, float* dk_out, cudaStream_t st, bool toeplitz = false, bool dw_umma = false) {
    if ((long long)p.B * esc::kMaxSlabs > 0x7fffffffLL) return ESC_ERR_UNSUPPORTED;
    const GapGrid grid = gap_grid(p.B, p.Ca, (long long)p.H * p.W, toeplitz, dw_umma);
    if (p.dtype == ESC_F32)
        return p.layout == ESC_NCHW ? launch_gap_t<float, esc::kNCHW>(p, x, est, w, dk_out, st, grid)
                                    : launch_gap_t<float, esc::kNHWC>(p, x, est, w, dk_out, st, grid);
    return p.layout == ESC_NCHW ? launch_gap_t<__nv_bfloat16, esc::kNCHW>(p, x, est, w, dk_out, st, grid)
                                : launch_gap_t<__nv_bfloat16, esc::kNHWC>(p, x, est, w, dk_out, st, grid);
}

int check_estimator(const Problem& p, const Estimator& e) {
    if (!e.w_last || !e.b_last) return ESC_ERR_NULL;
    if (!aligned(e.w_last, p.es()) || !aligned(e.b_last, p.es())) return ESC_ERR_ALIGN;
    if (e.hidden == 0) return ESC_OK;
    if (e.hidden < 0 || e.hidden > esc::kMaxHidden) return ESC_ERR_SHAPE;
    if (!e.w_down || !e.b_down) return ESC_ERR_NULL;
    if (!aligned(e.w_down, p.es()) || !aligned(e.b_down, p.es())) return ESC_ERR_ALIGN;
    return ESC_OK;
}

// ---- stage 2 ------------------------------------------------------------------------------
template <typename U>
int launch_copy_u(const void* x, void* out, long long rows, long long row_b, long long stride_b,
                  long long off_b, cudaStream_t st) {
    const long long u = sizeof(U);
    const long long total = rows * (row_b / u);
    if (total == 0) return ESC_OK;
    long long blocks = (total + 255) / 256;
    if (blocks > 16LL * sms_or_nominal()) blocks = 16LL * sms_or_nominal();
    esc::copy_through<U><<<(unsigned)blocks, 256, 0, st>>>(static_cast<const U*>(x), static_cast<U*>(out), rows,
                                                          row_b / u, stride_b / u, off_b / u);
    ESC_CUDA(cudaGetLastError());
    ++g_last_launches;
    return ESC_OK;
}

int launch_copy(const Problem& p, const void* x, void* out, cudaStream_t st) {
    if (p.Ca == p.C) return ESC_OK;
    const long long es = (long long)p.es(), HW = (long long)p.H * p.W;
    long long rows, row_b, stride_b, off_b;
    if (p.layout == ESC_NCHW) { rows = p.B; row_b = (p.C - p.Ca) * HW * es; stride_b = p.C * HW * es; off_b = p.Ca * HW * es; }
    else { rows = (long long)p.B * HW; row_b = (p.C - p.Ca) * es; stride_b = p.C * es; off_b = p.Ca * es; }
    if (row_b % 16 == 0 && stride_b % 16 == 0 && off_b % 16 == 0) return launch_copy_u<uint4>(x, out, rows, row_b, stride_b, off_b, st);
    if (row_b % 4 == 0 && stride_b % 4 == 0 && off_b % 4 == 0) return launch_copy_u<uint32_t>(x, out, rows, row_b, stride_b, off_b, st);
    return launch_copy_u<uint16_t>(x, out, rows, row_b, stride_b, off_b, st);
}

// The identity channels as a copy job for extra blocks of a stencil launch (blocks == 0: nothing to copy).
esc::CopyJob make_copy_job(const Problem& p, const void* x, void* out, long long first_block, int threads) {
    esc::CopyJob j = {};
    if (p.Ca == p.C || p.skip_copy) return j;
    const long long es = (long long)p.es(), HW = (long long)p.H * p.W;
    long long rows, row_b, stride_b, off_b;
    if (p.layout == ESC_NCHW) { rows = p.B; row_b = (p.C - p.Ca) * HW * es; stride_b = p.C * HW * es; off_b = p.Ca * HW * es; }
    else { rows = (long long)p.B * HW; row_b = (p.C - p.Ca) * es; stride_b = p.C * es; off_b = p.Ca * es; }
    const int u = (row_b % 16 == 0 && stride_b % 16 == 0 && off_b % 16 == 0) ? 16
                : (row_b % 4 == 0 && stride_b % 4 == 0 && off_b % 4 == 0) ? 4 : 2;
    j.src = x; j.dst = out;
    j.rows = rows; j.row_units = row_b / u; j.stride_units = stride_b / u; j.offset_units = off_b / u;
    j.unit_bytes = u;
    const long long total = rows * j.row_units;
    long long blocks = (total + (long long)threads * 4 - 1) / ((long long)threads * 4);   // about four units per thread
    if (blocks > 8LL * sms_or_nominal()) blocks = 8LL * sms_or_nominal();
    if (blocks < 1) blocks = 1;
    j.first_block = (unsigned)first_block;
    j.blocks = (unsigned)blocks;
    return j;
}

template <typename T, int LAYOUT, int KT, class G, int CB, int PER_SM>
int launch_regtile(const Problem& p, const void* x, const void* w_large, const float* dk, void* out, cudaStream_t st, bool dependent) {
    using L = esc::RtLayout<G, KT, CB>;
    const int tiles_x = (p.W + G::TX - 1) / G::TX, tiles_y = (p.H + G::TY - 1) / G::TY;
    const long long blocks = (long long)p.B * (p.Ca / CB) * tiles_x * tiles_y;
    const esc::CopyJob job = make_copy_job(p, x, out, blocks, L::Threads);
    if (blocks + job.blocks > 0x7fffffffLL) return ESC_ERR_UNSUPPORTED;
    const int smem = L::bytes(p.Ca, p.w_point != nullptr);
    static bool attr_set[esc::tma::kMaxDevices] = {};
    const int dev = esc::tma::current_device();
    if (dev < 0) return ESC_ERR_UNSUPPORTED;
    if (!attr_set[dev]) {
        ESC_CUDA(cudaFuncSetAttribute(esc::stencil_regtile<T, LAYOUT, KT, G, CB, PER_SM>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(blocks + job.blocks));   // the copy blocks come last
    cfg.blockDim = dim3(L::Threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    ESC_CUDA(cudaLaunchKernelEx(&cfg, esc::stencil_regtile<T, LAYOUT, KT, G, CB, PER_SM>, static_cast<const T*>(x), static_cast<T*>(out), p.C, p.Ca, p.H,
                                p.W, static_cast<const T*>(w_large), static_cast<const T*>(p.w_point), dk, tiles_x, tiles_y, job, p.bias));
    ++g_last_launches;
    return ESC_OK;
}
template <typename T, int LAYOUT, int KT>
int launch_regtile_k(const Problem& p, const void* x, const void* w_large, const float* dk, void* out, cudaStream_t st, bool dependent) {
    auto fewer = [&](int cb, long long per_sm) {           // blocks of the larger geometry
        using G = esc::RtSmall;
        return (long long)p.B * (p.Ca / cb) * ((p.W + G::TX - 1) / G::TX) * ((p.H + G::TY - 1) / G::TY) < per_sm * sms_or_nominal();
    };
    // four channels per block: whole groups of four, their pixels' loads aligned, and the point-wise filter within shared memory
    const bool four = p.Ca % 4 == 0 && (LAYOUT == esc::kNHWC ? p.C % 4 == 0 : p.w_point != nullptr) && (!p.w_point || p.Ca <= 1024);
    if (four) {
        if (fewer(4, 1)) return launch_regtile<T, LAYOUT, KT, esc::RtTiny, 4, 2>(p, x, w_large, dk, out, st, dependent);
        return launch_regtile<T, LAYOUT, KT, esc::RtSmall, 4, 2>(p, x, w_large, dk, out, st, dependent);
    }
    if (fewer(1, 2)) return launch_regtile<T, LAYOUT, KT, esc::RtTiny, 1, 6>(p, x, w_large, dk, out, st, dependent);
    if (fewer(1, 6)) return launch_regtile<T, LAYOUT, KT, esc::RtSmall, 1, 6>(p, x, w_large, dk, out, st, dependent);
    return launch_regtile<T, LAYOUT, KT, esc::RtSmall, 1, 8>(p, x, w_large, dk, out, st, dependent);
}
template <typename T, int LAYOUT>
int launch_generic_t(const Problem& p, const void* x, const void* w_large, const float* dk, void* out, cudaStream_t st, bool dependent) {
    switch (p.K) {
        case 3: return launch_regtile_k<T, LAYOUT, 3>(p, x, w_large, dk, out, st, dependent);
        case 5: return launch_regtile_k<T, LAYOUT, 5>(p, x, w_large, dk, out, st, dependent);
        case 7: return launch_regtile_k<T, LAYOUT, 7>(p, x, w_large, dk, out, st, dependent);
        case 9: return launch_regtile_k<T, LAYOUT, 9>(p, x, w_large, dk, out, st, dependent);
        case 11: return launch_regtile_k<T, LAYOUT, 11>(p, x, w_large, dk, out, st, dependent);
        case 13: return launch_regtile_k<T, LAYOUT, 13>(p, x, w_large, dk, out, st, dependent);
        case 15: return launch_regtile_k<T, LAYOUT, 15>(p, x, w_large, dk, out, st, dependent);
        case 17: return launch_regtile_k<T, LAYOUT, 17>(p, x, w_large, dk, out, st, dependent);
    }
    return ESC_ERR_UNSUPPORTED;
}

int launch_generic(const Problem& p, const void* x, const void* w_large, const float* dk, void* out,
                   cudaStream_t st, bool dependent) {
    g_last_path = 1;
    g_last_tile_w = 0;
    int rc;
    if (p.dtype == ESC_F32)
        rc = p.layout == ESC_NCHW ? launch_generic_t<float, esc::kNCHW>(p, x, w_large, dk, out, st, dependent)
                                  : launch_generic_t<float, esc::kNHWC>(p, x, w_large, dk, out, st, dependent);
    else
        rc = p.layout == ESC_NCHW ? launch_generic_t<__nv_bfloat16, esc::kNCHW>(p, x, w_large, dk, out, st, dependent)
                                  : launch_generic_t<__nv_bfloat16, esc::kNHWC>(p, x, w_large, dk, out, st, dependent);
    return rc;                                             // the identity channels went along as copy blocks
}

// The tensor-core depth-wise kernels are built for 13 x 13 taps.  A large kernel of odd size K < 13 is the 13 x 13 one with
// zeros around it -- exactly the same convolution -- so it is written, zero-padded, into the workspace once per call and
// handed to those kernels as a 13 x 13 kernel; every other kernel gets the weights as the caller gave them.
template <typename T>
__global__ void pad_large_kernel(const T* __restrict__ w, int Ca, int K, T* __restrict__ out) {
    const int off = (13 - K) / 2;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < Ca * 169; e += gridDim.x * blockDim.x) {
        const int c = e / 169, i = (e % 169) / 13 - off, j = e % 13 - off;
        out[e] = ((unsigned)i < (unsigned)K && (unsigned)j < (unsigned)K) ? w[((size_t)c * K + i) * K + j] : T(0.0f);
    }
}
struct TensorLk {
    const void* w;
    int K;
};
// Whether the depth-wise stage goes to the tcgen05 kernel: bf16 NHWC without the point-wise mix, unless the caller pinned the FP32
// kernel (by engine or by one of its tile widths), at least two groups of channels, and more work than the one-launch form of the
// mma.sync kernel takes.  (Forward, mma.sync / tcgen05, us, bursts of twenty: 1920x1080, 32 of 64 channels 325 / 237, with K = 9 329 / 265; 1280x720
// 168 / 123; 900x500, 48 of 192 218 / 114; 64 images of 160x64, 32 of 64 136 / 105, of 96x96, 48 of 192 307 / 155; 50 of 300x22, 32 of 128
// 169 / 69; 44 drawn sizes of two to six groups all faster, 5 to 70 %.  With one group the pooling and the copies weigh more: 1920x1080, 16 of 64 220 / 245,
// 16 of 48 180 / 192; only without identity channels (149 / 117) or on batches of small images (128 x (96x96), K = 9 152 / 126) it wins.)
// It takes every odd K up to 13 as it is.
bool dw_umma_follows(const Problem& p) {
    return !p.dense && !p.w_point && p.Ca >= 2 * esc::tma::CG && g_engine_policy != ESC_ENGINE_FP32 && g_tile_policy == 0 &&
           esc::tma::dwu::applies(p.C, p.Ca, p.K, p.dtype, p.layout) && esc::tma::dwu::fills(p.Ca, sms_or_nominal()) && (long long)p.B * p.H * p.W <= 0x7fffffffLL &&
           (long long)p.B * (p.W + esc::tma::dwu::GAPX) <= 0x3fffffffLL &&
           esc::tma::toep::units_of<esc::tma::toep::Shape64x16>(p.B, p.Ca, p.H, p.W) > (long long)esc::tma::toep::kMaxFusedUnits * sms_or_nominal();
}
TensorLk tensor_lk(const Problem& p, const void* x, const void* out, const void* w_large, void* pad, cudaStream_t st) {
    TensorLk t{w_large, p.K};
    if (p.dense || dw_umma_follows(p) || p.dtype != ESC_BF16 || p.K >= esc::tma::K13 || !pad || g_engine_policy == ESC_ENGINE_FP32 || g_tile_policy != 0) return t;
    if (!esc::tma::toep::applies(p.C, p.Ca, esc::tma::K13, p.dtype, p.layout) &&
        !esc::tma::toepn::takes(p.B, p.C, p.Ca, p.H, p.W, esc::tma::K13, p.dtype, p.layout, x, out))
        return t;
    pad_large_kernel<__nv_bfloat16><<<(p.Ca * 169 + 255) / 256, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(w_large), p.Ca, p.K,
                                                                            static_cast<__nv_bfloat16*>(pad));
    if (cudaGetLastError() != cudaSuccess) return t;
    ++g_last_launches;
    t.w = pad; t.K = esc::tma::K13;
    return t;
}

int launch_stencil(const Problem& p0, const void* x, const void* w_large0, const float* dk, void* out,
                   unsigned* ctrl, cudaStream_t st, bool dependent, const TensorLk* tl = nullptr) {
    // the tensor-core kernels see the (possibly padded) 13 x 13 kernel, everything else the caller's
    Problem p = p0;
    const void* w_large = w_large0;
    if (tl) { p.K = tl->K; w_large = tl->w; }
    if (dw_umma_follows(p0)) {
        const int rc = esc::tma::dwu::try_launch(p0.B, p0.C, p0.Ca, p0.H, p0.W, p0.K, p0.dtype, p0.layout, x, w_large0, dk, p0.bias, out, ctrl, st,
                                                        dependent, &g_last_launches, &g_last_error, p0.skip_copy);
        if (rc == ESC_OK) { g_last_path = 4; g_last_tile_w = esc::tma::dwu::WPX; return ESC_OK; }
        if (rc != esc::tma::kNotApplicable) return rc;
    }
    // Depth-wise K = 13 on NHWC bf16: the tensor-core (Toeplitz) kernel unless the caller pinned the FP32
    // kernel (by engine or by one of its tile widths) or asked for the point-wise mix, which only the
    // FP32 kernel carries.
    if ((!p.w_point || p.Ca == esc::tma::CG) && g_engine_policy != ESC_ENGINE_FP32 && g_tile_policy == 0) {
        int tw = 0;
        const int rc = esc::tma::toep::try_launch_toeplitz(p.B, p.C, p.Ca, p.H, p.W, p.K, p.dtype, p.layout, x, w_large, dk, p.bias,
                                                           out, ctrl, st, dependent, &g_last_launches, &g_last_error, &tw, p.skip_copy, p.w_point);
        if (rc == ESC_OK) { g_last_path = 4; g_last_tile_w = tw; return ESC_OK; }
        if (rc != esc::tma::kNotApplicable) return rc;
        {                                                    // the same arithmetic on NCHW tensors
            const int rn = esc::tma::toepn::try_launch(p.B, p.C, p.Ca, p.H, p.W, p.K, p.dtype, p.layout, x, w_large, dk, p.bias, out,
                                                       ctrl, st, dependent, &g_last_launches, &g_last_error, p.w_point, p.skip_copy);
            if (rn == ESC_OK) { g_last_path = 6; g_last_tile_w = esc::tma::toepn::TW; return ESC_OK; }
            if (rn != esc::tma::kNotApplicable) return rn;
        }
    }
    if (p.skip_copy && p.dtype != ESC_F32 && p.layout == ESC_NHWC) return ESC_ERR_UNSUPPORTED;   // of the kernels below only the generic one (all there is for fp32 and NCHW) can leave the identity channels out
    p.K = p0.K; w_large = w_large0;
    if (g_engine_policy == ESC_ENGINE_TENSOR) return launch_generic(p, x, w_large, dk, out, st, dependent);
    int tile_w = g_tile_policy;
    int rc = esc::tma::try_launch(p.B, p.C, p.Ca, p.H, p.W, p.K, p.dtype, p.layout, x, w_large, p.w_point, dk, p.bias, out,
                                  ctrl, st, dependent, &g_last_launches, &g_last_error, &tile_w);
    if (rc == ESC_OK) { g_last_path = 2; g_last_tile_w = tile_w; return ESC_OK; }
    if (rc != esc::tma::kNotApplicable) return rc;
    return launch_generic(p, x, w_large, dk, out, st, dependent);
}

// Whether launch_stencil will take the Toeplitz NHWC kernel, or for K = 13 the tcgen05 one in its place (same conditions).
bool tensor_stencil_follows(const Problem& p) {
    return !p.dense && (!p.w_point || (p.Ca == esc::tma::CG && !p.bias)) && g_engine_policy != ESC_ENGINE_FP32 && g_tile_policy == 0 &&
           esc::tma::toep::applies(p.C, p.Ca, p.K, p.dtype, p.layout);
}

// ---- library-owned scratch for the entry point that has no workspace argument --------------
struct Scratch { void* ptr = nullptr; size_t bytes = 0; };
std::mutex g_scratch_mu;
std::map<std::pair<int, void*>, Scratch> g_scratch;

int get_scratch(size_t need, cudaStream_t st, void** out) {
    int dev = 0;
    ESC_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    Scratch& s = g_scratch[{dev, (void*)st}];
    if (s.bytes < need) {
        if (s.ptr) { ESC_CUDA(cudaFree(s.ptr)); s.ptr = nullptr; s.bytes = 0; }   // cudaFree waits for pending work
        const size_t cap = round_up(need, 1 << 20);
        ESC_CUDA(cudaMalloc(&s.ptr, cap));
        ESC_CUDA(cudaMemset(s.ptr, 0, cap));
        ESC_CUDA(cudaStreamSynchronize(cudaStreamLegacy));   // st may be a stream that does not wait for that one
        s.bytes = cap;
    }
    *out = s.ptr;
    return ESC_OK;
}

template <typename T, int LAYOUT>
int launch_dense_generic_t(const Problem& p, const void* x, const void* w_dense, const float* dk, void* out,
                           cudaStream_t st, bool dependent) {
    const long long total = (long long)p.B * p.Ca * p.H * p.W;
    long long blocks = (total + 255) / 256;
    if (blocks > 8LL * sms_or_nominal()) blocks = 8LL * sms_or_nominal();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    ESC_CUDA(cudaLaunchKernelEx(&cfg, esc::tma::stencil_dense_generic<T, LAYOUT>, static_cast<const T*>(x),
                                static_cast<T*>(out), p.B, p.C, p.Ca, p.H, p.W, p.K, static_cast<const T*>(w_dense), dk));
    ++g_last_launches;
    return ESC_OK;
}

// Dense large kernel with 16 attention channels on the FP32 pipe; the identity channels go along as copy blocks.
template <typename T, int LAYOUT, int K>
int launch_dense_fp32_k(const Problem& p, const void* x, const void* w_dense, const float* dk, void* out, cudaStream_t st,
                        bool dependent) {
    namespace D = esc::dense32;
    const int tiles_x = (p.W + D::TX - 1) / D::TX, tiles_y = (p.H + D::TY - 1) / D::TY;
    const long long tiles = (long long)p.B * tiles_x * tiles_y;
    const int split = D::choose_split(tiles, sms_or_nominal());
    if (tiles * split > 0x3fffffffLL) return ESC_ERR_UNSUPPORTED;
    esc::CopyJob job = make_copy_job(p, x, out, tiles * split, D::kThreads);
    job.blocks = (job.blocks + split - 1) / split * split;               // whole clusters
    static bool attr_set[esc::tma::kMaxDevices] = {};
    const int dev = esc::tma::current_device();
    if (dev < 0) return ESC_ERR_UNSUPPORTED;
    if (!attr_set[dev]) {
        ESC_CUDA(cudaFuncSetAttribute(D::stencil_dense_fp32<T, LAYOUT, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)std::max(D::Geo<K>::smem_bytes(1), D::Geo<K>::smem_bytes(8))));
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * split + job.blocks));
    cfg.blockDim = dim3(D::kThreads);
    cfg.dynamicSmemBytes = D::Geo<K>::smem_bytes(split);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (dependent) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (split > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)split; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    ESC_CUDA(cudaLaunchKernelEx(&cfg, D::stencil_dense_fp32<T, LAYOUT, K>, static_cast<const T*>(x), static_cast<T*>(out), p.C, p.H, p.W,
                                static_cast<const T*>(w_dense), dk, p.bias, tiles_x, tiles_y, split, job));
    ++g_last_launches;
    return ESC_OK;
}
template <typename T, int LAYOUT>
int launch_dense_fp32_t(const Problem& p, const void* x, const void* w_dense, const float* dk, void* out, cudaStream_t st, bool dependent) {
    switch (p.K) {
        case 3: return launch_dense_fp32_k<T, LAYOUT, 3>(p, x, w_dense, dk, out, st, dependent);
        case 5: return launch_dense_fp32_k<T, LAYOUT, 5>(p, x, w_dense, dk, out, st, dependent);
        case 7: return launch_dense_fp32_k<T, LAYOUT, 7>(p, x, w_dense, dk, out, st, dependent);
        case 9: return launch_dense_fp32_k<T, LAYOUT, 9>(p, x, w_dense, dk, out, st, dependent);
        case 11: return launch_dense_fp32_k<T, LAYOUT, 11>(p, x, w_dense, dk, out, st, dependent);
        case 13: return launch_dense_fp32_k<T, LAYOUT, 13>(p, x, w_dense, dk, out, st, dependent);
        case 15: return launch_dense_fp32_k<T, LAYOUT, 15>(p, x, w_dense, dk, out, st, dependent);
        case 17: return launch_dense_fp32_k<T, LAYOUT, 17>(p, x, w_dense, dk, out, st, dependent);
    }
    return ESC_ERR_UNSUPPORTED;
}

// bf16 NCHW, dense form: the attention channels packed pixel by pixel, the identity planes copied (out may be null: packing only).
int launch_pack16(const Problem& p, const void* x, void* packed, void* out, cudaStream_t st) {
    const long long HW = (long long)p.H * p.W, pixels = (long long)p.B * HW;
    long long blocks = (pixels + esc::dense16::kThreads - 1) / esc::dense16::kThreads;
    if (blocks > 8LL * sms_or_nominal()) blocks = 8LL * sms_or_nominal();
    esc::CopyJob job = {};
    if (out) job = make_copy_job(p, x, out, blocks, esc::dense16::kThreads);
    esc::dense16::pack16<<<(unsigned)(blocks + job.blocks), esc::dense16::kThreads, 0, st>>>(
        static_cast<const __nv_bfloat16*>(x), static_cast<__nv_bfloat16*>(packed), p.C, HW, pixels, (unsigned)blocks, job);
    ESC_CUDA(cudaGetLastError());
    ++g_last_launches;
    return ESC_OK;
}
bool wants_packing(const Problem& p) {
    return p.pack_room && g_dense_engine == 0 && esc::dense16::nchw_wants_packing(p.B, p.Ca, p.H, p.W, p.K, p.dtype, p.layout);
}
// The tcgen05 kernel on a packed map, results into the NCHW tensor `out`.
int launch_umma_packed(const Problem& p, const void* packed, const void* w_dense, const float* dk, void* out, unsigned* ctrl,
                       cudaStream_t st, bool dependent, bool flip) {
    const int rc = esc::tma::umma::try_launch_dense_umma(p.B, esc::dense16::CA, p.Ca, p.H, p.W, p.K, p.dtype, ESC_NHWC, packed, w_dense, dk, out,
                                                         ctrl, st, dependent, &g_last_launches, &g_last_error, p.bias, flip, p.C, true);
    if (rc == ESC_OK) { g_last_path = 5; g_last_tile_w = esc::tma::umma::MW; }
    return rc;
}

// Dense large kernel: a tensor-core kernel where one applies, else the FP32-pipe kernel (16 attention channels) or one thread
// per output (any other channel count).
int launch_stencil_dense(const Problem& p, const void* x, const void* w_dense, const float* dk, void* out,
                         unsigned* ctrl, cudaStream_t st, bool dependent, bool flip = false) {
    // flip: w_dense is read with its channel axes swapped and its taps rotated, which the tcgen05 kernel alone can do
    g_last_tile_w = 0;
    if (g_dense_engine == 0) {
        const int urc = esc::tma::umma::try_launch_dense_umma(p.B, p.C, p.Ca, p.H, p.W, p.K, p.dtype, p.layout, x, w_dense, dk, out,
                                                              ctrl, st, dependent, &g_last_launches, &g_last_error, p.bias, flip);
        if (urc == ESC_OK) { g_last_path = 5; g_last_tile_w = esc::tma::umma::MW; return ESC_OK; }
        if (urc != esc::tma::kNotApplicable) return urc;
    }
    if (flip) return esc::tma::kNotApplicable;
    esc::CopyJob job = make_copy_job(p, x, out, 0, esc::tma::dense::kThreads);
    if (job.blocks > (unsigned)sms_or_nominal()) job.blocks = (unsigned)sms_or_nominal();   // every block of that launch takes a whole SM
    int rc = esc::tma::try_launch_dense(p.B, p.C, p.Ca, p.H, p.W, p.K, p.dtype, p.layout, x, w_dense, dk, out, ctrl,
                                        st, dependent, job, &g_last_launches, &g_last_error);
    if (rc == ESC_OK) {
        g_last_path = 3;
        g_last_tile_w = esc::tma::dense::TW;
        return ESC_OK;                                     // the identity channels went along as copy blocks
    } else if (rc == esc::tma::kNotApplicable) {
        g_last_path = 1;
        if (p.Ca == esc::dense32::CA) {
            if (p.dtype == ESC_F32)
                return p.layout == ESC_NCHW ? launch_dense_fp32_t<float, esc::kNCHW>(p, x, w_dense, dk, out, st, dependent)
                                            : launch_dense_fp32_t<float, esc::kNHWC>(p, x, w_dense, dk, out, st, dependent);
            return p.layout == ESC_NCHW ? launch_dense_fp32_t<__nv_bfloat16, esc::kNCHW>(p, x, w_dense, dk, out, st, dependent)
                                        : launch_dense_fp32_t<__nv_bfloat16, esc::kNHWC>(p, x, w_dense, dk, out, st, dependent);
        }
        if (p.dtype == ESC_F32)
            rc = p.layout == ESC_NCHW ? launch_dense_generic_t<float, esc::kNCHW>(p, x, w_dense, dk, out, st, dependent)
                                      : launch_dense_generic_t<float, esc::kNHWC>(p, x, w_dense, dk, out, st, dependent);
        else
            rc = p.layout == ESC_NCHW ? launch_dense_generic_t<__nv_bfloat16, esc::kNCHW>(p, x, w_dense, dk, out, st, dependent)
                                      : launch_dense_generic_t<__nv_bfloat16, esc::kNHWC>(p, x, w_dense, dk, out, st, dependent);
    }
    if (rc != ESC_OK) return rc;
    return launch_copy(p, x, out, st);
}

int forward_impl(const Problem& p0, const void* x, const void* w_large0, const Estimator& est,
                 void* out, void* ws, cudaStream_t st) {
    const Workspace w = carve(ws, p0.B, p0.Ca, (long long)p0.H * p0.W);
    int rc = clear_counters(w, p0.B, st);
    if (rc != ESC_OK) return rc;
    // what the tensor-core kernels see: a smaller large kernel zero-padded to 13 x 13 (launched first, so that the GAP
    // kernel stays the stencil kernel's immediate predecessor)
    const TensorLk tl = tensor_lk(p0, x, out, w_large0, w.lk_pad, st);
    Problem p = p0;
    p.K = tl.K;
    const void* w_large = tl.w;
    // Small problems on the tensor-core kernel: one launch, stage 1 inside the stencil kernel.
    if (g_fuse_stage1 && tensor_stencil_follows(p)) {
        const esc::tma::toep::Fused fu{est.w_last, est.b_last, est.w_down, est.b_down, est.hidden, w.unit_sums, w.arrivals, w.flags};
        int tw = 0;
        rc = esc::tma::toep::try_launch_fused(p.B, p.C, p.Ca, p.H, p.W, p.K, p.dtype, p.layout, x, w_large, fu, out,
                                              w.ctrl, st, &g_last_launches, &g_last_error, &tw, p.skip_copy, p.w_point);
        if (rc == ESC_OK) { g_last_path = 4; g_last_tile_w = tw; return ESC_OK; }
        if (rc != esc::tma::kNotApplicable) {
            // a cooperative launch can be refused (SMs held by another context): fall back to two kernels
            (void)cudaGetLastError();
            g_last_error.clear();
        }
    }
    if (g_fuse_stage1 && !p.dense && (!p.w_point || p.Ca == esc::tma::CG) && !p.bias && g_engine_policy != ESC_ENGINE_FP32 &&
        g_tile_policy == 0) {
        const esc::tma::toep::Fused fu{est.w_last, est.b_last, est.w_down, est.b_down, est.hidden, w.unit_sums, w.arrivals, w.flags};
        rc = esc::tma::toepn::try_launch_fused(p.B, p.C, p.Ca, p.H, p.W, p.K, p.dtype, p.layout, x, w_large, fu, out, w.ctrl, st,
                                               &g_last_launches, &g_last_error, p.w_point, p.skip_copy);
        if (rc == ESC_OK) { g_last_path = 6; g_last_tile_w = esc::tma::toepn::TW; return ESC_OK; }
        if (rc != esc::tma::kNotApplicable) { (void)cudaGetLastError(); g_last_error.clear(); }
    }
    const bool tensor_nchw = !p.dense && (!p.w_point || p.Ca == esc::tma::CG) && !p.bias && g_engine_policy != ESC_ENGINE_FP32 && g_tile_policy == 0 &&
                             esc::tma::toepn::takes(p.B, p.C, p.Ca, p.H, p.W, p.K, p.dtype, p.layout, x, out);
    const bool packed = p0.dense && wants_packing(p0);
    rc = packed ? launch_pack16(p0, x, w.packed, out, st) : ESC_OK;
    if (rc == ESC_OK) rc = launch_gap(p0, x, est, w, w.dk, st, tensor_stencil_follows(p) || tensor_nchw, dw_umma_follows(p0));
    if (rc != ESC_OK) return rc;
    if (packed) {
        rc = launch_umma_packed(p0, w.packed, w_large0, w.dk, out, w.ctrl, st, /*dependent=*/true, /*flip=*/false);
        if (rc != esc::tma::kNotApplicable) return rc;
    }
    if (p0.dense) return launch_stencil_dense(p0, x, w_large0, w.dk, out, w.ctrl, st, /*dependent=*/true);
    return launch_stencil(p0, x, w_large0, w.dk, out, w.ctrl, st, /*dependent=*/true, &tl);
}

// ---- backward pass -------------------------------------------------------------------------
// Workspace: [ctrl 256 B | per-tile partial tap gradients B*Ca*tiles*kSlot | tap gradients B*Ca*kSlot |
//             rotated LK Ca*169 elements | rotated dk B*Ca*9 | constants B*Ca], each part 256-byte aligned.
struct BackwardWs {
    unsigned* ctrl;
    float *part, *gtap, *dk_flip, *bias;
    esc::bwd::ImageValues iv;        // per image: g_dk [B][9 Ca], means [B][Ca], activations and g_t [B][kMaxHidden]
    void* lk_pad;                    // the rotated large kernel zero-padded to 13 x 13 for the tensor-core kernels
    void* w_flip;
    float *xs_part, *gp_part;        // decomposed form: per-chunk sums of x_att [B][chunks][Ca] and of g_P [B * chunks][Ca * Ca]
    int chunks;                      // chunks of pixels per image in those
    bool mixed;                      // the tap-gradient kernels ran on the mixed features: take the sums of x_att from xs_part
    size_t bytes;
    float* dense_part;               // dense large kernel: the blocks' tap sums [blocks][16][16][169]
    void* wd_flip;                   // the dense kernel with swapped channel axes and rotated taps
    void *x_packed, *go_packed;      // bf16 NCHW tensors: the attention channels of x and grad_out, [B][H][W][16]
    int dense_blocks;
    size_t bytes_dense;              // bytes with the first two behind the rest: what the dense form needs
    size_t bytes_packed;             // bytes with all of them
};
BackwardWs carve_backward(void* ws, const Problem& p) {
    // sized for whichever tiling of the tap-gradient kernels has more tiles (32x32, or 64x16 on the tensor cores)
    const int tiles = std::max(((p.W + esc::bwd::n8::TX - 1) / esc::bwd::n8::TX) * ((p.H + esc::bwd::n8::TY - 1) / esc::bwd::n8::TY),
                               esc::bwd::toep::tiles_of(p.H, p.W));
    BackwardWs w;
    char* base = static_cast<char*>(ws);
    size_t off = 256;
    w.ctrl = reinterpret_cast<unsigned*>(base);
    w.part = reinterpret_cast<float*>(base + off); off += round_up((size_t)p.B * p.Ca * tiles * esc::bwd::kSlot * 4, 256);
    w.gtap = reinterpret_cast<float*>(base + off); off += round_up((size_t)p.B * p.Ca * esc::bwd::kSlot * 4, 256);
    w.w_flip = base + off;                          off += round_up((size_t)p.Ca * esc::bwd::TAPS * 4, 256);
    w.dk_flip = reinterpret_cast<float*>(base + off); off += round_up((size_t)p.B * p.Ca * 9 * 4, 256);
    w.bias = reinterpret_cast<float*>(base + off);  off += round_up((size_t)p.B * p.Ca * 4, 256);
    w.iv.gdk = reinterpret_cast<float*>(base + off);  off += round_up((size_t)p.B * p.Ca * 9 * 4, 256);
    w.iv.mean = reinterpret_cast<float*>(base + off); off += round_up((size_t)p.B * p.Ca * 4, 256);
    w.iv.act = reinterpret_cast<float*>(base + off);  off += round_up((size_t)p.B * esc::kMaxHidden * 4, 256);
    w.iv.gt = reinterpret_cast<float*>(base + off);   off += round_up((size_t)p.B * esc::kMaxHidden * 4, 256);
    w.lk_pad = base + off;                          off += round_up((size_t)p.Ca * esc::bwd::TAPS * 4, 256);
    w.chunks = esc::bwd::pw::chunks_of((long long)p.H * p.W);
    w.mixed = false;
    w.xs_part = reinterpret_cast<float*>(base + off); off += round_up((size_t)p.B * w.chunks * p.Ca * 4, 256);
    w.gp_part = reinterpret_cast<float*>(base + off);
    if (esc::bwd::pw::supported(p.Ca)) off += round_up((size_t)p.B * w.chunks * p.Ca * p.Ca * 4, 256);
    w.bytes = off;
    w.dense_blocks = sms_or_nominal();
    w.dense_part = reinterpret_cast<float*>(base + off); off += round_up((size_t)w.dense_blocks * esc::bwd::dense::kPartFloats * 4, 256);
    w.wd_flip = base + off;                              off += round_up((size_t)esc::bwd::dense::CA * esc::bwd::dense::CA * esc::bwd::TAPS * 4, 256);
    w.bytes_dense = off;
    const size_t pk = round_up(esc::dense16::packed_bytes(p.B, p.Ca, (long long)p.H * p.W, p.K), 256);
    w.x_packed = base + off;  off += pk;
    w.go_packed = base + off; off += pk;
    w.bytes_packed = off;
    return w;
}

// A kernel that may be scheduled while the one before it drains; it waits (griddepcontrol) before it touches memory.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), unsigned grid, int threads, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Weight gradients the caller asked for (fp32, any may be null): of LK, and of the estimator's layers -- last layer
// (W_dyn, b_dyn, or W_up, b_up) and, for the two-layer estimator, W_down, b_down.
struct BackwardGrads {
    float *g_lk, *g_w_last, *g_b_last, *g_w_down, *g_b_down;
};

template <typename T, int LAYOUT>
int backward_t(const Problem& p, const void* x, const void* go, const void* w_large, const Estimator& est,
               const BackwardWs& w, const BackwardGrads& g, cudaStream_t st) {
    // bf16 NHWC with whole groups of 16 channels: the tensor-core kernel (all tap-gradient kernels form the 13 x 13 taps'
    // gradients, whatever the large kernel's size: a smaller one is their middle)
    int tiles_done = 0;
    if (g_engine_policy != ESC_ENGINE_FP32) {
        const int rt = esc::bwd::toep::try_launch(p.B, p.C, p.Ca, p.H, p.W, esc::bwd::K, p.dtype, p.layout, x, go, w.part, w.ctrl, st,
                                                  &g_last_launches, &g_last_error, /*centre_only=*/!g.g_lk);
        if (rt == ESC_OK) tiles_done = esc::bwd::toep::tiles_of(p.H, p.W);
        else if (rt != esc::tma::kNotApplicable) return rt;
        if (tiles_done == 0) {                               // the same on NCHW tensors
            const int rn = esc::bwd::toepn::try_launch(p.B, p.C, p.Ca, p.H, p.W, esc::bwd::K, p.dtype, p.layout, x, go, w.part, w.ctrl, st,
                                                       &g_last_launches, &g_last_error, /*centre_only=*/!g.g_lk);
            if (rn == ESC_OK) tiles_done = esc::bwd::toep::tiles_of(p.H, p.W);
            else if (rn != esc::tma::kNotApplicable) return rn;
        }
    }
    // NHWC with whole octets of channels: eight channels per block, 16-byte loads; else a block per channel
    const bool oct = LAYOUT == esc::kNHWC && p.Ca % 8 == 0 && p.C % 8 == 0;
    const int TXs = oct ? esc::bwd::n8::TX : esc::bwd::TX, TYs = oct ? esc::bwd::n8::TY : esc::bwd::TY;
    const int tiles_x = (p.W + TXs - 1) / TXs, tiles_y = (p.H + TYs - 1) / TYs;
    const long long blocks = (long long)p.B * (oct ? p.Ca / 8 : p.Ca) * tiles_x * tiles_y;
    if (blocks > 0x7fffffffLL) return ESC_ERR_UNSUPPORTED;
    const int ia = g.g_lk ? 0 : esc::bwd::P - 1, ib = g.g_lk ? esc::bwd::K : esc::bwd::P + 2;   // without g_lk only the middle is read
    if (tiles_done > 0) {
        // done above
    } else if (oct) {
        static bool attr_set[esc::tma::kMaxDevices] = {};
        const int dev = esc::tma::current_device();
        if (dev < 0) return ESC_ERR_UNSUPPORTED;
        if (!attr_set[dev]) {
            ESC_CUDA(cudaFuncSetAttribute(esc::bwd::tap_grad_nhwc8<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)esc::bwd::n8::kSmemBytes));
            attr_set[dev] = true;
        }
        const dim3 grid8((unsigned)blocks, (unsigned)esc::bwd::row_shares(blocks, 2, sms_or_nominal()));
        esc::bwd::tap_grad_nhwc8<T><<<grid8, esc::bwd::n8::kThreads, esc::bwd::n8::kSmemBytes, st>>>(
            static_cast<const T*>(x), static_cast<const T*>(go), p.C, p.Ca, p.H, p.W, tiles_x, tiles_y, ia, ib, w.part);
    } else {
        // fewer than two blocks an SM: four times the threads
        if (blocks < 2LL * sms_or_nominal())
            esc::bwd::tap_grad<T, LAYOUT, 4><<<(unsigned)blocks, 4 * esc::bwd::kThreads, 0, st>>>(
                static_cast<const T*>(x), static_cast<const T*>(go), p.C, p.Ca, p.H, p.W, tiles_x, tiles_y, ia, ib, w.part);
        else
            esc::bwd::tap_grad<T, LAYOUT, 1><<<(unsigned)blocks, esc::bwd::kThreads, 0, st>>>(
                static_cast<const T*>(x), static_cast<const T*>(go), p.C, p.Ca, p.H, p.W, tiles_x, tiles_y, ia, ib, w.part);
    }
    ESC_CUDA(cudaGetLastError());
    if (tiles_done == 0) ++g_last_launches;
    // the estimator's part, from the tap gradients; few tiles are added up on the way
    const int tiles = tiles_done > 0 ? tiles_done : tiles_x * tiles_y;
    esc::bwd::Taps taps{w.part, tiles};
    const float* xs_part = w.mixed ? w.xs_part : nullptr;
    if (tiles > esc::bwd::kDirectTiles) {
        ESC_CUDA(launch_pdl(esc::bwd::sum_tiles, (unsigned)(p.B * p.Ca), esc::bwd::kSumThreads, 0, st, w.part, tiles, xs_part, w.chunks, p.Ca,
                            w.gtap));
        ++g_last_launches;
        taps = esc::bwd::Taps{w.gtap, 1};
        xs_part = nullptr;                                   // the sums of x are in their place in gtap
    }
    const int ltaps = p.Ca * p.K * p.K;
    const bool weights = g.g_w_last || g.g_b_last || g.g_w_down || g.g_b_down;
    const int elems = weights ? 9 * p.Ca * (est.hidden > 0 ? est.hidden : p.Ca) + 9 * p.Ca + est.hidden * p.Ca + est.hidden : 0;
    const bool few = esc::bwd::few_images(p.B, p.Ca, est.hidden, p.dense, xs_part != nullptr);
    const size_t smem = (size_t)((p.Ca <= esc::bwd::kEstMaxCa ? 10 * p.Ca : 0) + 2 * est.hidden) * sizeof(float) * (few ? p.B : 1);
    const long long grid = (long long)p.B * (few ? 2 : 1) + (g.g_lk ? (ltaps + 31) / 32 : 0) + (p.dense ? 0 : esc::bwd::kFlipBlocks) +
                           (few ? (elems + esc::bwd::kEstThreads - 1) / esc::bwd::kEstThreads : 0);
    if (grid > 0x7fffffffLL) return ESC_ERR_UNSUPPORTED;
    ESC_CUDA(launch_pdl(few ? esc::bwd::estimator_image<T, true> : esc::bwd::estimator_image<T, false>, (unsigned)grid, esc::bwd::kEstThreads,
                        smem, st, taps, xs_part, w.chunks, p.B, p.Ca, est.hidden, p.H, p.W, p.K,
                        static_cast<const T*>(w_large), static_cast<const T*>(est.w_down), static_cast<const T*>(est.b_down),
                        static_cast<const T*>(est.w_last), static_cast<const T*>(est.b_last), w.iv, w.dk_flip, w.bias, g.g_lk,
                        p.dense ? (T*)nullptr : static_cast<T*>(w.w_flip),
                        esc::bwd::EstimatorGrads{g.g_w_last, g.g_b_last, g.g_w_down, g.g_b_down}));
    ++g_last_launches;
    if (weights && !few) {
        ESC_CUDA(launch_pdl(esc::bwd::estimator_weights, (unsigned)((elems + 31) / 32), esc::bwd::kEstThreads, 0, st, w.iv, p.B, p.Ca,
                            est.hidden, g.g_w_last, g.g_b_last, g.g_w_down, g.g_b_down));
        ++g_last_launches;
    }
    return ESC_OK;
}

// Decomposed form: the two per-pixel kernels around the depth-wise backward pass.
bool pw_vec(const Problem& p) { return p.layout == ESC_NHWC && ((size_t)p.C * p.es()) % 16 == 0 && ((size_t)p.Ca * p.es()) % 16 == 0; }

template <typename T, int LAYOUT, int CA>
int pw_mix_ca(const Problem& p, const void* x, const void* w_point, void* m, const BackwardWs& w, cudaStream_t st) {
    const unsigned blocks = (unsigned)((long long)p.B * w.chunks);
    esc::bwd::pw::mix<T, LAYOUT, CA><<<blocks, esc::bwd::pw::kThreads, 0, st>>>(
        static_cast<const T*>(x), static_cast<const T*>(w_point), static_cast<T*>(m), p.C, (long long)p.H * p.W, w.chunks,
        pw_vec(p) ? 1 : 0, w.xs_part);
    ESC_CUDA(cudaGetLastError());
    ++g_last_launches;
    return ESC_OK;
}
template <typename T, int LAYOUT>
int pw_mix_t(const Problem& p, const void* x, const void* w_point, void* m, const BackwardWs& w, cudaStream_t st) {
    switch (p.Ca) {
        case 4: return pw_mix_ca<T, LAYOUT, 4>(p, x, w_point, m, w, st);
        case 8: return pw_mix_ca<T, LAYOUT, 8>(p, x, w_point, m, w, st);
        case 16: return pw_mix_ca<T, LAYOUT, 16>(p, x, w_point, m, w, st);
        case 32: return pw_mix_ca<T, LAYOUT, 32>(p, x, w_point, m, w, st);
    }
    return ESC_ERR_UNSUPPORTED;
}

template <typename T, int LAYOUT, int CA>
int pw_back_ca(const Problem& p, const void* x, const void* w_point, void* gx, const BackwardWs& w, float* g_wp, cudaStream_t st) {
    constexpr size_t smem = esc::bwd::pw::back_smem_bytes<CA>();
    if (smem > 48 * 1024) {
        static bool attr_set[esc::tma::kMaxDevices] = {};
        const int dev = esc::tma::current_device();
        if (dev < 0) return ESC_ERR_UNSUPPORTED;
        if (!attr_set[dev]) {
            ESC_CUDA(cudaFuncSetAttribute(esc::bwd::pw::back<T, LAYOUT, CA>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            attr_set[dev] = true;
        }
    }
    const unsigned blocks = (unsigned)((long long)p.B * w.chunks);
    esc::bwd::pw::back<T, LAYOUT, CA><<<blocks, esc::bwd::pw::kThreads, smem, st>>>(
        static_cast<const T*>(x), static_cast<const T*>(w_point), static_cast<T*>(gx), w.bias, p.C, (long long)p.H * p.W,
        w.chunks, pw_vec(p) ? 1 : 0, w.gp_part);
    ESC_CUDA(cudaGetLastError());
    ++g_last_launches;
    if (g_wp) {
        const int elems = CA * CA;
        ESC_CUDA(launch_pdl(esc::bwd::pw::sum_gp, (unsigned)((elems + 31) / 32), esc::bwd::pw::kSumGpThreads, 0, st, (const float*)w.gp_part,
                            elems, (int)blocks, g_wp));
        ++g_last_launches;
    }
    return ESC_OK;
}
template <typename T, int LAYOUT>
int pw_back_t(const Problem& p, const void* x, const void* w_point, void* gx, const BackwardWs& w, float* g_wp, cudaStream_t st) {
    switch (p.Ca) {
        case 4: return pw_back_ca<T, LAYOUT, 4>(p, x, w_point, gx, w, g_wp, st);
        case 8: return pw_back_ca<T, LAYOUT, 8>(p, x, w_point, gx, w, g_wp, st);
        case 16: return pw_back_ca<T, LAYOUT, 16>(p, x, w_point, gx, w, g_wp, st);
        case 32: return pw_back_ca<T, LAYOUT, 32>(p, x, w_point, gx, w, g_wp, st);
    }
    return ESC_ERR_UNSUPPORTED;
}

// Dense large kernel: tap gradients of every channel pair.
template <typename T, int LAYOUT>
int dense_tap_grad_t(const Problem& p, const void* x, const void* go, const BackwardWs& w, float* g_wd, cudaStream_t st) {
    namespace D = esc::bwd::dense;
    static bool attr_set[esc::tma::kMaxDevices] = {};
    const int dev = esc::tma::current_device();
    if (dev < 0) return ESC_ERR_UNSUPPORTED;
    if (!attr_set[dev]) {
        ESC_CUDA(cudaFuncSetAttribute(D::tap_grad_dense<T, LAYOUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)D::kSmemBytes));
        attr_set[dev] = true;
    }
    const int tiles_x = (p.W + D::TX - 1) / D::TX, tiles_y = (p.H + D::TY - 1) / D::TY;
    bool g_wd_done = !g_wd;
    if (g_wd && g_engine_policy != ESC_ENGINE_FP32 && g_dense_engine == 0) {
        int blocks = 0;
        const int rc = D::umma::try_launch(p.B, p.C, p.Ca, p.H, p.W, p.dtype, p.layout, x, go, w.dense_part, w.dense_blocks, w.ctrl, st, &blocks,
                                           &g_last_launches, &g_last_error);
        if (rc == ESC_OK) {
            D::umma::sum_dense_umma<<<D::kPartFloats / 32, D::umma::kSumWarps * 32, 0, st>>>(w.dense_part, blocks, p.K, g_wd);
            ESC_CUDA(cudaGetLastError());
            ++g_last_launches;
            g_wd_done = true;
        } else if (rc != esc::tma::kNotApplicable) return rc;
    }
    if (!g_wd_done) {
        if (std::is_same<T, __nv_bfloat16>::value && g_engine_policy != ESC_ENGINE_FP32) {
            // bf16: a matrix product per tap on the tensor cores
            static bool attr_mma[esc::tma::kMaxDevices] = {};
            if (!attr_mma[dev]) {
                ESC_CUDA(cudaFuncSetAttribute(D::mma::tap_grad_dense_bf16<LAYOUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)D::mma::kSmemBytes));
                attr_mma[dev] = true;
            }
            const int vec = LAYOUT == esc::kNHWC && p.C % 8 == 0 ? 1 : 0;
            const int tiles_ym = (p.H + D::mma::TYM - 1) / D::mma::TYM;
            D::mma::tap_grad_dense_bf16<LAYOUT><<<(unsigned)w.dense_blocks, D::mma::kThreads, D::mma::kSmemBytes, st>>>(
                static_cast<const __nv_bfloat16*>(x), static_cast<const __nv_bfloat16*>(go), p.B, p.C, p.H, p.W, tiles_x, tiles_ym, vec,
                w.dense_part);
        } else {
            D::tap_grad_dense<T, LAYOUT><<<(unsigned)w.dense_blocks, D::kThreads, D::kSmemBytes, st>>>(
                static_cast<const T*>(x), static_cast<const T*>(go), p.B, p.C, p.H, p.W, tiles_x, tiles_y, w.dense_part);
        }
        ESC_CUDA(cudaGetLastError());
        const int elems = D::CA * D::CA * p.K * p.K;
        D::sum_dense<<<(unsigned)((elems + 255) / 256), 256, 0, st>>>(w.dense_part, w.dense_blocks, p.K, g_wd);
        ESC_CUDA(cudaGetLastError());
        g_last_launches += 2;
    }
    return ESC_OK;
}
// grad_x of the dense form: the forward's kernels on grad_out with the kernel's channel axes swapped and its taps rotated, plus
// the constants.  The tcgen05 kernel reads the weights that way and adds the constants itself; for the others the rotated
// kernel is written first, and the mma.sync kernel's result gets the constants in a pass of its own.
template <typename T, int LAYOUT>
int dense_grad_x_t(Problem p, const void* go, const void* w_dense, void* gx, const BackwardWs& w, bool packed, cudaStream_t st) {
    namespace D = esc::bwd::dense;
    p.dense = true;
    p.bias = w.bias;
    if (packed) {                                            // go_packed is there, and gx has its identity planes
        const int rp = launch_umma_packed(p, w.go_packed, w_dense, w.dk_flip, gx, w.ctrl, st, /*dependent=*/true, /*flip=*/true);
        if (rp != esc::tma::kNotApplicable) return rp;
    }
    // dependent: grad_out and the weights are older than the estimator's kernels, which alone it has to wait for
    int rc = launch_stencil_dense(p, go, w_dense, w.dk_flip, gx, w.ctrl, st, /*dependent=*/true, /*flip=*/true);
    if (rc != esc::tma::kNotApplicable) return rc;
    const int elems = D::CA * D::CA * p.K * p.K;
    D::flip_dense<T><<<(unsigned)((elems + 255) / 256), 256, 0, st>>>(static_cast<const T*>(w_dense), p.K, static_cast<T*>(w.wd_flip));
    ESC_CUDA(cudaGetLastError());
    ++g_last_launches;
    rc = launch_stencil_dense(p, go, w.wd_flip, w.dk_flip, gx, w.ctrl, st, /*dependent=*/false);
    if (rc != ESC_OK || g_last_path != 3) return rc;
    const long long total = (long long)p.B * p.Ca * p.H * p.W;
    long long blocks = (total + 255) / 256;
    if (blocks > 16LL * sms_or_nominal()) blocks = 16LL * sms_or_nominal();
    D::add_const<T, LAYOUT><<<(unsigned)blocks, 256, 0, st>>>(static_cast<T*>(gx), w.bias, p.B, p.C, p.Ca, (long long)p.H * p.W);
    ESC_CUDA(cudaGetLastError());
    ++g_last_launches;
    return ESC_OK;
}

// ---- Conv_fuse on the FP32 pipe: att | idt are the two parts of its input, kTrans: the matrix is read transposed; first: this
// is the call's first kernel ----
template <typename T, bool kTrans>
int launch_fuse_fp32(const Problem& p, const void* att, const void* idt, const void* w, const void* bias, const void* residual,
                     void* out, cudaStream_t st, bool first = false) {
    esc::fuse::f32::Params<T> fp;
    fp.att = static_cast<const T*>(att); fp.idt = static_cast<const T*>(idt); fp.w = static_cast<const T*>(w);
    fp.bias = static_cast<const T*>(bias); fp.residual = static_cast<const T*>(residual); fp.out = static_cast<T*>(out);
    fp.HW = (long long)p.H * p.W; fp.pixels = fp.HW * p.B; fp.B = p.B; fp.Ca = p.Ca; fp.vec = fp.HW % 4 == 0;
    ESC_CUDA(p.layout == ESC_NCHW ? (esc::fuse::f32::launch<T, esc::kNCHW, kTrans>(p.C, fp, st, first))
                                  : (esc::fuse::f32::launch<T, esc::kNHWC, kTrans>(p.C, fp, st, first)));
    ++g_last_launches;
    return ESC_OK;
}

// ---- backward pass of Conv_fuse -------------------------------------------------------------------------------
struct FuseBackwardWs {
    float* part;                     // [blocks][C * C + C]
    int passes, blocks;              // tensor-core kernels
    int passes32, blocks32;          // wgrad_fp32
    size_t bytes;
};
FuseBackwardWs carve_fuse_backward(void* ws, int C, long long pixels) {
    FuseBackwardWs w;
    // one block per SM at most (both kernels fill an SM), each with a run of pixels long enough to pay for its final sums
    const long long runs = (pixels + esc::fuse::bwd::kThreads - 1) / esc::fuse::bwd::kThreads, cap = sms_or_nominal();
    w.passes = (int)std::max(2LL, (runs + cap - 1) / cap);
    w.blocks = (int)((runs + w.passes - 1) / w.passes);
    // wgrad_fp32: two blocks per SM
    const long long runs32 = (pixels + esc::fuse::f32::kWPx - 1) / esc::fuse::f32::kWPx;
    w.passes32 = (int)std::max(2LL, (runs32 + 2 * cap - 1) / (2 * cap));
    w.blocks32 = (int)((runs32 + w.passes32 - 1) / w.passes32);
    char* base = static_cast<char*>(ws);
    size_t off = 0;
    w.part = reinterpret_cast<float*>(base + off);  off += round_up((size_t)std::max(w.blocks, w.blocks32) * ((size_t)C * C + C) * 4, 256);
    w.bytes = off;
    return w;
}

template <typename T, int LAYOUT, int C>
int fuse_wgrad_c(const void* cat, const void* go, long long HW, long long pixels, const FuseBackwardWs& w, cudaStream_t st) {
    namespace F = esc::fuse::f32;
    static bool attr_set[esc::tma::kMaxDevices] = {};
    const int dev = esc::tma::current_device();
    if (dev < 0) return ESC_ERR_UNSUPPORTED;
    if (!attr_set[dev]) {
        ESC_CUDA(cudaFuncSetAttribute(F::wgrad_fp32<T, LAYOUT, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F::WGeom<C>::kSmemBytes));
        attr_set[dev] = true;
    }
    F::wgrad_fp32<T, LAYOUT, C><<<(unsigned)w.blocks32, F::kWThreads, F::WGeom<C>::kSmemBytes, st>>>(
        static_cast<const T*>(cat), static_cast<const T*>(go), HW, pixels, w.passes32, w.part);
    ESC_CUDA(cudaGetLastError());
    ++g_last_launches;
    return ESC_OK;
}
template <typename T, int LAYOUT>
int fuse_wgrad_t(int C, const void* cat, const void* go, long long HW, long long pixels, const FuseBackwardWs& w, cudaStream_t st) {
    switch (C) {
        case 16: return fuse_wgrad_c<T, LAYOUT, 16>(cat, go, HW, pixels, w, st);
        case 32: return fuse_wgrad_c<T, LAYOUT, 32>(cat, go, HW, pixels, w, st);
        case 48: return fuse_wgrad_c<T, LAYOUT, 48>(cat, go, HW, pixels, w, st);
        case 64: return fuse_wgrad_c<T, LAYOUT, 64>(cat, go, HW, pixels, w, st);
    }
    return ESC_ERR_UNSUPPORTED;
}

// All three gradients in one pass on the tensor cores; `sums`: whether g_W or g_b is wanted.
template <int LAYOUT, int C>
int fuse_backward_mma_c(const void* cat, const void* go, const void* w_fuse, void* g_cat, long long HW, long long pixels,
                        const FuseBackwardWs& w, bool sums, cudaStream_t st) {
    namespace M = esc::fuse::bwd::mma;
    static bool attr_set[esc::tma::kMaxDevices] = {};
    const int dev = esc::tma::current_device();
    if (dev < 0) return ESC_ERR_UNSUPPORTED;
    if (!attr_set[dev]) {
        ESC_CUDA(cudaFuncSetAttribute(M::fuse_backward_bf16<LAYOUT, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)M::MGeom<LAYOUT, C>::kSmemBytes));
        attr_set[dev] = true;
    }
    M::fuse_backward_bf16<LAYOUT, C><<<(unsigned)w.blocks, esc::fuse::bwd::kThreads, M::MGeom<LAYOUT, C>::kSmemBytes, st>>>(
        static_cast<const __nv_bfloat16*>(cat), static_cast<const __nv_bfloat16*>(go), static_cast<const __nv_bfloat16*>(w_fuse),
        static_cast<__nv_bfloat16*>(g_cat), HW, pixels, w.passes, sums ? w.part : nullptr);
    ESC_CUDA(cudaGetLastError());
    ++g_last_launches;
    return ESC_OK;
}
template <int LAYOUT>
int fuse_backward_mma_t(int C, const void* cat, const void* go, const void* w_fuse, void* g_cat, long long HW, long long pixels,
                        const FuseBackwardWs& w, bool sums, cudaStream_t st) {
    switch (C) {
        case 32: return fuse_backward_mma_c<LAYOUT, 32>(cat, go, w_fuse, g_cat, HW, pixels, w, sums, st);
        case 48: return fuse_backward_mma_c<LAYOUT, 48>(cat, go, w_fuse, g_cat, HW, pixels, w, sums, st);
        case 64: return fuse_backward_mma_c<LAYOUT, 64>(cat, go, w_fuse, g_cat, HW, pixels, w, sums, st);
    }
    return ESC_ERR_UNSUPPORTED;
}

// ---- the bounded waits, run on purpose ----------------------------------------------------------------------
// One thread waits, with the kernels' own bounded waits, for a count that nothing raises and then on a barrier that nothing
// signals: each gives up after its poll limit (about a second) and records the status, and the kernel returns normally.  The first
// one's record is checked here: without it the second wait, whose record the host reads, is left out.
__global__ void bounded_wait_probe(unsigned* ctrl) {
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int count;
    __shared__ unsigned status[2];
    if (threadIdx.x == 0) {
        count = 2;
        status[0] = status[1] = 0;
        const bool enough = esc::tma::umma::wait_count(&count, 2, status, 0u) && status[0] == 0;
        const bool gave_up = !esc::tma::umma::wait_count(&count, 3, status, 0x5E1F0001u) && status[0] == esc::kDevTimeout && status[1] == 0x5E1F0001u;
        if (!enough || !gave_up) return;
        const uint32_t b = esc::tma::smem_u32(&bar);
        esc::tma::mbar_init(b, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        esc::tma::mbar_wait(b, 0, ctrl, 0x5E1F0000u);
    }
}

// ---- fixed scratch for the entry point that must not allocate ------------------------------
// Layout: [kStaticMaxImages arrival counters][kStaticMaxPartials partial sums].  The array lives in
// the library's device image: every GPU that loads the library holds these 64 KiB until exit.
constexpr int kStaticMaxImages = 1024;
constexpr int kStaticMaxPartials = 15360;
static __device__ __align__(256) unsigned g_static_scratch[kStaticMaxImages + kStaticMaxPartials];
constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
unsigned* g_static_addr[kMaxDevices] = {};   // device address of g_static_scratch, per device

// In host code `g_static_scratch` is only a handle; the address a kernel can use has to be asked
// for, once per device, with that device current.
int static_scratch_address(unsigned** out) {
    int dev = 0;
    ESC_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return ESC_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_addr[dev]) {
        void* ptr = nullptr;
        ESC_CUDA(cudaGetSymbolAddress(&ptr, g_static_scratch));
        g_static_addr[dev] = static_cast<unsigned*>(ptr);
    }
    *out = g_static_addr[dev];
    return ESC_OK;
}

// ---- host-buffer path ---------------------------------------------------------------------
struct HostPath {
    int dev = -1;
    cudaStream_t st = nullptr, compute = nullptr, down = nullptr;   // st: uploads, and the order of the slot's calls
    cudaEvent_t ev = nullptr;
    void *x = nullptr, *out = nullptr, *wts = nullptr, *ws = nullptr;
    size_t xbytes = 0, wbytes = 0, wsbytes = 0;
};
// NCHW keeps the identity channels of an image in one contiguous piece, which neither kernel needs: in a call that waits for its result
// they are uploaded behind the attention channels and go back, piece by piece, while the next piece comes in and the kernels run.
// (NHWC interleaves them with the attention channels pixel by pixel; strided copies of the two parts take longer than the overlap
// gains: 96 of every 128 bytes 0.60 ms and 32 of 128 0.44 ms against 0.52 ms for the whole map of 640x360x64 bf16.)
// Pieces of 4 MB, about 80 us each: part of an image, or several images as rows of one 2D copy.  From 1 MB of identity channels on, and
// 16 KB of them an image: shorter rows lose more than the overlap gains.  Blocking call, whole map up and down / overlapped, bf16:
// 640x360x64 1110 -> 870 us (1 MB pieces 1330), 320x180x64 315 -> 272; 64 x (64x64x64) 1260 -> 940 (a piece per image: 1390),
// 40 x (48x48x48) 369 -> 310, 800 x (16x16x64) 1100 -> 900, 800 x (16x16x24), rows of 4 KB, 527 -> 573; fp32 640x360x64 2210 -> 1570.
// Not between submit and wait: there the other slot's step fills both directions of the link, and pieces only add copies (640x360x64
// bf16, two slots 687 -> 780, 64 x (64x64x64) 775 -> 1335); nor for pageable buffers, whose copies hold up the submitting thread.
constexpr size_t kHostOverlapBytes = 1 << 20, kHostChunkBytes = 4 << 20, kHostMinRow = 16 << 10;
constexpr size_t kHostMaxPitch = 0x7fffffff;               // of a 2D copy
constexpr int kHostSlots = 2;
std::mutex g_host_mu;
HostPath g_host[kHostSlots];

// Whether parts of `out` may travel while parts of `x` are still to come: both pinned, and not the same memory.
bool host_buffers_allow(const void* x, const void* out, size_t bytes) {
    const char *a = static_cast<const char*>(x), *b = static_cast<const char*>(out);
    if (a < b + bytes && b < a + bytes) return false;
    for (const void* q : {x, out}) {
        cudaPointerAttributes at;
        if (cudaPointerGetAttributes(&at, q) != cudaSuccess) { (void)cudaGetLastError(); return false; }
        if (at.type != cudaMemoryTypeHost) return false;
    }
    return true;
}

}  // namespace

extern "C" {

int esc_version(void) { return 120; }

const char* esc_last_error(void) { return g_last_error.c_str(); }

int esc_convattn_last_path(void) { return g_last_path; }
int esc_convattn_last_tile_width(void) { return g_last_tile_w; }
int esc_convattn_set_tile_width(int tile_width) {
    if (tile_width != 0 && tile_width != esc::tma::Geom40::TW && tile_width != esc::tma::Geom64::TW) return ESC_ERR_UNSUPPORTED;
    g_tile_policy = tile_width;
    return ESC_OK;
}
int esc_convattn_set_stencil_engine(int engine) {
    if (engine != ESC_ENGINE_AUTO && engine != ESC_ENGINE_FP32 && engine != ESC_ENGINE_TENSOR) return ESC_ERR_UNSUPPORTED;
    g_engine_policy = engine;
    return ESC_OK;
}
int esc_convattn_set_dense_engine(int engine) {
    if (engine != 0 && engine != 1) return ESC_ERR_UNSUPPORTED;
    g_dense_engine = engine;
    return ESC_OK;
}
int esc_convattn_set_fused_stage1(int on) {
    g_fuse_stage1 = on != 0;
    return ESC_OK;
}
int esc_convattn_last_launches(void) { return g_last_launches; }

const char* esc_status_string(int s) {
    switch (s) {
        case ESC_OK: return "ok";
        case ESC_ERR_NULL: return "null pointer";
        case ESC_ERR_SHAPE: return "invalid shape";
        case ESC_ERR_UNSUPPORTED: return "unsupported configuration";
        case ESC_ERR_ALIGN: return "misaligned pointer";
        case ESC_ERR_ALIAS: return "out overlaps x";
        case ESC_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
        case ESC_ERR_CUDA: return "CUDA error";
        case ESC_DEV_TIMEOUT: return "device-side wait timed out";
        default: return "unknown status";
    }
}

size_t esc_convattn_workspace_bytes(int B, int C_a, int H, int W, int K) {
    if (B <= 0 || C_a <= 0 || H <= 0 || W <= 0 || K < 3 || (K & 1) == 0 || K > ESC_MAX_K) return 0;
    return workspace_bytes_packed(B, C_a, (long long)H * W, K);
}

int esc_convattn_workspace_init(void* workspace, size_t workspace_bytes_, void* stream) {
    if (!workspace || !aligned(workspace, 256) || workspace_bytes_ < 256) return ESC_ERR_WORKSPACE;
    ESC_CUDA(cudaMemsetAsync(workspace, 0, workspace_bytes_, static_cast<cudaStream_t>(stream)));
    return ESC_OK;
}

int esc_convattn_forward_ex(const void* x, int B, int C, int C_a, int H, int W, int K, const void* w_large,
                            const void* w_dyn, const void* b_dyn, void* out, int dtype, int layout,
                            void* workspace, size_t workspace_bytes_, void* stream) {
    g_last_launches = 0;
    const Problem p{B, C, C_a, H, W, K, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!w_large || !w_dyn || !b_dyn) return ESC_ERR_NULL;
    rc = check_tensors(p, x, out);
    if (rc != ESC_OK) return rc;
    if (!aligned(w_large, p.es()) || !aligned(w_dyn, p.es()) || !aligned(b_dyn, p.es())) return ESC_ERR_ALIGN;
    rc = check_workspace(p, workspace, workspace_bytes_);
    if (rc != ESC_OK) return rc;
    return forward_impl(p, x, w_large, Estimator{w_dyn, b_dyn, nullptr, nullptr, 0}, out, workspace,
                        static_cast<cudaStream_t>(stream));
}

int esc_convattn_forward(const void* x, int B, int C, int C_a, int H, int W, int K, const void* w_large,
                         const void* w_dyn, const void* b_dyn, void* out, void* stream) {
    g_last_launches = 0;
    const Problem p{B, C, C_a, H, W, K, ESC_F32, ESC_NCHW};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!w_large || !w_dyn || !b_dyn) return ESC_ERR_NULL;
    rc = check_tensors(p, x, out);
    if (rc != ESC_OK) return rc;
    if (!aligned(w_large, 4) || !aligned(w_dyn, 4) || !aligned(b_dyn, 4)) return ESC_ERR_ALIGN;
    void* ws = nullptr;
    rc = get_scratch(workspace_bytes(B, C_a, (long long)H * W), static_cast<cudaStream_t>(stream), &ws);
    if (rc != ESC_OK) return rc;
    return forward_impl(p, x, w_large, Estimator{w_dyn, b_dyn, nullptr, nullptr, 0}, out, ws, static_cast<cudaStream_t>(stream));
}

int esc_convattn_dynkernel(const void* x, int B, int C, int C_a, int H, int W, const void* w_dyn,
                           const void* b_dyn, float* dk_out, int dtype, int layout, void* workspace,
                           size_t workspace_bytes_, void* stream) {
    g_last_launches = 0;
    const Problem p{B, C, C_a, H, W, 3, dtype, layout};   // stage 1 has no large kernel: any valid K
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!x || !w_dyn || !b_dyn || !dk_out) return ESC_ERR_NULL;
    if (!aligned(x, 16) || !aligned(dk_out, 4) || !aligned(w_dyn, p.es()) || !aligned(b_dyn, p.es())) return ESC_ERR_ALIGN;
    rc = check_workspace(p, workspace, workspace_bytes_);
    if (rc != ESC_OK) return rc;
    const Workspace w = carve(workspace, B, C_a, (long long)H * W);
    rc = clear_counters(w, B, static_cast<cudaStream_t>(stream));
    if (rc != ESC_OK) return rc;
    return launch_gap(p, x, Estimator{w_dyn, b_dyn, nullptr, nullptr, 0}, w, dk_out, static_cast<cudaStream_t>(stream));
}

int esc_convattn_forward_mlp(const void* x, int B, int C, int C_a, int H, int W, int K, const void* w_large,
                             const void* w_down, const void* b_down, const void* w_up, const void* b_up, int hidden,
                             void* out, int dtype, int layout, void* workspace, size_t workspace_bytes_,
                             void* stream) {
    g_last_launches = 0;
    const Problem p{B, C, C_a, H, W, K, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (hidden < 1) return ESC_ERR_SHAPE;
    if (!w_large) return ESC_ERR_NULL;
    const Estimator est{w_up, b_up, w_down, b_down, hidden};
    rc = check_estimator(p, est);
    if (rc != ESC_OK) return rc;
    rc = check_tensors(p, x, out);
    if (rc != ESC_OK) return rc;
    if (!aligned(w_large, p.es())) return ESC_ERR_ALIGN;
    rc = check_workspace(p, workspace, workspace_bytes_);
    if (rc != ESC_OK) return rc;
    return forward_impl(p, x, w_large, est, out, workspace, static_cast<cudaStream_t>(stream));
}

int esc_convattn_dynkernel_mlp(const void* x, int B, int C, int C_a, int H, int W, const void* w_down,
                               const void* b_down, const void* w_up, const void* b_up, int hidden, float* dk_out,
                               int dtype, int layout, void* workspace, size_t workspace_bytes_, void* stream) {
    g_last_launches = 0;
    const Problem p{B, C, C_a, H, W, 3, dtype, layout};   // stage 1 has no large kernel: any valid K
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (hidden < 1) return ESC_ERR_SHAPE;
    if (!x || !dk_out) return ESC_ERR_NULL;
    const Estimator est{w_up, b_up, w_down, b_down, hidden};
    rc = check_estimator(p, est);
    if (rc != ESC_OK) return rc;
    if (!aligned(x, 16) || !aligned(dk_out, 4)) return ESC_ERR_ALIGN;
    rc = check_workspace(p, workspace, workspace_bytes_);
    if (rc != ESC_OK) return rc;
    const Workspace w = carve(workspace, B, C_a, (long long)H * W);
    rc = clear_counters(w, B, static_cast<cudaStream_t>(stream));
    if (rc != ESC_OK) return rc;
    return launch_gap(p, x, est, w, dk_out, static_cast<cudaStream_t>(stream));
}

int esc_convattn_dynkernel_static(const void* x, int B, int C, int C_a, int H, int W, const void* w_dyn,
                                  const void* b_dyn, float* dk_out, int dtype, int layout, void* stream) {
    g_last_launches = 0;
    const Problem p{B, C, C_a, H, W, 3, dtype, layout};   // stage 1 has no large kernel: any valid K
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!x || !w_dyn || !b_dyn || !dk_out) return ESC_ERR_NULL;
    if (!aligned(x, 16) || !aligned(dk_out, 4) || !aligned(w_dyn, p.es()) || !aligned(b_dyn, p.es())) return ESC_ERR_ALIGN;
    const int S = slabs_for(B, (long long)H * W, gap_grid(B, C_a, (long long)H * W, false, false) != GapGrid::Narrow);
    if (B > kStaticMaxImages || (long long)B * S * C_a > kStaticMaxPartials) {
        char buf[200];
        snprintf(buf, sizeof buf,
                 "esc_convattn_dynkernel_static: needs %d counters and %lld partial sums, the fixed scratch holds %d and %d",
                 B, (long long)B * S * C_a, kStaticMaxImages, kStaticMaxPartials);
        g_last_error = buf;
        return ESC_ERR_WORKSPACE;
    }
    unsigned* base = nullptr;
    rc = static_scratch_address(&base);
    if (rc != ESC_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // The counters must be zero when the kernel starts; a call that was cut short could have left them
    // otherwise, and the array is shared by every caller in the process.
    ESC_CUDA(cudaMemsetAsync(base, 0, (size_t)B * sizeof(unsigned), st));
    Workspace w;
    w.ctrl = nullptr;
    w.arrivals = base;
    w.dk = dk_out;
    w.partial = reinterpret_cast<float*>(base + kStaticMaxImages);
    return launch_gap(p, x, Estimator{w_dyn, b_dyn, nullptr, nullptr, 0}, w, dk_out, st);
}

int esc_convattn_stencil(const void* x, int B, int C, int C_a, int H, int W, int K, const void* w_large,
                         const float* dk, void* out, int dtype, int layout, void* workspace,
                         size_t workspace_bytes_, void* stream) {
    g_last_launches = 0;
    const Problem p{B, C, C_a, H, W, K, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!w_large || !dk) return ESC_ERR_NULL;
    rc = check_tensors(p, x, out);
    if (rc != ESC_OK) return rc;
    if (!aligned(w_large, p.es()) || !aligned(dk, 4)) return ESC_ERR_ALIGN;
    unsigned* ctrl = nullptr;
    void* pad = nullptr;
    if (workspace) {
        rc = check_workspace(p, workspace, workspace_bytes_);
        if (rc != ESC_OK) return rc;
        const Workspace w = carve(workspace, B, C_a, (long long)H * W);
        ctrl = w.ctrl; pad = w.lk_pad;
    }
    const TensorLk tl = tensor_lk(p, x, out, w_large, pad, static_cast<cudaStream_t>(stream));
    return launch_stencil(p, x, w_large, dk, out, ctrl, static_cast<cudaStream_t>(stream), /*dependent=*/false, &tl);
}

int esc_convattn_stencil_pw(const void* x, int B, int C, int C_a, int H, int W, int K, const void* w_large,
                            const void* w_point, const float* dk, void* out, int dtype, int layout, void* workspace,
                            size_t workspace_bytes_, void* stream) {
    g_last_launches = 0;
    Problem p{B, C, C_a, H, W, K, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!w_large || !w_point || !dk) return ESC_ERR_NULL;
    rc = check_tensors(p, x, out);
    if (rc != ESC_OK) return rc;
    if (!aligned(w_large, p.es()) || !aligned(w_point, p.es()) || !aligned(dk, 4)) return ESC_ERR_ALIGN;
    p.w_point = w_point;
    unsigned* ctrl = nullptr;
    void* pad = nullptr;
    if (workspace) {
        rc = check_workspace(p, workspace, workspace_bytes_);
        if (rc != ESC_OK) return rc;
        const Workspace w = carve(workspace, B, C_a, (long long)H * W);
        ctrl = w.ctrl; pad = w.lk_pad;
    }
    const TensorLk tl = tensor_lk(p, x, out, w_large, pad, static_cast<cudaStream_t>(stream));
    return launch_stencil(p, x, w_large, dk, out, ctrl, static_cast<cudaStream_t>(stream), /*dependent=*/false, &tl);
}

int esc_convattn_forward_pw(const void* x, int B, int C, int C_a, int H, int W, int K, const void* w_large,
                            const void* w_point, const void* w_dyn, const void* b_dyn, void* out, int dtype,
                            int layout, void* workspace, size_t workspace_bytes_, void* stream) {
    g_last_launches = 0;
    Problem p{B, C, C_a, H, W, K, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!w_large || !w_point || !w_dyn || !b_dyn) return ESC_ERR_NULL;
    rc = check_tensors(p, x, out);
    if (rc != ESC_OK) return rc;
    if (!aligned(w_large, p.es()) || !aligned(w_point, p.es()) || !aligned(w_dyn, p.es()) || !aligned(b_dyn, p.es()))
        return ESC_ERR_ALIGN;
    rc = check_workspace(p, workspace, workspace_bytes_);
    if (rc != ESC_OK) return rc;
    p.w_point = w_point;
    return forward_impl(p, x, w_large, Estimator{w_dyn, b_dyn, nullptr, nullptr, 0}, out, workspace,
                        static_cast<cudaStream_t>(stream));
}

int esc_convattn_stencil_dense(const void* x, int B, int C, int C_a, int H, int W, int K, const void* w_dense,
                               const float* dk, void* out, int dtype, int layout, void* workspace,
                               size_t workspace_bytes_, void* stream) {
    g_last_launches = 0;
    Problem p{B, C, C_a, H, W, K, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!w_dense || !dk) return ESC_ERR_NULL;
    rc = check_tensors(p, x, out);
    if (rc != ESC_OK) return rc;
    if (!aligned(w_dense, p.es()) || !aligned(dk, 4)) return ESC_ERR_ALIGN;
    p.dense = true;
    unsigned* ctrl = nullptr;
    if (workspace) {
        rc = check_workspace(p, workspace, workspace_bytes_);
        if (rc != ESC_OK) return rc;
        const Workspace w = carve(workspace, B, C_a, (long long)H * W);
        ctrl = w.ctrl;
        p.pack_room = workspace_bytes_ >= workspace_bytes_packed(B, C_a, (long long)H * W, K);
        if (wants_packing(p)) {
            cudaStream_t st = static_cast<cudaStream_t>(stream);
            rc = launch_pack16(p, x, w.packed, out, st);
            if (rc == ESC_OK) rc = launch_umma_packed(p, w.packed, w_dense, dk, out, ctrl, st, /*dependent=*/false, /*flip=*/false);
            if (rc != esc::tma::kNotApplicable) return rc;
        }
    }
    return launch_stencil_dense(p, x, w_dense, dk, out, ctrl, static_cast<cudaStream_t>(stream), /*dependent=*/false);
}

int esc_convattn_forward_dense(const void* x, int B, int C, int C_a, int H, int W, int K, const void* w_dense,
                               const void* w_dyn, const void* b_dyn, void* out, int dtype, int layout,
                               void* workspace, size_t workspace_bytes_, void* stream) {
    g_last_launches = 0;
    Problem p{B, C, C_a, H, W, K, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!w_dense || !w_dyn || !b_dyn) return ESC_ERR_NULL;
    rc = check_tensors(p, x, out);
    if (rc != ESC_OK) return rc;
    if (!aligned(w_dense, p.es()) || !aligned(w_dyn, p.es()) || !aligned(b_dyn, p.es())) return ESC_ERR_ALIGN;
    rc = check_workspace(p, workspace, workspace_bytes_);
    if (rc != ESC_OK) return rc;
    p.dense = true;
    p.pack_room = workspace_bytes_ >= workspace_bytes_packed(B, C_a, (long long)H * W, K);
    return forward_impl(p, x, w_dense, Estimator{w_dyn, b_dyn, nullptr, nullptr, 0}, out, workspace,
                        static_cast<cudaStream_t>(stream));
}

int esc_convattn_forward_variant(const void* x, int B, int C, int C_a, int H, int W, int K, int large_kernel,
                                 const void* w_large, const void* w_point, const void* w_down, const void* b_down,
                                 const void* w_up, const void* b_up, int hidden, void* out, int dtype, int layout,
                                 void* workspace, size_t workspace_bytes_, void* stream) {
    g_last_launches = 0;
    Problem p{B, C, C_a, H, W, K, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (large_kernel != ESC_LK_DEPTHWISE && large_kernel != ESC_LK_DECOMPOSED && large_kernel != ESC_LK_DENSE)
        return ESC_ERR_UNSUPPORTED;
    if (hidden < 0) return ESC_ERR_SHAPE;
    if (!w_large || (large_kernel == ESC_LK_DECOMPOSED && !w_point)) return ESC_ERR_NULL;
    const Estimator est{w_up, b_up, hidden > 0 ? w_down : nullptr, hidden > 0 ? b_down : nullptr, hidden};
    rc = check_estimator(p, est);
    if (rc != ESC_OK) return rc;
    rc = check_tensors(p, x, out);
    if (rc != ESC_OK) return rc;
    if (!aligned(w_large, p.es()) || (large_kernel == ESC_LK_DECOMPOSED && !aligned(w_point, p.es()))) return ESC_ERR_ALIGN;
    rc = check_workspace(p, workspace, workspace_bytes_);
    if (rc != ESC_OK) return rc;
    if (large_kernel == ESC_LK_DECOMPOSED) p.w_point = w_point;
    p.dense = large_kernel == ESC_LK_DENSE;
    p.pack_room = workspace_bytes_ >= workspace_bytes_packed(B, C_a, (long long)H * W, K);
    return forward_impl(p, x, w_large, est, out, workspace, static_cast<cudaStream_t>(stream));
}

int esc_convattn_forward_fused(const void* x, int B, int C, int C_a, int H, int W, int K, const void* w_large,
                               const void* w_dyn, const void* b_dyn, const void* w_fuse, const void* b_fuse,
                               const void* residual, void* out, int dtype, int layout, void* workspace,
                               size_t workspace_bytes_, void* stream) {
    g_last_launches = 0;
    Problem p{B, C, C_a, H, W, K, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!w_large || !w_dyn || !b_dyn || !w_fuse) return ESC_ERR_NULL;
    rc = check_tensors(p, x, out);
    if (rc != ESC_OK) return rc;
    if (!aligned(w_large, p.es()) || !aligned(w_dyn, p.es()) || !aligned(b_dyn, p.es()) || !aligned(w_fuse, p.es()) ||
        (b_fuse && !aligned(b_fuse, p.es())))
        return ESC_ERR_ALIGN;
    if (residual) {
        if (!aligned(residual, 16)) return ESC_ERR_ALIGN;
        const uintptr_t ra = reinterpret_cast<uintptr_t>(residual), oa = reinterpret_cast<uintptr_t>(out);
        const size_t bytes = p.elems() * p.es();
        if (ra < oa + bytes && oa < ra + bytes) return ESC_ERR_ALIAS;        // out is rewritten pixel block by pixel block
    }
    rc = check_workspace(p, workspace, workspace_bytes_);
    if (rc != ESC_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const Estimator est{w_dyn, b_dyn, nullptr, nullptr, 0};
    const long long pixels = (long long)B * H * W;
    // Fast path: the tensor-core stencil writes only the attention channels; the 1x1 kernel takes the identity
    // channels straight from x, so they are never copied.
    if (esc::fuse::fast_applies(C, C_a, dtype, layout) && aligned(w_fuse, 16) && tensor_stencil_follows(p)) {
        p.skip_copy = true;
        rc = forward_impl(p, x, w_large, est, out, workspace, st);
        if (rc != ESC_OK) return rc;
        esc::fuse::Params fp;
        fp.att = static_cast<const __nv_bfloat16*>(out); fp.idt = static_cast<const __nv_bfloat16*>(x);
        fp.w = static_cast<const __nv_bfloat16*>(w_fuse); fp.bias = static_cast<const __nv_bfloat16*>(b_fuse);
        fp.residual = static_cast<const __nv_bfloat16*>(residual); fp.out = static_cast<__nv_bfloat16*>(out);
        fp.pixels = pixels; fp.C = C; fp.Ca = C_a;
        ESC_CUDA(esc::fuse::launch_fast(fp, st));
        ++g_last_launches;
        return ESC_OK;
    }
    // The same on NCHW tensors: the NCHW tensor-core stencil without its copy of the identity planes, then the NCHW 1x1 kernel.
    if (K == esc::tma::K13 && g_engine_policy != ESC_ENGINE_FP32 && g_tile_policy == 0 &&
        esc::fuse::nchw::applies(C, C_a, (long long)H * W, dtype, layout, x, out, residual, w_fuse) &&
        esc::tma::toepn::takes(B, C, C_a, H, W, K, dtype, layout, x, out)) {
        p.skip_copy = true;
        rc = forward_impl(p, x, w_large, est, out, workspace, st);
        if (rc != ESC_OK) return rc;
        esc::fuse::nchw::Params fp;
        fp.att = static_cast<const __nv_bfloat16*>(out); fp.idt = static_cast<const __nv_bfloat16*>(x);
        fp.w = static_cast<const __nv_bfloat16*>(w_fuse); fp.bias = static_cast<const __nv_bfloat16*>(b_fuse);
        fp.residual = static_cast<const __nv_bfloat16*>(residual); fp.out = static_cast<__nv_bfloat16*>(out);
        fp.HW = (long long)H * W; fp.B = B; fp.C = C; fp.Ca = C_a;
        ESC_CUDA(esc::fuse::nchw::launch(fp, st));
        ++g_last_launches;
        return ESC_OK;
    }
    if (esc::fuse::f32::supported(C)) {
        // The FP32-pipe 1x1 kernel.  For fp32 the identity channels are read from x and never copied; a bf16 forward may run on a
        // kernel that always copies them, so there the whole concatenated map is in out.
        p.skip_copy = dtype == ESC_F32;
        rc = forward_impl(p, x, w_large, est, out, workspace, st);
        if (rc != ESC_OK) return rc;
        return dtype == ESC_F32 ? launch_fuse_fp32<float, false>(p, out, x, w_fuse, b_fuse, residual, out, st)
                                : launch_fuse_fp32<__nv_bfloat16, false>(p, out, out, w_fuse, b_fuse, residual, out, st);
    }
    rc = forward_impl(p, x, w_large, est, out, workspace, st);
    if (rc != ESC_OK) return rc;
    const size_t smem = (size_t)esc::fuse::kGenPix * C * sizeof(float);
    if (smem > 48 * 1024) return ESC_ERR_UNSUPPORTED;
    const unsigned blocks = (unsigned)((pixels + esc::fuse::kGenPix - 1) / esc::fuse::kGenPix);
#define ESC_FUSE_GENERIC(T, L) esc::fuse::conv_fuse_generic<T, L><<<blocks, esc::fuse::kGenThreads, smem, st>>>( \
        static_cast<T*>(out), static_cast<const T*>(w_fuse), static_cast<const T*>(b_fuse), static_cast<const T*>(residual), B, C, H, W)
    if (dtype == ESC_F32) { if (layout == ESC_NCHW) ESC_FUSE_GENERIC(float, esc::kNCHW); else ESC_FUSE_GENERIC(float, esc::kNHWC); }
    else { if (layout == ESC_NCHW) ESC_FUSE_GENERIC(__nv_bfloat16, esc::kNCHW); else ESC_FUSE_GENERIC(__nv_bfloat16, esc::kNHWC); }
#undef ESC_FUSE_GENERIC
    ESC_CUDA(cudaGetLastError());
    ++g_last_launches;
    return ESC_OK;
}

size_t esc_convattn_backward_workspace_bytes(int B, int C_a, int H, int W, int K) {
    if (B <= 0 || C_a <= 0 || H <= 0 || W <= 0 || K < 3 || K > esc::bwd::K || (K & 1) == 0) return 0;
    const Problem p{B, C_a, C_a, H, W, K, ESC_F32, ESC_NCHW};
    return carve_backward(nullptr, p).bytes;
}

namespace {
int backward_entry(const void* x, const void* grad_out, int B, int C, int C_a, int H, int W, int K, const void* w_large,
                   const Estimator& est, void* grad_x, const BackwardGrads& g, int dtype, int layout, void* workspace,
                   size_t workspace_bytes_, void* stream, const void* w_point = nullptr, float* g_wp = nullptr,
                   bool dense = false, float* g_wd = nullptr) {
    g_last_launches = 0;
    Problem p{B, C, C_a, H, W, K, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (K > esc::bwd::K) return ESC_ERR_UNSUPPORTED;         // the tap-gradient kernels hold 13 x 13 taps; a smaller LK is their middle
    if ((long long)B * C_a > 0x7fffffffLL / esc::bwd::kSlot) return ESC_ERR_UNSUPPORTED;
    if (!x || !grad_out || !grad_x || !w_large) return ESC_ERR_NULL;
    rc = check_estimator(p, est);
    if (rc != ESC_OK) return rc;
    rc = check_tensors(p, grad_out, grad_x);                 // the stencil pass reads grad_out and writes grad_x
    if (rc != ESC_OK) return rc;
    if (!aligned(x, 16)) return ESC_ERR_ALIGN;
    {
        const uintptr_t xa = reinterpret_cast<uintptr_t>(x), oa = reinterpret_cast<uintptr_t>(grad_x);
        const size_t bytes = p.elems() * p.es();
        if (xa < oa + bytes && oa < xa + bytes) return ESC_ERR_ALIAS;
    }
    if (!aligned(w_large, p.es())) return ESC_ERR_ALIGN;
    for (const float* q : {g.g_lk, g.g_w_last, g.g_b_last, g.g_w_down, g.g_b_down, g_wp})
        if (q && !aligned(q, 4)) return ESC_ERR_ALIGN;
    if (w_point) {
        if (!aligned(w_point, p.es())) return ESC_ERR_ALIGN;
        if (!esc::bwd::pw::supported(C_a)) return ESC_ERR_UNSUPPORTED;
        if ((long long)B * esc::bwd::pw::chunks_of((long long)H * W) > 0x7fffffffLL) return ESC_ERR_UNSUPPORTED;
    }
    if (!workspace || !aligned(workspace, 256)) return ESC_ERR_WORKSPACE;
    if (dense && (C_a != esc::bwd::dense::CA || w_point)) return ESC_ERR_UNSUPPORTED;
    if (g_wd && !aligned(g_wd, 4)) return ESC_ERR_ALIGN;
    BackwardWs w = carve_backward(workspace, p);
    if (workspace_bytes_ < (dense ? w.bytes_dense : w.bytes)) return ESC_ERR_WORKSPACE;
    p.pack_room = dense && workspace_bytes_ >= w.bytes_packed;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (w_point) {
        // decomposed form (Eq. 5): the mixed features go into grad_x's attention channels, where the tap-gradient kernels
        // read them; grad_x is rewritten by the stencil pass and the last kernel below
        rc = dtype == ESC_F32 ? (layout == ESC_NCHW ? pw_mix_t<float, esc::kNCHW>(p, x, w_point, grad_x, w, st)
                                                    : pw_mix_t<float, esc::kNHWC>(p, x, w_point, grad_x, w, st))
                              : (layout == ESC_NCHW ? pw_mix_t<__nv_bfloat16, esc::kNCHW>(p, x, w_point, grad_x, w, st)
                                                    : pw_mix_t<__nv_bfloat16, esc::kNHWC>(p, x, w_point, grad_x, w, st));
        if (rc != ESC_OK) return rc;
        w.mixed = true;
    }
    const void* x_taps = w_point ? grad_x : x;             // what the depth-wise stage saw
    bool packed = false;
    if (dense) {
        // w_large is the dense kernel [16][16][K][K]: its gradient here; the depth-wise kernels
        // below give g_dk (the middle 3 x 3 of their tap gradients) and what follows from it
        packed = wants_packing(p) && g_engine_policy != ESC_ENGINE_FP32;
        if (packed) {
            // bf16 NCHW: everything that follows reads the packed attention channels, as NHWC tensors of 16 channels
            rc = launch_pack16(p, x, w.x_packed, nullptr, st);
            if (rc == ESC_OK) rc = launch_pack16(p, grad_out, w.go_packed, grad_x, st);
            if (rc != ESC_OK) return rc;
            Problem q = p;
            q.C = esc::dense16::CA; q.layout = ESC_NHWC; q.dense = true;
            rc = dense_tap_grad_t<__nv_bfloat16, esc::kNHWC>(q, w.x_packed, w.go_packed, w, g_wd, st);
            if (rc == ESC_OK) rc = backward_t<__nv_bfloat16, esc::kNHWC>(q, w.x_packed, w.go_packed, w_large, est, w, g, st);
            if (rc != ESC_OK) return rc;
            return dense_grad_x_t<__nv_bfloat16, esc::kNCHW>(p, grad_out, w_large, grad_x, w, true, st);
        }
        rc = dtype == ESC_F32 ? (layout == ESC_NCHW ? dense_tap_grad_t<float, esc::kNCHW>(p, x, grad_out, w, g_wd, st)
                                                    : dense_tap_grad_t<float, esc::kNHWC>(p, x, grad_out, w, g_wd, st))
                              : (layout == ESC_NCHW ? dense_tap_grad_t<__nv_bfloat16, esc::kNCHW>(p, x, grad_out, w, g_wd, st)
                                                    : dense_tap_grad_t<__nv_bfloat16, esc::kNHWC>(p, x, grad_out, w, g_wd, st));
        if (rc != ESC_OK) return rc;
    }
    p.dense = dense;
    if (dtype == ESC_F32)
        rc = layout == ESC_NCHW ? backward_t<float, esc::kNCHW>(p, x_taps, grad_out, w_large, est, w, g, st)
                                : backward_t<float, esc::kNHWC>(p, x_taps, grad_out, w_large, est, w, g, st);
    else
        rc = layout == ESC_NCHW ? backward_t<__nv_bfloat16, esc::kNCHW>(p, x_taps, grad_out, w_large, est, w, g, st)
                                : backward_t<__nv_bfloat16, esc::kNHWC>(p, x_taps, grad_out, w_large, est, w, g, st);
    if (rc != ESC_OK) return rc;
    // grad_x: the forward stencil on grad_out with both kernels rotated by 180 degrees, plus the constants (in the
    // decomposed form the constants belong behind the transposed mix: the last kernel adds them)
    if (dense)
        return dtype == ESC_F32 ? (layout == ESC_NCHW ? dense_grad_x_t<float, esc::kNCHW>(p, grad_out, w_large, grad_x, w, packed, st)
                                                      : dense_grad_x_t<float, esc::kNHWC>(p, grad_out, w_large, grad_x, w, packed, st))
                                : (layout == ESC_NCHW ? dense_grad_x_t<__nv_bfloat16, esc::kNCHW>(p, grad_out, w_large, grad_x, w, packed, st)
                                                      : dense_grad_x_t<__nv_bfloat16, esc::kNHWC>(p, grad_out, w_large, grad_x, w, packed, st));
    p.bias = w_point ? nullptr : w.bias;
    const TensorLk tl = tensor_lk(p, grad_out, grad_x, w.w_flip, w.lk_pad, st);
    rc = launch_stencil(p, grad_out, w.w_flip, w.dk_flip, grad_x, w.ctrl, st, /*dependent=*/false, &tl);
    if (rc != ESC_OK || !w_point) return rc;
    rc = dtype == ESC_F32 ? (layout == ESC_NCHW ? pw_back_t<float, esc::kNCHW>(p, x, w_point, grad_x, w, g_wp, st)
                                                : pw_back_t<float, esc::kNHWC>(p, x, w_point, grad_x, w, g_wp, st))
                          : (layout == ESC_NCHW ? pw_back_t<__nv_bfloat16, esc::kNCHW>(p, x, w_point, grad_x, w, g_wp, st)
                                                : pw_back_t<__nv_bfloat16, esc::kNHWC>(p, x, w_point, grad_x, w, g_wp, st));
    return rc;
}
}  // namespace

int esc_convattn_backward(const void* x, const void* grad_out, int B, int C, int C_a, int H, int W, int K,
                          const void* w_large, const void* w_dyn, const void* b_dyn, void* grad_x,
                          float* grad_w_large, float* grad_w_dyn, float* grad_b_dyn, int dtype, int layout,
                          void* workspace, size_t workspace_bytes_, void* stream) {
    const Estimator est{w_dyn, b_dyn, nullptr, nullptr, 0};
    const BackwardGrads g{grad_w_large, grad_w_dyn, grad_b_dyn, nullptr, nullptr};
    return backward_entry(x, grad_out, B, C, C_a, H, W, K, w_large, est, grad_x, g, dtype, layout, workspace, workspace_bytes_, stream);
}

int esc_convattn_backward_mlp(const void* x, const void* grad_out, int B, int C, int C_a, int H, int W, int K,
                              const void* w_large, const void* w_down, const void* b_down, const void* w_up,
                              const void* b_up, int hidden, void* grad_x, float* grad_w_large, float* grad_w_down,
                              float* grad_b_down, float* grad_w_up, float* grad_b_up, int dtype, int layout,
                              void* workspace, size_t workspace_bytes_, void* stream) {
    if (hidden <= 0) return ESC_ERR_SHAPE;
    const Estimator est{w_up, b_up, w_down, b_down, hidden};
    const BackwardGrads g{grad_w_large, grad_w_up, grad_b_up, grad_w_down, grad_b_down};
    return backward_entry(x, grad_out, B, C, C_a, H, W, K, w_large, est, grad_x, g, dtype, layout, workspace, workspace_bytes_, stream);
}

int esc_convattn_backward_pw(const void* x, const void* grad_out, int B, int C, int C_a, int H, int W, int K,
                             const void* w_large, const void* w_point, const void* w_dyn, const void* b_dyn, void* grad_x,
                             float* grad_w_large, float* grad_w_point, float* grad_w_dyn, float* grad_b_dyn, int dtype,
                             int layout, void* workspace, size_t workspace_bytes_, void* stream) {
    if (!w_point) return ESC_ERR_NULL;
    const Estimator est{w_dyn, b_dyn, nullptr, nullptr, 0};
    const BackwardGrads g{grad_w_large, grad_w_dyn, grad_b_dyn, nullptr, nullptr};
    return backward_entry(x, grad_out, B, C, C_a, H, W, K, w_large, est, grad_x, g, dtype, layout, workspace, workspace_bytes_, stream,
                          w_point, grad_w_point);
}

size_t esc_convattn_backward_dense_workspace_bytes(int B, int C_a, int H, int W, int K) {
    if (B <= 0 || C_a != esc::bwd::dense::CA || H <= 0 || W <= 0 || K < 3 || K > esc::bwd::K || (K & 1) == 0) return 0;
    const Problem p{B, C_a, C_a, H, W, K, ESC_F32, ESC_NCHW};
    return carve_backward(nullptr, p).bytes_packed;
}

int esc_convattn_backward_dense(const void* x, const void* grad_out, int B, int C, int C_a, int H, int W, int K,
                                const void* w_dense, const void* w_dyn, const void* b_dyn, void* grad_x,
                                float* grad_w_dense, float* grad_w_dyn, float* grad_b_dyn, int dtype, int layout,
                                void* workspace, size_t workspace_bytes_, void* stream) {
    const Estimator est{w_dyn, b_dyn, nullptr, nullptr, 0};
    const BackwardGrads g{nullptr, grad_w_dyn, grad_b_dyn, nullptr, nullptr};
    return backward_entry(x, grad_out, B, C, C_a, H, W, K, w_dense, est, grad_x, g, dtype, layout, workspace, workspace_bytes_, stream,
                          nullptr, nullptr, /*dense=*/true, grad_w_dense);
}

int esc_convattn_backward_variant(const void* x, const void* grad_out, int B, int C, int C_a, int H, int W, int K,
                                  int large_kernel, const void* w_large, const void* w_point, const void* w_down,
                                  const void* b_down, const void* w_up, const void* b_up, int hidden, void* grad_x,
                                  float* grad_w_large, float* grad_w_point, float* grad_w_down, float* grad_b_down,
                                  float* grad_w_up, float* grad_b_up, int dtype, int layout, void* workspace,
                                  size_t workspace_bytes_, void* stream) {
    if (large_kernel != ESC_LK_DEPTHWISE && large_kernel != ESC_LK_DECOMPOSED && large_kernel != ESC_LK_DENSE)
        return ESC_ERR_UNSUPPORTED;
    if (hidden < 0) return ESC_ERR_SHAPE;
    if (large_kernel == ESC_LK_DECOMPOSED && !w_point) return ESC_ERR_NULL;
    const Estimator est{w_up, b_up, hidden > 0 ? w_down : nullptr, hidden > 0 ? b_down : nullptr, hidden};
    const bool dense = large_kernel == ESC_LK_DENSE;
    const BackwardGrads g{dense ? nullptr : grad_w_large, grad_w_up, grad_b_up, hidden > 0 ? grad_w_down : nullptr,
                          hidden > 0 ? grad_b_down : nullptr};
    return backward_entry(x, grad_out, B, C, C_a, H, W, K, w_large, est, grad_x, g, dtype, layout, workspace, workspace_bytes_, stream,
                          large_kernel == ESC_LK_DECOMPOSED ? w_point : nullptr,
                          large_kernel == ESC_LK_DECOMPOSED ? grad_w_point : nullptr, dense, dense ? grad_w_large : nullptr);
}

size_t esc_conv_fuse_backward_workspace_bytes(int B, int C, int H, int W) {
    if (B <= 0 || H <= 0 || W <= 0 || !esc::fuse::bwd::supported(C)) return 0;
    return carve_fuse_backward(nullptr, C, (long long)B * H * W).bytes;
}

int esc_conv_fuse_backward(const void* cat, const void* grad_out, int B, int C, int H, int W, const void* w_fuse,
                           void* grad_cat, float* grad_w_fuse, float* grad_b_fuse, int dtype, int layout,
                           void* workspace, size_t workspace_bytes_, void* stream) {
    g_last_launches = 0;
    const Problem p{B, C, C, H, W, 3, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!esc::fuse::bwd::supported(C)) return ESC_ERR_UNSUPPORTED;
    if (!cat || !grad_out || !w_fuse || !grad_cat) return ESC_ERR_NULL;
    rc = check_tensors(p, grad_out, grad_cat);
    if (rc != ESC_OK) return rc;
    if (!aligned(cat, 16) || !aligned(w_fuse, p.es())) return ESC_ERR_ALIGN;
    {
        const uintptr_t xa = reinterpret_cast<uintptr_t>(cat), oa = reinterpret_cast<uintptr_t>(grad_cat);
        const size_t bytes = p.elems() * p.es();
        if (xa < oa + bytes && oa < xa + bytes) return ESC_ERR_ALIAS;
    }
    for (const float* q : {grad_w_fuse, grad_b_fuse})
        if (q && !aligned(q, 4)) return ESC_ERR_ALIGN;
    if (!workspace || !aligned(workspace, 256)) return ESC_ERR_WORKSPACE;
    const long long HW = (long long)H * W, pixels = (long long)B * HW;
    const FuseBackwardWs w = carve_fuse_backward(workspace, C, pixels);
    if (workspace_bytes_ < w.bytes) return ESC_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool sums = grad_w_fuse || grad_b_fuse;
    int blocks = w.blocks32;
    if (esc::fuse::bwd::mma::applies(C, HW, dtype, layout, w_fuse) && g_engine_policy != ESC_ENGINE_FP32) {
        blocks = w.blocks;
        rc = layout == ESC_NCHW ? fuse_backward_mma_t<esc::kNCHW>(C, cat, grad_out, w_fuse, grad_cat, HW, pixels, w, sums, st)
                                : fuse_backward_mma_t<esc::kNHWC>(C, cat, grad_out, w_fuse, grad_cat, HW, pixels, w, sums, st);
    } else {
        if (sums) {
            if (dtype == ESC_F32)
                rc = layout == ESC_NCHW ? fuse_wgrad_t<float, esc::kNCHW>(C, cat, grad_out, HW, pixels, w, st)
                                        : fuse_wgrad_t<float, esc::kNHWC>(C, cat, grad_out, HW, pixels, w, st);
            else
                rc = layout == ESC_NCHW ? fuse_wgrad_t<__nv_bfloat16, esc::kNCHW>(C, cat, grad_out, HW, pixels, w, st)
                                        : fuse_wgrad_t<__nv_bfloat16, esc::kNHWC>(C, cat, grad_out, HW, pixels, w, st);
            if (rc != ESC_OK) return rc;
        }
        // grad_cat = W_fuse^T grad_out per pixel: the 1x1 kernel with the matrix read transposed, no bias, no residual
        rc = dtype == ESC_F32 ? launch_fuse_fp32<float, true>(p, grad_out, grad_out, w_fuse, nullptr, nullptr, grad_cat, st, /*first=*/!sums)
                              : launch_fuse_fp32<__nv_bfloat16, true>(p, grad_out, grad_out, w_fuse, nullptr, nullptr, grad_cat, st, !sums);
    }
    if (rc != ESC_OK || !sums) return rc;
    const int elems = C * C + C;
    ESC_CUDA(launch_pdl(esc::fuse::bwd::sum_wgrad, (unsigned)((elems + 31) / 32), esc::fuse::bwd::kSumWarps * 32, 0, st, w.part, C, blocks, grad_w_fuse, grad_b_fuse));
    ESC_CUDA(cudaGetLastError());
    ++g_last_launches;
    return ESC_OK;
}

int esc_convattn_selftest_bounded_wait(void* workspace, void* stream) {
    if (!workspace || !aligned(workspace, 256)) return ESC_ERR_WORKSPACE;
    bounded_wait_probe<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<unsigned*>(workspace));
    ESC_CUDA(cudaGetLastError());
    return ESC_OK;
}

int esc_convattn_device_status(void* workspace, void* stream) {
    if (!workspace) return ESC_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned word[2] = {0, 0};
    ESC_CUDA(cudaMemcpyAsync(word, workspace, sizeof word, cudaMemcpyDeviceToHost, st));
    ESC_CUDA(cudaStreamSynchronize(st));
    if (word[0] != 0) {
        char buf[96];
        snprintf(buf, sizeof buf, "device status %u, detail 0x%x", word[0], word[1]);
        g_last_error = buf;
        ESC_CUDA(cudaMemsetAsync(workspace, 0, sizeof word, st));
        ESC_CUDA(cudaStreamSynchronize(st));
    }
    return (int)word[0];
}

namespace {
// alone: the caller waits for this step before it submits another
int host_submit(int slot, const void* x_host, int B, int C, int C_a, int H, int W, int K, const void* w_large_host, const void* w_dyn_host,
                const void* b_dyn_host, void* out_host, int dtype, int layout, bool alone) {
    g_last_launches = 0;
    if (slot < 0 || slot >= kHostSlots) return ESC_ERR_UNSUPPORTED;
    const Problem p{B, C, C_a, H, W, K, dtype, layout};
    int rc = check_shape(p);
    if (rc != ESC_OK) return rc;
    if (!x_host || !w_large_host || !w_dyn_host || !b_dyn_host || !out_host) return ESC_ERR_NULL;
    std::lock_guard<std::mutex> lock(g_host_mu);
    HostPath& h = g_host[slot];
    int dev = 0;
    ESC_CUDA(cudaGetDevice(&dev));
    if (h.dev != dev) {   // first use, or the caller switched device: start over
        if (h.dev >= 0) {
            ESC_CUDA(cudaSetDevice(h.dev));
            if (h.st) cudaStreamSynchronize(h.st);
            cudaFree(h.x); cudaFree(h.out); cudaFree(h.wts); cudaFree(h.ws);
            if (h.st) cudaStreamDestroy(h.st);
            if (h.compute) cudaStreamDestroy(h.compute);
            if (h.down) cudaStreamDestroy(h.down);
            if (h.ev) cudaEventDestroy(h.ev);
            ESC_CUDA(cudaSetDevice(dev));
        }
        h = HostPath();
        h.dev = dev;
        ESC_CUDA(cudaStreamCreateWithFlags(&h.st, cudaStreamNonBlocking));
        ESC_CUDA(cudaStreamCreateWithFlags(&h.compute, cudaStreamNonBlocking));
        ESC_CUDA(cudaStreamCreateWithFlags(&h.down, cudaStreamNonBlocking));
        ESC_CUDA(cudaEventCreateWithFlags(&h.ev, cudaEventDisableTiming));
    }
    const size_t es = p.es(), xbytes = p.elems() * es;
    const size_t n_wl = (size_t)C_a * K * K, n_wd = (size_t)9 * C_a * C_a, n_bd = (size_t)9 * C_a;
    const size_t off_wd = round_up(n_wl * es, 256), off_bd = off_wd + round_up(n_wd * es, 256);
    const size_t wbytes = off_bd + round_up(n_bd * es, 256);
    const size_t wsbytes = workspace_bytes(B, C_a, (long long)H * W);
    if (h.xbytes < xbytes || h.wbytes < wbytes || h.wsbytes < wsbytes)
        ESC_CUDA(cudaStreamSynchronize(h.st));               // nothing of this slot may still use the old buffers
    if (h.xbytes < xbytes) {
        cudaFree(h.x); cudaFree(h.out); h.x = h.out = nullptr; h.xbytes = 0;
        ESC_CUDA(cudaMalloc(&h.x, xbytes));
        ESC_CUDA(cudaMalloc(&h.out, xbytes));
        h.xbytes = xbytes;
    }
    if (h.wbytes < wbytes) {
        cudaFree(h.wts); h.wts = nullptr; h.wbytes = 0;
        ESC_CUDA(cudaMalloc(&h.wts, wbytes));
        h.wbytes = wbytes;
    }
    if (h.wsbytes < wsbytes) {
        cudaFree(h.ws); h.ws = nullptr; h.wsbytes = 0;
        ESC_CUDA(cudaMalloc(&h.ws, wsbytes));
        ESC_CUDA(cudaMemsetAsync(h.ws, 0, wsbytes, h.st));
        h.wsbytes = wsbytes;
    }
    char* wts = static_cast<char*>(h.wts);
    const size_t image = xbytes / B, att = (size_t)C_a * H * W * es, identity = image - att;
    const bool overlap = alone && layout == ESC_NCHW && identity * B >= kHostOverlapBytes && identity >= kHostMinRow && image <= kHostMaxPitch &&
                         host_buffers_allow(x_host, out_host, xbytes);
    if (overlap) ESC_CUDA(cudaMemcpy2DAsync(h.x, image, x_host, image, att, B, cudaMemcpyHostToDevice, h.st));
    else ESC_CUDA(cudaMemcpyAsync(h.x, x_host, xbytes, cudaMemcpyHostToDevice, h.st));
    ESC_CUDA(cudaMemcpyAsync(wts, w_large_host, n_wl * es, cudaMemcpyHostToDevice, h.st));
    ESC_CUDA(cudaMemcpyAsync(wts + off_wd, w_dyn_host, n_wd * es, cudaMemcpyHostToDevice, h.st));
    ESC_CUDA(cudaMemcpyAsync(wts + off_bd, b_dyn_host, n_bd * es, cudaMemcpyHostToDevice, h.st));
    const Estimator est{wts + off_wd, wts + off_bd, nullptr, nullptr, 0};
    if (!overlap) {
        rc = forward_impl(p, h.x, wts, est, h.out, h.ws, h.st);
        if (rc != ESC_OK) return rc;
        ESC_CUDA(cudaMemcpyAsync(out_host, h.out, xbytes, cudaMemcpyDeviceToHost, h.st));
        return ESC_OK;
    }
    // `to` goes on only when what `from` has been given so far is done
    auto follow = [&](cudaStream_t to, cudaStream_t from) -> int {
        ESC_CUDA(cudaEventRecord(h.ev, from));
        ESC_CUDA(cudaStreamWaitEvent(to, h.ev, 0));
        return ESC_OK;
    };
    auto enqueue = [&]() -> int {
        int r = follow(h.compute, h.st);
        if (r != ESC_OK) return r;
        Problem pa = p;
        pa.skip_copy = true;
        r = forward_impl(pa, h.x, wts, est, h.out, h.ws, h.compute);
        if (r != ESC_OK) return r;
        ESC_CUDA(cudaMemcpy2DAsync(out_host, image, h.out, image, att, B, cudaMemcpyDeviceToHost, h.compute));
        // pieces of about kHostChunkBytes: part of an image's identity channels, or those of several images
        const size_t cols = identity < kHostChunkBytes ? identity : kHostChunkBytes;
        const int rows = (int)std::min((size_t)B, kHostChunkBytes / cols);
        for (int b = 0; b < B; b += rows)
            for (size_t at = att; at < image; at += cols) {
                const size_t off = (size_t)b * image + at, n = std::min(cols, image - at);
                const int nb = std::min(rows, B - b);
                ESC_CUDA(cudaMemcpy2DAsync(static_cast<char*>(h.x) + off, image, static_cast<const char*>(x_host) + off, image, n, nb, cudaMemcpyHostToDevice, h.st));
                r = follow(h.down, h.st);
                if (r != ESC_OK) return r;
                ESC_CUDA(cudaMemcpy2DAsync(static_cast<char*>(out_host) + off, image, static_cast<char*>(h.x) + off, image, n, nb, cudaMemcpyDeviceToHost, h.down));
            }
        return ESC_OK;
    };
    rc = enqueue();
    // the slot's stream ends behind the other two, also after an error: who waits for it waits for all
    const int r1 = follow(h.st, h.compute), r2 = follow(h.st, h.down);
    return rc != ESC_OK ? rc : r1 != ESC_OK ? r1 : r2;
}
}  // namespace

int esc_convattn_forward_host_submit(int slot, const void* x_host, int B, int C, int C_a, int H, int W, int K,
                                     const void* w_large_host, const void* w_dyn_host, const void* b_dyn_host,
                                     void* out_host, int dtype, int layout) {
    return host_submit(slot, x_host, B, C, C_a, H, W, K, w_large_host, w_dyn_host, b_dyn_host, out_host, dtype, layout, /*alone=*/false);
}

int esc_convattn_forward_host_wait(int slot) {
    if (slot < 0 || slot >= kHostSlots) return ESC_ERR_UNSUPPORTED;
    cudaStream_t st = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_host_mu);
        if (g_host[slot].dev < 0) return ESC_OK;             // nothing was ever submitted here
        st = g_host[slot].st;
    }
    ESC_CUDA(cudaStreamSynchronize(st));
    return ESC_OK;
}

int esc_convattn_forward_host(const void* x_host, int B, int C, int C_a, int H, int W, int K,
                              const void* w_large_host, const void* w_dyn_host, const void* b_dyn_host,
                              void* out_host, int dtype, int layout) {
    const int rc = host_submit(0, x_host, B, C, C_a, H, W, K, w_large_host, w_dyn_host, b_dyn_host, out_host, dtype, layout, /*alone=*/true);
    if (rc != ESC_OK) return rc;
    return esc_convattn_forward_host_wait(0);
}

}  // extern "C"
