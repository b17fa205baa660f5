// Kernel (b) on the fifth-generation tensor cores: the depth-wise stage of ConvAttn (ESC paper, Section 3.3, Eq. 4 lines 3-4) for
// bf16 tensors and odd K up to 13, with tcgen05.mma and accumulators in tensor memory.
//
//   out[b,c,y,x] = sum_{i,j} w[c,i,j] x[b,c,y+i-P,x+j-P]  +  sum_{i,j} dk[b,c,i,j] x[b,c,y+i-1,x+j-1] (+ bias[b,c])
//
// Formulation.  A unit is eight channels.  PAIRS of neighbouring pixels are the rows of A: M = 128 pairs, K = 16 = two pixels of eight
// channels, so one instruction multiplies 256 staged pixels.  B stacks all 13 kernel rows, both pixels of the output pair and the eight
// output channels: N = 13 x 2 x 8 = 208 columns,
//   B_q[(s, k)][(12 - i) * 16 + e * 8 + n] = w[n][i][2q + s - e]   where k == n and 0 <= 2q + s - e <= 12, else 0,
// and seven instructions (q = 0 .. 6, A one pair further each time) are all an input row needs.  Column block c of the result belongs
// to output row (input row) - 6 + c: the accumulators of 32 output rows lie side by side in the 512 columns of tensor memory, an
// input row is staged once and nothing is unfolded or transposed.  A channel meets only itself, so seven eighths of B are zero;
// with 16 channels and single pixels (the dense kernel's form) it would be fifteen sixteenths, 13 instructions for the same outputs.
//
// Staged row: even and odd pixels in planes of their own, [2][134 pairs][8 channels], which is the tensor core's K-major layout
// without swizzle; a pair further on is 16 bytes.  NHWC pixels go there as they are, 16 bytes at a time with cp.async (zero fill = the padding).
//
// Window.  The pixel rows of all images, and of S row segments of each image, are laid end to end with six zeros between
// neighbours (the padding of both); a window is 256 consecutive positions of that line, whatever images and segments they belong to, and is
// walked over the R rows of a segment.  So 64-pixel patches and odd widths fill the instruction as well as wide maps do.
// The rows of all windows are dealt evenly to the CTAs (a CTA may end one window and begin another).
//
// A non-finite input makes NaN of accumulators outside its window too (zero times infinity).  The epilogue sees that -- the sum of a
// pixel's accumulators is not finite -- and notes the row, unless the 3x3 part is NaN as well; behind its last row it evaluates what
// is not finite in those rows directly, so what leaves the kernel has the window of the definition.  1920x1080, 32 of 64 channels,
// stage alone: finite 182 us, one bad pixel 458, a map of NaN 178; a bad pixel in every 16 x 16 13.9 ms, one channel of NaN beside
// finite ones 20 ms, 4 ms where all is infinite.  (A forward whose attention channels hold NaN or infinity has NaN in dk, hence in
// every output of that image: 239 - 259 us.)
//
// Roles (512 threads, one CTA per SM):
//   warps 0-7    epilogue: one pixel x eight channels per thread and row: tcgen05.ld, the dynamic 3x3 kernel in fp32 on the CUDA cores, one
//                rounding, a 16-byte store
//   warps 8-11   input rows into a ring of 24
//   warp 12      issues the instructions; warps 12-15 build B before that
//   warp 13      copies the identity channels, TMA in / TMA out
//
// What bounds it: the shared-memory / L1 data pipe, and under sustained load the board's power.  Of 1,290 cycles per input row of a
// window the tensor core's operands take 640 wavefronts (48 %), loads and stores 500 (39 %: every 16-byte pixel part of a 128-byte line is
// one), TMA copies most of the rest; the tensor pipe is 63 % busy, DRAM 42 %.  1920x1080, C_a = 32 of 64 channels, stage alone, 303 k
// cycles on random data: 183 us in bursts of twenty launches against 264 for the mma.sync Toeplitz kernel (169 against 254 without identity
// channels), 208 against 263 back to back, where 1,000 W hold the clock at about 1.46 GHz; the whole forward 325 -> 237 and 323 -> 256.
// On the way (bursts): one output row at a time in the epilogue and waits by one lane
// 316; loads ahead of the arithmetic, rows by two 241 (by four 282); slots counted on and tensor memory asked for by four rows in the
// issuing warp, identity channels beside the same rows 185 (chunks of the whole map in turn instead: 297, the parts of a line then reach
// DRAM one by one); those copied once each and up to 24 rows ahead 178 - 183.  No difference: L2 prefetch sizes on the loads.
#pragma once
#include "stencil_dense_umma.cuh"
#include "gap_dynkernel.cuh"
#include <type_traits>

namespace esc { namespace tma { namespace dwu {

constexpr int OCT = 8;                              // channels of a unit
constexpr int WPX = 256;                            // output pixels of a window row: two per row of A
constexpr int SPX = WPX + K13 - 1;                  // staged pixels
constexpr int GAPX = P6;                            // zeros between neighbours on the line
constexpr int PAR_BYTES = 2240;                     // a parity plane: 134 pairs of 16 bytes; 64 modulo 128, so that neighbouring pixels' stores do not share banks
constexpr int ROW_BYTES = 2 * PAR_BYTES;
constexpr int NRING = 24;
constexpr int DEPTH = 8;                            // rows in flight, two a producer warp
constexpr int NQ = (K13 + 1) / 2;                   // instructions per input row
constexpr int NBC = 2 * OCT;                        // columns per output row
constexpr int BHALF_BYTES = K13 * NBC * 16;         // [208 rows][8 k-values]
constexpr int BQ_BYTES = 2 * BHALF_BYTES;
constexpr int B_BYTES = NQ * BQ_BYTES;              // 46,592
constexpr int SLOTS = 512 / NBC;
constexpr int kEpiWarps = 8, kEpiThreads = kEpiWarps * 32, kProdWarps = 4, kThreads = 512;
constexpr int kLaunchRegs = 128, kEpiRegs = 200, kRestRegs = 56;   // 256 * 200 + 256 * 56 = 512 * 128
constexpr int kMaxImages = 40;                      // images a window can touch: 256 / 7 + 2
constexpr int kCopyBytes = 49152, kCopyChunkBytes = 16384, kCopySlots = 12;   // identity channels: the ring, a chunk, and chunks in the ring at most
constexpr int kCopyLead = 24;                       // rows the copies may be ahead of the epilogue
constexpr int kOffB = NRING * ROW_BYTES, kOffCopy = kOffB + B_BYTES, kOffDk = kOffCopy + kCopyBytes,
              kOffTaps = kOffDk + kMaxImages * 9 * OCT * 4, kOffBars = kOffTaps + K13 * K13 * OCT * 2, kSmemBytes = kOffBars + 1152;
constexpr int kBars = 2 * NRING + 2 * SLOTS + kCopySlots + 2;
static_assert(SPX / 2 * 16 <= PAR_BYTES && PAR_BYTES % 128 == 64, "parity plane");
static_assert(kOffB % 128 == 0 && kOffCopy % 128 == 0 && kOffTaps % 16 == 0 && kOffBars % 16 == 0, "alignment");
static_assert(kBars * 8 + 8 + 4 * kCopySlots <= 1152 && kSmemBytes <= 227 * 1024, "shared memory");
static_assert(DEPTH + 5 <= NRING && DEPTH == 2 * kProdWarps, "rows the epilogue needs are signalled before a slot is waited for");

struct Params {
    int B, C, Ca, H, W, K;
    int pitch, S, R, pieces;          // the line: pieces = B * S neighbours, pitch = W + 6 apart; R rows per segment
    int rows, Q, octets;              // rows of all windows, rows per CTA
    const __nv_bfloat16 *x, *w_large; // [Ca][K][K]
    const float* dk;                  // [B][Ca][9]
    const float* bias;                // [B][Ca] or nullptr
    __nv_bfloat16* out;
    unsigned* ctrl;
    int wait_first;
    int copy_cc, copy_shift, copy_slots, copy_chunks, copy_rows;   // identity channels, log2 of a chunk's pixels, chunks in the ring and in all; copied row by row
};

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_zero8(uint32_t taddr) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(taddr), "r"(0u) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(map), "r"(src), "r"(c0), "r"(c1) : "memory");
}
// The seven instructions of an input row, all 13 or fewer column blocks at once, by the lane that elect.sync names (see umma::mma_f16).
__device__ __forceinline__ void mma_row(uint32_t d, unsigned long long da, unsigned long long db, uint32_t idesc) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 p, 1, 0;\n\telect.sync _|q, 0xffffffff;\n\tmov.b64 a, %1;\n\tmov.b64 b, %2;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\tadd.s64 a, a, 1;\n\tadd.s64 b, b, %4;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\tadd.s64 a, a, 1;\n\tadd.s64 b, b, %4;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\tadd.s64 a, a, 1;\n\tadd.s64 b, b, %4;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\tadd.s64 a, a, 1;\n\tadd.s64 b, b, %4;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\tadd.s64 a, a, 1;\n\tadd.s64 b, b, %4;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\tadd.s64 a, a, 1;\n\tadd.s64 b, b, %4;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}"
        ::"r"(d), "l"(da), "l"(db), "r"(idesc), "n"(BQ_BYTES >> 4) : "memory");
}
__device__ __forceinline__ void unpack8(const uint4& v, float (&f)[OCT]) {
    const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) { f[2 * q] = __uint_as_float(w[q] << 16); f[2 * q + 1] = __uint_as_float(w[q] & 0xffff0000u); }
}
__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 2, %0;" ::"n"(kEpiThreads) : "memory"); }

// Outputs that are not finite, straight from the definition: a warp looks at its pixels again in the rows [first, last) of the CTA's
// windows (taps: [K * K][8] weights).  Eight lanes take a pixel: a lane sums kernel rows k and k + 8 of all channels, of which the
// sums over the lanes leave it one, to which it adds the 3x3 part.  Of its own and behind the main loop, so that the registers it
// takes are not missing there (called from the loop, 180 -> 245 us) and no wait of another warp runs out meanwhile.
__device__ __noinline__ void direct(const Params& p, const uint4* taps, int oct, int r_begin, int r_end, int m2, int first, int last) {
    const int lane = threadIdx.x & 31, k = lane & 7, P = p.K / 2;
    first = __reduce_min_sync(0xffffffffu, first);
    last = __reduce_max_sync(0xffffffffu, last);
    int o = 0;
    for (int r = r_begin; r < r_end;) {
        const int t = r / p.R, row0 = r - t * p.R, L = min(p.R - row0, r_end - r);
        const int f = t * WPX + m2, piece = f / p.pitch, x = f - piece * p.pitch, b = piece / p.S, y0 = (piece - b * p.S) * p.R + row0;
        const bool valid = piece < p.pieces && x < p.W;
        for (int yr = max(0, first - o); yr < min(L, last - o); ++yr) {
            unsigned bad = 0;                                // channels of this lane's pixel
            if (valid && y0 + yr < p.H) {
                float v[OCT];
                unpack8(*reinterpret_cast<const uint4*>(p.out + (((size_t)b * p.H + y0 + yr) * p.W + x) * p.C + oct * OCT), v);
#pragma unroll
                for (int n = 0; n < OCT; ++n) bad |= (fabsf(v[n]) < INFINITY ? 0u : 1u) << n;
            }
            for (unsigned todo = __ballot_sync(0xffffffffu, bad != 0); todo != 0;) {
                // the next four pixels, one per group of eight lanes
                int src = -1;
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    if (g == lane >> 3 && todo != 0) src = __ffs(todo) - 1;
                    todo &= todo - 1;
                }
                const int from = max(src, 0), py = __shfl_sync(0xffffffffu, y0, from) + yr, pxx = __shfl_sync(0xffffffffu, x, from),
                          pb = __shfl_sync(0xffffffffu, b, from);
                const unsigned from_bad = __shfl_sync(0xffffffffu, bad, from), pbad = src < 0 ? 0u : from_bad;
                const __nv_bfloat16* img = p.x + (size_t)(pbad ? pb : 0) * p.H * p.W * p.C + oct * OCT;
                float s3 = 0.f;                              // the 3x3 part of channel k, as the main loop has it
                if (pbad >> k & 1) {
                    const size_t bc = (size_t)pb * p.Ca + oct * OCT + k;
                    if (p.bias) s3 = __ldcg(p.bias + bc);
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        const int yy = py + i / 3 - 1, xx = pxx + i % 3 - 1;
                        const bool in = yy >= 0 && yy < p.H && xx >= 0 && xx < p.W;
                        s3 = fmaf(__ldcg(p.dk + bc * 9 + i), in ? __bfloat162float(img[((size_t)yy * p.W + xx) * p.C + k]) : 0.f, s3);
                    }
                }
                const bool open = (pbad >> k & 1) && s3 == s3;                   // else NaN whatever the large kernel's sum
                const bool group = (__ballot_sync(0xffffffffu, open) >> (lane & 24) & 0xffu) != 0;
                float s[OCT] = {};
                if (group)
                    for (int i = k; i < p.K; i += 8) {
                        const int yy = py + i - P;
                        if (yy < 0 || yy >= p.H) continue;
                        const __nv_bfloat16* row = img + (size_t)yy * p.W * p.C;
                        uint4 v[K13];
#pragma unroll
                        for (int j = 0; j < K13; ++j) {
                            const int xx = pxx + j - P;
                            v[j] = make_uint4(0u, 0u, 0u, 0u);
                            if (j < p.K && xx >= 0 && xx < p.W) v[j] = __ldg(reinterpret_cast<const uint4*>(row + (size_t)xx * p.C));
                        }
#pragma unroll
                        for (int j = 0; j < K13; ++j) {
                            const int xx = pxx + j - P;
                            if (j < p.K && xx >= 0 && xx < p.W) {
                                float fv[OCT], w[OCT];
                                unpack8(v[j], fv);
                                unpack8(taps[i * p.K + j], w);
#pragma unroll
                                for (int n = 0; n < OCT; ++n) s[n] = fmaf(w[n], fv[n], s[n]);
                            }
                        }
                    }
                // sums over the eight lanes; lane k keeps channel k
#pragma unroll
                for (int h = 4; h > 0; h >>= 1)
#pragma unroll
                    for (int n = 0; n < h; ++n) {
                        const bool up = (lane & h) != 0;
                        const float keep = up ? s[n + h] : s[n];
                        s[n] = keep + __shfl_xor_sync(0xffffffffu, up ? s[n] : s[n + h], h);
                    }
                if (open) p.out[(((size_t)pb * p.H + py) * p.W + pxx) * p.C + oct * OCT + k] = __float2bfloat16_rn(s[0] + s3);
            }
        }
        o += L;
        r += L;
    }
}

__global__ void __maxnreg__(kLaunchRegs)
stencil_dw_umma_nhwc_bf16(const __grid_constant__ CUtensorMap map_cin, const __grid_constant__ CUtensorMap map_cout, const __grid_constant__ Params p)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* ring = smem;
    unsigned char* btab = smem + kOffB;
    unsigned char* cring = smem + kOffCopy;
    float* dks = reinterpret_cast<float*>(smem + kOffDk);                   // [image of the window][9 taps][8 channels]
    u64* bars = reinterpret_cast<u64*>(smem + kOffBars);
    const uint32_t rowfull0 = smem_u32(bars), rowfree0 = rowfull0 + 8 * NRING, accfull0 = rowfree0 + 8 * NRING, accfree0 = accfull0 + 8 * SLOTS,
                   cfull0 = accfree0 + 8 * SLOTS, cleared = cfull0 + 8 * kCopySlots, drained = cleared + 8;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kBars);
    int* progress = reinterpret_cast<int*>(tmem_slot + 1);                  // output rows the first epilogue warp has finished

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < NRING; ++s) { mbar_init(rowfull0 + 8 * s, 1); mbar_init(rowfree0 + 8 * s, 1 + kEpiWarps); }
        for (int s = 0; s < SLOTS; ++s) { mbar_init(accfull0 + 8 * s, 1); mbar_init(accfree0 + 8 * s, kEpiWarps); }
        for (int s = 0; s < kCopySlots; ++s) mbar_init(cfull0 + 8 * s, 1);
        mbar_init(cleared, kEpiWarps);
        mbar_init(drained, 1);
        *progress = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 12) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    umma::tc_fence_before();
    __syncthreads();
    umma::tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    if (p.wait_first) pdl_wait_primary();
    pdl_launch_dependents();

    // ---- this CTA's rows [r_begin, r_end) of the windows' rows, for channels oct * 8 .. + 7 -------------------
    const int oct = (int)(blockIdx.x % (unsigned)p.octets);
    const int r_begin = (int)(blockIdx.x / (unsigned)p.octets) * p.Q, r_end = min(p.rows, r_begin + p.Q);
    const int off = (K13 - p.K) / 2;

    if (warp >= kEpiWarps && warp < kEpiWarps + kProdWarps) {
        // ======================= input rows ==========================================================
        // A warp takes every fourth row, a lane every 32nd pixel of it.  It signals a row when it has asked for its next one, so that
        // DEPTH rows are in flight.  Row g's slot is free when output row g - NRING - 7 is done, for which the rows up to
        // g - NRING + 5 must have been signalled: DEPTH + 5 <= NRING.
        reg_dec<kRestRegs>();
        constexpr int kPer = (SPX + 31) / 32;
        const int pw = warp - kEpiWarps;
        const uint32_t ring_a = smem_u32(ring) + (lane & 1) * PAR_BYTES + (lane >> 1) * 16;
        const long long row_stride = (long long)p.W * p.C;
        int g = 0, pending = -1;                             // rows so far; the row asked for and not signalled
        bool alive = true;
        auto signal = [&](int row) {
            fence_async_smem();                              // the tensor core reads through the async proxy
            __syncwarp();
            if (lane == 0) mbar_arrive(rowfull0 + 8 * (row % NRING));
        };
        for (int r = r_begin; r < r_end;) {
            const int t = r / p.R, row0 = r - t * p.R, L = min(p.R - row0, r_end - r), n_in = L + K13 - 1;
            unsigned src[kPer];                              // in pixels
            int y0[kPer];
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const int px = lane + 32 * k, f = t * WPX + px - P6;
                const int piece = f < 0 ? 0 : f / p.pitch, xx = f < 0 ? p.W : f - piece * p.pitch;
                const bool ok = px < SPX && xx < p.W && piece < p.pieces;
                const int b = piece / p.S, s = piece - b * p.S;
                y0[k] = ok ? s * p.R + row0 - P6 : -(1 << 30);
                src[k] = (unsigned)(ok ? b : 0) * (unsigned)(p.H * p.W) + (unsigned)(ok ? xx : 0);
            }
            const __nv_bfloat16* base = p.x + oct * OCT;
            for (int n = (pw - g) & 3; n < n_in; n += 4) {
                const int row = g + n, slot = row % NRING;
                if (row >= NRING && alive)
                    alive = umma::mbar_wait_warp(rowfree0 + 8 * slot, (unsigned)((row / NRING - 1) & 1), p.ctrl, 0xE0000000u | (unsigned)(row & 0xffff));
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    if (k == kPer - 1 && lane >= SPX - 32 * (kPer - 1)) continue;
                    const int y = y0[k] + n;
                    const bool ok = y >= 0 && y < p.H;
                    cp_async16(ring_a + slot * ROW_BYTES + k * 256, base + (ok ? (long long)src[k] * p.C + y * row_stride : 0), ok);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
                if (pending >= 0) {
                    asm volatile("cp.async.wait_group %0;" ::"n"(DEPTH / kProdWarps - 1) : "memory");
                    signal(pending);
                }
                pending = row;
            }
            g += n_in;
            r += L;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (pending >= 0) signal(pending);
    } else if (warp >= kEpiWarps + kProdWarps) {
        reg_dec<kRestRegs>();
        // ======================= B: zeros, then each tap at its two places ===============================
        {
            const int bt = tid - (kEpiThreads + kProdWarps * 32), taps = p.K * p.K, items = OCT * taps;
            const unsigned short* wg = reinterpret_cast<const unsigned short*>(p.w_large) + (size_t)oct * items;
            unsigned short v[11];                            // 1,352 taps at most, all loads in flight before the zeros
            constexpr int kT = 128;
#pragma unroll
            for (int u = 0; u < 11; ++u) v[u] = bt + u * kT < items ? __ldg(wg + bt + u * kT) : 0;
            for (int e = bt; e < B_BYTES / 16; e += kT) reinterpret_cast<uint4*>(btab)[e] = make_uint4(0u, 0u, 0u, 0u);
            asm volatile("bar.sync 3, %0;" ::"n"(kT) : "memory");
#pragma unroll
            for (int u = 0; u < 11; ++u) {
                const int it = bt + u * kT;
                if (it < items) {
                    const int n = it / taps, rem = it - n * taps, i = rem / p.K + off, j = rem % p.K + off;
                    *reinterpret_cast<unsigned short*>(smem + kOffTaps + (rem * OCT + n) * 2) = v[u];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int tt = j + e;
                        *reinterpret_cast<unsigned short*>(btab + (tt >> 1) * BQ_BYTES + (tt & 1) * BHALF_BYTES +
                                                           ((K13 - 1 - i) * NBC + e * OCT + n) * 16 + n * 2) = v[u];
                    }
                }
            }
            fence_async_smem();
            asm volatile("bar.sync 3, %0;" ::"n"(kT) : "memory");
            asm volatile("bar.arrive 4, %0;" ::"n"(kT + kEpiThreads) : "memory");   // the epilogue may read the taps
        }
        if (warp == 12) {
            // ======================= tensor-core instructions =========================================
            bool alive = umma::mbar_wait_warp(cleared, 0, p.ctrl, 0xE1000000u);
            const uint32_t ring_a = smem_u32(ring), btab_a = smem_u32(btab);
            const int q_lo = off >> 1, q_hi = (K13 - off) >> 1;
            // What the warp does beside issuing is not hidden by the few instructions that the tensor core keeps waiting, so
            // slots are counted on, and the tensor memory of four output rows is asked for at a time.
            unsigned slot = 0, full_parity = 0, o = 0, free_rows = SLOTS;      // o: output rows so far; those below free_rows may be opened
            const unsigned long long da0 = umma::smem_desc(ring_a, PAR_BYTES, 128), db0 = umma::smem_desc(btab_a, BHALF_BYTES, 128);
            unsigned long long da = da0;
            for (int r = r_begin; r < r_end;) {
                const int t = r / p.R, row0 = r - t * p.R, L = min(p.R - row0, r_end - r);
                for (int n = 0; n < L + K13 - 1; ++n) {
                    if (alive) alive = umma::mbar_wait_warp(rowfull0 + 8 * slot, full_parity, p.ctrl, 0xE2000000u | (unsigned)(n & 0xffff));
                    if (n < L && o + n >= free_rows) {           // the columns of the output row this input row opens, and of the next three
                        const unsigned last = o + n + 3 - SLOTS;
                        if (alive) alive = umma::mbar_wait_warp(accfree0 + 8 * (last % SLOTS), (last / SLOTS) & 1, p.ctrl, 0xE3000000u | (unsigned)(n & 0xffff));
                        free_rows = last + SLOTS + 1;
                    }
                    umma::tc_fence_after();
                    // input row n feeds output rows n - 12 + c, c = off .. 12 - off (kernel row 12 - c), those inside [0, L)
                    const int c_lo = max(off, (K13 - 1) - n), c_hi = min(K13 - 1 - off, L - 1 - n + (K13 - 1));
                    if (c_lo <= c_hi) {
                        const unsigned s0 = (o + (unsigned)(n - (K13 - 1) + c_lo)) % SLOTS;
                        const int cnt = c_hi - c_lo + 1, cnt1 = min(cnt, (int)(SLOTS - s0)), cnt2 = cnt - cnt1;
                        const uint32_t id1 = umma::instr_desc(cnt1 * NBC), d1 = tmem + s0 * NBC;
                        const unsigned long long db = db0 + (unsigned long long)(c_lo * NBC);
                        if (cnt2 == 0 && off == 0) {
                            mma_row(d1, da, db, id1);
                        } else if (off == 0) {                   // the row slots wrap around at 32; the halves do not meet in tensor memory
                            mma_row(d1, da, db, id1);
                            mma_row(tmem, da, db + (unsigned long long)(cnt1 * NBC), umma::instr_desc(cnt2 * NBC));
                        } else {
                            const uint32_t id2 = umma::instr_desc(cnt2 * NBC);
                            for (int q = q_lo; q <= q_hi; ++q) {
                                const unsigned long long aq = da + (unsigned long long)q, bq = db + (unsigned long long)(q * (BQ_BYTES >> 4));
                                umma::mma_f16(d1, aq, bq, id1);
                                if (cnt2) umma::mma_f16(tmem, aq, bq + (unsigned long long)(cnt1 * NBC), id2);
                            }
                        }
                    }
                    umma::mma_commit(rowfree0 + 8 * slot);
                    if (n >= K13 - 1) umma::mma_commit(accfull0 + 8 * ((o + (unsigned)(n - (K13 - 1))) % SLOTS));
                    da += ROW_BYTES >> 4;
                    if (++slot == NRING) { slot = 0; full_parity ^= 1; da = da0; }
                }
                o += (unsigned)L;
                r += L;
            }
            umma::mma_commit(drained);                           // nothing is in flight when tensor memory is given back
            umma::mbar_wait_warp(drained, 0, p.ctrl, 0xE4000000u);
        } else if (warp == 13 && lane == 0 && p.copy_cc != 0) {
            // ======================= copy-through of the identity channels ==============================
            // Chunks of a power of two of pixels, the pixels of all images counted through, in a ring that is loaded up to one slot
            // ahead of the store.  Wide maps: a chunk goes with the row of a window that its first pixel lies in, dealt among the CTAs
            // of the same rows and other channels, not far ahead of the epilogue, so that the parts of a line reach L2
            // together.  Narrow maps: the chunks dealt in turn to the CTAs.  Each chunk is copied once: with chunks cut at the ends of
            // a window's part of a row, and whole ones copied for every part, 16 x (320x320) copied 1.75 times as much as there is
            // (stage 191 -> 150 us, 480x500 with 64 of 96 channels 133 -> 115, 900x500 with 144 of 192 109 -> 92).  Up to 8 rows
            // ahead 1920x1080 takes 183 us, 16 180, 24 or 32 178; chunks of 8 KB 186, of 4 KB 212.
            const unsigned bytes = (unsigned)(p.copy_cc * 2) << p.copy_shift, slot_bytes = (bytes + 127) & ~127u;
            int* pend = progress + 1;                        // first pixel of each slot's chunk
            bool alive = true;
            int load_slot = 0, store_slot = 0, lag = 0;      // lag: loads that are not stored yet
            unsigned parity = 0;
            // A wait that gave up ends the copying: what was asked for is waited for, but not stored, and nothing more is asked for.
            auto store = [&]() {                             // the oldest load
                const bool landed = mbar_wait(cfull0 + 8 * store_slot, parity, p.ctrl, 0xE5000000u);
                alive = alive && landed;
                if (alive) {
                    tma_store_2d(&map_cout, smem_u32(cring) + store_slot * slot_bytes, p.Ca, pend[store_slot]);
                    bulk_commit();
                }
                if (++store_slot == p.copy_slots) { store_slot = 0; parity ^= 1; }
                --lag;
            };
            auto copy = [&](unsigned chunk) {
                if (!alive) return;
                if (lag == p.copy_slots - 1) { store(); bulk_wait_read<1>(); if (!alive) return; }   // the store before that one has read its slot
                const int px = (int)(chunk << p.copy_shift);
                mbar_expect_tx(cfull0 + 8 * load_slot, bytes);
                tma_load_2d(smem_u32(cring) + load_slot * slot_bytes, &map_cin, cfull0 + 8 * load_slot, p.Ca, px);
                pend[load_slot] = px;
                if (++load_slot == p.copy_slots) load_slot = 0;
                ++lag;
            };
            if (p.copy_rows) {
                int o = 0;
                for (int r = r_begin; r < r_end && alive;) {
                    const int t = r / p.R, row0 = r - t * p.R, L = min(p.R - row0, r_end - r);
                    for (int yr = 0; yr < L && alive; ++yr) {
                        if ((row0 + yr) % p.octets != oct) continue;
                        alive = umma::wait_count(progress, o + yr - kCopyLead, p.ctrl, 0xE8000000u | (unsigned)(yr & 0xffff));
                        for (int f = t * WPX; f < t * WPX + WPX;) {
                            const int piece = f / p.pitch, x = f - piece * p.pitch, end = min(t * WPX + WPX, (piece + 1) * p.pitch);
                            const int b = piece / p.S, y = (piece - b * p.S) * p.R + row0 + yr, n = min(p.W - x, end - f);
                            if (piece < p.pieces && y < p.H && n > 0) {
                                const unsigned px = (unsigned)((b * p.H + y) * p.W + x), up = (1u << p.copy_shift) - 1;
                                for (unsigned k = (px + up) >> p.copy_shift; k < (px + (unsigned)n + up) >> p.copy_shift; ++k) copy(k);
                            }
                            f = end;
                        }
                    }
                    o += L;
                    r += L;
                }
            } else {
                for (unsigned k = blockIdx.x; k < (unsigned)p.copy_chunks && alive; k += gridDim.x) copy(k);
            }
            while (lag > 0) store();
            bulk_wait_all<0>();
        }
        __syncwarp();
    } else {
        // ======================= epilogue warps ========================================================
        reg_inc<kEpiRegs>();
        const int quad = warp & 3, e = warp >> 2, m = quad * 32 + lane;         // tensor-memory lane m, pixel 2m + e of the window
        const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(e * OCT);
        for (int s = 0; s < SLOTS; ++s) umma::tmem_zero16(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(s * NBC));
        umma::tmem_wait_st();
        umma::tc_fence_before();
        __syncwarp();
        if (lane == 0) {
            mbar_arrive(cleared);
#pragma unroll
            for (int n = 0; n < 5; ++n) mbar_arrive(rowfree0 + 8 * n);           // the 3x3 part reads rows 5 .. L + 6 of a window
        }

        if (!p.wait_first) pdl_wait_primary();                   // dk comes from the kernel before this one

        int g0 = 0, o = 0, first_bad = 0x7fffffff, last_bad = 0;                // rows with sums that are not finite
        bool alive = true;
        for (int r = r_begin; r < r_end;) {
            const int t = r / p.R, row0 = r - t * p.R, L = min(p.R - row0, r_end - r);
            const int f = t * WPX + 2 * m + e, piece = f / p.pitch, x = f - piece * p.pitch;
            const bool valid = piece < p.pieces && x < p.W;
            const int b0 = min(t * WPX / p.pitch, p.pieces - 1) / p.S, b1 = min((t * WPX + WPX - 1) / p.pitch, p.pieces - 1) / p.S, nimg = b1 - b0 + 1;
            const int b = valid ? piece / p.S : b0, y0 = (valid ? piece - b * p.S : 0) * p.R + row0;
            // ---- dk of the window's images for this CTA's channels
            epi_bar();                                           // everybody has the previous window's values
            for (int i = tid; i < nimg * 9 * OCT; i += kEpiThreads) {
                const int im = i / (9 * OCT), tap = i % (9 * OCT) / OCT, c = i % OCT;
                dks[i] = __ldcg(p.dk + ((size_t)(b0 + im) * p.Ca + oct * OCT + c) * 9 + tap);
            }
            epi_bar();
            u64 kk[9][4], d1[4], d2[4], c0[4];
            {
                const u64* src = reinterpret_cast<const u64*>(dks + (b - b0) * 9 * OCT);
#pragma unroll
                for (int i = 0; i < 9; ++i)
#pragma unroll
                    for (int v = 0; v < 4; ++v) kk[i][v] = src[i * 4 + v];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const float* bp = p.bias + (size_t)b * p.Ca + oct * OCT + 2 * v;
                    c0[v] = p.bias ? pack2(__ldcg(bp), __ldcg(bp + 1)) : 0ull;
                }
            }
            // pixels x - 1, x, x + 1 of a staged row: positions 2m + e + 5 .. 7
            const int pos = 2 * m + e + 5;
            const unsigned char* in0 = ring + (pos & 1) * PAR_BYTES + (pos >> 1) * 16;
            const unsigned char* in1 = ring + ((pos + 1) & 1) * PAR_BYTES + ((pos + 1) >> 1) * 16;
            // An input row is read once: it completes an output row and is added to the two that follow.
            auto load_row = [&](int g, uint4 (&v)[3]) {
                const int ro = (g % NRING) * ROW_BYTES;
                v[0] = *reinterpret_cast<const uint4*>(in0 + ro);
                v[1] = *reinterpret_cast<const uint4*>(in1 + ro);
                v[2] = *reinterpret_cast<const uint4*>(in0 + ro + 16);
            };
            auto add_row = [&](const uint4 (&v)[3], u64 (&s0)[4], u64 (&s1)[4], u64 (&s2)[4], int rows) {
#pragma unroll
                for (int bb = 0; bb < 3; ++bb) {
                    const unsigned w[4] = {v[bb].x, v[bb].y, v[bb].z, v[bb].w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const u64 fv = pack2(__uint_as_float(w[q] << 16), __uint_as_float(w[q] & 0xffff0000u));
                        if (rows > 1) fma2(s0[q], kk[6 + bb][q], fv);
                        if (rows > 0) fma2(s1[q], kk[3 + bb][q], fv);
                        fma2(s2[q], kk[bb][q], fv);
                    }
                }
            };
            __nv_bfloat16* dst = p.out + (((size_t)b * p.H + y0) * p.W + (valid ? x : 0)) * p.C + oct * OCT;
            const size_t row_stride = (size_t)p.W * p.C;
            // N output rows from yr on: one wait, N reads of tensor memory under way together, one signal
            auto rows = [&](auto count, int yr) {
                constexpr int N = decltype(count)::value;
                const int last = o + yr + N - 1, g = g0 + yr + 7;
                if (alive) alive = umma::mbar_wait_warp(accfull0 + 8 * (last % SLOTS), (unsigned)((last / SLOTS) & 1), p.ctrl, 0xE6000000u | (unsigned)(yr & 0xffff));
                if (alive) alive = umma::mbar_wait_warp(rowfull0 + 8 * ((g + N - 1) % NRING), (unsigned)(((g + N - 1) / NRING) & 1), p.ctrl, 0xE7000000u);   // long complete
                umma::tc_fence_after();
                uint32_t a[N][8];
                uint4 in[N][3];
#pragma unroll
                for (int i = 0; i < N; ++i) { tmem_ld8(lane_base + (uint32_t)((o + yr + i) % SLOTS * NBC), a[i]); load_row(g + i, in[i]); }
                if (yr == 0) {
                    u64 none[4];
                    uint4 v5[3], v6[3];
                    load_row(g - 2, v5); load_row(g - 1, v6);
#pragma unroll
                    for (int q = 0; q < 4; ++q) { d1[q] = d2[q] = c0[q]; none[q] = 0ull; }
                    add_row(v5, none, none, d1, 0);
                    add_row(v6, none, d1, d2, 1);
                }
                // rows that nobody needs any more: their slots may be filled again once the tensor core has read them too
                __syncwarp();
                if (yr == 0 && lane < 7 && (g0 > 0 || lane >= 5)) mbar_arrive(rowfree0 + 8 * ((g0 + lane) % NRING));
                if (lane < N) mbar_arrive(rowfree0 + 8 * ((g + lane) % NRING));
                if (yr + N == L && lane < 5) mbar_arrive(rowfree0 + 8 * ((g + N + lane) % NRING));
                u64 d0[N][4];
#pragma unroll
                for (int i = 0; i < N; ++i) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) { d0[i][q] = d1[q]; d1[q] = d2[q]; d2[q] = c0[q]; }
                    add_row(in[i], d0[i], d1, d2, 2);
                }
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < N; ++i) tmem_zero8(lane_base + (uint32_t)((o + yr + i) % SLOTS * NBC));
                float check = 0.f;
#pragma unroll
                for (int i = 0; i < N; ++i)
#pragma unroll
                    for (int q = 0; q < 8; ++q) check += __uint_as_float(a[i][q]);
                if (!(fabsf(check) < INFINITY) && valid) {
                    bool open = false;                       // not finite, and the 3x3 part does not make the result NaN anyway
#pragma unroll
                    for (int i = 0; i < N; ++i)
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            float lo, hi;
                            unpack2(d0[i][q], lo, hi);
                            open |= !(fabsf(__uint_as_float(a[i][2 * q])) < INFINITY) && lo == lo;
                            open |= !(fabsf(__uint_as_float(a[i][2 * q + 1])) < INFINITY) && hi == hi;
                        }
                    if (open) { first_bad = min(first_bad, o + yr); last_bad = o + yr + N; }
                }
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    uint32_t ov[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float lo, hi;
                        unpack2(d0[i][q], lo, hi);
                        ov[q] = pack_bf16x2(__uint_as_float(a[i][2 * q]) + lo, __uint_as_float(a[i][2 * q + 1]) + hi);
                    }
                    if (valid && y0 + yr + i < p.H) *reinterpret_cast<uint4*>(dst) = make_uint4(ov[0], ov[1], ov[2], ov[3]);
                    dst += row_stride;
                }
                __syncwarp();
                umma::tmem_wait_st();                            // the rows' columns are cleared
                umma::tc_fence_before();
                __syncwarp();
                if (lane < N) mbar_arrive(accfree0 + 8 * ((o + yr + lane) % SLOTS));
                if (tid == 0) umma::st_release_cta(progress, o + yr + N);
            };
            int yr = 0;
            for (; yr + 2 <= L; yr += 2) rows(std::integral_constant<int, 2>{}, yr);
            if (yr < L) rows(std::integral_constant<int, 1>{}, yr);
            g0 += L + K13 - 1;
            o += L;
            r += L;
        }
        asm volatile("bar.sync 4, %0;" ::"n"(128 + kEpiThreads) : "memory");    // the taps are in place
        __syncwarp();
        if (__any_sync(0xffffffffu, last_bad > 0))
            direct(p, reinterpret_cast<const uint4*>(smem + kOffTaps), oct, r_begin, r_end, 2 * m + e, first_bad, last_bad);
    }
    umma::tc_fence_before();
    __syncthreads();
    if (warp == 12) {
        umma::tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// ---- host side ------------------------------------------------------------------------------------
inline bool applies(int C, int Ca, int K, int dtype, int layout) {
    return K <= K13 && dtype == 1 /*bf16*/ && layout == kNHWC && Ca % CG == 0 && C % 8 == 0 && C - Ca <= 256;
}

// Whether the CTAs, as many groups of one for each eight channels as fit, take at least three quarters of the SMs.  Stage, us, mma.sync /
// this kernel: 304 channels (114 of 148 SMs) 90 / 84, 352 (132) 100 / 84, 512 (128) 139 / 131, 1024 (128) 140 / 133; but 400 (100) 109 / 131,
// 608 (76) 165 / 236, 800 (100) 110 / 134, 1200 (150 CTAs, two rounds) 166 / 259.
inline bool fills(int Ca, int sms) {
    const int octets = Ca / OCT, ctas = octets < sms ? sms / octets * octets : octets, rounds = (ctas + sms - 1) / sms;
    return 4LL * ctas >= 3LL * rounds * sms;
}

// Segments per image S, rows per segment R, rows per CTA Q: the fewest rows for the CTA that has most, a new window counted as
// five rows (its first and last twelve input rows feed only some of the columns).
struct Plan { int S, R, T, Q, parts; };
inline bool make_plan(int B, int Ca, int H, int W, Plan& best) {
    const int sms = sm_count(), octets = Ca / OCT, groups = octets < sms ? sms / octets : 1;
    long long best_cost = -1;
    for (int S = 1; S <= 64 && S <= H; ++S) {
        const int R = (H + S - 1) / S;
        if ((H + R - 1) / R != S) continue;
        const long long line = (long long)B * S * (W + GAPX) - GAPX, T = (line + WPX - 1) / WPX, rows = T * R;
        if (line > 0x3fffffffLL || rows > 0x3fffffffLL || (long long)B * H * W > 0x7fffffffLL) break;
        long long Q = (rows + groups - 1) / groups;
        if (Q < 2) Q = 2;
        const long long windows = R % Q == 0 ? 1 : (Q - 1) / R + 2, cost = Q + 5 * windows;
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = Plan{S, R, (int)T, (int)Q, (int)((rows + Q - 1) / Q)};
        }
    }
    return best_cost >= 0;
}

// Launches the kernel if the problem fits it: 0 on success, kNotApplicable otherwise, or an ESC_ERR_* code.
inline int try_launch(int B, int C, int Ca, int H, int W, int K, int dtype, int layout, const void* x, const void* w_large, const float* dk,
                      const float* bias, void* out, unsigned* ctrl, cudaStream_t st, bool dependent, int* launches, std::string* err,
                      bool skip_copy) {
    if (!applies(C, Ca, K, dtype, layout) || sm_count() <= 0) return kNotApplicable;
    Plan plan;
    if (!make_plan(B, Ca, H, W, plan)) return kNotApplicable;
    Params p = {};
    p.B = B; p.C = C; p.Ca = Ca; p.H = H; p.W = W; p.K = K;
    p.pitch = W + GAPX; p.S = plan.S; p.R = plan.R; p.pieces = B * plan.S;
    p.rows = plan.T * plan.R; p.Q = plan.Q; p.octets = Ca / OCT;
    const long long grid = (long long)plan.parts * p.octets;
    if (grid > 0x7fffffffLL) return kNotApplicable;
    p.x = static_cast<const __nv_bfloat16*>(x); p.w_large = static_cast<const __nv_bfloat16*>(w_large);
    p.dk = dk; p.bias = bias; p.out = static_cast<__nv_bfloat16*>(out); p.ctrl = ctrl;
    p.wait_first = dependent ? 0 : 1;
    const int cc = skip_copy ? 0 : C - Ca;
    CUtensorMap m_cin = {}, m_cout = {};
    if (cc > 0) {
        // the pixels of all images as one axis
        const long long px = (long long)B * H * W;
        if (px > 0x7fffffffLL) return kNotApplicable;
        p.copy_cc = cc;
        p.copy_shift = 8;
        while (p.copy_shift > 0 && cc * 2 << p.copy_shift > kCopyChunkBytes) --p.copy_shift;
        const int slot_bytes = ((cc * 2 << p.copy_shift) + 127) & ~127;
        p.copy_slots = std::min(kCopySlots, kCopyBytes / slot_bytes);
        p.copy_chunks = (int)((px + (1 << p.copy_shift) - 1) >> p.copy_shift);
        p.copy_rows = W >= WPX;
        EncodeTiledFn fn = encode_fn();
        if (!fn) return kNotApplicable;
        const cuuint64_t dims[2] = {(cuuint64_t)C, (cuuint64_t)px}, strides[1] = {(cuuint64_t)C * 2};
        const cuuint32_t box[2] = {(cuuint32_t)cc, 1u << p.copy_shift}, estr[2] = {1, 1};
        const void* base[2] = {x, out};
        for (int i = 0; i < 2; ++i)
            if (fn(i ? &m_cout : &m_cin, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base[i]), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return kNotApplicable;
    }
    static bool attr_set[kMaxDevices] = {};
    const int dev = current_device();
    if (dev < 0) return kNotApplicable;
    if (!attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(stencil_dw_umma_nhwc_bf16, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e != cudaSuccess) { (void)cudaGetLastError(); return kNotApplicable; }
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, stencil_dw_umma_nhwc_bf16, m_cin, m_cout, p);
    if (e != cudaSuccess) {
        char buf[256];
        snprintf(buf, sizeof buf, "stencil_dw_umma_nhwc_bf16 launch: %s (%s)", cudaGetErrorName(e), cudaGetErrorString(e));
        *err = buf;
        return 7;  // ESC_ERR_CUDA
    }
    ++*launches;
    return 0;
}

}}}  // namespace esc::tma::dwu
