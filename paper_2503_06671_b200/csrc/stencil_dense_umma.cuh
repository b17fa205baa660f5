// Dense large kernel (ESC paper, Section 3.2: LK in R^{13x13x16x16}; Eq. 4 line 3 with that LK) for NHWC bf16
// tensors with 16 attention channels on the fifth-generation tensor cores (tcgen05.mma, accumulators in
// tensor memory):
//
//   out[b,n,y,x] = sum_{k,i,j} w_dense[n,k,i,j] x[b,k,y+i-6,x+j-6]  +  sum_{i,j} dk[b,n,i,j] x[b,n,y+i-1,x+j-1]
//
// Formulation.  One INPUT row of a 128-pixel-wide strip, shifted by a tap column j, is the A operand
// (M = 128 pixels, K = 16 input channels) of ONE instruction whose B operand stacks all 13 kernel rows:
// B_j[k][(12 - i) * 16 + n] = w_dense[n][k][i][j], N = 13 x 16 = 208.  Column block c of the result belongs to
// output row (input row) - 6 + c, so the accumulators of 32 output rows live side by side in the 512 columns
// of tensor memory (row y in columns (y mod 32) * 16 ..) and an input row is used once -- 13 instructions,
// one per tap column -- and never again.  Per instruction 128 x 208 x 16 multiply-adds against 4 KB + 6.5 KB
// of shared-memory operands: the tensor pipe, not shared memory, is the bound, and nothing is unfolded.
// At the ends of a CTA's row range the instruction takes only the column blocks that exist (N = 16 .. 192).
//
// Operands are K-major.  A: a staged input row is [pixel][16 channels], 32 bytes per pixel, written by ONE TMA load
// per row (zero fill = the padding) with the 32-byte swizzle, and described to the tensor core with the same
// swizzle; the swizzle is a function of the shared-memory address, so the descriptor may start at ANY pixel and
// the tap column j is a shift of its start address by 32 * j bytes (verified output by output against
// a direct fp64 evaluation).  B: the weights, without swizzle ([half of K][row][8 k-values], rows 16 bytes apart).
// What bounds it: an instruction takes 104 cycles at N = 208 and 39 to 96 for the 12 input rows above and below a CTA's range,
// which feed only some of the 13 column blocks: with 13 output rows per CTA (640x360 on 148 SMs) 20.6 k cycles for 17.6 k
// cycles' worth of results; larger maps give longer ranges.  Its operands are 10.7 KB of shared memory per 104 cycles, so what
// else moves through shared memory (the copy-through, the 3x3 part) is felt: 120 cycles in place of 104.  640x360 alone, cold:
// 36.9 -> 28.7 us (B table 12 k -> 8.3 k cycles, of them 4 k until the weights have landed; 137 -> 120 cycles per instruction by
// the way the issuing warp waits; 3x3 part read row by row); 64 patches of 64x64: 53 -> 44 us.
//
// Roles (224 threads, one CTA per SM, each CTA one range of rows of one strip):
//   warp 0   lane 0 requests input rows by TMA (one load per row) into a ring of 16; the warp allocates and frees tensor memory
//   warp 1   issues the instructions (one elected lane) and commits them to mbarriers (ring slot consumed / output row complete)
//   warps 2-5  epilogue: tcgen05.ld of a finished row (one pixel per thread, 16 channels), constants, the dynamic 3x3
//            kernel in fp32 on the CUDA cores from the same ring, one rounding to bf16, 32-byte store;
//            the row's columns are cleared for their next user.
//   warp 6   lane 0 copies the identity channels of the CTA's rows, TMA in / TMA out through a ring of two slots.
#pragma once
#include "stencil_generic.cuh"
#include "stencil_tma.cuh"

namespace esc { namespace tma { namespace umma {

constexpr int MW = 128;                       // output pixels per strip row = M of the instruction
constexpr int SPX = 144;                      // staged pixels per row: 128 + 12, padded to keep half-rows 128-byte aligned
constexpr int HALF_BYTES = SPX * 16;
constexpr int ROW_BYTES = 2 * HALF_BYTES;     // one staged row: SPX pixels x 32 bytes
constexpr int NRING = 16;                     // input rows in flight / kept for the 3x3 part
constexpr int NBLK = K13;                     // column blocks of 16 (kernel rows) in a B operand
constexpr int BHALF_BYTES = NBLK * CG * 16;   // 3,328: one tap column, one channel half: [208 rows][8 k]
constexpr int BJ_BYTES = 2 * BHALF_BYTES + 16;   // tap columns 16 bytes apart modulo 128: the table's stores spread over the banks
constexpr int B_BYTES = (K13 * BJ_BYTES + 127) / 128 * 128;   // 86,784
constexpr int SLOTS = 32;                     // output rows whose accumulators fit tensor memory (512 columns)
constexpr int kThreads = 224;                 // producer, issuer, four epilogue warps, copy-through warp
constexpr int kEpiThreads = 128;
constexpr int kCopySlotBytes = 16384, kCopySlots = 2;
constexpr unsigned kPollLimit = 1u << 22;
constexpr int kMiscBytes = 1024;               // dk, progress word, tensor-memory base
constexpr int kBarBytes = 1024;                // 2 * NRING + SLOTS + kCopySlots + 1 mbarriers
constexpr int kCopyRingOffset = NRING * ROW_BYTES + B_BYTES + kMiscBytes + kBarBytes;
constexpr size_t kSmemBytes = (size_t)kCopyRingOffset + kCopySlots * kCopySlotBytes;
static_assert((2 * NRING + SLOTS + kCopySlots + 1) * 8 <= kBarBytes && kCopyRingOffset % 128 == 0, "barriers fit; the copy ring is a TMA destination");
// While the B table is built the weights as they are lie behind the first three rows of the ring (eleven of sixteen leading
// channels) and in the copy ring (five).
constexpr int kRawRows = 3, kRawSplit = 11, kRawChannelBytes = CG * K13 * K13 * 2;
static_assert(kRawSplit * kRawChannelBytes <= (NRING - kRawRows) * ROW_BYTES && (CG - kRawSplit) * kRawChannelBytes <= kCopySlots * kCopySlotBytes, "staging");
static_assert(HALF_BYTES % 128 == 0, "TMA destinations are 128-byte aligned");

struct Params {
    int B, C, H, W;
    int strips, segs, seg_rows;       // per image: strips of 128 pixels x row ranges of seg_rows rows
    const __nv_bfloat16* w_dense;     // [16][16][KK][KK]  (output channel, input channel, row, column)
    int KK;                           // odd, at most 13: a smaller kernel is the middle of the table, and only that is multiplied
    int raw_bulk;                     // w_dense is 16-byte aligned: it is staged with bulk copies
    int flip;                         // the gradient's form: channel axes of w_dense swapped, taps rotated by 180 degrees
    const float* dk;                  // [B][16][9]
    const float* bias;                // [B][16] added to every output of an (image, channel), or nullptr
    __nv_bfloat16* out;
    int out_c;                        // channels of out; its layout: NHWC, or NCHW (x then is the packed map of 16 channels)
    int out_nchw;
    unsigned* ctrl;
    int wait_first;
    int copy_cc, copy_pw;             // identity channels; pixels of a strip row per copy chunk (0: nothing to copy)
};

// Shared-memory matrix descriptor, K-major, no swizzle: 8 rows x 16 bytes are contiguous (rows 16 bytes apart),
// the next 8 rows follow `sbo` bytes on, the second half of K (k = 8..15) `lbo` bytes on.
__device__ __forceinline__ unsigned long long smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (unsigned long long)((addr >> 4) & 0x3FFFu) | ((unsigned long long)((lbo >> 4) & 0x3FFFu) << 16) |
           ((unsigned long long)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// A operand: K-major with the 32-byte swizzle -- a row (pixel) is 32 contiguous bytes, its two 16-byte halves swapped
// where bit 7 of the shared-memory address is set -- exactly what a TMA load with CU_TENSOR_MAP_SWIZZLE_32B writes for
// a 32-byte inner box.  Rows are 32 bytes apart, 8-row groups 256 bytes.
__device__ __forceinline__ unsigned long long smem_desc_sw32(uint32_t addr) {
    return (unsigned long long)((addr >> 4) & 0x3FFFu) | (1ull << 16) | ((unsigned long long)(256u >> 4) << 32) | (1ull << 46) |
           (6ull << 61);
}
// Instruction descriptor of kind::f16: D fp32, A and B bf16, both K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t instr_desc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(MW >> 4) << 24);
}
// Executed by a whole warp with the same arguments in every lane; one elected lane issues.  (Issued from a branch that a single
// lane takes, an instruction occupied the issuing thread for about 112 cycles whatever its N; this way it costs what the
// tensor pipe takes: 39 cycles for N = 16, 48 for 64, N / 2 from 128 on.)
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, unsigned long long da, unsigned long long db, uint32_t idesc) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, 1, 0;\n\telect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(da), "l"(db), "r"(idesc) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {         // the same elected lane: it tracks what that lane issued
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
                 "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar) : "memory");
}
// The issuing warp's bounded wait, by all its lanes: a phase that is complete costs about 85 cycles this way, hidden behind the
// instructions in flight; one lane asking for the warp costs 280 (the branch, and what the compiler no longer takes for uniform).
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, unsigned parity, unsigned* ctrl, unsigned where) {
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (__all_sync(0xffffffffu, ok)) return true;
    for (unsigned n = 0; n < kSpinLimit; ++n) {
        ok = mbar_try_wait(bar, parity);
        if (__all_sync(0xffffffffu, ok)) return true;
    }
    if (ctrl && (threadIdx.x & 31) == 0) { atomicExch(ctrl, kDevTimeout); atomicExch(ctrl + 1, where); }
    return false;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_zero16(uint32_t taddr) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};"
                 ::"r"(taddr), "r"(0u) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ int ld_acquire_cta(const int* p) {
    int v;
    asm volatile("ld.acquire.cta.shared.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_cta(int* p, int v) {
    asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
// One lane's bounded wait for a count that another warp of the CTA publishes; records where it gave up, as mbar_wait does.
__device__ __forceinline__ bool wait_count(const int* count, int need, unsigned* ctrl, unsigned where) {
    for (unsigned polls = 0; polls < kPollLimit; ++polls) {
        if (ld_acquire_cta(count) >= need) return true;
        __nanosleep(200);
    }
    if (ctrl) { atomicExch(ctrl, kDevTimeout); atomicExch(ctrl + 1, where); }
    return false;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, unsigned bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// kSmall: K < 13.  Of its own, so that the unrolled issue loop of the full size keeps its constants (with both in one kernel 640x360
// took 28.8 us for 28.2).
template <bool kSmall>
__global__ void __launch_bounds__(kThreads, 1)
stencil_dense_umma_nhwc_bf16(const __grid_constant__ CUtensorMap map_half, const __grid_constant__ CUtensorMap map_cin,
                             const __grid_constant__ CUtensorMap map_cout, const Params p)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* ring = smem;                                             // [NRING][SPX pixels][32 bytes], 32-byte swizzle
    unsigned char* btab = smem + NRING * ROW_BYTES;                         // [13 tap columns][2 halves][208 rows][16 bytes]
    float* dks = reinterpret_cast<float*>(btab + B_BYTES);                  // [9 taps][16 channels]
    int* prog = reinterpret_cast<int*>(dks + 9 * CG);                       // output rows the epilogue has finished
    int* aborted = prog + 1;
    uint32_t* tmem_base_slot = reinterpret_cast<uint32_t*>(prog + 2);
    u64* bars = reinterpret_cast<u64*>(btab + B_BYTES + 1024);
    const uint32_t rowfull0 = smem_u32(bars), rowdone0 = rowfull0 + 8 * NRING, accfull0 = rowdone0 + 8 * NRING,
                   cfull0 = accfull0 + 8 * SLOTS, wfull = cfull0 + 8 * kCopySlots;
    unsigned char* cring = smem + kCopyRingOffset;

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // warp: known to be uniform
    if (tid == 0) {
        for (int s = 0; s < NRING; ++s) { mbar_init(rowfull0 + 8 * s, 1); mbar_init(rowdone0 + 8 * s, 1); }
        for (int s = 0; s < SLOTS; ++s) mbar_init(accfull0 + 8 * s, 1);
        for (int s = 0; s < kCopySlots; ++s) mbar_init(cfull0 + 8 * s, 1);
        mbar_init(wfull, 1);
        *prog = 0; *aborted = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {                                        // all 512 columns of this SM's tensor memory (one CTA per SM)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_base_slot, 0);
    if (p.wait_first) pdl_wait_primary();
    pdl_launch_dependents();

    // ---- this CTA's rows: image b, strip sx, rows [ya, yb) -------------------------------------------
    unsigned u = blockIdx.x;
    const int seg = (int)(u % (unsigned)p.segs); u /= (unsigned)p.segs;
    const int sx = (int)(u % (unsigned)p.strips);
    const int b = (int)(u / (unsigned)p.strips);
    const int ya = seg * p.seg_rows, yb = min(p.H, ya + p.seg_rows), L = yb - ya;
    const int x0 = sx * MW;
    const int n_in = L + K13 - 1;                           // input rows ya - 6 .. yb + 5, index n = row - (ya - 6)

    auto request_rows = [&](int n0, int n1) {
        for (int n = n0; n < min(n_in, n1); ++n) {
            mbar_expect_tx(rowfull0 + 8 * n, ROW_BYTES);
            tma_load_4d(smem_u32(ring + (size_t)n * ROW_BYTES), &map_half, rowfull0 + 8 * n, 0, x0 - P6, ya - P6 + n, b);
        }
    };
    // ---- B operands: btab[j][half][(12 - i) * 16 + n][k % 8] = w[n][half * 8 + k % 8][i][j] -----------------------
    // The weights come as they are with two bulk copies, behind the first rows of the ring and in the copy ring.  Then a warp
    // takes 32 consecutive taps of an output channel n and half of the input channels: eight 2-byte reads per lane, 64
    // contiguous bytes over the warp, and one 16-byte store.
    const int taps = p.KK * p.KK, chan = CG * taps;                              // elements of one leading channel of w_dense
    if (p.raw_bulk) {
        if (tid == 0) {
            mbar_expect_tx(wfull, (unsigned)(CG * chan * 2));
            bulk_load(smem_u32(ring + kRawRows * ROW_BYTES), p.w_dense, (unsigned)(kRawSplit * chan * 2), wfull);
            bulk_load(smem_u32(cring), p.w_dense + kRawSplit * chan, (unsigned)((CG - kRawSplit) * chan * 2), wfull);
            request_rows(0, kRawRows);
        }
    }
    // clear the accumulators: every instruction accumulates, a row's columns are cleared again after it is read
    if (warp >= 2) {
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        for (int s = 0; s < SLOTS; ++s) tmem_zero16(lane_base + (uint32_t)(s * CG));
        tmem_wait_st();
    }
    if (p.raw_bulk) mbar_wait(wfull, 0, p.ctrl, 0xD7000000u);
    {
        // a lane's place in the table depends on its tap alone: worked out once per 32 taps, not per item
        const int off = (K13 - p.KK) / 2;
        auto build = [&](auto value) {                                            // value(leading channel, offset behind it)
            for (int t0 = 0; t0 < taps; t0 += 32) {
                const int t = t0 + lane, tc = min(t, taps - 1), r = tc / p.KK, c = tc - r * p.KK;
                const int i = off + (p.flip ? p.KK - 1 - r : r), j = off + (p.flip ? p.KK - 1 - c : c);
                unsigned char* dst = btab + j * BJ_BYTES + (K13 - 1 - i) * CG * 16;
                constexpr int kWarps = kThreads / 32, kItems = (2 * CG + kWarps - 1) / kWarps;
                unsigned v[kItems][8];
#pragma unroll
                for (int u = 0; u < kItems; ++u) {                                // all reads of the 32 taps, then the stores
                    const int nh = min(warp + u * kWarps, 2 * CG - 1), n = nh >> 1, h = nh & 1;
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        v[u][q] = p.flip ? value(8 * h + q, n * taps + tc) : value(n, (8 * h + q) * taps + tc);
                }
#pragma unroll
                for (int u = 0; u < kItems; ++u) {
                    const int nh = warp + u * kWarps;
                    if (nh < 2 * CG && t < taps)
                        *reinterpret_cast<uint4*>(dst + (nh & 1) * BHALF_BYTES + (nh >> 1) * 16) =
                            make_uint4(v[u][0] | (v[u][1] << 16), v[u][2] | (v[u][3] << 16), v[u][4] | (v[u][5] << 16), v[u][6] | (v[u][7] << 16));
                }
            }
        };
        if (p.raw_bulk) {
            const unsigned short* lo = reinterpret_cast<const unsigned short*>(ring + kRawRows * ROW_BYTES);
            const int hi = (int)((cring - (ring + kRawRows * ROW_BYTES)) / 2) - kRawSplit * chan;   // where channel 0 would lie for the second piece
            build([&](int a, int o) { return (unsigned)lo[a * chan + o + (a < kRawSplit ? 0 : hi)]; });
        } else {
            build([&](int a, int o) { return (unsigned)__ldg(reinterpret_cast<const unsigned short*>(p.w_dense) + a * chan + o); });
        }
    }
    fence_async_smem();                                     // the B table is read through the async proxy
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0) request_rows(p.raw_bulk ? kRawRows : 0, NRING);

    if (warp == 0) {
        // ======================= input rows by TMA (the first sixteen are under way) ===================
        if (lane == 0) {
            bool alive = true;
            for (int n = NRING; n < n_in && alive; ++n) {
                const int slot = n % NRING;
                // the slot's previous row (n - 16) must have been consumed by the tensor cores and, if the 3x3 part reads it, by
                // the epilogue: rows 5 and 6 with output row 0, row q >= 7 with output row q - 7
                alive = mbar_wait(rowdone0 + 8 * slot, (unsigned)(((n - NRING) / NRING) & 1), p.ctrl, 0xD0000000u | (unsigned)n);
                const int need = n < NRING + 5 ? 0 : min(max(1, n - NRING - 6), L);
                unsigned polls = 0;
                while (alive && ld_acquire_cta(prog) < need) {
                    __nanosleep(64);
                    if (++polls > kPollLimit || ld_acquire_cta(aborted)) alive = false;
                }
                if (!alive) { if (p.ctrl) { atomicExch(p.ctrl, kDevTimeout); atomicExch(p.ctrl + 1, 0xD1000000u | (unsigned)n); } st_release_cta(aborted, 1); break; }
                const uint32_t dst = smem_u32(ring + (size_t)slot * ROW_BYTES), bar = rowfull0 + 8 * slot;
                mbar_expect_tx(bar, ROW_BYTES);
                tma_load_4d(dst, &map_half, bar, 0, x0 - P6, ya - P6 + n, b);
            }
        }
    } else if (warp == 1) {
        // ======================= tensor-core instructions =============================================
        bool alive = true;
        const uint32_t ring_a = smem_u32(ring), btab_a = smem_u32(btab);
        const int off = kSmall ? (K13 - p.KK) / 2 : 0;                         // first tap column and kernel row of a smaller kernel
        for (int n = 0; n < n_in; ++n) {
            const int slot = n % NRING;
            alive = mbar_wait_warp(rowfull0 + 8 * slot, (unsigned)((n / NRING) & 1), p.ctrl, 0xD2000000u | (unsigned)n);
            // the columns of the output row this input row opens (n, if it exists) were cleared by the epilogue of row n - 32
            if (n >= SLOTS && n < L) {
                unsigned polls = 0;
                while (alive && __any_sync(0xffffffffu, ld_acquire_cta(prog) < n - SLOTS + 1)) {
                    __nanosleep(64);
                    if (++polls > kPollLimit || __any_sync(0xffffffffu, ld_acquire_cta(aborted))) alive = false;
                }
            }
            if (!alive) {
                if (lane == 0) { if (p.ctrl) { atomicExch(p.ctrl, kDevTimeout); atomicExch(p.ctrl + 1, 0xD3000000u | (unsigned)n); } st_release_cta(aborted, 1); }
                break;
            }
            tc_fence_after();
            // input row n feeds output rows n - 12 + c, c = off .. 12 - off (kernel row 12 - c), those inside [0, L)
            const int c_lo = max(off, (K13 - 1) - n), c_hi = min(K13 - 1 - off, L - 1 - n + (K13 - 1));
            if (c_lo <= c_hi) {
                const int cnt = c_hi - c_lo + 1, s0 = (n - (K13 - 1) + c_lo) % SLOTS;
                const int cnt1 = min(cnt, SLOTS - s0), cnt2 = cnt - cnt1;          // the row slots wrap around at 32
                const uint32_t id1 = instr_desc(cnt1 * CG);
                unsigned long long da = smem_desc_sw32(ring_a + (uint32_t)(slot * ROW_BYTES));
                unsigned long long db = smem_desc(btab_a + (uint32_t)(c_lo * CG * 16), BHALF_BYTES, 128);
                if (!kSmall && cnt2 == 0) {
#pragma unroll
                    for (int j = 0; j < K13; ++j)                              // one pixel (32 bytes) and one tap column further on
                        mma_f16(tmem + (uint32_t)(s0 * CG), da + (unsigned long long)(2 * j), db + (unsigned long long)(j * (BJ_BYTES >> 4)), id1);
                } else {
                    const uint32_t id2 = instr_desc(cnt2 * CG);
                    if (kSmall) { da += 2 * off; db += off * (BJ_BYTES >> 4); }
                    for (int j = 0; j < (kSmall ? p.KK : K13); ++j) {
                        mma_f16(tmem + (uint32_t)(s0 * CG), da, db, id1);
                        if (!kSmall || cnt2) mma_f16(tmem, da, db + (unsigned long long)(cnt1 * CG), id2);
                        da += 2; db += BJ_BYTES >> 4;
                    }
                }
            }
            mma_commit(rowdone0 + 8 * slot);                                   // arrives when the instructions above have read the row
            if (n >= K13 - 1) mma_commit(accfull0 + 8 * ((n - (K13 - 1)) % SLOTS));   // output row n - 12 is complete
        }
    } else if (warp == 6) {
        // ======================= copy-through of the identity channels: TMA in, TMA out ================
        // this CTA's rows of its strip, a strip row (or a part of it) per chunk, through a ring of two slots
        if (lane == 0 && p.copy_cc != 0) {
            bool alive = true;
            const int per_row = MW / p.copy_pw, chunks = L * per_row;
            const unsigned bytes = (unsigned)(p.copy_cc * p.copy_pw * 2);
            auto coords = [&](int ch, int& cx, int& cy) { cy = ya + ch / per_row; cx = x0 + (ch % per_row) * p.copy_pw; };
            auto issue = [&](int ch, int n) {                               // the n-th chunk that is copied
                int cx, cy; coords(ch, cx, cy);
                const int slot = n % kCopySlots;
                mbar_expect_tx(cfull0 + 8 * slot, bytes);
                tma_load_4d(smem_u32(cring + slot * kCopySlotBytes), &map_cin, cfull0 + 8 * slot, CG, cx, cy, b);
            };
            // chunks wholly outside the image (right of W) are skipped, so slots and phases go by the count of those that are not
            auto inside = [&](int ch) { int cx, cy; coords(ch, cx, cy); return cx < p.W; };
            int next = 0;
            while (next < chunks && !inside(next)) ++next;
            if (next < chunks) issue(next, 0);
            int cur = next;
            for (int n = 0; cur < chunks; ++n) {
                int nx = cur + 1;
                while (nx < chunks && !inside(nx)) ++nx;
                if (nx < chunks) {
                    bulk_wait_read<0>();                                    // the store that last used the other slot has read it
                    issue(nx, n + 1);
                }
                if (alive) alive = mbar_wait(cfull0 + 8 * (n % kCopySlots), (unsigned)((n / kCopySlots) & 1), p.ctrl, 0xD6000000u | (unsigned)cur);
                int cx, cy; coords(cur, cx, cy);
                tma_store_4d(&map_cout, smem_u32(cring + (n % kCopySlots) * kCopySlotBytes), CG, cx, cy, b);
                bulk_commit();
                cur = nx;
            }
            bulk_wait_all<0>();
        }
    } else {
        // ======================= epilogue: one pixel per thread =======================================
        const int et = tid - 64, m = ((warp & 3) * 32) + lane;              // tensor-memory lane = pixel of the strip row
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        if (!p.wait_first) pdl_wait_primary();                               // dk comes from the kernel before this one
        for (int e = et; e < 9 * CG; e += kEpiThreads) dks[e] = __ldcg(p.dk + ((size_t)b * CG + (e % CG)) * 9 + e / CG);
        asm volatile("bar.sync 2, %0;" ::"n"(kEpiThreads) : "memory");
        // the constant of this (image, channel), added to the accumulators
        float c0[CG];
#pragma unroll
        for (int c = 0; c < CG; ++c) c0[c] = p.bias ? __ldcg(p.bias + (size_t)b * CG + c) : 0.f;
        bool alive = true;
        const int x = x0 + m;
        // Dynamic 3x3 kernel, depth-wise, fp32 (Eq. 4 line 3, second term).  Output row yr reads input rows yr + 5 .. yr + 7
        // of the ring, pixels m + 5 .. m + 7 of the staged row.  An input row is read once: it completes one output row and
        // is added to the two that follow, whose sums wait in registers (shared-memory bandwidth is what the instructions
        // live on: 10.7 KB per 104 cycles).
        float d1[CG], d2[CG];                                                // output rows yr + 1, yr + 2 so far
#pragma unroll
        for (int c = 0; c < CG; ++c) d1[c] = d2[c] = 0.f;
        auto add_row = [&](int n, float (&s0)[CG], float (&s1)[CG], float (&s2)[CG], int rows) {
            // input row n into s0 (its kernel row 2), s1 (1), s2 (0); `rows` says which of the first two exist
            const int rslot = n % NRING;
            const unsigned char* rowp = ring + (size_t)rslot * ROW_BYTES;
#pragma unroll
            for (int bb = 0; bb < 3; ++bb) {
                // the pixel's two 16-byte halves are swapped where bit 7 of its address is set (32-byte swizzle)
                const int px = m + 5 + bb, sw = ((rslot * (ROW_BYTES / 128) + (px >> 2)) & 1) * 16;
                const uint4 lo = *reinterpret_cast<const uint4*>(rowp + (size_t)px * 32 + sw);
                const uint4 hi = *reinterpret_cast<const uint4*>(rowp + (size_t)px * 32 + (16 - sw));
                float f[16];
                unpack16<__nv_bfloat16>(lo, f);
                unpack16<__nv_bfloat16>(hi, f + 8);
                const float4* k2 = reinterpret_cast<const float4*>(dks + (6 + bb) * CG);
                const float4* k1 = reinterpret_cast<const float4*>(dks + (3 + bb) * CG);
                const float4* k0 = reinterpret_cast<const float4*>(dks + bb * CG);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (rows > 1) {
                        const float4 d = k2[q];
                        s0[4 * q] = fmaf(d.x, f[4 * q], s0[4 * q]); s0[4 * q + 1] = fmaf(d.y, f[4 * q + 1], s0[4 * q + 1]);
                        s0[4 * q + 2] = fmaf(d.z, f[4 * q + 2], s0[4 * q + 2]); s0[4 * q + 3] = fmaf(d.w, f[4 * q + 3], s0[4 * q + 3]);
                    }
                    if (rows > 0) {
                        const float4 d = k1[q];
                        s1[4 * q] = fmaf(d.x, f[4 * q], s1[4 * q]); s1[4 * q + 1] = fmaf(d.y, f[4 * q + 1], s1[4 * q + 1]);
                        s1[4 * q + 2] = fmaf(d.z, f[4 * q + 2], s1[4 * q + 2]); s1[4 * q + 3] = fmaf(d.w, f[4 * q + 3], s1[4 * q + 3]);
                    }
                    const float4 d = k0[q];
                    s2[4 * q] = fmaf(d.x, f[4 * q], s2[4 * q]); s2[4 * q + 1] = fmaf(d.y, f[4 * q + 1], s2[4 * q + 1]);
                    s2[4 * q + 2] = fmaf(d.z, f[4 * q + 2], s2[4 * q + 2]); s2[4 * q + 3] = fmaf(d.w, f[4 * q + 3], s2[4 * q + 3]);
                }
            }
        };
        for (int yr = 0; yr < L; ++yr) {
            const int slot = yr % SLOTS;
            // one lane asks (a wait that all 32 lanes execute costs the warp over a hundred cycles)
            if (lane == 0 && alive) alive = mbar_wait(accfull0 + 8 * slot, (unsigned)((yr / SLOTS) & 1), p.ctrl, 0xD4000000u | (unsigned)yr);
            if (lane == 0 && !alive) st_release_cta(aborted, 1);
            __syncwarp();
            tc_fence_after();
            uint32_t r[16];
            tmem_ld16(lane_base + (uint32_t)(slot * CG), r);
            tmem_zero16(lane_base + (uint32_t)(slot * CG));
            float d0[CG];                                                    // this output row's 3x3 sums so far
            if (yr == 0) {
                float none[CG];
#pragma unroll
                for (int c = 0; c < CG; ++c) none[c] = 0.f;
                add_row(5, none, none, d1, 0);
                add_row(6, none, d1, d2, 1);
            }
#pragma unroll
            for (int c = 0; c < CG; ++c) { d0[c] = d1[c]; d1[c] = d2[c]; d2[c] = 0.f; }
            add_row(yr + 7, d0, d1, d2, 2);
            float acc[CG];
#pragma unroll
            for (int c = 0; c < CG; ++c) acc[c] = __uint_as_float(r[c]) + (d0[c] + c0[c]);
            if (x < p.W && p.out_nchw) {                                      // 64 contiguous bytes of a plane per warp and store
                const size_t plane = (size_t)p.H * p.W;
                __nv_bfloat16* dst = p.out + (size_t)b * p.out_c * plane + (size_t)(ya + yr) * p.W + x;
#pragma unroll
                for (int c = 0; c < CG; ++c) dst[c * plane] = __float2bfloat16_rn(acc[c]);
            } else if (x < p.W) {
                uint32_t o[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const __nv_bfloat162 h2 = __floats2bfloat162_rn(acc[2 * q], acc[2 * q + 1]);
                    o[q] = *reinterpret_cast<const uint32_t*>(&h2);
                }
                uint4* dst = reinterpret_cast<uint4*>(p.out + (((size_t)b * p.H + ya + yr) * p.W + x) * p.out_c);
                dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
                dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
            }
            tmem_wait_st();                                                   // the row's columns are cleared
            tc_fence_before();
            asm volatile("bar.sync 2, %0;" ::"n"(kEpiThreads) : "memory");
            if (et == 0) st_release_cta(prog, yr + 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// ---- host side ------------------------------------------------------------------------------------
// [B][H][W][C] bf16 as a 4-D map {C, W, H, B} with a box of 8 channels x SPX pixels x 1 row.
inline int try_launch_dense_umma(int B, int C, int Ca, int H, int W, int K, int dtype, int layout, const void* x,
                                 const void* w_dense, const float* dk, void* out, unsigned* ctrl, cudaStream_t st,
                                 bool dependent, int* launches, std::string* err, const float* bias = nullptr, bool flip = false,
                                 int out_c = 0, bool out_nchw = false) {
    if (K > K13 || dtype != 1 /*bf16*/ || layout != kNHWC || Ca != CG || C % 8 != 0) return kNotApplicable;
    if ((reinterpret_cast<uintptr_t>(w_dense) & 1) != 0) return kNotApplicable;
    const int sms = sm_count();
    if (sms <= 0) return kNotApplicable;
    Params p;
    p.B = B; p.C = C; p.H = H; p.W = W;
    p.strips = (W + MW - 1) / MW;
    // row ranges: about one CTA per SM, at least 8 rows each (12 more are read above and below a range)
    long long want = (long long)sms / ((long long)B * p.strips);
    if (want < 1) want = 1;
    int rows = (int)((H + want - 1) / want);
    if (rows < 8) rows = H < 8 ? H : 8;
    p.seg_rows = rows;
    p.segs = (H + rows - 1) / rows;
    const long long ctas = (long long)B * p.strips * p.segs;
    if (ctas > 0x3fffffffLL) return kNotApplicable;
    p.w_dense = static_cast<const __nv_bfloat16*>(w_dense);
    p.dk = dk; p.out = static_cast<__nv_bfloat16*>(out); p.ctrl = ctrl;
    p.out_c = out_c > 0 ? out_c : C; p.out_nchw = out_nchw ? 1 : 0;
    p.wait_first = dependent ? 0 : 1;
    p.raw_bulk = (reinterpret_cast<uintptr_t>(w_dense) & 15) == 0 ? 1 : 0;
    p.KK = K; p.flip = flip ? 1 : 0; p.bias = bias;
    const int cc = C - Ca;
    p.copy_cc = cc; p.copy_pw = 0;
    if (cc > 256) return kNotApplicable;
    if (cc > 0) {
        int pw = MW;
        while (pw > 8 && cc * 2 * pw > kCopySlotBytes) pw >>= 1;
        if (cc * 2 * pw > kCopySlotBytes) return kNotApplicable;
        p.copy_pw = pw;
    }
    CUtensorMap m_half, m_cin, m_cout;
    {   // one staged row per load: 16 channels x SPX pixels, written with the 32-byte swizzle the A descriptor names
        EncodeTiledFn fn = encode_fn();
        if (!fn) return kNotApplicable;
        const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
        const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
        const cuuint32_t box[4] = {(cuuint32_t)CG, (cuuint32_t)SPX, 1, 1};
        const cuuint32_t estr[4] = {1, 1, 1, 1};
        if (fn(&m_half, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_64B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return kNotApplicable;
    }
    if (cc > 0) {
        if (!make_map(&m_cin, x, B, C, H, W, cc, p.copy_pw, 1)) return kNotApplicable;
        if (!make_map(&m_cout, out, B, C, H, W, cc, p.copy_pw, 1)) return kNotApplicable;
    } else {
        m_cin = m_half; m_cout = m_half;
    }
    const bool small = K < K13;
    auto* kernel = small ? stencil_dense_umma_nhwc_bf16<true> : stencil_dense_umma_nhwc_bf16<false>;
    static bool attr_set[2][kMaxDevices] = {};
    const int dev = current_device();
    if (dev < 0) return kNotApplicable;
    if (!attr_set[small][dev]) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
        if (e != cudaSuccess) { (void)cudaGetLastError(); return kNotApplicable; }
        attr_set[small][dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, m_half, m_cin, m_cout, p);
    if (e != cudaSuccess) {
        char buf[256];
        snprintf(buf, sizeof buf, "stencil_dense_umma_nhwc_bf16 launch: %s (%s)", cudaGetErrorName(e), cudaGetErrorString(e));
        *err = buf;
        return 7;  // ESC_ERR_CUDA
    }
    ++*launches;
    return 0;
}

}}}  // namespace esc::tma::umma
