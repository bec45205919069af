// 3x3 convolution as an implicit GEMM on the 5th-generation tensor cores
// (tcgen05.mma, accumulators in TMEM, operands staged by TMA), BF16 or
// FP8-E4M3 operands with FP32 accumulation, and the weight gradient of the
// same convolution (k_wgrad_tc, below).
//
// The convolution (k_conv_fold) folds the three kernel ROWS into the MMA N
// dimension; see the comment above the kernel for the schedule.  Each
// activation row (64 channels) is 128 bytes (bf16) or 64 bytes (fp8), stored
// with the matching TMA swizzle (128B / 64B) so that the shared-memory
// descriptors address it directly; out-of-range parts of a TMA box are
// zero-filled, which is the convolution's zero padding.  All 9 taps of the
// layer's weights stay resident in shared memory for the whole persistent CTA.
//
// Warp roles (640 threads, one CTA per SM):
//   warp 0: TMA producer (weights once, then one A box per input row through
//           an S-stage ring)
//   warp 1: TMEM allocator and MMA issuer (all lanes form the operands, one issues)
//   warps 2-17: epilogue; warp w reads TMEM lanes 32 (w % 4) .. + 31 and 16 of
//           the 64 output channels: dequantisation (fp8), bias, ReLU /
//           residual / mask / FP32 partial sum / bilinear skip, BF16 results
//           written into the staging slot (swizzled) and sent out by one TMA
//           store per tile, or FP32 results stored directly
//   warp 18: residual prefetch into one of three or four staging slots
//   warp 19: output TMA stores from the staging slots
// Every wait is bounded (no hardware barrier inside the role loops): on
// timeout the kernel sets *err, all roles unwind, TMEM is freed, and the host
// reports MRS_ERR_TIMEOUT.
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <queue>
#include <type_traits>
#include <utility>
#include <vector>

#include "conv_tc.cuh"

namespace mrs {
namespace {

constexpr int kEpiWarps = 16;                  // 4 per TMEM lane quarter
constexpr int kResWarp = 2 + kEpiWarps;        // residual-prefetch warp
constexpr int kStoreWarp = kResWarp + 1;       // output-store warp
constexpr int kThreads = 32 * (kStoreWarp + 1);  // A-TMA, MMA, epilogue, residual, store warps
// residual / output staging slots; epilogue warps of one row.  kAlt: the warps
// form two groups that take alternate rows (each slot then belongs to one group)
constexpr int fold_slots(bool alt) { return alt ? 4 : 3; }
constexpr int fold_row_warps(bool alt) { return alt ? kEpiWarps / 2 : kEpiWarps; }
constexpr long long kTimeoutCycles = 4000000000LL;   // ~2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// as above, but the thread may be suspended (up to `ns` nanoseconds) until the
// phase completes instead of spinning in a loop that takes issue slots from
// the working warps
__device__ __forceinline__ bool mbar_try_wait_sleep(uint64_t* bar, uint32_t parity, uint32_t ns)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(ns)
        : "memory");
    return ok != 0;
}
// bounded wait; false if this or another role gave up.  Each poll lets the
// hardware suspend the thread (1 ms limit) until the phase completes; the
// error word and the clock are consulted between polls
__device__ __forceinline__ bool mbar_wait_limit(uint64_t* bar, uint32_t parity, int* err,
                                                long long limit_cycles, uint32_t sleep_ns)
{
    if (mbar_try_wait(bar, parity)) return true;
    long long t0 = clock64();
    for (;;) {
        if (mbar_try_wait_sleep(bar, parity, sleep_ns)) return true;
        if (*(volatile int*)err) return false;
        if (clock64() - t0 > limit_cycles) {
            atomicExch(err, 1);
            return false;
        }
    }
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* err)
{
    return mbar_wait_limit(bar, parity, err, kTimeoutCycles, 1000000u);
}

// every lane polls; the answer is the same for the whole warp.  (Lane 0 polling
// for the warp, a shuffle and a second look by all lanes took some 500 cycles
// more a wait; polling without the suspending wait takes issue slots and made
// the convolutions 4 to 10% slower.)
__device__ __forceinline__ bool mbar_wait_all(uint64_t* bar, uint32_t parity, int* err)
{
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, err));
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1,
                                            int c2, int c3, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
        "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int c0, int c1,
                                            uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}

// tcgen05 shared-memory matrix descriptor, K-major, swizzled rows of
// `row_bytes` (128 -> SWIZZLE_128B, 64 -> SWIZZLE_64B), 8-row groups.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, int row_bytes)
{
    uint64_t d = (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;                                  // LBO (unused when swizzled)
    d |= (uint64_t)((8 * row_bytes) >> 4) << 32;              // SBO: next 8-row group
    d |= (uint64_t)1 << 46;                                  // descriptor version
    d |= (uint64_t)(row_bytes == 128 ? 2 : 4) << 61;         // swizzle mode
    return d;
}

// executed by the lane whose `leader` is set; the whole warp runs the code that
// forms the operands, so that they stay in uniform registers
__device__ __forceinline__ void mma_f16(bool leader, uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc,
                                        uint32_t accum)
{
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accum), "r"((uint32_t)leader));
}
__device__ __forceinline__ void mma_f8(bool leader, uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc,
                                       uint32_t accum)
{
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accum), "r"((uint32_t)leader));
}
__device__ __forceinline__ void mma_commit(uint64_t* bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15,%16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// bilinear x s upsampling of LRHS at HR pixel (x, y): half-pixel centres,
// clamped at the borders
__device__ __forceinline__ void bilinear(const float* __restrict__ lr, int h, int w, int s, int x,
                                         int y, float out[3])
{
    float inv = 1.0f / (float)s;
    float sy = fmaxf(((float)y + 0.5f) * inv - 0.5f, 0.0f);
    float sx = fmaxf(((float)x + 0.5f) * inv - 0.5f, 0.0f);
    int y0 = min((int)sy, h - 1), x0 = min((int)sx, w - 1);
    int y1 = min(y0 + 1, h - 1), x1 = min(x0 + 1, w - 1);
    float ly = sy - (float)y0, lx = sx - (float)x0;
    const float* a = lr + ((size_t)y0 * w + x0) * 3;
    const float* b = lr + ((size_t)y0 * w + x1) * 3;
    const float* c = lr + ((size_t)y1 * w + x0) * 3;
    const float* d = lr + ((size_t)y1 * w + x1) * 3;
    for (int k = 0; k < 3; ++k) {
        float top = __ldg(a + k) * (1.0f - lx) + __ldg(b + k) * lx;
        float bot = __ldg(c + k) * (1.0f - lx) + __ldg(d + k) * lx;
        out[k] = top * (1.0f - ly) + bot * ly;
    }
}

__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, const void* src, int c0,
                                             int c1, int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
            (uint64_t)map),
        "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Work split: the layer is T = N * XB * H tiles (one tile = one output row of
// one 128-pixel column strip; N counts groups of tc_images images, narrow
// images sharing the strip), flattened as f = (n * XB + xb) * H + y.  CTA c
// takes the contiguous run [T c / G, T (c + 1) / G), cut at strip boundaries
// into pieces; a piece is a run of rows of one strip, streamed through the
// input-row ring with its own halo rows.  piece_rows returns the piece that
// starts at f (< f1) and advances f past it.
__device__ __forceinline__ void piece_rows(long long& f, long long f1, int XB, int H, int& xb,
                                           int& n, int& y0, int& y1)
{
    const long long k = f / H;
    y0 = (int)(f - k * H);
    const long long left = f1 - f;
    y1 = (int)((long long)y0 + left < (long long)H ? (long long)y0 + left : (long long)H);
    xb = (int)(k % XB);
    n = (int)(k / XB);
    f += y1 - y0;
}

// byte offset of 16-byte chunk j of row m in a SWIZZLE_128B tile
__device__ __forceinline__ uint32_t sw128(int m, int j) { return m * 128 + ((j ^ (m & 7)) << 4); }

// ---------------------------------------------------------------------------
// 3x3 convolution with the kernel ROWS folded into the MMA N dimension.
//
// Input row r of a column strip meets the weights of all three kernel rows in
// one MMA: B = [w(dy 0, dx); w(dy 1, dx); w(dy 2, dx)] (3 NOUT rows) gives
// column block j = the contribution of row r to output row r + 1 - j.  The
// accumulators of consecutive output rows sit in consecutive NOUT-column
// slots of TMEM in DEcreasing order (slot(t) = (-t) mod NS for the CTA's t-th
// output row), so one MMA with D at slot(r + 1) adds to output rows r + 1, r,
// r - 1 at once; where the three slots wrap around the end of TMEM the MMA is
// split in two.  The column taps dx are row-shifted A descriptors into one
// 130-pixel box per input row (x0 - 1 .. x0 + 128), so an output pixel's sum
// is complete in its own TMEM lane: the epilogue reads one NOUT-column slot
// per output row, without cross-lane shuffles, and zeroes it for reuse (every
// MMA accumulates onto zeroed TMEM).  Each input row is consumed by the 12
// MMAs (3 dx x 4 K steps) issued right after it lands and then released, so
// the whole ring is prefetch depth.  An output tile is 128 pixels of one row.
// FP8 operands (kind::f8f6f4, K = 32 per MMA, 64-byte rows with the 64B
// swizzle) follow the same schedule with one-row (64-byte) descriptor shifts,
// per-output-channel weight scales and a per-layer activation scale; their
// BF16 outputs also leave an FP8 copy for the next layer's operand.
// Consecutive MMAs into different D regions do not pipeline, so the wrap
// rows issue all MMAs of one region before the other.
constexpr int kFoldTile = 128;               // output pixels per tile (= MMA M)
constexpr int kFoldABox = kFoldTile + 2;     // input pixels per row box (one halo each side)
constexpr int kFoldMaxRows = 6;              // output rows per sub-piece of a multi-chunk conv
// bytes per activation row of the operand type, ring slot (1024-aligned)
constexpr int fold_rowb(int oper) { return oper == TC_BF16 ? 128 : 64; }
constexpr int fold_aslot(int oper) { return ((kFoldABox * fold_rowb(oper) + 1023) / 1024) * 1024; }

template <int NOUT, int OPER, bool kAlt> size_t fold_smem_bytes(int stages)
{
    constexpr int kSlots = fold_slots(kAlt);
    return 1024 + ((9 * NOUT * fold_rowb(OPER) + 1023) & ~1023) + (size_t)stages * fold_aslot(OPER) +
           (size_t)kSlots * kFoldTile * 128 + 2 * 64 * 4 + 8 * (2 * stages + 2 + 2 * (512 / NOUT) + 3 * kSlots) + 16;
}

__device__ __forceinline__ const TcConvArgs& more_of(const TcConvArgs& a) { return a; }
__device__ __forceinline__ TcConvArgs more_of(const TcConvBase&) { return TcConvArgs{}; }

// kImages: several images a tile (tc_images).  kMore: also groups, masked sums
// and second results (TcConvArgs::ng, mask, op2).  Variants, because the tests
// for them cost a layer that has neither: 3% on an image of 256 x 128 (fusion
// network 171 against 166 us in BF16, 165 against 159 in FP8), 2% on a large one.
// kAlt: the epilogue's two groups have two rows' time for one row's latency, but
// each row takes twice as long (a warp has 32 of its 64 channels): for CTAs with
// rows enough (see tc_conv3x3).
template <int NOUT, int OPER, bool kImages, bool kMore, bool kAlt>
__global__ void __launch_bounds__(kThreads, 1)
    k_conv_fold(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
                const __grid_constant__ CUtensorMap tmap_res,
                const __grid_constant__ CUtensorMap tmap_out,
                const std::conditional_t<kMore, TcConvArgs, TcConvBase> a, int stages)
{
    const auto& more = more_of(a);
    constexpr int kSlots = fold_slots(kAlt), kRowWarps = fold_row_warps(kAlt);
    constexpr int NS = 512 / NOUT;                            // TMEM accumulator slots
    constexpr int ROWB = fold_rowb(OPER);                     // bytes per operand row
    constexpr int ASLOT = fold_aslot(OPER);
    constexpr int KSTEPS = OPER == TC_BF16 ? 4 : 2;           // MMAs per 64 input channels (K 16 / 32)
    constexpr int WBYTES = 9 * NOUT * ROWB;
    constexpr int SBYTES = kFoldTile * 128;
    constexpr int BROWS = 3 * NOUT;                           // B rows per dx: dy 0, 1, 2
    constexpr uint32_t kTmemCols = 512;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sW = smem;
    uint8_t* sA = smem + ((WBYTES + 1023) & ~1023);
    uint8_t* sS = sA + stages * ASLOT;
    float* sBias = (float*)(sS + kSlots * SBYTES);
    float* sScale = sBias + 64;                               // FP8: dequantisation factor by channel
    uint64_t* bars = (uint64_t*)(sScale + 64);
    uint64_t* full = bars;
    uint64_t* empty = bars + stages;
    uint64_t* wbar = bars + 2 * stages;                       // weights landed
    uint64_t* wempty = wbar + 1;                              // weight buffer free
    uint64_t* tfull = wempty + 1;                             // [NS] output row complete
    uint64_t* sfree = tfull + NS;                             // [NS] slot read and zeroed
    uint64_t* rfull = sfree + NS;
    uint64_t* rempty = rfull + kSlots;
    uint64_t* edone = rempty + kSlots;
    uint32_t* tslot = (uint32_t*)(edone + kSlots);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int XB = (a.W + kFoldTile - 1) / kFoldTile;
    const int im = kImages ? tc_images(a.N, a.W) : 1, pitch = a.W + 2;      // images per tile, their rows apart
    const long long T = (long long)((a.N + im - 1) / im) * XB * a.H;
    // the CTA's group (of ng convolutions of the same input) and its place in it
    const int ng = kMore && more.ng > 1 ? more.ng : 1, group = kMore ? (int)blockIdx.x * ng / (int)gridDim.x : 0;
    const int cta0 = kMore ? (group * (int)gridDim.x + ng - 1) / ng : 0;
    const int cta1 = kMore ? ((group + 1) * (int)gridDim.x + ng - 1) / ng : (int)gridDim.x;
    const long long f0 = T * ((int)blockIdx.x - cta0) / (cta1 - cta0), f1 = T * ((int)blockIdx.x - cta0 + 1) / (cta1 - cta0);
    const int mode = kMore && ng > 1 ? more.gmode[min(group, 3)] : a.mode, w_row0 = a.w_row0 + 9 * NOUT * group;
    const CUtensorMap* mres = kMore && ng > 1 ? more.gmaps + 2 * group : &tmap_res;
    const CUtensorMap* mout = kMore && ng > 1 ? more.gmaps + 2 * group + 1 : &tmap_out;
    const bool bf_out = mode == TC_RELU_BF16 || mode == TC_RESID_BF16 ||
                        mode == TC_LIN_BF16 || mode == TC_MASK_BF16 ||
                        mode == TC_RESRELU_BF16;
    const bool loads_res = mode == TC_RESID_BF16 || mode == TC_MASK_BF16 ||
                           mode == TC_RESRELU_BF16;
    // a bf16 result that nobody reads (fp8 operands: only the fp8 copy) is
    // neither staged nor stored
    const bool stores_bf = bf_out && !(a.fp8_only && a.out_fp8);

    if (threadIdx.x == 0) {
        for (int i = 0; i < stages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        mbar_init(wbar, 1);
        mbar_init(wempty, 1);
        for (int i = 0; i < NS; ++i) {
            mbar_init(&tfull[i], 1);
            mbar_init(&sfree[i], kRowWarps);
        }
        for (int i = 0; i < kSlots; ++i) {
            mbar_init(&rfull[i], 1);
            mbar_init(&rempty[i], 1);
            mbar_init(&edone[i], kRowWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (threadIdx.x < 64) sBias[threadIdx.x] = threadIdx.x < NOUT ? a.bias[threadIdx.x + (kMore && more.gbias ? 64 * group : 0)] : 0.0f;
    if (OPER == TC_FP8 && threadIdx.x < NOUT) sScale[threadIdx.x] = a.wscale[threadIdx.x] * a.xscale;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tslot)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *(volatile uint32_t*)tslot;
    // every accumulator slot starts at zero (the MMAs always accumulate)
    if (warp >= 2 && warp < 2 + kEpiWarps) {
        const int q = warp & 3, grp = (warp - 2) >> 2;
        uint32_t z[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) z[e] = 0u;
        for (int c = grp * 16; c < (int)kTmemCols; c += 64) tmem_st16(tmem + ((uint32_t)(q * 32) << 16) + c, z);
        tmem_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // programmatic dependent launch: the next conv may be scheduled now; every
    // access to data of the previous kernel in the stream waits for its
    // completion (griddepcontrol.wait).  The weights and biases come from
    // before the previous kernel (packed at set-up or by a non-overlapping
    // kernel), so the weight load is issued before that wait.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (!(warp == 0 && lane == 0)) asm volatile("griddepcontrol.wait;" ::: "memory");

    // A convolution over kc > 1 inputs (64-channel chunks, each its own tensor
    // map in a.amaps, weights chunk after chunk in tmap_w) accumulates all
    // chunks in TMEM: a piece is cut into sub-pieces of at most kMaxRows
    // output rows, whose accumulators all stay live while the chunks pass
    // (chunk-major order; the weight buffer is reloaded per chunk).
    const int kc = a.kc > 1 ? a.kc : 1;
    const int maxr = kc > 1 ? kFoldMaxRows : (1 << 30);
    if (warp == 0) {
        if (lane == 0) {
            // A producer: per (sub-piece, chunk), input rows ys-1 .. ye, 130
            // pixels from x0-1; the first weights are loaded here, before the
            // wait for the previous kernel
            mbar_expect_tx(wbar, WBYTES);
            // tap (dy, dx) at B row (3 dx + dy) NOUT: per dx the three kernel rows are contiguous
            for (int t = 0; t < 9; ++t)
                tma_load_2d(sW + ((t % 3) * 3 + t / 3) * NOUT * ROWB, &tmap_w, 0, w_row0 + t * NOUT, wbar);
            asm volatile("griddepcontrol.wait;" ::: "memory");
            const uint32_t abytes = (uint32_t)((im > 1 ? im * pitch : kFoldABox) * ROWB);
            uint32_t it = 0;
            bool ok = true;
            for (long long f = f0; ok && f < f1;) {
                int xb, n, y0, y1;
                piece_rows(f, f1, XB, a.H, xb, n, y0, y1);
                for (int ys = y0; ok && ys < y1; ys += maxr) {
                    const int ye = min(y1, ys + maxr);
                    for (int j = 0; ok && j < kc; ++j) {
                        const CUtensorMap* am = kc > 1 ? a.amaps + j : &tmap_x;
                        // a map in global memory, written by the host before
                        // the launch: acquire it for the tensor-map proxy
                        if (kc > 1)
                            asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(
                                             (uint64_t)am)
                                         : "memory");
                        for (int r = ys - 1; r <= ye; ++r, ++it) {
                            int s = it % stages;
                            if (!mbar_wait(&empty[s], ((it / stages) & 1) ^ 1, a.err)) { ok = false; break; }
                            mbar_expect_tx(&full[s], abytes);
                            tma_load_4d(sA + s * ASLOT, am, 0, xb * kFoldTile - 1, r, n * im, &full[s]);
                        }
                    }
                }
            }
        } else if (lane == 16 && kc > 1) {
            // weight loader for every (sub-piece, chunk) pass after the first:
            // waits for the MMAs of the previous pass to finish with the buffer
            uint32_t k = 0;
            bool ok = true;
            for (long long f = f0; ok && f < f1;) {
                int xb, n, y0, y1;
                piece_rows(f, f1, XB, a.H, xb, n, y0, y1);
                for (int ys = y0; ok && ys < y1; ys += maxr)
                    for (int j = 0; ok && j < kc; ++j, ++k) {
                        if (k == 0) continue;
                        if (!mbar_wait(wempty, (k - 1) & 1, a.err)) { ok = false; break; }
                        mbar_expect_tx(wbar, WBYTES);
                        for (int t = 0; t < 9; ++t)
                            tma_load_2d(sW + ((t % 3) * 3 + t / 3) * NOUT * ROWB, &tmap_w, 0,
                                        a.w_row0 + (j * 9 + t) * NOUT, wbar);
                    }
            }
        }
    } else if (warp == kResWarp) {
        if (lane == 0) {
            if (kMore && ng > 1 && loads_res)
                asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"((uint64_t)mres) : "memory");
            uint32_t j = 0;
            bool ok = true;
            for (long long f = f0; ok && f < f1;) {
                int xb, n, y0, y1;
                piece_rows(f, f1, XB, a.H, xb, n, y0, y1);
                for (int y = y0; y < y1; ++y, ++j) {
                    uint32_t slot = j % kSlots, use = j / kSlots;
                    if (!mbar_wait(&rempty[slot], (use & 1) ^ 1, a.err)) { ok = false; break; }
                    if (loads_res) {
                        mbar_expect_tx(&rfull[slot], im > 1 ? (uint32_t)(im * pitch * 128) : (uint32_t)SBYTES);
                        tma_load_4d(sS + slot * SBYTES, mres, 0, xb * kFoldTile, y, n * im, &rfull[slot]);
                    } else {
                        mbar_arrive(&rfull[slot]);
                    }
                }
            }
        }
    } else if (warp == kStoreWarp) {
        if (lane == 0) {
            if (kMore && ng > 1 && stores_bf)
                asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"((uint64_t)mout) : "memory");
            uint32_t j = 0;
            bool ok = true;
            for (long long f = f0; ok && f < f1;) {
                int xb, n, y0, y1;
                piece_rows(f, f1, XB, a.H, xb, n, y0, y1);
                for (int y = y0; y < y1; ++y, ++j) {
                    uint32_t slot = j % kSlots, use = j / kSlots;
                    if (!mbar_wait(&edone[slot], use & 1, a.err)) { ok = false; break; }
                    if (stores_bf) {
                        tma_store_4d(mout, sS + slot * SBYTES, 0, xb * kFoldTile, y, n * im);
                        bulk_commit();
                        bulk_wait_read0();
                    }
                    mbar_arrive(&rempty[slot]);
                }
            }
            bulk_wait_all();
        }
    } else if (warp == 1) {
        // MMA issuer: for each input row r of a piece, the blocks j whose output
        // row r + 1 - j lies in the piece, in one MMA per (dx, K step) (two
        // where the slots wrap)
        {
            const bool leader = lane == 0;
            bool ok = true;
            uint32_t it = 0, k = 0;
            int s = 0;                                          // ring slot of row `it`
            uint32_t ph = 0;                                    // its fill phase parity
            long long t0 = 0;                                   // CTA output-row counter at sub-piece start
            const uint32_t wbase = smem_u32(sW), abase = smem_u32(sA);
            // descriptors differ only in their start-address field (address / 16,
            // bits 0-13): each MMA's pair is a base pair plus a constant offset
            const uint64_t adesc0 = sdesc(abase, ROWB), bdesc0 = sdesc(wbase, ROWB);
            for (long long f = f0; ok && f < f1;) {
                int xb, n, y0, y1;
                piece_rows(f, f1, XB, a.H, xb, n, y0, y1);
                for (int ys = y0; ok && ys < y1; ys += maxr) {
                  const int ye = min(y1, ys + maxr);
                  for (int j = 0; ok && j < kc; ++j, ++k) {
                    // weights of this pass (loaded once when kc == 1)
                    if ((kc > 1 || k == 0) && !mbar_wait_all(wbar, k & 1, a.err)) { ok = false; break; }
                    for (int r = ys - 1; ok && r <= ye; ++r, ++it, s = (s + 1 == stages ? 0 : s + 1),
                                                        ph ^= (s == 0 ? 1u : 0u)) {
                        const int jlo = max(0, r + 2 - ye), jhi = min(2, r + 1 - ys);
                        // output row of block jb: CTA counter t0 + (r + 1 - jb - ys)
                        const long long tlo = t0 + (r + 1 - jlo - ys);   // newest row (highest t)
                        if (jlo == 0 && j == 0) {
                            // block 0 of the first chunk starts output row tlo: its slot must
                            // have been read and zeroed by the epilogue of row tlo - NS
                            const int sl = (int)(tlo % NS);
                            const uint32_t use = (uint32_t)(tlo / NS);
                            if (!mbar_wait_all(&sfree[(NS - sl) % NS], (use & 1) ^ 1, a.err)) { ok = false; break; }
                        }
                        if (!mbar_wait_all(&full[s], ph, a.err)) { ok = false; break; }
                        tc_fence_after();
                        const int nb = jhi - jlo + 1;
                        const int c0 = (int)((NS - (int)(tlo % NS)) % NS);   // slot of block jlo
                        const int n1 = min(nb, NS - c0);                    // blocks before the wrap
                        // all MMAs of one D region back to back: the region before
                        // the wrap, then (rarely) the one after it; consecutive
                        // MMAs into different regions do not pipeline
                        for (int part = 0; part < (n1 < nb ? 2 : 1); ++part) {
                            const uint32_t dcol = part ? 0u : (uint32_t)(c0 * NOUT);
                            const int b0 = part ? n1 : 0, nbp = part ? nb - n1 : n1;
                            const uint32_t idesc = (1u << 4) | ((OPER == TC_BF16 ? 1u : 0u) << 7) |
                                                   ((OPER == TC_BF16 ? 1u : 0u) << 10) |
                                                   ((uint32_t)((nbp * NOUT) >> 3) << 17) |
                                                   ((uint32_t)(kFoldTile >> 4) << 24);
                            const uint64_t arow = adesc0 + (uint64_t)((s * ASLOT) >> 4);
                            const uint64_t brow0 = bdesc0 + (uint64_t)(((jlo + b0) * NOUT * ROWB) >> 4);
#pragma unroll
                            for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
                                for (int kk = 0; kk < KSTEPS; ++kk) {
                                    const uint64_t ad = arow + (uint64_t)((dx * ROWB + kk * 32) >> 4);
                                    const uint64_t bd = brow0 + (uint64_t)((dx * BROWS * ROWB + kk * 32) >> 4);
                                    if (OPER == TC_BF16) mma_f16(leader, tmem + dcol, ad, bd, idesc, 1u);
                                    else mma_f8(leader, tmem + dcol, ad, bd, idesc, 1u);
                                }
                            }
                        }
                        if (leader) mma_commit(&empty[s]);
                        if (jhi == 2 && j == kc - 1) {
                            // output row r - 1 (block 2 of the last chunk) is complete
                            const long long td = tlo - (2 - jlo);
                            if (leader) mma_commit(&tfull[(NS - (int)(td % NS)) % NS]);
                        }
                    }
                    // the weight buffer is free once this pass's MMAs complete
                    if (kc > 1 && leader) mma_commit(wempty);
                  }
                  t0 += ye - ys;
                }
            }
        }
    } else {
        // epilogue: warp w reads TMEM lanes 32 q .. 32 q + 31 (output pixels
        // x0 + 32 q + lane) and channels [ch0, ch0 + 16 kBlk) of the finished
        // output row's slot, then zeroes them.  (FP8: the factors come from shared
        // memory and values are converted in pairs; loading a factor and converting
        // value by value bound the row: the network at 512 x 288 0.255 -> 0.238 ms)
        const int q = warp & 3, grp = (warp - 2) >> 2;
        constexpr int kBlk = kAlt && NOUT >= 64 ? 2 : 1;       // 16-channel blocks of a warp
        const int ch0 = (kAlt ? grp >> 1 : grp) * 16 * kBlk;
        const int j = q * 32 + lane;
        const bool active = ch0 < NOUT;
        // the lane's image in its tile and pixel in the strip
        const bool masked = kMore && more.mask && group == ng - 1 && mode == TC_RESID_BF16;
        const __nv_bfloat16* aux = (const __nv_bfloat16*)(masked ? more.mask : kMore && more.op2 ? more.x2 : nullptr);
        const int ji = im > 1 ? j / pitch : 0, jx = j - ji * pitch;
        uint32_t lt = 0;
        bool stop = false;
        for (long long f = f0; !stop && f < f1;) {
          int xb, n, y0, y1;
          piece_rows(f, f1, XB, a.H, xb, n, y0, y1);
          for (int y = y0; y < y1; ++y, ++lt) {
            if (kAlt && (int)(lt & 1) != (grp & 1)) continue;
            const int sl = (int)((NS - (int)(lt % NS)) % NS);
            const uint32_t use = lt / NS;
            const uint32_t slot = lt % kSlots, suse = lt / kSlots;
            const int x = xb * kFoldTile + jx, img = n * im + ji;
            const bool valid = x < a.W && ji < im && img < a.N;
            const size_t p = valid ? ((size_t)img * a.H + y) * a.W + x : 0;
            // the mask's or second result's operand, read while the row is computed
            uint4 ux[2 * kBlk];
            if (kMore && aux && active && valid)
#pragma unroll
                for (int e = 0; e < 2 * kBlk; ++e) ux[e] = *(const uint4*)(aux + p * 64 + ch0 + 8 * e);
            // the staging slot first: it is usually free, and off the row's critical path
            if (!mbar_wait_all(&rfull[slot], suse & 1, a.err)) { stop = true; break; }
            if (!mbar_wait_all(&tfull[sl], use & 1, a.err)) { stop = true; break; }
            tc_fence_after();
            uint8_t* srow = sS + slot * SBYTES;
            if (active) {
              const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(sl * NOUT);
              uint32_t rr[kBlk][16];
#pragma unroll
              for (int blk = 0; blk < kBlk; ++blk) tmem_ld16(trow + ch0 + 16 * blk, rr[blk]);
              tmem_wait_ld();
#pragma unroll
              for (int blk = 0; blk < kBlk; ++blk) {
                const int c0 = ch0 + 16 * blk;
                const uint32_t taddr = trow + c0;
                const uint4* u2 = ux + 2 * blk;
                const uint32_t (&r0)[16] = rr[blk];
                uint32_t z[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) z[e] = 0u;
                tmem_st16(taddr, z);
                float v[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) v[e] = __uint_as_float(r0[e]);
                if (OPER == TC_FP8) {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        v[e] = v[e] * sScale[c0 + e];
                }
                if (bf_out) {
                    float o[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) o[e] = v[e] + sBias[c0 + e];
                    if (mode == TC_RELU_BF16) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) o[e] = fmaxf(o[e], 0.0f);
                    } else if (mode == TC_MASK_BF16) {
#pragma unroll
                        for (int jj = 0; jj < 2; ++jj) {
                            uint4 u = *(const uint4*)(srow + sw128(j, c0 / 8 + jj));
                            const __nv_bfloat162* h2 = (const __nv_bfloat162*)&u;
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                float2 fv = __bfloat1622float2(h2[e]);
                                if (!(fv.x > 0.0f)) o[8 * jj + 2 * e] = 0.0f;
                                if (!(fv.y > 0.0f)) o[8 * jj + 2 * e + 1] = 0.0f;
                            }
                        }
                    } else if (mode == TC_RESID_BF16 || mode == TC_RESRELU_BF16) {
                        const bool rl = mode == TC_RESRELU_BF16;
#pragma unroll
                        for (int jj = 0; jj < 2; ++jj) {
                            uint4 u = *(const uint4*)(srow + sw128(j, c0 / 8 + jj));
                            const __nv_bfloat162* h2 = (const __nv_bfloat162*)&u;
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                float2 fv = __bfloat1622float2(h2[e]);
                                float o0 = o[8 * jj + 2 * e], o1 = o[8 * jj + 2 * e + 1];
                                if (rl) { o0 = fmaxf(o0, 0.0f); o1 = fmaxf(o1, 0.0f); }
                                o[8 * jj + 2 * e] = fv.x + o0;
                                o[8 * jj + 2 * e + 1] = fv.y + o1;
                            }
                        }
                        if (kMore && masked && valid) {
                            const __nv_bfloat16* h = (const __nv_bfloat16*)u2;
#pragma unroll
                            for (int e = 0; e < 16; ++e)
                                if (!(__bfloat162float(h[e]) > 0.0f)) o[e] = 0.0f;
                        }
                    }
                    if (kMore && more.op2 && valid) {
                        const __nv_bfloat162* h2 = (const __nv_bfloat162*)u2;
                        __nv_bfloat162 t2[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const float2 x2 = __bfloat1622float2(h2[e]);
                            float2 b2 = __bfloat1622float2(__floats2bfloat162_rn(o[2 * e], o[2 * e + 1]));
                            if (more.op2 == 1) {
                                if (!(x2.x > 0.0f)) b2.x = 0.0f;
                                if (!(x2.y > 0.0f)) b2.y = 0.0f;
                            } else {
                                b2.x = x2.x + b2.x;
                                b2.y = x2.y + b2.y;
                            }
                            t2[e] = __floats2bfloat162_rn(b2.x, b2.y);
                        }
                        __nv_bfloat16* o2 = (__nv_bfloat16*)more.out2 + p * 64 + c0;
                        *(uint4*)o2 = ((const uint4*)t2)[0];
                        *(uint4*)(o2 + 8) = ((const uint4*)t2)[1];
                    }
                    if (stores_bf) {
#pragma unroll
                        for (int jj = 0; jj < 2; ++jj) {
                            uint4 u;
                            __nv_bfloat162* h2 = (__nv_bfloat162*)&u;
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                h2[e] = __floats2bfloat162_rn(o[8 * jj + 2 * e], o[8 * jj + 2 * e + 1]);
                            *(uint4*)(srow + sw128(j, c0 / 8 + jj)) = u;
                        }
                    }
                    if (a.out_fp8 && valid) {
                        // the next layer's FP8 operand row
                        uint4 u;
                        __nv_fp8x2_storage_t* b8 = (__nv_fp8x2_storage_t*)&u;
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            b8[e] = __nv_cvt_float2_to_fp8x2(make_float2(o[2 * e] * a.out_fp8_inv_scale,
                                                                         o[2 * e + 1] * a.out_fp8_inv_scale),
                                                             __NV_SATFINITE, __NV_E4M3);
                        *(uint4*)((uint8_t*)a.out_fp8 + p * 64 + c0) = u;
                    }
                } else if (valid) {
                    if (mode == TC_FINAL_F32) {
                        if (c0 == 0) {
                            float up[3];
                            bilinear(a.lrhs + (size_t)img * (a.H / a.scale) * (a.W / a.scale) * 3,
                                     a.H / a.scale, a.W / a.scale, a.scale, x, y, up);
                            float* op = (float*)a.out + p * 3;
                            for (int c = 0; c < 3; ++c) op[c] = (v[c] + sBias[c]) + up[c];
                        }
                    } else if (a.cout == 64 && ((uintptr_t)a.out & 15) == 0) {
                        float4* op = (float4*)((float*)a.out + p * 64 + c0);
#pragma unroll
                        for (int i4 = 0; i4 < 4; ++i4) {
                            float4 t = make_float4(v[4 * i4] + sBias[c0 + 4 * i4],
                                                   v[4 * i4 + 1] + sBias[c0 + 4 * i4 + 1],
                                                   v[4 * i4 + 2] + sBias[c0 + 4 * i4 + 2],
                                                   v[4 * i4 + 3] + sBias[c0 + 4 * i4 + 3]);
                            if (a.relu) {
                                t.x = fmaxf(t.x, 0.0f); t.y = fmaxf(t.y, 0.0f);
                                t.z = fmaxf(t.z, 0.0f); t.w = fmaxf(t.w, 0.0f);
                            }
                            op[i4] = t;
                        }
                    } else {
                        float* op = (float*)a.out + p * a.cout;
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            if (c0 + e < a.cout) {
                                float o = v[e] + sBias[c0 + e];
                                op[c0 + e] = a.relu ? fmaxf(o, 0.0f) : o;
                            }
                        }
                    }
                }
              }
              tmem_wait_st();
            }
            // the slot is read and zeroed; the staging slot goes to the store warp
            tc_fence_before();
            if (stores_bf) fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&sfree[sl]);
                mbar_arrive(&edone[slot]);
            }
          }
        }
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kTmemCols));
    }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void* p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

// input-row ring depth of the conv (0: the most that fits shared memory)
std::atomic<int> g_fold_ring{0};

template <int NOUT, int OPER, bool kImages, bool kMore, bool kAlt>
mrs_status launch_fold(const TcConvArgs& a, cudaStream_t st)
{
    int smax = 4;
    while (fold_smem_bytes<NOUT, OPER, kAlt>(smax + 1) <= 227 * 1024 && smax < 12) ++smax;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_conv_fold<NOUT, OPER, kImages, kMore, kAlt>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)fold_smem_bytes<NOUT, OPER, kAlt>(smax));
        if (e != cudaSuccess) return cuda_status(e, "conv smem attribute");
        attr = true;
    }
    const int want = g_fold_ring.load(std::memory_order_relaxed);
    const int stages = want >= 3 ? (want < smax ? want : smax) : smax;
    size_t smem = fold_smem_bytes<NOUT, OPER, kAlt>(stages);
    const std::conditional_t<kMore, TcConvArgs, TcConvBase> b = a;
    const int im = tc_images(a.N, a.W);
    const long long T = (long long)((a.N + im - 1) / im) * ((a.W + kFoldTile - 1) / kFoldTile) * a.H;
    const long long tiles = T * (a.ng > 1 ? a.ng : 1);
    int grid = tiles < sm_count() ? (int)tiles : sm_count();
    if (grid < 1) return MRS_OK;
    const CUtensorMap* res = a.tmap_res ? a.tmap_res : a.tmap_x;
    const CUtensorMap* out = a.tmap_out ? a.tmap_out : a.tmap_x;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute la[1];
    la[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    la[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = la;
    cfg.numAttrs = 1;
    cudaError_t le = cudaSuccess;
    MRS_TIMED(PK_CONV_TC, st, (le = cudaLaunchKernelEx(&cfg, k_conv_fold<NOUT, OPER, kImages, kMore, kAlt>, *a.tmap_x, *a.tmap_w, *res, *out, b, stages)));
    MRS_LAUNCHED(1);
    if (le != cudaSuccess) return cuda_status(le, "conv launch");
    return cuda_status(cudaGetLastError(), "conv launch");
}

// images of a box: a conv's operand or output box (tc_images), else one
int conv_box(int& box_px, int box_rows, int N, int W)
{
    const int im = box_rows == 1 && (box_px == kABox || box_px == kOutBox) ? tc_images(N, W) : 1;
    if (im > 1) box_px = W + 2;
    return im;
}

}  // namespace

mrs_status tc_make_act_map(CUtensorMap* m, const void* ptr, int N, int H, int W, int operand,
                           int box_px)
{
    auto fn = encode_fn();
    if (!fn) { set_error("cuTensorMapEncodeTiled unavailable"); return MRS_ERR_CUDA; }
    int rowb = operand == TC_BF16 ? 128 : 64;
    cuuint64_t dims[4] = {64, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    cuuint64_t strides[3] = {(cuuint64_t)rowb, (cuuint64_t)rowb * W, (cuuint64_t)rowb * W * H};
    const int im = conv_box(box_px, 1, N, W);
    cuuint32_t box[4] = {64, (cuuint32_t)box_px, 1, (cuuint32_t)im};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = fn(m, operand == TC_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8,
                    4, const_cast<void*>(ptr), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    operand == TC_BF16 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { set_error("cuTensorMapEncodeTiled(act) failed: %d", (int)r); return MRS_ERR_CUDA; }
    return MRS_OK;
}

mrs_status tc_make_view_map(CUtensorMap* m, const void* ptr, int N, int H, int W,
                            long long px_stride, long long row_stride, long long img_stride,
                            int box_px, int box_rows)
{
    auto fn = encode_fn();
    if (!fn) { set_error("cuTensorMapEncodeTiled unavailable"); return MRS_ERR_CUDA; }
    if (((uintptr_t)ptr & 15) || (px_stride & 15) || (row_stride & 15) || (img_stride & 15)) {
        set_error("tc_make_view_map: base and strides must be multiples of 16 bytes");
        return MRS_ERR_ARG;
    }
    cuuint64_t dims[4] = {64, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    cuuint64_t strides[3] = {(cuuint64_t)px_stride, (cuuint64_t)row_stride, (cuuint64_t)img_stride};
    const int im = conv_box(box_px, box_rows, N, W);
    cuuint32_t box[4] = {64, (cuuint32_t)box_px, (cuuint32_t)box_rows, (cuuint32_t)im};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(ptr), dims, strides,
                    box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { set_error("cuTensorMapEncodeTiled(view) failed: %d", (int)r); return MRS_ERR_CUDA; }
    return MRS_OK;
}

mrs_status tc_make_w_map(CUtensorMap* m, const void* ptr, int rows, int nout, int operand)
{
    auto fn = encode_fn();
    if (!fn) { set_error("cuTensorMapEncodeTiled unavailable"); return MRS_ERR_CUDA; }
    int rowb = operand == TC_BF16 ? 128 : 64;
    cuuint64_t dims[2] = {64, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)rowb};
    cuuint32_t box[2] = {64, (cuuint32_t)nout};
    cuuint32_t es[2] = {1, 1};
    CUresult r = fn(m, operand == TC_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8,
                    2, const_cast<void*>(ptr), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    operand == TC_BF16 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { set_error("cuTensorMapEncodeTiled(w) failed: %d", (int)r); return MRS_ERR_CUDA; }
    return MRS_OK;
}

namespace {
// waits on an mbarrier that nothing completes; the bounded wait must give up,
// raise the error word and return (exercises the kernels' timeout path)
__global__ void k_wait_selftest(int* err, long long limit_cycles, int* gave_up)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        bool ok = mbar_wait_limit(&bar, 0, err, limit_cycles, 1000u);
        *gave_up = ok ? 0 : 1;
    }
}
}  // namespace

mrs_status tc_wait_selftest(long long limit_cycles, int* gave_up, cudaStream_t st)
{
    int* d = nullptr;
    MRS_CHECK(cudaMalloc(&d, 2 * sizeof(int)));
    MRS_CHECK(cudaMemsetAsync(d, 0, 2 * sizeof(int), st));
    k_wait_selftest<<<1, 32, 0, st>>>(d, limit_cycles, d + 1);
    MRS_LAUNCHED(1);
    int h[2] = {0, 0};
    mrs_status rc = cuda_status(cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, st), "selftest copy");
    if (rc == MRS_OK) rc = cuda_status(cudaStreamSynchronize(st), "selftest sync");
    cudaFree(d);
    if (rc != MRS_OK) return rc;
    *gave_up = h[1] && h[0];
    return MRS_OK;
}

void tc_set_ring(int stages) { g_fold_ring.store(stages, std::memory_order_relaxed); }

mrs_status tc_conv3x3(const TcConvArgs& a, cudaStream_t st)
{
    if (a.kc > 1 && (!a.amaps || ((uintptr_t)a.amaps & 63))) {
        set_error("tc_conv3x3: kc > 1 needs a 64-byte aligned device array of kc maps");
        return MRS_ERR_ARG;
    }
    if (a.ng > 1 && (a.kc > 1 || a.op2 || a.ng > sm_count() || !a.gmaps || ((uintptr_t)a.gmaps & 63))) {
        set_error("tc_conv3x3: a group of convs takes one input chunk and a 64-byte aligned device array of maps");
        return MRS_ERR_ARG;
    }
    if (a.mask && a.op2) {
        set_error("tc_conv3x3: mask and op2 exclude each other");
        return MRS_ERR_ARG;
    }
    if (a.ng > 1 || a.mask || a.op2) {
        if (a.nout == 64 && a.operand == TC_BF16) return launch_fold<64, TC_BF16, true, true, false>(a, st);
        set_error("tc_conv3x3: groups, masks and second results need 64 BF16 channels");
        return MRS_ERR_ARG;
    }
    if (a.nout != 64 && a.nout != 16) {
        set_error("tc_conv3x3: nout must be 64 or 16");
        return MRS_ERR_ARG;
    }
    const bool wide = a.nout == 64, bf = a.operand == TC_BF16;
    if (tc_images(a.N, a.W) > 1) {
        if (wide) return bf ? launch_fold<64, TC_BF16, true, false, false>(a, st) : launch_fold<64, TC_FP8, true, false, false>(a, st);
        return bf ? launch_fold<16, TC_BF16, true, false, false>(a, st) : launch_fold<16, TC_FP8, true, false, false>(a, st);
    }
    // alternating epilogue groups from 3 rows a CTA.  The fusion network in BF16
    // at 1024^2 (54 rows) 1.212 -> 1.183 ms, 512 x 288 (7.6) 0.265 -> 0.262, in
    // FP8 512 x 288 0.246 -> 0.240, 384 x 216 (4.3) 0.195 -> 0.193, 256 x 128 (1.7)
    // 0.147 -> 0.151; the two-encoder network at 256^2 (3.4) 1.576 -> 1.568
    const long long tiles = (long long)a.N * ((a.W + kFoldTile - 1) / kFoldTile) * a.H;
    if (tiles >= 3LL * sm_count()) {
        if (wide)
            return bf ? launch_fold<64, TC_BF16, false, false, true>(a, st) : launch_fold<64, TC_FP8, false, false, true>(a, st);
        return bf ? launch_fold<16, TC_BF16, false, false, true>(a, st) : launch_fold<16, TC_FP8, false, false, true>(a, st);
    }
    if (wide)
        return bf ? launch_fold<64, TC_BF16, false, false, false>(a, st) : launch_fold<64, TC_FP8, false, false, false>(a, st);
    return bf ? launch_fold<16, TC_BF16, false, false, false>(a, st) : launch_fold<16, TC_FP8, false, false, false>(a, st);
}


// ---------------------------------------------------------------------------
// Weight gradient on the tensor cores: the GEMM
//     D[(t, c)][o] = sum_p x[p + shift_t][c] * dy[p][o]
// with K = pixels.  Both tensors keep their [pixel][64-channel] layout, which
// for this GEMM is MN-major (the M or N index is the contiguous one): a TMA
// box of pixels with 128-byte swizzled rows is the canonical MN-major
// SWIZZLE_128B operand, one 128-byte row per K index, 8-row groups 1024 bytes
// apart.  M = 128 is made of two 64-channel MN atoms LBO bytes apart, so one
// MMA covers two taps:
//   MMA dx     (dx = 0..2): rows 0-63 tap (ky 0, dx), rows 64-127 tap (ky 1, dx)
//                           (input rows y-1 and y lie one box row apart)
//   MMA 3 + dx            : rows 0-63 tap (ky 2, dx), rows 64-127 read a
//                           region of ones, which makes those rows db[o]
// A job is kWgKB output pixels of one image row.  Per job the producer loads
// input rows y-1, y, y+1 (kWgKB + 2 pixels from x0 - 1, one TMA box, zero-filled
// outside the image: the zero padding) and dy row y (kWgKB pixels); the kx shift
// is a descriptor start offset of kx 128-byte rows.  MMAs into different D
// regions do not pipeline, so a job issues one MMA's four K steps after the
// other; K steps wholly outside the image are left out.
// The accumulators of a run (6 x 64 FP32 columns) go to the epilogue's
// registers, which add up the runs of one class: an earlier form wrote every
// run's 147 KB as a partial sum, 178 launches and 10,400 partials for a step of
// the two-encoder network, whose writing, re-reading and launch gaps cost
// several times the MMAs.  A (tile, class) pair is the unit of work, or one
// half of it (MMAs 0-2 or 3-5) where the whole would outlast an even share of
// all work; the host deals the units to the CTAs, largest first.
// Warps (16): 2 TMA producer, 3 MMA issuer (lane 0), 7 TMEM allocator, the
// others epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31; lanes 0-63 have
// 384 useful columns (4 warps x 96), lanes 64-127 192 (2 x 96) and the bias
// row's 64 (warp 6).
namespace {

constexpr int kWgThreads = 512;
constexpr int kWgXRow = (kWgKB + 2) * 128;                   // bytes of one input row of a job
constexpr int kWgXBytes = 3 * kWgXRow;
constexpr int kWgYBytes = kWgKB * 128;
constexpr int kWgYOff = (kWgXBytes + 1023) & ~1023;
constexpr int kWgStage = kWgYOff + kWgYBytes;
constexpr int kWgStages = 6;
constexpr int kWgOnes = (kWgXRow + 1023) & ~1023;
constexpr size_t kWgSmem = 1024 + (size_t)kWgStages * kWgStage + kWgOnes + 8 * (2 * kWgStages + 2) + 16;
static_assert(kWgSmem <= 227 * 1024, "wgrad shared memory");
// kind::f16, D f32, A and B bf16, both MN-major, N = 64, M = 128
constexpr uint32_t kWgIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                              ((uint32_t)(64 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

struct alignas(64) WgDesc {
    CUtensorMap x, dy;
    int njobs, runs, H, W, XS, cin, cout;
};
struct WgUnit { int tile, w, half; };   // half: 0 MMAs 0-5, 1 MMAs 0-2, 2 MMAs 3-5

// MN-major SWIZZLE_128B descriptor: `lbo` = bytes to the next 64-element MN
// atom, SBO = 1024 bytes to the next group of 8 K rows
__device__ __forceinline__ uint64_t sdesc_mn(uint32_t saddr, uint32_t lbo)
{
    uint64_t d = (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// waits for a phase regardless of the error word (used to drain copies in
// flight before the CTA exits); gives up after `limit_cycles`
__device__ __forceinline__ void mbar_drain(uint64_t* bar, uint32_t parity, long long limit_cycles)
{
    long long t0 = clock64();
    while (!mbar_try_wait_sleep(bar, parity, 100000u))
        if (clock64() - t0 > limit_cycles) return;
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

// first job of run g
__device__ __forceinline__ int wg_run(const WgDesc& d, int g) { return (int)((long long)d.njobs * g / d.runs); }

// MMAs QA .. QB - 1 of a job: a01 / a2 are the A descriptors of MMAs 0 and 3
// (one 128-byte row further per dx), bd the B descriptor; ks K steps of 16
// pixels, each 2048 bytes (+ 128 in the start-address field, bits 0-13;
// shared-memory addresses stay far below the field's 256 KB) into every operand
template <int QA, int QB>
__device__ __forceinline__ void wg_issue(uint32_t tmem, uint64_t a01, uint64_t a2, uint64_t bd, int ks, uint32_t more)
{
    if (ks == kWgKB / 16) {
#pragma unroll
        for (int q = QA; q < QB; ++q)
#pragma unroll
            for (int kk = 0; kk < kWgKB / 16; ++kk)
                mma_f16(true, tmem + q * 64, (q < 3 ? a01 : a2) + (uint64_t)((q % 3) * 8 + kk * 128),
                        bd + (uint64_t)(kk * 128), kWgIdesc, kk ? 1u : more);
    } else {
#pragma unroll
        for (int q = QA; q < QB; ++q)
#pragma unroll
            for (int kk = 0; kk < kWgKB / 16 - 1; ++kk)
                if (kk < ks)
                    mma_f16(true, tmem + q * 64, (q < 3 ? a01 : a2) + (uint64_t)((q % 3) * 8 + kk * 128),
                            bd + (uint64_t)(kk * 128), kWgIdesc, kk ? 1u : more);
    }
}

// kOne: a launch of one tile, described by its parameter instead of lists in device
// memory; CTA c takes class c, or a half of class c / 2 (halves set: up to half as
// many classes as SMs), and classes = runs.  Through the lists, which the host makes
// and whose upload the kernel waits for, the call for a layer's gradient took 108 us
// with 8 images of 30 x 30, so 84.
struct WgNone {};
template <bool kOne>
__global__ void __launch_bounds__(kWgThreads, 1)
    k_wgrad_tc(const __grid_constant__ std::conditional_t<kOne, WgDesc, WgNone> one, int halves,
               const WgDesc* __restrict__ tiles, const WgUnit* __restrict__ units, const int* __restrict__ first,
               int classes, float* __restrict__ part, float* __restrict__ dbpart, int* err)
{
    auto unit = [&](int u) -> WgUnit {
        if constexpr (kOne) return halves ? WgUnit{0, (int)blockIdx.x / 2, 1 + (int)blockIdx.x % 2} : WgUnit{0, (int)blockIdx.x, 0};
        else return units[u];
    };
    auto desc = [&](const WgUnit& w) -> const WgDesc& {
        if constexpr (kOne) return one;
        else return tiles[w.tile];
    };
    constexpr uint32_t kTmemCols = 512;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sOnes = smem + (size_t)kWgStages * kWgStage;
    uint64_t* full = (uint64_t*)(sOnes + kWgOnes);
    uint64_t* empty = full + kWgStages;
    uint64_t* done = empty + kWgStages;      // a run's MMAs have completed
    uint64_t* tfree = done + 1;              // its accumulators have been read
    uint32_t* tslot = (uint32_t*)(tfree + 1);
    constexpr int kWgEpiWarps = 13;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u0 = kOne ? 0 : first[blockIdx.x], u1 = kOne ? 1 : first[blockIdx.x + 1];

    for (int i = threadIdx.x; i < kWgOnes / 4; i += kWgThreads) ((uint32_t*)sOnes)[i] = 0x3F803F80u;  // bf16 1.0
    fence_async_smem();
    if (threadIdx.x == 0) {
        for (int i = 0; i < kWgStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        mbar_init(done, 1);
        mbar_init(tfree, kWgEpiWarps);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    if (warp == 7) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tslot)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *(volatile uint32_t*)tslot;

    if (warp == 2) {
        if (lane == 0) {
            uint32_t it = 0, ph = 0;
            int s = 0;
            bool ok = true;
            for (int u = u0; ok && u < u1; ++u) {
                const WgUnit un = unit(u);
                const WgDesc& d = desc(un);
                if constexpr (!kOne) {
                    // maps in global memory, written by the host before the launch
                    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"((uint64_t)&d.x) : "memory");
                    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"((uint64_t)&d.dy) : "memory");
                }
                const int XS = d.XS, H = d.H;
                for (int g = un.w; ok && g < d.runs; g += classes) {
                    const int je = wg_run(d, g + 1);
                    for (int j = wg_run(d, g); j < je;
                         ++j, ++it, s = (s + 1 == kWgStages ? 0 : s + 1), ph ^= (s == 0 ? 1u : 0u)) {
                        const int xs = j % XS, r = j / XS, y = r % H, n = r / H;
                        if (!mbar_wait(&empty[s], ph ^ 1, err)) { ok = false; break; }
                        mbar_expect_tx(&full[s], kWgXBytes + kWgYBytes);
                        uint8_t* sb = smem + (size_t)s * kWgStage;
                        tma_load_4d(sb, &d.x, 0, xs * kWgKB - 1, y - 1, n, &full[s]);
                        tma_load_4d(sb + kWgYOff, &d.dy, 0, xs * kWgKB, y, n, &full[s]);
                    }
                }
            }
            // no copy may still be landing when the CTA exits
            for (uint32_t i = it > (uint32_t)kWgStages ? it - kWgStages : 0; i < it; ++i)
                mbar_drain(&full[i % kWgStages], (i / kWgStages) & 1, kTimeoutCycles);
        }
    } else if (warp == 3) {
        if (lane == 0) {
            // MMA issuer
            const uint32_t ones = smem_u32(sOnes), sbase = smem_u32(smem);
            uint32_t ph = 0, k = 0;
            int s = 0;
            bool ok = true;
            for (int u = u0; ok && u < u1; ++u) {
                const WgUnit un = unit(u);
                const WgDesc& d = desc(un);
                const int XS = d.XS, W = d.W;
                const int half = un.half;
                for (int g = un.w; ok && g < d.runs; g += classes, ++k) {
                    const int jb = wg_run(d, g), je = wg_run(d, g + 1);
                    // the previous run's accumulators have been read
                    if (k > 0 && !mbar_wait(tfree, (k - 1) & 1, err)) { ok = false; break; }
                    tc_fence_after();
                    int xs = jb % XS;
                    for (int j = jb; j < je; ++j) {
                        if (!mbar_wait(&full[s], ph, err)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t base = sbase + (uint32_t)s * kWgStage, top2 = base + 2 * kWgXRow;
                        const uint64_t a01 = sdesc_mn(base, kWgXRow), a2 = sdesc_mn(top2, ones - top2);
                        const uint64_t bd = sdesc_mn(base + kWgYOff, kWgYBytes);
                        const int ks = min(kWgKB / 16, (W - xs * kWgKB + 15) / 16);
                        const uint32_t more = j > jb ? 1u : 0u;
                        if (half == 0) wg_issue<0, 6>(tmem, a01, a2, bd, ks, more);
                        else if (half == 1) wg_issue<0, 3>(tmem, a01, a2, bd, ks, more);
                        else wg_issue<3, 6>(tmem, a01, a2, bd, ks, more);
                        mma_commit(&empty[s]);
                        if (++s == kWgStages) { s = 0; ph ^= 1u; }
                        if (++xs == XS) xs = 0;
                    }
                    mma_commit(done);   // arrives once every MMA issued above has completed
                }
            }
        }
    } else if (warp != 7) {
        const int quarter = warp & 3, m = 32 * quarter + lane, c = m & 63;
        // this warp's columns: 96 from col0, or the bias row's 64
        const bool bias = warp == 6;
        const int col0 = bias ? 192 : 96 * (quarter < 2 ? warp >> 2 : (warp >> 2) - 2);
        uint32_t k = 0;
        bool ok = true;
        for (int u = u0; ok && u < u1; ++u) {
            const WgUnit un = unit(u);
            const WgDesc& d = desc(un);
            const int w = un.w, half = un.half, runs = d.runs, cin = d.cin, cout = d.cout;
            const bool mine = half == 0 || (half == 1 ? col0 < 192 : col0 >= 192);
            float acc[96];
#pragma unroll
            for (int i = 0; i < 96; ++i) acc[i] = 0.0f;
            for (int g = w; g < runs; g += classes, ++k) {
                if (!mbar_wait_all(done, k & 1, err)) { ok = false; break; }
                tc_fence_after();
#pragma unroll
                for (int h = 0; h < 12; ++h) {
                    if (!mine || (h >= 8 && bias)) continue;
                    uint32_t r[8];
                    tmem_ld8(tmem + ((uint32_t)(32 * quarter) << 16) + col0 + 8 * h, r);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 8; ++i) acc[8 * h + i] += __uint_as_float(r[i]);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tfree);
            }
            if (!ok) break;
            if (!mine) continue;
            const size_t slot = (size_t)un.tile * classes + w;
            float* P = part + slot * kWgPart;
            if (bias) {
                if (lane == 0)
#pragma unroll
                    for (int o = 0; o < 64; ++o)
                        if (o < cout) dbpart[slot * 64 + o] = acc[o];
            } else {
#pragma unroll
                for (int i = 0; i < 96; ++i) {
                    // TMEM lane m of MMA q: tap t
                    const int q = (col0 + i) >> 6, o = (col0 + i) & 63;
                    const int t = q < 3 ? (m < 64 ? q : 3 + q) : 3 + q;
                    if (o < cout && c < cin) P[((size_t)t * cout + o) * cin + c] = acc[i];
                }
            }
        }
        // on the error path MMAs may still run: TMEM is freed only after them
        if (!ok && warp == 0 && lane == 0) mbar_drain(done, k & 1, kTimeoutCycles);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 7) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kTmemCols));
    }
}

}  // namespace

mrs_status tc_make_wg_x_map(CUtensorMap* m, const void* ptr, int N, int H, int W, long long px_stride,
                            long long row_stride, long long img_stride)
{
    return tc_make_view_map(m, ptr, N, H, W, px_stride, row_stride, img_stride, kWgKB + 2, 3);
}
mrs_status tc_make_wg_dy_map(CUtensorMap* m, const void* ptr, int N, int H, int W, long long px_stride,
                             long long row_stride, long long img_stride)
{
    return tc_make_view_map(m, ptr, N, H, W, px_stride, row_stride, img_stride, kWgKB);
}

static mrs_status wg_desc(const WgTile& w, WgDesc& e)
{
    if (w.cin < 1 || w.cin > 64 || w.cout < 1 || w.cout > 64 || w.runs < 1) {
        set_error("tensor-core weight gradient: cin, cout must be in [1, 64], runs >= 1");
        return MRS_ERR_ARG;
    }
    memset(&e, 0, sizeof(e));
    e.x = w.x; e.dy = w.dy; e.H = w.H; e.W = w.W; e.cin = w.cin; e.cout = w.cout;
    e.XS = (w.W + kWgKB - 1) / kWgKB;
    const long long nj = (long long)w.N * w.H * e.XS;
    if (nj > 0x7fffffff) { set_error("tensor-core weight gradient: too many jobs"); return MRS_ERR_CAPACITY; }
    e.njobs = (int)nj;
    e.runs = (int)std::min<long long>(nj, w.runs);
    return MRS_OK;
}

mrs_status tc_wgrad_plan(const std::vector<WgTile>& tiles, int classes, WgPlan& plan)
{
    const int nt = (int)tiles.size();
    std::vector<WgDesc> d(nt);
    struct Sized { long long cost; WgUnit u; };
    std::vector<Sized> units;
    plan.ntiles = nt;
    plan.classes = classes;
    long long total = 0;
    plan.np.assign(nt, 0);
    for (int t = 0; t < nt; ++t) {
        const WgTile& w = tiles[t];
        WgDesc& e = d[t];
        const mrs_status rc = wg_desc(w, e);
        if (rc != MRS_OK) return rc;
        const long long nj = e.njobs;
        plan.np[t] = std::min(e.runs, classes);
        for (int c = 0; c < plan.np[t]; ++c) {
            long long cost = 0;
            // K steps of the class's runs, and about six for each emptying
            for (int g = c; g < e.runs; g += classes)
                cost += (nj * (g + 1) / e.runs - nj * g / e.runs) * ((w.W + 15) / 16) / e.XS + 6;
            units.push_back({cost, {t, c, 0}});
            total += cost;
        }
    }
    // a unit well above an SM's even share is done in two halves
    for (size_t i = 0, n = units.size(); i < n; ++i)
        if (units[i].cost * 4 * sm_count() > 5 * total) {
            Sized b = units[i];
            units[i].u.half = 1;
            b.u.half = 2;
            units[i].cost = b.cost = b.cost / 2 + 1;
            units.push_back(b);
        }
    // the units to the CTAs, largest first, each to the least loaded
    plan.units = (int)units.size();
    plan.ctas = (int)std::min<size_t>(units.size(), (size_t)sm_count());
    std::stable_sort(units.begin(), units.end(), [](const Sized& a, const Sized& b) { return a.cost > b.cost; });
    std::vector<std::vector<WgUnit>> mine(plan.ctas);
    typedef std::pair<long long, int> Load;
    std::priority_queue<Load, std::vector<Load>, std::greater<Load>> load;
    for (int g = 0; g < plan.ctas; ++g) load.push({0, g});
    for (const Sized& s : units) {
        Load l = load.top();
        load.pop();
        mine[l.second].push_back(s.u);
        load.push({l.first + s.cost, l.second});
    }
    std::vector<WgUnit> list;
    std::vector<int> first;
    for (const auto& m : mine) {
        first.push_back((int)list.size());
        list.insert(list.end(), m.begin(), m.end());
    }
    first.push_back((int)list.size());
    const size_t a = nt * sizeof(WgDesc), b = list.size() * sizeof(WgUnit);
    plan.blob.resize(a + b + first.size() * sizeof(int));
    memcpy(plan.blob.data(), d.data(), a);
    memcpy(plan.blob.data() + a, list.data(), b);
    memcpy(plan.blob.data() + a + b, first.data(), first.size() * sizeof(int));
    return MRS_OK;
}

// a unit a (tile, class) pair, or its two halves; a first unit for each CTA and the end
size_t tc_wgrad_blob_max(int ntiles, int classes)
{
    return ntiles * (sizeof(WgDesc) + 2 * (size_t)classes * sizeof(WgUnit)) + ((size_t)sm_count() + 1) * sizeof(int);
}

template <bool kOne>
static mrs_status launch_wgrad(const std::conditional_t<kOne, WgDesc, WgNone>& one, int halves, int ctas, const WgDesc* d,
                               const WgUnit* u, const int* first, int classes, float* part, float* dbpart, int* err,
                               cudaStream_t st)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_wgrad_tc<kOne>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWgSmem);
        if (e != cudaSuccess) return cuda_status(e, "wgrad smem attribute");
        attr = true;
    }
    MRS_TIMED(PK_WGRAD_TC, st, (k_wgrad_tc<kOne><<<ctas, kWgThreads, kWgSmem, st>>>(one, halves, d, u, first, classes, part, dbpart, err)));
    MRS_LAUNCHED(1);
    return cuda_status(cudaGetLastError(), "wgrad launch");
}

mrs_status tc_conv3x3_wgrad(const WgPlan& plan, const void* d_blob, float* part, float* dbpart, int* err,
                            cudaStream_t st)
{
    if (plan.ctas < 1) return MRS_OK;
    const WgDesc* d = (const WgDesc*)d_blob;
    const WgUnit* u = (const WgUnit*)(d + plan.ntiles);
    return launch_wgrad<false>({}, 0, plan.ctas, d, u, (const int*)(u + plan.units), plan.classes, part, dbpart, err, st);
}

mrs_status tc_conv3x3_wgrad(const WgTile& tile, float* part, float* dbpart, int* np, int* err, cudaStream_t st)
{
    WgDesc d;
    const mrs_status rc = wg_desc(tile, d);
    if (rc != MRS_OK) return rc;
    *np = d.runs;
    if (d.runs < 1) return MRS_OK;
    const int halves = 2 * d.runs <= sm_count();
    return launch_wgrad<true>(d, halves, d.runs * (1 + halves), nullptr, nullptr, nullptr, d.runs, part, dbpart, err, st);
}

}  // namespace mrs
