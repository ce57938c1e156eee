// 3x3 convolution with replicated borders as an implicit GEMM on the sm_103a
// tensor cores (tcgen05): the dense contraction of the MultiScale CNN
// (Sec. 3.1).  BF16 activations and weights, FP32 accumulation in tensor
// memory, bias + optional ReLU + BF16 rounding in the epilogue.
//
// GEMM view of one tile: M = 128 output pixels (flattened over batch, rows
// and columns), N = Cout, K = 9 taps x Cin.  For every tap the A operand is
// the gathered neighbour pixel of each output pixel (replicated borders
// handled by clamping the coordinates), written to shared memory in the
// canonical no-swizzle K-major layout: core matrices of 8 rows x 16 bytes,
// [tap][channel chunk of 8][row][8 channels].  The weights are packed the
// same way once per CTA: [tap][chunk][cout][8 channels].  One thread issues
// the 9 x Cin/16 MMAs (M = 128, N = Cout, K = 16) into one TMEM accumulator,
// commits them to an mbarrier, and the 128 threads read their row back with
// tcgen05.ld.  This gather form serves widths below 32; wider images use the
// warp-specialised row walk further down.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "hproj_internal.cuh"

namespace hp {

namespace {

constexpr int kConvThreads = 128;  // one thread per GEMM row (output pixel)
constexpr int kTileM = 128;
constexpr uint32_t kSpinLimit = 1u << 26;  // bounded mbarrier wait

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor (tcgen05): start address, leading-dimension
// byte offset (between core matrices along K), stride-dimension byte offset
// (between core matrices along M or N), descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// The same for a K-major operand whose rows (pitch 32, 64 or 128 bytes) are
// swizzled as a TMA tile of that inner width: groups of eight rows are
// contiguous; K steps and whole-row shifts move the start address.
__device__ __forceinline__ uint64_t smem_desc_swizzled(uint32_t addr, int pitch)
{
    const uint64_t mode = pitch == 128 ? 2 : pitch == 64 ? 4 : 6;
    return smem_desc(addr, 16, 8 * pitch) | mode << 61;
}

// Instruction descriptor, kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N = n, M = m.
__host__ __device__ constexpr uint32_t mma_idesc(int m, int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

// The same issued by one lane of a warp whose lanes all run the call with the
// same arguments: in uniform control flow the descriptors stay in uniform
// registers.  (From a branch of one lane every MMA first moved its operands
// there, 107-125 cycles per MMA, at N = 96 twice what the MMA takes.)
__device__ __forceinline__ void mma_bf16_warp(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                              uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p, one;\n\telect.sync _|one, 0xffffffff;\n\t"
        "setp.eq.b32 p, 0, 0;\n\t"
        "@one tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc)
        : "memory");
}

__device__ __forceinline__ void mma_commit_warp(uint32_t mbar)
{
    asm volatile(
        "{\n\t.reg .pred one;\n\telect.sync _|one, 0xffffffff;\n\t"
        "@one tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::
            "r"(mbar)
        : "memory");
}

__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t phase)
{
    for (uint32_t it = 0; it < kSpinLimit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(mbar), "r"(phase)
            : "memory");
        if (done) return true;
    }
    return false;
}

// 32 consecutive FP32 accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v)
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
        "%28, %29, %30, %31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

template <int CIN, int COUT>
struct ConvSmem {
    static constexpr int kChunks = CIN / 8;
    static constexpr int kABytes = 9 * kChunks * kTileM * 16;  // all taps of one tile
    static constexpr int kBBytes = 9 * kChunks * COUT * 16;    // all weights
    static constexpr int kBytes = kABytes + kBBytes;
    static constexpr int kTmemCols = COUT < 32 ? 32 : COUT;
};

// x: [P][CIN] bf16 with P = B*H*W pixels (NHWC); w: [9][COUT][CIN] bf16 (tap
// = 3*dy + dx, dy, dx in 0..2 for offsets -1..1); y: [P][COUT] bf16.
template <int CIN, int COUT>
__global__ void __launch_bounds__(kConvThreads, 1)
    conv3x3_tc_kernel(const uint4* __restrict__ x, const uint4* __restrict__ w,
                      const float* __restrict__ bias, __nv_bfloat16* __restrict__ y, int B,
                      int H, int W, int relu, int ntiles, int* err)
{
    using S = ConvSmem<CIN, COUT>;
    constexpr int NCH = S::kChunks;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* sA = smem;
    uint8_t* sB = smem + S::kABytes;
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ float s_bias[COUT];

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const uint32_t mbar_a = smem_u32(&mbar);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_base)),
                     "r"((uint32_t)S::kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_a), "r"(1u));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    for (int i = tid; i < COUT; i += kConvThreads) s_bias[i] = bias[i];
    // weights -> [tap][chunk][cout][8]
    for (int i = tid; i < 9 * COUT * NCH; i += kConvThreads) {
        const int ch = i % NCH;
        const int n = (i / NCH) % COUT;
        const int tap = i / (NCH * COUT);
        const uint4 v = w[(size_t)(tap * COUT + n) * NCH + ch];
        *reinterpret_cast<uint4*>(sB + ((tap * NCH + ch) * COUT + n) * 16) = v;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    // a programmatic dependent of the layer before it: inputs read and outputs
    // written once that layer has completed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const long P = (long)B * H * W;
    const uint32_t idesc = mma_idesc(kTileM, COUT);
    const uint32_t a_base = smem_u32(sA), b_base = smem_u32(sB);
    uint32_t phase = 0;
    bool ok = true;

    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        // gather the 9 tap rows of this thread's output pixel
        const long p = (long)tile * kTileM + tid;
        const bool valid = p < P;
        int b = 0, yy = 0, xx = 0;
        if (valid) {
            b = (int)(p / ((long)H * W));
            const int r = (int)(p - (long)b * H * W);
            yy = r / W;
            xx = r - yy * W;
        }
#pragma unroll 1
        for (int dy = 0; dy < 3; ++dy) {
            const int sy = min(max(yy + dy - 1, 0), H - 1);
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                const int sx = min(max(xx + dx - 1, 0), W - 1);
                const uint4* src = x + (((size_t)b * H + sy) * W + sx) * NCH;
                const int tap = dy * 3 + dx;
#pragma unroll
                for (int ch = 0; ch < NCH; ++ch) {
                    const uint4 v = valid ? src[ch] : make_uint4(0u, 0u, 0u, 0u);
                    *reinterpret_cast<uint4*>(sA + ((tap * NCH + ch) * kTileM + tid) * 16) = v;
                }
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
#pragma unroll
                for (int ks = 0; ks < NCH / 2; ++ks) {
                    const uint64_t ad = smem_desc(a_base + (tap * NCH + 2 * ks) * kTileM * 16,
                                                  kTileM * 16, 128);
                    const uint64_t bd =
                        smem_desc(b_base + (tap * NCH + 2 * ks) * COUT * 16, COUT * 16, 128);
                    mma_bf16(tmem, ad, bd, idesc, (tap | ks) != 0);
                }
            }
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    mbar_a)
                : "memory");
        }
        // a timed-out wait (never expected) ends the kernel on every thread
        ok = __syncthreads_and(mbar_wait(mbar_a, phase) ? 1 : 0) != 0;
        if (!ok) {
            // the MMAs must land before their accumulator is freed: wait once
            // more (bounded) before leaving
            mbar_wait(mbar_a, phase);
            __syncthreads();
            break;
        }
        phase ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // epilogue: this thread's row = TMEM lane tid
        const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll
        for (int c0 = 0; c0 < COUT; c0 += 32) {
            float acc[32];
            tmem_ld32(lane_addr + c0, acc);
            if (valid) {
                __nv_bfloat16* out = y + (size_t)p * COUT + c0;
#pragma unroll
                for (int j = 0; j < 32; j += 8) {
                    __align__(16) __nv_bfloat16 o[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        float vq = acc[j + q] + s_bias[c0 + j + q];
                        if (relu) vq = fmaxf(vq, 0.0f);
                        o[q] = __float2bfloat16_rn(vq);
                    }
                    *reinterpret_cast<uint4*>(out + j) = *reinterpret_cast<const uint4*>(o);
                }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
    }
    if (!ok && err) atomicOr(err, 1);
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"((uint32_t)S::kTmemCols));
    }
}

// Row-walking layout: a CTA walks a 128-pixel column strip down its rows.
// Input rows live once in a ring in shared memory, [slot][130 pixels][channels]
// (pixels x0 - 1 .. x0 + 128, replicated at the borders), each one TMA copy
// swizzled by the channels' width, so the A operand of tap (dy, dx) is a
// descriptor view of the slot holding row y + dy - 1 that starts dx pixels on.
constexpr int kHaloPx = kTileM + 2;

// Warp-specialised persistent row walk.  Each CTA loops over items (grid,
// 128-pixel column strip, rows of it); the input rows of all its items form
// one stream through a kWsSlots-deep ring of halo rows in shared memory (the
// layout and descriptor views above).
//
// One input row r feeds three output rows: r + 1 through the kernel row
// dy = 0, r through dy = 1 and r - 1 through dy = 2.  The weights are staged
// as [dx][dy][cout][cin], so for each (dx, K step) the three
// dy blocks are adjacent along N, and the accumulators of consecutive output
// rows sit in adjacent TMEM column blocks of a ring of kAccSlots (output o of
// the CTA's stream at columns Cout * (kAccSlots - 1 - o % kAccSlots)).  One
// MMA with N = 3 Cout then adds row r's contribution to all three outputs:
// the A operand (the 4 KB input view) is read once for three output rows,
// and each input row needs 3 x Cin/16 MMAs.  At the first and last rows of an
// item only the dy blocks whose output lies in it are issued, and an
// MMA whose column range would wrap around the ring is split in two; this
// plan is made once per input row, so the unrolled issue loop costs two
// descriptor additions per MMA.  Accumulator slots are pre-filled with the
// bias, so every MMA accumulates.
//
// Roles, overlapping through mbarriers:
//   warp 5 (producer): the copy of input row j into slot j % kWsSlots once the
//     MMAs that read the slot's previous row have completed (empty[slot],
//     arrived by tcgen05.commit);
//   warp 6 (borders): replicates the border pixel of rows that need it;
//   warp 4 (MMA, all lanes in step, one issues): per input row waits for the
//     row and, when it starts a new output row, for that accumulator slot to
//     be refilled; issues the MMAs, commits to empty[] of the row and, when an
//     output row is complete, to out_full[] of its slot;
//   warps 0-3 (epilogue): wait out_full, tcgen05.ld their 32 TMEM lanes,
//     refill the slot with the bias (tcgen05.st) and release it (slot_free),
//     then ReLU + BF16 rounding in one conversion and a store staged through
//     shared memory so that each warp writes contiguous 512-byte runs.
// The weights are staged once per CTA.  Every wait is bounded; on a timeout
// the CTA raises the error flag and all roles leave their loops.
constexpr int kWsSlots = 6;
// Narrower images use the gather kernel.  Measured on 256 images, 64 -> 64:
// width 64 0.171 ms (gather 0.434 ms), width 32 0.088 ms (gather 0.119 ms).
constexpr int kWsMinWidth = 32;
constexpr int kAccSlots = 8;
constexpr int kWsThreads = 224;
constexpr uint32_t kWsSpinLimit = 1u << 22;

// CTAs per SM: the edge layers of a branch (16 -> 32 and the 32 -> 1 layer
// as 32 -> 16) and 32 -> 32 leave room in shared memory, registers and tensor
// memory for two or three CTAs, whose pipelines then hide each other's
// latency; the 64-channel layers take one.
template <int CIN, int COUT, bool OUT1>
constexpr int ws_ctas_per_sm()
{
    return OUT1 ? 3 : (CIN == 16 || (CIN == 32 && COUT == 32)) ? 2 : 1;
}

// OUT1: the layer has one output channel (the last convolution of a
// branch), computed as channel 0 of COUT = 16 (the other weights are zero)
// and stored as FP32 [P] without rounding.
template <int CIN, int COUT, bool OUT1 = false>
struct WsSmem {
    static constexpr int kChunks = CIN / 8;
    static constexpr int kPitch = 2 * CIN;  // bytes of a pixel
    static constexpr int kRowBytes = kHaloPx * kPitch;
    static constexpr int kSlotBytes = (kRowBytes + 1023) / 1024 * 1024;
    static constexpr int kRingBytes = kWsSlots * kSlotBytes;
    static constexpr int kBBytes = 9 * kChunks * COUT * 16;
    // per epilogue warp: its 32 output pixels in BF16, 16-byte chunks XOR-swizzled
    static constexpr int kStageBytes = OUT1 ? 0 : 4 * 32 * COUT * 2;
    static constexpr int kBytes = kRingBytes + kBBytes + kStageBytes;
    static constexpr int kTmemCols = kAccSlots * COUT;  // 128, 256 or 512
    static constexpr int kCtas = ws_ctas_per_sm<CIN, COUT, OUT1>();
    // shared memory requested per CTA: enough that no more than kCtas CTAs
    // share an SM (228 KB, 1 KB reserved per CTA), so their tensor memory
    // (kCtas x kTmemCols <= 512 columns) always fits
    static constexpr int kSmemRequest =
        kCtas == 1 || kBytes > 228 * 1024 / (kCtas + 1) ? kBytes : 228 * 1024 / (kCtas + 1) + 1;
    static_assert(COUT == 32 || COUT == 64 || (COUT == 16 && OUT1),
                  "accumulator ring sized for 32 or 64 channels (16 for one output)");
    static_assert(CIN % 16 == 0, "K steps of 16 channels");
    static_assert(kCtas * kTmemCols <= 512, "tensor memory of the CTAs that share an SM");
    static_assert(kCtas * (kSmemRequest + 1024) <= 228 * 1024, "shared memory per SM");
};

// A bounded wait on an mbarrier phase: gives up after `limit` polls, or
// earlier once another role of the CTA has raised abort_flag.
__device__ __forceinline__ bool mbar_wait_ws(uint32_t mbar, uint32_t parity,
                                             const volatile int* abort_flag,
                                             uint32_t limit = kWsSpinLimit)
{
    // a limit of the caller's counts plain looks; the compiled one counts
    // waits that the hardware may suspend for a while
    if (limit != kWsSpinLimit) {
        for (uint32_t it = 0; it < limit; ++it) {
            uint32_t done;
            asm volatile(
                "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                "selp.u32 %0, 1, 0, p;\n\t}\n"
                : "=r"(done)
                : "r"(mbar), "r"(parity)
                : "memory");
            if (done) return true;
            if ((it & 1023u) == 1023u && *abort_flag) return false;
        }
        return false;
    }
    for (uint32_t it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 1023u) == 1023u && *abort_flag) return false;
    }
    return false;
}

// The same for four barriers and all lanes of a warp, looked at together.
__device__ __forceinline__ bool mbar_wait4(const uint32_t (&mbar)[4], const uint32_t (&parity)[4],
                                           const volatile int* abort_flag, uint32_t limit)
{
    bool ok = true;
    if (limit == kWsSpinLimit) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred a, b, c, d;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 a, [%1], %2;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 b, [%3], %4;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 c, [%5], %6;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 d, [%7], %8;\n\t"
            "and.pred a, a, b;\n\tand.pred c, c, d;\n\tand.pred a, a, c;\n\t"
            "selp.u32 %0, 1, 0, a;\n\t}"
            : "=r"(done)
            : "r"(mbar[0]), "r"(parity[0]), "r"(mbar[1]), "r"(parity[1]), "r"(mbar[2]),
              "r"(parity[2]), "r"(mbar[3]), "r"(parity[3])
            : "memory");
        if (__all_sync(0xffffffffu, done != 0)) return true;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
        ok = ok && __all_sync(0xffffffffu, mbar_wait_ws(mbar[i], parity[i], abort_flag, limit));
    return ok;
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// 32 consecutive 32-bit TMEM columns of this thread's lane, without the wait.
__device__ __forceinline__ void tmem_ld32_raw(uint32_t taddr, uint32_t* r)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
        "%28, %29, %30, %31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr));
}

// Write 32 consecutive 32-bit TMEM columns of this thread's lane.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, "
        "%10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, "
        "%27, %28, %29, %30, %31, %32};\n" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
        "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]),
        "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]),
        "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}

// 16 consecutive 32-bit TMEM columns of this thread's lane.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, "
        "%10, %11, %12, %13, %14, %15, %16};\n" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
        "r"(r[15])
        : "memory");
}

// One 32-bit TMEM column of this thread's lane, without the wait.
__device__ __forceinline__ uint32_t tmem_ld1_raw(uint32_t taddr)
{
    uint32_t r;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n" : "=r"(r) : "r"(taddr));
    return r;
}

// An accumulator slot (COUT columns) set to the given 32-bit values.
template <int COUT>
__device__ __forceinline__ void tmem_fill(uint32_t taddr, const uint32_t* bits)
{
    if (COUT % 32 == 0) {
#pragma unroll
        for (int c0 = 0; c0 < COUT; c0 += 32) tmem_st32(taddr + c0, bits + c0);
    } else {
        tmem_st16(taddr, bits);
    }
}

// Two FP32 values to packed BF16 (lo in the low half), round to nearest even,
// optionally with ReLU in the same conversion.
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi, bool relu)
{
    uint32_t d;
    if (relu)
        asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    else
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// Two packed BF16 values v kept where the matching BF16 value of a is
// positive, zeroed elsewhere.
__device__ __forceinline__ uint32_t relu_mask2(uint32_t v, uint32_t a)
{
    uint32_t m = 0;
    if ((a & 0xFFFFu) != 0u && !(a & 0x8000u)) m |= 0xFFFFu;
    if ((a >> 16) != 0u && !(a & 0x80000000u)) m |= 0xFFFF0000u;
    return v & m;
}

template <bool F>
struct Flag {
    static constexpr bool value = F;
};

struct WsItem {
    int b, x0, y0, y1;
};

// The rows of all strips (grid, 128-pixel column) form one sequence of `rows`
// rows, and CTA k of n takes the k-th of n equal pieces of it, so that no CTA
// has more than one row above the mean; an item is what of a piece lies in one
// strip.  (Bands of a common height left 8 x 512^2 with 1,184 items for 152
// CTAs, 8 x 14 rows with a halo of two each, where the mean is 107.8 rows.)
struct WsRows {
    int at, end;
};

__device__ __forceinline__ WsRows ws_rows(int rows)
{
    return {(int)((long long)rows * blockIdx.x / gridDim.x),
            (int)((long long)rows * (blockIdx.x + 1) / gridDim.x)};
}

__device__ __forceinline__ WsItem ws_next(WsRows& piece, int segs, int H)
{
    WsItem it;
    const int strip = piece.at / H;
    it.b = strip / segs;
    it.x0 = (strip - it.b * segs) * kTileM;
    it.y0 = piece.at - strip * H;
    it.y1 = min(H, it.y0 + piece.end - piece.at);
    piece.at += it.y1 - it.y0;
    return it;
}

__device__ __forceinline__ uint32_t idesc_for_rows(int n_out, int cout)
{
    return n_out == 1 ? mma_idesc(kTileM, cout)
           : n_out == 2 ? mma_idesc(kTileM, 2 * cout)
                        : mma_idesc(kTileM, 3 * cout);
}

// DGRAD: the input gradient of a convolution as the convolution of the output
// gradient x with the flipped, transposed weights w: zero padding instead of
// replicated borders (the border terms of the replicated padding are added
// by a separate pass), and in the epilogue every value whose activation in
// act (same layout as the output) is not positive is zeroed (the ReLU
// derivative of the layer that produced act; act may be null).
template <int CIN, int COUT, bool OUT1, bool DGRAD = false>
__global__ void __launch_bounds__(kWsThreads, (ws_ctas_per_sm<CIN, COUT, OUT1>()))
    conv3x3_tc_ws_kernel(const float* __restrict__ bias, void* __restrict__ yout, int H, int W,
                         int segs, int rows, int relu, int* err,
                         uint32_t wait_limit, const uint4* __restrict__ act,
                         const __grid_constant__ CUtensorMap xmap,
                         const __grid_constant__ CUtensorMap wmap)
{
    using S = WsSmem<CIN, COUT, OUT1>;
    // polls of each pipeline wait before it gives up (0: the compiled limit);
    // the final waits for issued MMAs always use the compiled limit
    const uint32_t lim = wait_limit ? wait_limit : kWsSpinLimit;
    __nv_bfloat16* __restrict__ y = reinterpret_cast<__nv_bfloat16*>(yout);
    constexpr int NCH = S::kChunks;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* ring = smem;
    uint8_t* sB = smem + S::kRingBytes;
    __shared__ __align__(8) uint64_t full_bar[kWsSlots];
    __shared__ __align__(8) uint64_t w_bar;              // the weights are there
    __shared__ __align__(8) uint64_t raw_bar[kWsSlots];  // copied, borders not replicated yet
    __shared__ __align__(8) uint64_t empty_bar[kWsSlots];
    __shared__ __align__(8) uint64_t outf_bar[kAccSlots];
    __shared__ __align__(8) uint64_t free_bar[kAccSlots];
    __shared__ uint32_t tmem_base;
    __shared__ float s_bias[COUT];
    __shared__ volatile int s_abort;

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_base)),
                     "r"((uint32_t)S::kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int s = 0; s < kWsSlots; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full_bar[s])),
                         "r"(1u));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&raw_bar[s])),
                         "r"(1u));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&empty_bar[s])),
                         "r"(1u));
        }
        for (int k = 0; k < kAccSlots; ++k) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&outf_bar[k])),
                         "r"(1u));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&free_bar[k])),
                         "r"(4u));
        }
        s_abort = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&w_bar)), "r"(1u));
        asm volatile("fence.mbarrier_init.release.cluster;");
        // weights [tap = 3 dy + dx][cout][cin] -> [dx][dy][cout][cin], each
        // tap one swizzled copy: for one dx the three dy blocks are adjacent
        // along N.  They do not depend on the kernel before this one.
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&w_bar)),
                     "r"((uint32_t)S::kBBytes)
                     : "memory");
        for (int tap = 0; tap < 9; ++tap)
            asm volatile(
                "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
                "[%0], [%1, {%2, %3}], [%4];" ::"r"(
                    smem_u32(sB) + (uint32_t)((tap % 3 * 3 + tap / 3) * COUT * S::kPitch)),
                "l"(&wmap), "r"(0), "r"(tap * COUT), "r"(smem_u32(&w_bar))
                : "memory");
    }
    for (int i = tid; i < COUT; i += kWsThreads) s_bias[i] = bias[i];
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
    // the bias as raw bits, the value every accumulator slot starts from
    uint32_t bias_bits[COUT];
#pragma unroll
    for (int c = 0; c < COUT; ++c) bias_bits[c] = __float_as_uint(s_bias[c]);
    if (warp < 4) {
#pragma unroll
        for (int sl = 0; sl < kAccSlots; ++sl)
            tmem_fill<COUT>(tmem + lane_off + (uint32_t)(sl * COUT), bias_bits);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // Launched as a programmatic dependent of the layer before it, the
    // prologue above (tensor memory, barriers, weights, bias) overlaps that
    // layer's end; the inputs are read, and the outputs written, only once it
    // has completed.  The next layer may then start its own prologue.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool ok = true;

    // a tile whose halo crosses the image's left or right border gets the
    // replicated pixel there by hand (the copy fills it with zeros)
    auto at_border = [&](const WsItem& it) {
        return !DGRAD && (it.x0 == 0 || it.x0 + kHaloPx - 1 > W);
    };
    if (warp == 5) {
        // ---------------------------------------------------------- producer
        if (lane == 0) {
            uint32_t jg = 0, raw = 0;  // raw: parity of the next phase of raw_bar[s]
            uint32_t last_raw = 0;     // bit s: the last copy into slot s signalled raw_bar
            for (WsRows piece = ws_rows(rows); piece.at < piece.end && ok;) {
                const WsItem it = ws_next(piece, segs, H);
                const bool border = at_border(it);
                for (int r = it.y0 - 1; r <= it.y1 && ok; ++r, ++jg) {
                    const uint32_t s = jg % kWsSlots, u = jg / kWsSlots;
                    if (u > 0)
                        ok = mbar_wait_ws(smem_u32(&empty_bar[s]), (u - 1) & 1u, &s_abort, lim);
                    if (!ok) break;
                    const uint32_t bar = smem_u32(border ? &raw_bar[s] : &full_bar[s]);
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                                 "r"((uint32_t)S::kRowBytes)
                                 : "memory");
                    // the input gradient reads zeros outside the image, the
                    // forward the nearest row
                    const int sr = DGRAD ? r : min(max(r, 0), H - 1);
                    asm volatile(
                        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::"
                        "complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(
                            smem_u32(ring + s * S::kSlotBytes)),
                        "l"(&xmap), "r"(0), "r"(it.x0 - 1), "r"(sr), "r"(it.b), "r"(bar)
                        : "memory");
                    if (border) raw ^= 1u << s;
                    last_raw = (last_raw & ~(1u << s)) | ((border ? 1u : 0u) << s);
                }
            }
            // no copy may land after this CTA has left
            const volatile int no_abort = 0;
            for (uint32_t j = jg > kWsSlots ? jg - kWsSlots : 0; j < jg; ++j) {
                const uint32_t s = j % kWsSlots;
                const bool landed =
                    last_raw >> s & 1u
                        ? mbar_wait_ws(smem_u32(&raw_bar[s]), (raw >> s & 1u) ^ 1u, &no_abort)
                        : mbar_wait_ws(smem_u32(&full_bar[s]), (j / kWsSlots) & 1u, &no_abort);
                ok = ok && landed;
            }
        }
    } else if (warp == 6) {
        // ----------------------------------------------------------- borders
        if constexpr (!DGRAD) {
            constexpr int CPX = S::kPitch / 16;  // 16-byte chunks of a pixel
            // chunk c of pixel p within a slot, as the swizzled copy places it
            auto chunk_at = [](int p, int c) {
                const int f = CPX == 8 ? p & 7 : CPX == 4 ? p >> 1 & 3 : p >> 2 & 1;
                return p * S::kPitch + (c ^ f) * 16;
            };
            uint32_t jg = 0, raw = 0;
            for (WsRows piece = ws_rows(rows); piece.at < piece.end && ok;) {
                const WsItem it = ws_next(piece, segs, H);
                const int halo_rows = it.y1 - it.y0 + 2;
                if (!at_border(it)) {
                    jg += halo_rows;
                    continue;
                }
                for (int i = 0; i < halo_rows && ok; ++i, ++jg) {
                    const uint32_t s = jg % kWsSlots;
                    ok = __all_sync(0xffffffffu, mbar_wait_ws(smem_u32(&raw_bar[s]), raw >> s & 1u,
                                                              &s_abort, lim));
                    if (!ok) break;
                    raw ^= 1u << s;
                    uint8_t* slot = ring + s * S::kSlotBytes;
                    const int last = W - it.x0;  // ring pixel of the image's last one
                    if (lane < CPX && it.x0 == 0)
                        *reinterpret_cast<uint4*>(slot + chunk_at(0, lane)) =
                            *reinterpret_cast<const uint4*>(slot + chunk_at(1, lane));
                    if (lane < CPX && last + 1 < kHaloPx)
                        *reinterpret_cast<uint4*>(slot + chunk_at(last + 1, lane)) =
                            *reinterpret_cast<const uint4*>(slot + chunk_at(last, lane));
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&full_bar[s]));
                }
            }
        }
    } else if (warp == 4) {
        // --------------------------------------------------------------- MMA
        // every lane walks the rows (uniform control flow), one issues
        {
            // (the OR over the warp lands in a uniform register)
            const uint32_t tmem_u = __reduce_or_sync(0xffffffffu, tmem);
            const uint64_t a_hi = smem_desc_swizzled(0, S::kPitch);
            const uint64_t bd_base = smem_desc_swizzled(smem_u32(sB), S::kPitch);
            constexpr uint64_t kBlock = COUT * S::kPitch / 16;  // one dy block, 16-byte units
            const volatile int never = 0;
            ok = __all_sync(0xffffffffu, mbar_wait_ws(smem_u32(&w_bar), 0u, &never));
            const uint32_t ring_a = smem_u32(ring);
            uint32_t jg = 0, og = 0;
            int last_row = -1, last_out = -1;
            for (WsRows piece = ws_rows(rows); piece.at < piece.end && ok;) {
                const WsItem it = ws_next(piece, segs, H);
                for (int r = it.y0 - 1; r <= it.y1 && ok; ++r, ++jg) {
                    // dy blocks whose output row r + 1 - dy lies in [y0, y1)
                    const int dlo = max(0, r + 2 - it.y1), dhi = min(2, r + 1 - it.y0);
                    const int nd = dhi - dlo + 1;
                    const uint32_t o_first = og + (uint32_t)(r + 1 - dlo - it.y0);
                    // the barriers of two rows are looked at together: a look
                    // costs about 180 cycles (of 1,152 that a row's MMAs take)
                    if (((r - it.y0) & 1) != 0) {
                        const int n = r < it.y1 ? 2 : 1;  // rows r, r + 1
                        uint32_t bar[4], par[4];
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const uint32_t j = jg + (i < n ? i : 0);
                            bar[2 * i] = smem_u32(&full_bar[j % kWsSlots]);
                            par[2 * i] = (j / kWsSlots) & 1u;
                            // output row r + 1 + i starts with this row, if the band has it
                            const uint32_t o = og + (uint32_t)(r + 1 + i - it.y0);
                            const bool starts = r + 1 + i < it.y1 && o >= (uint32_t)kAccSlots;
                            bar[2 * i + 1] = starts ? smem_u32(&free_bar[o % kAccSlots]) : bar[0];
                            par[2 * i + 1] = starts ? ((o / kAccSlots) - 1) & 1u : par[0];
                        }
                        ok = mbar_wait4(bar, par, &s_abort, lim);
                    }
                    if (!ok) break;
                    // plan: outputs o_first, o_first - 1, ... in at most two
                    // runs of adjacent TMEM column blocks (split at the wrap)
                    const int m = (int)(o_first % kAccSlots);
                    const int len0 = nd < m + 1 ? nd : m + 1;
                    const int len1 = nd - len0;
                    const uint32_t d0 = tmem_u + (uint32_t)(COUT * (kAccSlots - 1 - m));
                    const uint32_t d1 = tmem_u;  // the run after the wrap starts at slot 0
                    const uint32_t id0 = idesc_for_rows(len0, COUT);
                    const uint32_t id1 = idesc_for_rows(len1 > 0 ? len1 : 1, COUT);
                    // B: the first dy block of each run
                    const uint64_t b0 = bd_base + (uint64_t)dlo * kBlock;
                    const uint64_t b1 = bd_base + (uint64_t)(dlo + len0) * kBlock;
                    const uint64_t ad_row =
                        a_hi | (uint64_t)((ring_a + (jg % kWsSlots) * S::kSlotBytes) >> 4);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    auto issue = [&](auto two) {
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
                            for (int ks = 0; ks < NCH / 2; ++ks) {
                                // A: input view shifted by dx pixels, channels from 16 ks;
                                // B: weights of dx, channels from 16 ks
                                const uint64_t ad =
                                    ad_row + (uint64_t)((dx * S::kPitch + 32 * ks) >> 4);
                                const uint64_t boff = 3 * dx * kBlock + 2 * ks;
                                mma_bf16_warp(d0, ad, b0 + boff, id0);
                                if (two.value) mma_bf16_warp(d1, ad, b1 + boff, id1);
                            }
                        }
                    };
                    if (len1 == 0) issue(Flag<false>{});
                    else issue(Flag<true>{});
                    if constexpr (DGRAD) {
                        // ghost output rows -1 and H of the zero-padded
                        // transpose, folded into rows 0 and H - 1 (the
                        // replicated border); both are still accumulating
                        // while input rows 0 and H - 1 are issued
                        for (int f = 0; f < 2; ++f) {
                            const bool fold = f == 0 ? (r == 0 && it.y0 == 0)
                                                     : (r == H - 1 && it.y1 == H);
                            if (!fold) continue;
                            const int o = f == 0 ? 0 : H - 1;
                            const int dsrc = f == 0 ? 2 : 0;  // block of output row -1 / H
                            const uint32_t sl =
                                (og + (uint32_t)(o - it.y0)) % (uint32_t)kAccSlots;
                            const uint32_t dd = tmem_u + (uint32_t)(COUT * (kAccSlots - 1 - (int)sl));
                            const uint32_t idf = idesc_for_rows(1, COUT);
#pragma unroll
                            for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                                for (int ks = 0; ks < NCH / 2; ++ks) {
                                    const uint64_t ad = ad_row + (uint64_t)((dx * S::kPitch + 32 * ks) >> 4);
                                    const uint64_t boff = (3 * dx + dsrc) * kBlock + 2 * ks;
                                    mma_bf16_warp(dd, ad, bd_base + boff, idf);
                                }
                        }
                    }
                    mma_commit_warp(smem_u32(&empty_bar[jg % kWsSlots]));
                    last_row = (int)jg;
                    if (dhi == 2) {
                        // output row r - 1 has all three contributions
                        const uint32_t o_done = og + (uint32_t)(r - 1 - it.y0);
                        mma_commit_warp(smem_u32(&outf_bar[o_done % kAccSlots]));
                        last_out = (int)o_done;
                    }
                }
                og += (uint32_t)(it.y1 - it.y0);
            }
            // the MMAs and the arrivals of the last commits must have landed
            // before the accumulators are freed and the CTA exits (also on
            // the error path)
            const volatile int no_abort = 0;
            bool drained = true;
            if (last_row >= 0)
                drained = mbar_wait_ws(smem_u32(&empty_bar[last_row % kWsSlots]),
                                       ((uint32_t)last_row / kWsSlots) & 1u, &no_abort);
            if (last_out >= 0 && drained)
                drained = mbar_wait_ws(smem_u32(&outf_bar[last_out % kAccSlots]),
                                       ((uint32_t)last_out / kAccSlots) & 1u, &no_abort);
            ok = ok && drained;
        }
    } else {
        // ---------------------------------------------------------- epilogue
        constexpr int CPP = COUT / 8;  // 16-byte chunks per pixel
        auto stage_swz = [](int p) { return (p / (8 / CPP)) & (CPP - 1); };
        uint8_t* stage = sB + S::kBBytes + warp * 32 * COUT * 2;
        const bool do_relu = relu != 0;
        uint32_t og = 0;
        for (WsRows piece = ws_rows(rows); piece.at < piece.end && ok;) {
            const WsItem it = ws_next(piece, segs, H);
            for (int yy = it.y0; yy < it.y1; ++yy, ++og) {
                const uint32_t sl = og % kAccSlots;
                // DGRAD: this lane's activation chunks of the row, loaded while
                // the MMAs of the row are still running
                uint4 act_r[DGRAD ? CPP : 1];
                if constexpr (DGRAD) {
                    if (act) {
#pragma unroll
                        for (int i = 0; i < CPP; ++i) {
                            const int k = lane + 32 * i;
                            const int p = k / CPP, c = k % CPP;
                            const int xo = it.x0 + warp * 32 + p;
                            act_r[i] = xo < W ? act[(((size_t)it.b * H + yy) * W + xo) * CPP + c]
                                              : make_uint4(0u, 0u, 0u, 0u);
                        }
                    }
                }
                // one decision per warp: the tcgen05.ld below is warp-collective
                ok = __all_sync(0xffffffffu, mbar_wait_ws(smem_u32(&outf_bar[sl]),
                                                          (og / kAccSlots) & 1u, &s_abort, lim));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t taddr =
                    tmem + lane_off + (uint32_t)(COUT * (kAccSlots - 1 - (int)sl));
                if constexpr (OUT1) {
                    // channel 0 only, FP32 (bias included by the slot's fill)
                    const uint32_t v = tmem_ld1_raw(taddr);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    tmem_fill<COUT>(taddr, bias_bits);
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&free_bar[sl]));
                    const int xo = it.x0 + warp * 32 + lane;
                    if (xo < W)
                        reinterpret_cast<float*>(yout)[((size_t)it.b * H + yy) * W + xo] =
                            __uint_as_float(v);
                    continue;
                } else {
                uint32_t acc[COUT];
#pragma unroll
                for (int c0 = 0; c0 < COUT; c0 += 32) tmem_ld32_raw(taddr + c0, acc + c0);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                // refill the slot with the bias for the output row that reuses it
                tmem_fill<COUT>(taddr, bias_bits);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&free_bar[sl]));
                // the warp's 32 pixels go through shared memory so that the
                // global stores are contiguous: chunk c of pixel p (16 bytes,
                // 8 channels) sits at position c ^ swz(p), conflict-free on
                // both sides
#pragma unroll
                for (int c = 0; c < CPP; ++c) {
                    uint4 o;
                    o.x = pack_bf16x2(__uint_as_float(acc[8 * c + 0]),
                                      __uint_as_float(acc[8 * c + 1]), do_relu);
                    o.y = pack_bf16x2(__uint_as_float(acc[8 * c + 2]),
                                      __uint_as_float(acc[8 * c + 3]), do_relu);
                    o.z = pack_bf16x2(__uint_as_float(acc[8 * c + 4]),
                                      __uint_as_float(acc[8 * c + 5]), do_relu);
                    o.w = pack_bf16x2(__uint_as_float(acc[8 * c + 6]),
                                      __uint_as_float(acc[8 * c + 7]), do_relu);
                    *reinterpret_cast<uint4*>(stage + lane * (COUT * 2) +
                                              ((c ^ stage_swz(lane)) * 16)) = o;
                }
                __syncwarp();
                __nv_bfloat16* row = y + (((size_t)it.b * H + yy) * W + it.x0 + warp * 32) * COUT;
#pragma unroll
                for (int i = 0; i < CPP; ++i) {
                    const int k = lane + 32 * i;
                    const int p = k / CPP, c = k % CPP;
                    uint4 v = *reinterpret_cast<const uint4*>(
                        stage + p * (COUT * 2) + ((c ^ stage_swz(p)) * 16));
                    if (it.x0 + warp * 32 + p < W) {
                        if constexpr (DGRAD) {
                            if (act) {
                                const uint4 a = act_r[i];
                                v.x = relu_mask2(v.x, a.x);
                                v.y = relu_mask2(v.y, a.y);
                                v.z = relu_mask2(v.z, a.z);
                                v.w = relu_mask2(v.w, a.w);
                            }
                        }
                        *reinterpret_cast<uint4*>(row + (size_t)p * COUT + 8 * c) = v;
                    }
                }
                __syncwarp();
                }
            }
        }
    }
    if (!ok) {
        s_abort = 1;
        if (err) atomicOr(err, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"((uint32_t)S::kTmemCols));
    }
}

// cuTensorMapEncodeTiled, by way of the runtime (no link to the driver library)
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                         cudaEnableDefault, &found);
        if (e == cudaSuccess && found != cudaDriverEntryPointSuccess) e = cudaErrorNotSupported;
        if (e != cudaSuccess) set_cuda_error(e);
        else encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    }
    return encode;
}

// A map of BF16 data whose inner dimension is the channels of one pixel or
// filter, swizzled by their width.
hp_status channel_map(const void* p, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                      const cuuint32_t* box, CUtensorMap* map)
{
    const auto encode = tensor_map_encoder();
    if (!encode) return HP_ERR_CUDA;
    const cuuint32_t one[4] = {1, 1, 1, 1};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank,
                              const_cast<void*>(p), dims, strides, box, one,
                              CU_TENSOR_MAP_INTERLEAVE_NONE,
                              dims[0] == 64   ? CU_TENSOR_MAP_SWIZZLE_128B
                              : dims[0] == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                              : CU_TENSOR_MAP_SWIZZLE_32B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? HP_OK : HP_ERR_INVALID_ARG;
}

// The copy of one row: all channels x px pixels of one row of one image of
// x [B][H][W][cin].
hp_status row_map(const void* x, int cin, int W, int H, int B, int px, CUtensorMap* map)
{
    const cuuint64_t pix = 2ull * cin;
    const cuuint64_t dims[4] = {(cuuint64_t)cin, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
    const cuuint64_t strides[3] = {pix, pix * W, pix * W * H};
    const cuuint32_t box[4] = {(cuuint32_t)cin, (cuuint32_t)px, 1, 1};
    return channel_map(x, 4, dims, strides, box, map);
}

// The copy of one tap of the weights [9][cout][cin].
hp_status weight_map(const void* w, int cin, int cout, CUtensorMap* map)
{
    const cuuint64_t dims[2] = {(cuuint64_t)cin, 9ull * cout};
    const cuuint64_t strides[1] = {2ull * cin};
    const cuuint32_t box[2] = {(cuuint32_t)cin, (cuuint32_t)cout};
    return channel_map(w, 2, dims, strides, box, map);
}

// warp-specialised row walk, kCtas persistent CTAs per SM (an image narrower
// than 128 pixels is one strip whose pixels past its width are not stored)
template <int CIN, int COUT, bool OUT1, bool DGRAD = false>
hp_status launch_ws(const void* x, const void* w, const float* bias, void* y, int B, int H,
                    int W, int relu, int* err, int nsm, cudaStream_t st,
                    const void* act = nullptr, uint32_t wait_limit = 0, bool pdl = false)
{
    using R = WsSmem<CIN, COUT, OUT1>;
    CUtensorMap xmap, wmap;
    hp_status mrc = row_map(x, CIN, W, H, B, kHaloPx, &xmap);
    if (mrc == HP_OK) mrc = weight_map(w, CIN, COUT, &wmap);
    if (mrc != HP_OK) return mrc;
    static bool rattr = false;
    if (!rattr) {
        cudaError_t e = cudaFuncSetAttribute(conv3x3_tc_ws_kernel<CIN, COUT, OUT1, DGRAD>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             R::kSmemRequest);
        if (e != cudaSuccess) { set_cuda_error(e); return HP_ERR_CUDA; }
        rattr = true;
    }
    const int segs = (W + kTileM - 1) / kTileM;
    const long rows = (long)B * H * segs;
    const long ctas = (long)R::kCtas * nsm;
    if (rows > 0x7fffffffL) return HP_ERR_INVALID_ARG;
    const int grid = rows < ctas ? (int)rows : (int)ctas;
    // pdl: a programmatic dependent of the kernel before it in the stream
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kWsThreads);
    cfg.dynamicSmemBytes = R::kSmemRequest;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, conv3x3_tc_ws_kernel<CIN, COUT, OUT1, DGRAD>,
                                       bias, y, H, W, segs, (int)rows, relu, err,
                                       wait_limit, (const uint4*)act, xmap, wmap);
    if (e != cudaSuccess) { set_cuda_error(e); return HP_ERR_CUDA; }
    return check_launch();
}

// ---------------------------------------------------------------------------
// Weight gradient of a 3 x 3 convolution with replicated borders on the
// tensor cores:
//     gW[dy][dx][co][ci] = sum over pixels p of gy[p][co] * x[clamp(p + (dy, dx))][ci]
// Per input row r and 128-pixel segment this is a GEMM over K = the segment's
// output-gradient pixels (8 steps of 16, fewer at the image's right end):
//   A = the input row, M = 128 = kShifts blocks of CI channels, block i the
//       row shifted by i pixels: the rows are single TMA copies (130 pixels,
//       the border pixels replicated by a helper warp), MN-major and swizzled
//       by the channels' width, so a shift by one pixel is a stride of one
//       pixel between the blocks;
//   B = the gradient rows r - 1, r, r + 1 as far as the CTA has them, up to
//       three consecutive slots of a ring of TMA copies, N = 3 CO;
//   D = TMEM, lane (dx, ci), column (2 - dy, co), accumulating over every row
//       and segment the CTA visits.
// CI = 64: two tiles, dx 0 and 1, then dx 2 (the other half of the second is
// not read out); CI = 32: one tile of dx 0..3 (3 is not read out).  Each
// gradient pixel is a K index once, so no operand is staged in shifted copies.
//
// What bounds it: the MMAs, 2 x 8 x 96 cycles per row and segment at 64 -> 64
// (N / 2 each), of which 3/4 are useful.  The gradient of a training batch of
// 64 x 128^2 (13 of these layers) took 4.33 ms with three shifted copies of
// the gradient row staged by cp.async, 18 MMAs per row issued from a branch of
// one lane and bands of a common height, and takes 3.40 ms in this form.
//
// Roles: warp 5 copies the rows; warp 6 replicates the border pixels; warp 4
// issues the MMAs, all lanes in step as in the forward; warps 0-3 add the
// gradient rows up for the bias gradient while they are in shared memory, and
// finally read the accumulators out to per-CTA partial sums
// part[cta][3 dy + dx][co][ci].
constexpr int kWgXSlots = 4;
constexpr int kWgGSlots = 8;
constexpr int kWgThreads = 224;

template <int CI, int CO>
struct WgSmem {
    static constexpr int kPitchX = 2 * CI, kPitchG = 2 * CO;  // bytes of a pixel
    static constexpr int kShifts = 128 / CI;
    static constexpr int kTiles = kShifts == 2 ? 2 : 1;
    static constexpr int kXRowBytes = kHaloPx * kPitchX, kGRowBytes = kTileM * kPitchG;
    // the last tile's unread block reaches one pixel past the halo row
    static constexpr int kXSlotBytes = ((kHaloPx + 1) * kPitchX + 1023) / 1024 * 1024;
    static constexpr int kGOffset = kWgXSlots * kXSlotBytes;
    static constexpr int kBytes = kGOffset + kWgGSlots * kGRowBytes;
    static constexpr int kN = 3 * CO;
    static constexpr int kTmemCols = kTiles * kN <= 128 ? 128 : kTiles * kN <= 256 ? 256 : 512;
    static_assert(CI == 32 || CI == 64, "input channels 32 or 64");
    static_assert(CO == 32 || CO == 64, "output channels 32 or 64");
    static_assert(kGRowBytes % 1024 == 0, "gradient slots on swizzle atoms");
    static_assert(kBytes <= 227 * 1024, "shared memory");
};

// Descriptor of an MN-major operand of pixels (K) by channels, swizzled by
// the pixel pitch: `block` bytes between blocks of one pitch along M or N,
// groups of eight pixels contiguous.
__device__ __forceinline__ uint64_t smem_desc_pixels(uint32_t addr, int pitch, uint32_t block)
{
    return smem_desc(addr, block, 8 * pitch) | (pitch == 128 ? 2ull : 4ull) << 61;
}

template <int CI, int CO>
__global__ void __launch_bounds__(kWgThreads, 1)
    conv3x3_wgrad_tc_kernel(float* __restrict__ part, float* __restrict__ partb, int H, int W,
                            int segs, int rows, int* err, uint32_t wait_limit,
                            const __grid_constant__ CUtensorMap xmap,
                            const __grid_constant__ CUtensorMap gmap)
{
    using S = WgSmem<CI, CO>;
    // polls of each pipeline wait before it gives up (0: the compiled limit);
    // the waits for issued MMAs and copies always use the compiled limit
    const uint32_t lim = wait_limit ? wait_limit : kWsSpinLimit;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* xring = smem;
    uint8_t* gring = smem + S::kGOffset;
    __shared__ __align__(8) uint64_t xfull[kWgXSlots];
    __shared__ __align__(8) uint64_t xraw[kWgXSlots];  // copied, borders not replicated yet
    __shared__ __align__(8) uint64_t xempty[kWgXSlots];
    __shared__ __align__(8) uint64_t gfull[kWgGSlots];
    __shared__ __align__(8) uint64_t gempty[kWgGSlots];
    __shared__ __align__(8) uint64_t done_bar;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int s_abort;
    __shared__ float s_bias[128][8];

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_base)),
                     "r"((uint32_t)S::kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        auto init = [](uint64_t* bar, uint32_t count) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
        };
        for (int i = 0; i < kWgXSlots; ++i) {
            init(&xfull[i], 1);
            init(&xraw[i], 1);
            init(&xempty[i], 1);
        }
        for (int i = 0; i < kWgGSlots; ++i) {
            init(&gfull[i], 1);
            init(&gempty[i], 5);  // the MMAs and the four bias warps
        }
        init(&done_bar, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    if (warp < 4) {  // every MMA accumulates
        uint32_t zero[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) zero[i] = 0u;
        for (int c = 0; c < S::kTiles * S::kN; c += 32)
            tmem_st32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c, zero);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    bool ok = true;
    const volatile int no_abort = 0;
    float bacc[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};

    auto at_border = [&](const WsItem& it) { return it.x0 == 0 || it.x0 + kHaloPx - 1 > W; };
    if (warp == 5) {
        // ---------------------------------------------------------- producer
        if (lane == 0) {
            uint32_t jx = 0, jg = 0, raw = 0;  // raw: parity of the next phase of xraw[s]
            uint32_t last_raw = 0;  // bit s: the last copy into slot s signalled xraw
            auto copy_row = [&](uint32_t dst, const CUtensorMap& map, uint32_t bytes, int x, int y,
                                int b, uint32_t bar) {
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                             "r"(bytes)
                             : "memory");
                asm volatile(
                    "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::"
                    "complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
                    "l"(&map), "r"(0), "r"(x), "r"(y), "r"(b), "r"(bar)
                    : "memory");
            };
            for (WsRows piece = ws_rows(rows); piece.at < piece.end && ok;) {
                const WsItem it = ws_next(piece, segs, H);
                const bool border = at_border(it);
                for (int r = it.y0 - 1; r <= it.y1 && ok; ++r) {
                    if (r + 1 < it.y1) {  // the gradient row that input row r is the first to need
                        const uint32_t s = jg % kWgGSlots, u = jg / kWgGSlots;
                        if (u > 0)
                            ok = mbar_wait_ws(smem_u32(&gempty[s]), (u - 1) & 1u, &s_abort, lim);
                        if (!ok) break;
                        copy_row(smem_u32(gring + s * S::kGRowBytes), gmap, S::kGRowBytes, it.x0,
                                 r + 1, it.b, smem_u32(&gfull[s]));
                        ++jg;
                    }
                    const uint32_t s = jx % kWgXSlots, u = jx / kWgXSlots;
                    if (u > 0)
                        ok = mbar_wait_ws(smem_u32(&xempty[s]), (u - 1) & 1u, &s_abort, lim);
                    if (!ok) break;
                    copy_row(smem_u32(xring + s * S::kXSlotBytes), xmap, S::kXRowBytes, it.x0 - 1,
                             min(max(r, 0), H - 1), it.b, smem_u32(border ? &xraw[s] : &xfull[s]));
                    ++jx;
                    if (border) raw ^= 1u << s;
                    last_raw = (last_raw & ~(1u << s)) | ((border ? 1u : 0u) << s);
                }
            }
            if (!ok) s_abort = 1;
            // no copy may land after this CTA has left
            for (uint32_t j = jx > kWgXSlots ? jx - kWgXSlots : 0; j < jx; ++j) {
                const uint32_t s = j % kWgXSlots;
                const bool landed =
                    last_raw >> s & 1u
                        ? mbar_wait_ws(smem_u32(&xraw[s]), (raw >> s & 1u) ^ 1u, &no_abort)
                        : mbar_wait_ws(smem_u32(&xfull[s]), (j / kWgXSlots) & 1u, &no_abort);
                ok = ok && landed;
            }
            for (uint32_t j = jg > kWgGSlots ? jg - kWgGSlots : 0; j < jg; ++j)
                ok = mbar_wait_ws(smem_u32(&gfull[j % kWgGSlots]), (j / kWgGSlots) & 1u, &no_abort) &&
                     ok;
        }
    } else if (warp == 6) {
        // ----------------------------------------------------------- borders
        constexpr int CPX = S::kPitchX / 16;  // 16-byte chunks of a pixel
        // chunk c of pixel p within a slot, as the swizzled copy places it
        auto chunk_at = [](int p, int c) {
            return p * S::kPitchX + (c ^ (CPX == 8 ? p & 7 : p >> 1 & 3)) * 16;
        };
        uint32_t jx = 0, raw = 0;
        for (WsRows piece = ws_rows(rows); piece.at < piece.end && ok;) {
            const WsItem it = ws_next(piece, segs, H);
            const int halo_rows = it.y1 - it.y0 + 2;
            if (!at_border(it)) {
                jx += halo_rows;
                continue;
            }
            for (int i = 0; i < halo_rows && ok; ++i, ++jx) {
                const uint32_t s = jx % kWgXSlots;
                ok = __all_sync(0xffffffffu,
                                mbar_wait_ws(smem_u32(&xraw[s]), raw >> s & 1u, &s_abort, lim));
                if (!ok) break;
                raw ^= 1u << s;
                uint8_t* slot = xring + s * S::kXSlotBytes;
                const int last = W - it.x0;  // ring pixel of the image's last one
                if (lane < CPX && it.x0 == 0)
                    *reinterpret_cast<uint4*>(slot + chunk_at(0, lane)) =
                        *reinterpret_cast<const uint4*>(slot + chunk_at(1, lane));
                if (lane < CPX && last + 1 < kHaloPx)
                    *reinterpret_cast<uint4*>(slot + chunk_at(last + 1, lane)) =
                        *reinterpret_cast<const uint4*>(slot + chunk_at(last, lane));
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&xfull[s]));
            }
        }
    } else if (warp == 4) {
        // --------------------------------------------------------------- MMA
        constexpr uint32_t kMnMajor = (1u << 15) | (1u << 16);
        const uint32_t tmem_u = __reduce_or_sync(0xffffffffu, tmem);
        const uint64_t a_base = smem_desc_pixels(smem_u32(xring), S::kPitchX, S::kPitchX);
        const uint64_t b_base = smem_desc_pixels(smem_u32(gring), S::kPitchG, S::kGRowBytes);
        uint32_t jx = 0, jg = 0;  // jg: ring position of the item's first gradient row
        for (WsRows piece = ws_rows(rows); piece.at < piece.end && ok;) {
            const WsItem it = ws_next(piece, segs, H);
            const int ksteps = (min(W - it.x0, kTileM) + 15) / 16;
            for (int r = it.y0 - 1; r <= it.y1 && ok; ++r, ++jx) {
                const uint32_t xs = jx % kWgXSlots;
                // the row and the gradient row that it is the first to need
                const bool more = r + 1 < it.y1;
                const uint32_t gn = jg + (uint32_t)(r + 1 - it.y0);
                uint32_t bar[4], par[4];
                bar[0] = bar[2] = bar[3] = smem_u32(&xfull[xs]);
                par[0] = par[2] = par[3] = (jx / kWgXSlots) & 1u;
                bar[1] = more ? smem_u32(&gfull[gn % kWgGSlots]) : bar[0];
                par[1] = more ? (gn / kWgGSlots) & 1u : par[0];
                ok = mbar_wait4(bar, par, &s_abort, lim);
                if (!ok) break;
                // gradient rows g0 .. g0 + n - 1, at most two runs of
                // adjacent slots (split where the ring wraps)
                const int g0 = max(r - 1, it.y0), n = min(r + 1, it.y1 - 1) - g0 + 1;
                const uint32_t s0 = (jg + (uint32_t)(g0 - it.y0)) % kWgGSlots;
                const int len0 = min(n, kWgGSlots - (int)s0), len1 = n - len0;
                const uint32_t d0 = tmem_u + (uint32_t)((g0 - r + 1) * CO);
                const uint32_t d1 = d0 + (uint32_t)(len0 * CO);
                const uint32_t id0 = idesc_for_rows(len0, CO) | kMnMajor;
                const uint32_t id1 = idesc_for_rows(len1 > 0 ? len1 : 1, CO) | kMnMajor;
                const uint64_t a = a_base + (uint64_t)(xs * S::kXSlotBytes >> 4);
                const uint64_t b0 = b_base + (uint64_t)(s0 * S::kGRowBytes >> 4);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                auto step = [&](int ks, auto two) {
#pragma unroll
                    for (int t = 0; t < S::kTiles; ++t) {
                        const uint64_t ad = a + (uint64_t)((16 * ks + 2 * t) * S::kPitchX >> 4);
                        const uint64_t boff = (uint64_t)(16 * ks * S::kPitchG >> 4);
                        mma_bf16_warp(d0 + (uint32_t)(t * S::kN), ad, b0 + boff, id0);
                        if (two.value)  // continues at slot 0
                            mma_bf16_warp(d1 + (uint32_t)(t * S::kN), ad, b_base + boff, id1);
                    }
                };
                auto issue = [&](auto two) {
                    if (ksteps == kTileM / 16) {
#pragma unroll
                        for (int ks = 0; ks < kTileM / 16; ++ks) step(ks, two);
                    } else {
                        for (int ks = 0; ks < ksteps; ++ks) step(ks, two);
                    }
                };
                if (len1 == 0) issue(Flag<false>{});
                else issue(Flag<true>{});
                mma_commit_warp(smem_u32(&xempty[xs]));
                // gradient row r - 1 is not read again
                if (r > it.y0) {
                    const uint32_t gd = jg + (uint32_t)(r - 1 - it.y0);
                    mma_commit_warp(smem_u32(&gempty[gd % kWgGSlots]));
                }
            }
            jg += (uint32_t)(it.y1 - it.y0);
        }
        if (!ok) s_abort = 1;
        // every MMA issued must have landed before the accumulators are read
        // or freed, also on the error path
        mma_commit_warp(smem_u32(&done_bar));
        ok = __all_sync(0xffffffffu, mbar_wait_ws(smem_u32(&done_bar), 0u, &no_abort)) && ok;
    } else {
        // -------------------------------------- bias gradient, then epilogue
        // thread: channels 8 (tid % NG) .. + 7 of the pixels tid / NG + 128 / NG i
        constexpr int NG = CO / 8;
        const int chb = tid % NG;
        uint32_t jg = 0;
        for (WsRows piece = ws_rows(rows); piece.at < piece.end && ok;) {
            const WsItem it = ws_next(piece, segs, H);
            for (int r = it.y0; r < it.y1; ++r, ++jg) {
                const uint32_t s = jg % kWgGSlots;
                ok = __all_sync(0xffffffffu, mbar_wait_ws(smem_u32(&gfull[s]),
                                                          (jg / kWgGSlots) & 1u, &s_abort, lim));
                if (!ok) break;
                const uint8_t* slot = gring + s * S::kGRowBytes;
#pragma unroll
                for (int i = 0; i < NG; ++i) {
                    const int p = tid / NG + i * (128 / NG);
                    const int c = chb ^ (NG == 8 ? p & 7 : p >> 1 & 3);
                    const uint4 v =
                        *reinterpret_cast<const uint4*>(slot + p * S::kPitchG + c * 16);
                    const uint32_t e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        bacc[2 * h] += __uint_as_float(e[h] << 16);
                        bacc[2 * h + 1] += __uint_as_float(e[h] & 0xFFFF0000u);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&gempty[s]));
            }
        }
        if (!ok) s_abort = 1;
        // the MMA warp commits done_bar on every path, so this wait ends once
        // its MMAs have landed
        const bool landed =
            __all_sync(0xffffffffu, mbar_wait_ws(smem_u32(&done_bar), 0u, &no_abort));
        ok = ok && landed;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int L = warp * 32 + lane;  // TMEM lane
        const int ci = L % CI;
        const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
        float* dst = part + (size_t)blockIdx.x * 9 * CO * CI;
#pragma unroll
        for (int t = 0; t < S::kTiles; ++t) {
            const int dx = 2 * t + L / CI;
#pragma unroll
            for (int c0 = 0; c0 < S::kN; c0 += 32) {
                uint32_t v[32];
                tmem_ld32_raw(tmem + lane_off + (uint32_t)(t * S::kN + c0), v);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (landed && dx < 3) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const int dy = 2 - (c0 + j) / CO, co = (c0 + j) % CO;
                        dst[((size_t)(3 * dy + dx) * CO + co) * CI + ci] = __uint_as_float(v[j]);
                    }
                }
            }
        }
    }
    if (!ok) {
        s_abort = 1;
        if (err) atomicOr(err, 1);
    }
    if (warp < 4) {
#pragma unroll
        for (int k = 0; k < 8; ++k) s_bias[tid][k] = bacc[k];
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"((uint32_t)S::kTmemCols));
    }
    // bias partial of the CTA: the threads of each channel chunk, in a fixed
    // order
    if (tid < CO) {
        const int k = tid % 8;
        float t = 0.0f;
        for (int q = tid / 8; q < 128; q += CO / 8) t += s_bias[q][k];
        partb[(size_t)blockIdx.x * CO + tid] = t;
    }
}

template <int CI, int CO>
hp_status launch_wgrad_t(const void* x, const void* gy, float* part, size_t part_len,
                         float* partb, size_t partb_len, int B, int H, int W, int* err, int nsm,
                         int* grid_out, cudaStream_t st, uint32_t wait_limit)
{
    using S = WgSmem<CI, CO>;
    CUtensorMap xmap, gmap;
    hp_status mrc = row_map(x, CI, W, H, B, kHaloPx, &xmap);
    if (mrc == HP_OK) mrc = row_map(gy, CO, W, H, B, kTileM, &gmap);
    if (mrc != HP_OK) return mrc;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(conv3x3_wgrad_tc_kernel<CI, CO>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, S::kBytes);
        if (e != cudaSuccess) { set_cuda_error(e); return HP_ERR_CUDA; }
        attr = true;
    }
    const int segs = (W + kTileM - 1) / kTileM;
    const long rows = (long)B * H * segs;
    if (rows > 0x7fffffffL) return HP_ERR_INVALID_ARG;
    const int grid = rows < nsm ? (int)rows : nsm;
    if ((size_t)grid * 9 * CO * CI > part_len || (size_t)grid * CO > partb_len)
        return HP_ERR_INVALID_ARG;
    conv3x3_wgrad_tc_kernel<CI, CO><<<grid, kWgThreads, S::kBytes, st>>>(
        part, partb, H, W, segs, (int)rows, err, wait_limit, xmap, gmap);
    *grid_out = grid;
    return check_launch();
}

template <int CIN, int COUT>
hp_status launch_conv_t(const void* x, const void* w, const float* bias, void* y, int B, int H,
                        int W, int relu, int* err, int nsm, cudaStream_t st, uint32_t wait_limit,
                        bool pdl)
{
    if (W >= kWsMinWidth) return launch_ws<CIN, COUT, false>(x, w, bias, y, B, H, W, relu, err,
                                                            nsm, st, nullptr, wait_limit, pdl);
    using S = ConvSmem<CIN, COUT>;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(conv3x3_tc_kernel<CIN, COUT>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, S::kBytes);
        if (e != cudaSuccess) { set_cuda_error(e); return HP_ERR_CUDA; }
        attr = true;
    }
    const long P = (long)B * H * W;
    const int ntiles = (int)((P + kTileM - 1) / kTileM);
    const int grid = ntiles < nsm ? ntiles : nsm;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kConvThreads);
    cfg.dynamicSmemBytes = S::kBytes;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, conv3x3_tc_kernel<CIN, COUT>, (const uint4*)x,
                                       (const uint4*)w, bias, (__nv_bfloat16*)y, B, H, W, relu,
                                       ntiles, err);
    if (e != cudaSuccess) { set_cuda_error(e); return HP_ERR_CUDA; }
    return check_launch();
}

}  // namespace

hp_status launch_conv3x3_tc(const void* x, const void* w, const float* bias, void* y, int B,
                            int H, int W, int cin, int cout, int relu, int* err, int nsm,
                            cudaStream_t st, uint32_t wait_limit, bool pdl)
{
    if (cin == 32 && cout == 32)
        return launch_conv_t<32, 32>(x, w, bias, y, B, H, W, relu, err, nsm, st, wait_limit, pdl);
    if (cin == 32 && cout == 64)
        return launch_conv_t<32, 64>(x, w, bias, y, B, H, W, relu, err, nsm, st, wait_limit, pdl);
    if (cin == 64 && cout == 32)
        return launch_conv_t<64, 32>(x, w, bias, y, B, H, W, relu, err, nsm, st, wait_limit, pdl);
    if (cin == 64 && cout == 64)
        return launch_conv_t<64, 64>(x, w, bias, y, B, H, W, relu, err, nsm, st, wait_limit, pdl);
    // first layer of a branch, input padded to 16 channels (warp-specialised
    // kernel only; narrower images take the CUDA-core layer)
    if (cin == 16 && cout == 32 && W >= kWsMinWidth)
        return launch_ws<16, 32, false>(x, w, bias, y, B, H, W, relu, err, nsm, st, nullptr,
                                        wait_limit, pdl);
    return HP_ERR_UNSUPPORTED;
}

int conv_tc_min_width() { return kWsMinWidth; }

// Input gradient of a tensor-core layer (cin -> cout): the convolution of the
// output gradient gy (BF16 [P][cout]) with wdg = the flipped, transposed
// weights (BF16 [9][cin][cout], tap 8 - t of the forward's tap t), zero
// padding, zero bias (cout floats), the ReLU derivative of act (BF16
// [P][cin], may be null) applied; gx BF16 [P][cin].  Widths from
// conv_tc_min_width() up.
hp_status launch_conv3x3_tc_dgrad(const void* gy, const void* wdg, const float* zero_bias,
                                  const void* act, void* gx, int B, int H, int W, int cin,
                                  int cout, int* err, int nsm, cudaStream_t st,
                                  uint32_t wait_limit)
{
    if (W < kWsMinWidth) return HP_ERR_UNSUPPORTED;
    if (cin == 64 && cout == 64)
        return launch_ws<64, 64, false, true>(gy, wdg, zero_bias, gx, B, H, W, 0, err, nsm, st, act,
                                               wait_limit);
    if (cin == 32 && cout == 64)
        return launch_ws<64, 32, false, true>(gy, wdg, zero_bias, gx, B, H, W, 0, err, nsm, st, act,
                                               wait_limit);
    if (cin == 64 && cout == 32)
        return launch_ws<32, 64, false, true>(gy, wdg, zero_bias, gx, B, H, W, 0, err, nsm, st, act,
                                               wait_limit);
    if (cin == 32 && cout == 32)
        return launch_ws<32, 32, false, true>(gy, wdg, zero_bias, gx, B, H, W, 0, err, nsm, st, act,
                                               wait_limit);
    return HP_ERR_UNSUPPORTED;
}

// Weight- and bias-gradient partial sums of a tensor-core layer (cin ->
// cout) into part[g][9][cout][cin] and partb[g][cout] for g < *grid_out (one
// per CTA); x BF16 [P][cin], gy BF16 [P][cout].
hp_status launch_conv3x3_tc_wgrad(const void* x, const void* gy, float* part, size_t part_len,
                                  float* partb, size_t partb_len, int B, int H, int W, int cin,
                                  int cout, int* err, int nsm, int* grid_out, cudaStream_t st,
                                  uint32_t wait_limit)
{
    if (cin == 64 && cout == 64)
        return launch_wgrad_t<64, 64>(x, gy, part, part_len, partb, partb_len, B, H, W, err, nsm,
                                      grid_out, st, wait_limit);
    if (cin == 32 && cout == 64)
        return launch_wgrad_t<32, 64>(x, gy, part, part_len, partb, partb_len, B, H, W, err, nsm,
                                      grid_out, st, wait_limit);
    if (cin == 64 && cout == 32)
        return launch_wgrad_t<64, 32>(x, gy, part, part_len, partb, partb_len, B, H, W, err, nsm,
                                      grid_out, st, wait_limit);
    if (cin == 32 && cout == 32)
        return launch_wgrad_t<32, 32>(x, gy, part, part_len, partb, partb_len, B, H, W, err, nsm,
                                      grid_out, st, wait_limit);
    return HP_ERR_UNSUPPORTED;
}

// Last layer of a branch, 32 -> 1, as channel 0 of a 32 -> 16 convolution
// (w: BF16 [9][16][32], rows 1..15 zero; bias: 16 floats) written as FP32
// [B][H][W] without rounding; HP_ERR_UNSUPPORTED below the width the
// warp-specialised kernel serves.
hp_status launch_conv3x3_tc_out1(const void* x, const void* w, const float* bias, float* y,
                                 int B, int H, int W, int* err, int nsm, cudaStream_t st,
                                 uint32_t wait_limit, bool pdl)
{
    if (W < kWsMinWidth) return HP_ERR_UNSUPPORTED;
    return launch_ws<32, 16, true>(x, w, bias, y, B, H, W, 0, err, nsm, st, nullptr, wait_limit,
                                   pdl);
}

}  // namespace hp

extern "C" hp_status hp_conv3x3_bf16(const uint16_t* x, const uint16_t* w, const float* bias,
                                     uint16_t* y, int32_t batch, int32_t height, int32_t width,
                                     int32_t cin, int32_t cout, int32_t relu, int32_t* err,
                                     void* stream)
{
    if (!x || !w || !bias || !y || batch <= 0 || height <= 0 || width <= 0) return HP_ERR_INVALID_ARG;
    if ((uintptr_t)x % 16 || (uintptr_t)w % 16 || (uintptr_t)y % 16) return HP_ERR_INVALID_ARG;
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) { hp::set_cuda_error(e); return HP_ERR_CUDA; }
    return hp::launch_conv3x3_tc(x, w, bias, y, batch, height, width, cin, cout, relu, err, nsm,
                                 (cudaStream_t)stream);
}
