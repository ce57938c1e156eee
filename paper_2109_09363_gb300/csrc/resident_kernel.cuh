// Grid-resident masked Jacobi sweeps for sm_103a (Sec. 2.2 Jacobi iteration,
// stop rule of Sec. 3.3 / 4.1): the kernel, instantiated by resident_*.cu.
//
// A grid stays on chip for all of its sweeps.  It is cut into horizontal
// strips of whole rows, one CTA (one SM) each, up to 512 cells wide; the CTAs
// of one grid form a group, and one cooperative launch holds as many groups as
// fit on the device, each working through grids of the batch.  A CTA has 8 sweep
// warps in WX columns of 32 C cells and 8 / WX warp rows; thread (warp, lane)
// holds R rows x C columns of phi in registers, div and four bits of open-face
// count per cell sit in shared memory.  A ninth warp does the E rounds, two more
// receive the neighbours' rows.  Per sweep and warp:
//   - the rows next to the warp's block come from shared memory (double
//     buffered), or, at the edge of the strip, from the neighbouring CTA
//     through the L2: every 32-bit value travels with the number of its
//     message in one 64-bit word, so the receiver polls the data itself and
//     no fence or flag is needed;
//   - warps of the lower half hold their rows bottom up, so that the row at
//     the strip's edge is register row 0 in every edge warp: it is computed
//     and sent first, and travels while the other rows are computed;
//   - groups of rows whose cells all have the open-face count of an
//     unobstructed row of that column take the update without the closed-face
//     terms (bit for bit the same result: the left-out product is an exact
//     zero), the others look 4 - n and 1/n up by the cell's bits.
// The only barrier of a sweep is the CTA's own.
//
// What bounds it: latency, with two sweep warps per scheduler (the registers
// hold phi, so there is no room for more).  At 16 x 512^2 the schedulers issue in
// 45 % of their cycles; an instruction waits 1.2 cycles at the CTA barrier, 0.7 for
// fixed latencies, 0.5 for shared memory and 0.4 for instructions to be fetched.
//
// Grids wider than 512 cells are also cut into columns of 240 cells: a CTA then
// holds 256 columns, the outer 8 on each side copies of its neighbours' cells.
// A copy is good for one column less after every sweep, so they are fetched
// anew every 8 sweeps (through the L2 as well), which costs two exposed round
// trips in 8 sweeps instead of one more exchange in each.
//
// E_k: FP32 |r| per thread and group of eight lanes (1,024 cells at most; over
// whole warps the mean error against FP64 was up to 1.6 times that of FP64 sums
// of 1,024 cells each, at 2048^2, and is now 0.5 to 1.1 times it), then sums of
// float pairs (TwoSum, 48 bits; an FP64 addition of a warp occupies its
// scheduler's FP64 unit for 64 cycles here, and four dependent ones per round
// cost 0.6 us a sweep) per CTA (32 sums) and per group (CTA partials in rank
// order), in rounds of four sweeps.  Round q holds sweeps 4q..4q+3; one warp of
// every CTA posts the CTA partials, that of rank 0 adds them and posts the stop
// decision, which every CTA reads at the same sweep (res_lag), so all CTAs of a
// group leave the loop together and go back to the last checkpoint of phi at or below
// k* (ckpt_step), from which they replay the sweeps to k* exactly.
// The comparison with the threshold is made in FP64 whenever the FP32 head of
// the sum is within 1e-6 of it.  phi at the cap is kept aside as it passes, so
// a grid that reaches its cap replays nothing; a run of fixed length needs
// neither E nor a decision.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "hproj_internal.cuh"

namespace hp {

constexpr int kResWarps = 8;       // sweep warps: two warpgroups
constexpr int kResSweepers = kResWarps * 32;
constexpr int kResThreads = kResSweepers + 128;  // and one of helpers
constexpr int kResMaxCtas = 192;   // CTAs of one launch (one per SM)
// registers a thread: 384 x 168 at launch, then 232 for the sweep warps and 40
// for the helpers: 128 x (2 x 232 + 40) = 384 x 168
constexpr int kResRegs = 168, kResRegsSweep = 232, kResRegsHelp = 40;
static_assert(kResSweepers * kResRegsSweep + 128 * kResRegsHelp <= kResThreads * kResRegs,
              "the split waits forever for registers the launch does not have");
// A decision about sweep j is known everywhere before sweep 4 (j / 4 + lag), for
// the lag of the loop index at which it is read.  A single CTA has it within a
// sweep.  Between CTAs it takes up to 8 us (144 of them), more than two sweeps:
// waiting for it costs that much in each round (2048^2: 3.6 us a sweep with a lag
// of three, 4.5 with two), sweeping on costs four more sweeps once.  So the first
// two rounds, where most hybrid projections stop, are waited for and the others
// are not.
constexpr int kResLag = 3;
__device__ __forceinline__ int res_lag(int k, int n) { return n == 1 || k < 12 ? 2 : kResLag; }
constexpr int kResRing = 4;        // > kResLag: rounds between the sweeps and the decision
constexpr int kWsumRing = 4 * kResRing;  // warp sums, by sweep
constexpr int kResSums = 4;        // of one warp: each over eight lanes
// A wait gives up after so many polls: of a word in the L2 (a round trip, half
// a microsecond, so about ten seconds) or of a barrier (suspended for a
// microsecond at most); of a word in shared memory, which waits for a warp that
// waits for the others.  Long enough for a CTA that starts late because kernels
// of other streams hold its SM.  The CTA then marks the launch, waits no longer than one poll
// each for the rest of its grid (whose result is void) and takes no other grid.
constexpr int kResPolls = 1 << 24, kResLooks = 1 << 30;
// the sums of pairs are scaled (exactly) so that no sum of finite warp sums overflows
constexpr float kSumScale = 1.0f / 8192.0f;
static_assert(kResMaxCtas * kResWarps * kResSums <= 8192, "FP32 sums of one grid");

// Exchange area in global memory (one per context, cleared before every
// launch): messages between neighbouring CTAs, E partials, decisions, queue.
struct ResBox {
    // row messages: [receiver][side: from above, from below][parity]
    uint4 row[kResMaxCtas][2][2][256];  // [word][lanes of the strip's width]
    uint4 part[kResMaxCtas][kResRing][4];  // E partial of one sweep: head, tag, tail, tag
    uint4 dec[kResMaxCtas][kResRing];      // by group: decision, tag, sweep, tag
    uint4 next[kResMaxCtas][2];            // by group: grid, tag
    uint32_t queue;                        // grids handed out beyond the first of each group
};

// Columns of a strip that are copies, on each side, and sweeps they last.
constexpr int kResGhost = 8;

// Columns from the CTAs beside (grids wider than 512 cells): [receiver][side:
// from the left, from the right][parity][warp][word][lane]
struct ResColumns {
    uint4 w[kResMaxCtas][2][2][kResWarps][2][32];
};

struct ResArgs {
    const float* phi0;  // phi_0 of the caller (cells without an open face ignored), null = 0
    // phi_{k*} out, and phi at the cap as it passes: not phi0, since a strip with
    // copied columns reads its neighbours' cells of phi_0 (again for a replay
    // from it) when these may already be storing phi_{k*}
    float* phi;
    // checkpoint buffers [B][ny][nx]; phi0 may be ck[1], which is first written
    // at sweep 32, when every strip has read phi_0 and no replay starts from it
    float* ck[2];
    const float* div;   // [B][ny][nx]
    const uint8_t* mask;
    GridState* gs;
    ResBox* box;
    ResColumns* cols;   // null unless ntx > 1
    int32_t* err;       // both set to 1 when a wait gave up
    int32_t polls, looks;  // limits of the waits (kResPolls, kResLooks)
    double* e_hist;     // [B][hist_len] or null
    int32_t hist_len;
    int32_t B, ny, nx;
    int32_t n, ntx;     // CTAs per grid, side by side
    int32_t groups;
    int32_t cap;
    int32_t phi0_vec;   // phi0 allows 16-byte loads
    uint32_t epoch;     // of this launch (GridState::wild)
    int32_t fixed;      // exactly cap sweeps; E only for grids whose values could overflow
    double threshold;   // < 0: never stops before the cap
    float sum_near;     // sums of |r| above it are above the threshold
};

template <int C, int R, int WX>
struct ResLayout {
    static constexpr int WY = kResWarps / WX;
    static constexpr int V = C / 4;                                      // 16-byte words per row
    static constexpr int kDiv = 0;                                       // [8][R][V][32] float4
    static constexpr int kCode = kDiv + kResWarps * R * V * 512;         // [8][R][32] u32, 4 bits a cell
    // rows next to a block: [2 parities][8 warps x 2 rows + a zero row][V][32] float4
    static constexpr int kRow = kCode + kResWarps * R * 128;
    static constexpr int kRowSlot = V * 512;
    static constexpr int kRowPar = (2 * kResWarps + 1) * kRowSlot;
    // columns next to a block: [2][8 warps x 2 columns + a zero column][R] float
    static constexpr int kCol = kRow + 2 * kRowPar;
    static constexpr int kColPar = (2 * kResWarps + 1) * R * 4;
    // rows received from the neighbouring CTAs: [2 sides][2 parities][WX][V][32] float4
    static constexpr int kHalo = kCol + 2 * kColPar;
    static constexpr int kHaloPar = WX * kRowSlot;
    static constexpr int kLut = kHalo + 4 * kHaloPar;                    // [5] float2
    static constexpr int kWsum = kLut + 64;                              // [16][8][4] float
    // copied columns in transit: [warp][2 sides][R][8] float
    static constexpr int kGhost = kWsum + kWsumRing * kResWarps * kResSums * 4;
    static constexpr int kBytes = kGhost + kResWarps * 2 * R * kResGhost * 4;
    static_assert(R % 4 == 0 && C % 4 == 0, "rows and columns go out four values at a time");
    static_assert(kBytes <= 227 * 1024 - 64, "shared memory of one CTA");
};

// ---- 16-byte words through the L2: two 64-bit elements, each a value and its
// tag.  A vector access promises nothing beyond its elements (PTX models it as
// one access per element, in any order), so the pair has to be one element.

__device__ __forceinline__ uint4 ld_box(const uint4* p)
{
    uint4 v;
    asm volatile("{\n\t.reg .b64 lo, hi;\n\tld.relaxed.gpu.global.v2.b64 {lo, hi}, [%4];\n\t"
                 "mov.b64 {%0, %1}, lo;\n\tmov.b64 {%2, %3}, hi;\n\t}"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

__device__ __forceinline__ void st_box(uint4* p, uint32_t a, uint32_t b, uint32_t tag)
{
    asm volatile("{\n\t.reg .b64 lo, hi;\n\tmov.b64 lo, {%1, %2};\n\tmov.b64 hi, {%3, %2};\n\t"
                 "st.relaxed.gpu.global.v2.b64 [%0], {lo, hi};\n\t}" ::"l"(p), "r"(a), "r"(tag), "r"(b)
                 : "memory");
}

// ---- barriers in shared memory
__device__ __forceinline__ uint32_t res_smem(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void bar_init(uint64_t* b, int count)
{
    asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(res_smem(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void bar_arrive(uint64_t* b)
{
    asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.shared.b64 t, [%0];\n\t}" ::"r"(res_smem(b))
                 : "memory");
}

// whether the phase of this parity has completed; a poll is suspended for a
// microsecond at most
__device__ __forceinline__ bool bar_try(uint64_t* b, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(res_smem(b)), "r"(parity), "r"(1000u)  // ns
        : "memory");
    return done != 0;
}

// the same, after up to `limit` polls
__device__ __forceinline__ bool bar_wait(uint64_t* b, uint32_t parity, const volatile int& limit)
{
    bool done = bar_try(b, parity);
    if (!done) {
        int polls = limit;
        while (!done && --polls > 0) done = bar_try(b, parity);
    }
    return done;
}

// named barriers: 1 the sweep warps, 2 these and the helper of the E rounds
__device__ __forceinline__ void sync_sweepers()
{
    asm volatile("barrier.cta.sync 1, %0;" ::"n"(kResSweepers) : "memory");
}
__device__ __forceinline__ void sync_grid()
{
    asm volatile("barrier.cta.sync 2, %0;" ::"n"(kResSweepers + 32) : "memory");
}

// ---- sums of float pairs: h + l, |l| <= ulp(h) / 2 (TwoSum, Knuth)
struct Pair {
    float h, l;
};

__device__ __forceinline__ Pair pair_add(Pair a, Pair b)
{
    const float s = __fadd_rn(a.h, b.h);
    if (!(fabsf(s) <= 3.402823466e38f)) return {s, 0.0f};  // the error of an infinite sum is NaN
    const float t = __fsub_rn(s, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
    const float f = __fadd_rn(e, __fadd_rn(a.l, b.l));
    const float h = __fadd_rn(s, f);
    return {h, __fsub_rn(f, __fsub_rn(h, s))};
}

// over the eight lanes of a group, result in its first lane
__device__ __forceinline__ Pair pair_tree(Pair v)
{
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
        const Pair o = {__shfl_down_sync(0xffffffffu, v.h, off, 8),
                        __shfl_down_sync(0xffffffffu, v.l, off, 8)};
        v = pair_add(v, o);
    }
    return v;
}

// A wait of this CTA ran out: the others wait for one poll only from now on.
__device__ __forceinline__ void give_up(const ResArgs& a, volatile int& limit)
{
    a.err[0] = a.err[1] = 1;
    limit = 1;
}

template <int C, int R, int WX>
struct ResWarp {
    using L = ResLayout<C, R, WX>;
    static constexpr int V = C / 4;
    uint8_t* sm;
    int lane, wid, wx, wy;
    bool flip;        // register row r is image row y0 + R - 1 - r
    bool rem;         // the row beside register row 0 comes from another CTA
    bool out;         // this lane lies outside the grid
    bool mute;        // its residuals are not this CTA's to sum
    uint32_t gen;     // bit g: some cell of rows 4g..4g+3 differs from its column's default
    uint32_t skip;    // bit g: rows 4g..4g+3 lie outside the grid
    float c0, inv0, invm, inv3, c3;  // column defaults (first, inner and last cell; inner c = 0)
    int in_f, in_l;   // byte offsets (parity 0) of the rows beside rows 0 and R - 1
    int in_c;         // of the column beside this lane's edge (left, lane 31: right)
    int out_r, out_c; // of this warp's own rows and column
    int in_h;         // of the row received from the neighbouring CTA
    uint64_t* full;   // [parity]: it is there
    volatile int* limit;  // ResShared::limit
    uint4* tx;        // [parity][word] to the neighbouring CTA, this lane
    uint32_t t;       // messages sent (= received and being waited for) so far

    __device__ __forceinline__ void ld_row(int off, float (&v)[C]) const
    {
#pragma unroll
        for (int h = 0; h < V; ++h) {
            const float4 f = *reinterpret_cast<const float4*>(sm + off + 512 * h);
            v[4 * h] = f.x; v[4 * h + 1] = f.y; v[4 * h + 2] = f.z; v[4 * h + 3] = f.w;
        }
    }
    __device__ __forceinline__ void st_row(int off, const float (&v)[C]) const
    {
#pragma unroll
        for (int h = 0; h < V; ++h)
            *reinterpret_cast<float4*>(sm + off + 512 * h) =
                make_float4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
    }
    static constexpr int kMsgLanes = 32 * WX;
    // the row of message t, from the helper that receives it; bounded
    __device__ __forceinline__ void receive(float (&v)[C], const ResArgs& a)
    {
        if (!bar_wait(full + (t & 1u), (t - 1) >> 1 & 1u, *limit)) give_up(a, *limit);
        ld_row(in_h + (t & 1u ? L::kHaloPar : 0), v);
    }
    __device__ __forceinline__ void send(const float (&v)[C], uint32_t tag) const
    {
        uint4* p = tx + (tag & 1u) * 256;
#pragma unroll
        for (int i = 0; i < 2 * V; ++i)
            st_box(p + kMsgLanes * i, __float_as_uint(v[2 * i]), __float_as_uint(v[2 * i + 1]), tag);
    }
    // boundary values of phi into the buffers of message t + 1
    __device__ __forceinline__ void publish(const float (&phi)[R][C])
    {
        ++t;
        const int pr = (t & 1u) ? L::kRowPar : 0, pc = (t & 1u) ? L::kColPar : 0;
        st_row(out_r + pr, phi[0]);
        st_row(out_r + pr + L::kRowSlot, phi[R - 1]);
        if (rem) send(phi[0], t);
        if (WX > 1) {
#pragma unroll
            for (int r = 0; r < R; r += 4) {
                const bool q = lane == 31;
                const float4 c = make_float4(
                    q ? phi[r][C - 1] : phi[r][0], q ? phi[r + 1][C - 1] : phi[r + 1][0],
                    q ? phi[r + 2][C - 1] : phi[r + 2][0], q ? phi[r + 3][C - 1] : phi[r + 3][0]);
                if (lane == 0 || lane == 31)
                    *reinterpret_cast<float4*>(sm + out_c + pc + 4 * r) = c;
            }
        }
    }
    // every message is received, also the one no sweep uses: the sender counts on it
    __device__ __forceinline__ void drain(const ResArgs& a)
    {
        if (rem) {
            float v[C];
            receive(v, a);
        }
    }

    // phi_{k+1} from phi_k and the boundary values of message t; sends message
    // t + 1.  WITH_E: `pending` (this thread's FP32 sum of |r(phi_{k-1})|) is
    // summed over groups of eight lanes while the rows are computed, stored in
    // *wsum by lanes 0..3, and becomes the sum of |r(phi_k)|.
    template <bool WITH_E>
    __device__ __forceinline__ void update(float (&phi)[R][C], float& pending, float* wsum,
                                           const ResArgs& a)
    {
        const int pr = (t & 1u) ? L::kRowPar : 0, pc = (t & 1u) ? L::kColPar : 0;
        const int qr = L::kRowPar - pr, qc = L::kColPar - pc;
        // a warp-wide OR lands in a uniform register: the branches below stay
        // uniform (a fifth of the instructions were their divergence handling)
        const uint32_t cls = __reduce_or_sync(0xffffffffu, gen | skip << 8 | (rem ? 1u << 16 : 0u));
        const uint32_t any = cls | cls >> 8;
        const bool far = (cls >> 16) != 0;
        // ds of the row before: south difference, the negated north one of this row
        float dsp[C];
        if (far) receive(dsp, a);
        else ld_row(in_f + pr, dsp);
#pragma unroll
        for (int q = 0; q < C; ++q) dsp[q] = __fsub_rn(phi[0][q], dsp[q]);
        const int s_div = L::kDiv + (wid * R * V * 32 + lane) * 16;
        const int s_code = L::kCode + (wid * R * 32 + lane) * 4;
        // |r| in four chains, by column; with 128 cells a thread they would be 32
        // values long, so every four rows are added up by themselves
        constexpr bool kSplit = R * C > 64;
        float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        float sum[2] = {0.0f, 0.0f};
        float s = pending;
        // one row: differences of phi_k (each formed once: south of row r is
        // minus north of row r + 1, east of a cell minus west of the next),
        // then the update in one of two forms
        auto row = [&](auto plain, int r, float halo) {
            float d[C];
            ld_row(s_div + r * L::kRowSlot, d);
            float left = __shfl_up_sync(0xffffffffu, phi[r][C - 1], 1);
            float right = __shfl_down_sync(0xffffffffu, phi[r][0], 1);
            if (lane == 0) left = halo;
            if (lane == 31) right = halo;
            float below[C];
            if (r + 1 == R) ld_row(in_l + pr, below);
            float exw = __fsub_rn(phi[r][0], left);
            uint32_t even = 0, odd = 0;  // 8 n of the even and of the odd cells, a byte each
            if (!plain.value) {
                const uint32_t code = *reinterpret_cast<const uint32_t*>(sm + s_code + r * 128);
                even = (code << 3) & 0x78787878u;
                odd = (code >> 1) & 0x78787878u;
            }
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const float pc0 = phi[r][q];
                const float exe = __fsub_rn(q + 1 < C ? phi[r][q + 1] : right, pc0);
                const float ds = __fsub_rn(r + 1 < R ? phi[r + 1 < R ? r + 1 : r][q] : below[q], pc0);
                float lap = __fadd_rn(__fsub_rn(exe, exw), __fsub_rn(ds, dsp[q]));
                exw = exe;
                dsp[q] = ds;
                float res;
                if (plain.value) {
                    float inv = invm;
                    if (q == 0) {
                        lap = __fmaf_rn(c0, pc0, lap);
                        inv = inv0;
                    } else if (q == C - 1) {
                        lap = __fmaf_rn(c3, pc0, lap);
                        inv = inv3;
                    }
                    res = __fsub_rn(d[q], lap);
                    phi[r][q] = __fmaf_rn(-res, inv, pc0);
                } else {
                    const float2 k = *reinterpret_cast<const float2*>(
                        sm + L::kLut + (((q & 1 ? odd : even) >> (8 * (q / 2))) & 0xffu));
                    // [n > 0] from 1/n in {0, 1/4, 1/3, 1/2, 1}: saturate(4/n) is 0 or 1
                    lap = __fmaf_rn(k.x, pc0, lap);
                    res = __fmaf_rn(-__saturatef(k.y * 4.0f), lap, d[q]);
                    phi[r][q] = __fmaf_rn(-res, k.y, pc0);
                }
                if (WITH_E) acc[q % 4] = __fadd_rn(acc[q % 4], fabsf(res));
            }
        };
#pragma unroll
        for (int g = 0; g < R / 4; ++g) {
            float h[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (WX > 1) {
                const float4 hv = *reinterpret_cast<const float4*>(sm + in_c + pc + 16 * g);
                h[0] = hv.x; h[1] = hv.y; h[2] = hv.z; h[3] = hv.w;
            }
            // after row i of the group: the boundary rows go out, a level of
            // the warp sum of the sweep before
            auto after = [&](int i) {
                const int r = 4 * g + i;
                if (r == 0) {
                    if (far) send(phi[0], t + 1);
                    st_row(out_r + qr, phi[0]);
                }
                if (r == R - 1) st_row(out_r + qr + L::kRowSlot, phi[R - 1]);
            };
            if (WITH_E) {
#pragma unroll
                for (int i = 0; i < 3; ++i) {  // three levels over the groups there are
                    if (i * (R / 4) / 3 == g)
                        s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, 16 >> i));
                }
            }
            if (!(any & (1u << g))) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    row(Bool<true>{}, 4 * g + i, h[i]);
                    after(i);
                }
            } else if (!(cls & (256u << g))) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    row(Bool<false>{}, 4 * g + i, h[i]);
                    after(i);
                }
            } else {  // phi stays 0; the next group's north differences
#pragma unroll
                for (int q = 0; q < C; ++q)
                    dsp[q] = 4 * g + 4 < R ? phi[4 * g + 4 < R ? 4 * g + 4 : 0][q] : 0.0f;
#pragma unroll
                for (int i = 0; i < 4; ++i) after(i);
            }
            if (WITH_E && kSplit) {
                sum[g / 2] = __fadd_rn(sum[g / 2], __fadd_rn(__fadd_rn(acc[0], acc[1]),
                                                             __fadd_rn(acc[2], acc[3])));
                acc[0] = acc[1] = acc[2] = acc[3] = 0.0f;
            }
            if (WX > 1) {
                const bool q = lane == 31;
                // predicated, not branched around
                asm volatile(
                    "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %5, 0;\n\t"
                    "@p st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n\t}" ::"r"(
                        (uint32_t)__cvta_generic_to_shared(sm + out_c + qc + 16 * g)),
                    "f"(q ? phi[4 * g][C - 1] : phi[4 * g][0]),
                    "f"(q ? phi[4 * g + 1][C - 1] : phi[4 * g + 1][0]),
                    "f"(q ? phi[4 * g + 2][C - 1] : phi[4 * g + 2][0]),
                    "f"(q ? phi[4 * g + 3][C - 1] : phi[4 * g + 3][0]),
                    "r"((int)(lane == 0 || q))
                    : "memory");
            }
        }
        ++t;
        if (WITH_E) {
            if (lane < kResSums) *wsum = s;
            pending = mute ? 0.0f : __fadd_rn(
                kSplit ? sum[0] : __fadd_rn(acc[0], acc[1]),
                kSplit ? sum[1] : __fadd_rn(acc[2], acc[3]));
        }
    }
    template <bool P>
    struct Bool {
        static constexpr bool value = P;
    };
};

// Shared by the sweep warps and the helpers of one CTA.
struct ResShared {
    uint64_t full[2][2];       // [side][parity]: a neighbour's row is there
    uint64_t sums[kResRing];   // the warp sums of a round are there
    volatile uint32_t end;     // messages in all, once the CTA is done
    volatile int rounds;       // rounds of this grid decided
    volatile int stop;         // the round that stopped it
    int kstar, code;           // k*; 1 converged, 2 not
    double estar;
    int act;                   // 1: leave the sweep loop
    int begun;                 // rounds begun by then
    volatile int limit;        // polls of a wait; 1 once one has given up
    int grid;                  // next grid of the group
};

// Sweeps from checkpoint k to the next.  A store of a strip costs two to four of
// its sweeps, a stop replays half a step on average, so the step grows as the
// root of the sweeps done; 16 sweeps or more, since a decision may take 12.
// (With 32 from the start, a stop at sweep 20 or 60 took up to 1.4 times as
// long: 256 x 128^2 323 and 243 us, 410 and 330 us.)
__device__ __forceinline__ int ckpt_step(int k)
{
    return k < 64 ? 16 : k < 256 ? 32 : k < 1024 ? 64 : 128;
}

// Helper warp: rows from the neighbouring CTA on one side into shared memory.
template <int C, int R, int WX>
__device__ __forceinline__ void res_receiver(const ResArgs& a, uint8_t* sm, ResShared& sh, int cta,
                                             int side)
{
    using L = ResLayout<C, R, WX>;
    constexpr int W = 2 * L::V;  // words per source lane
    const int lane = threadIdx.x & 31;
    for (uint32_t t = 1;; ++t) {
        const int limit = __shfl_sync(0xffffffffu, sh.limit, 0);  // the warp's
#pragma unroll 1
        for (int x = 0; x < WX; ++x) {
            const uint4* p = &a.box->row[cta][side][t & 1u][32 * x + lane];
            uint4 v[W];
            int left = limit;
            for (;;) {
                bool ok = true;
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    v[i] = ld_box(p + i * 32 * WX);
                    ok = ok && v[i].y == t && v[i].w == t;
                }
                if (__all_sync(0xffffffffu, ok)) break;
                const uint32_t end = sh.end;
                if (__any_sync(0xffffffffu, end != 0 && t > end)) return;
                if (--left <= 0) {
                    give_up(a, sh.limit);
                    return;
                }
            }
            uint8_t* dst = sm + L::kHalo + (side * 2 + (t & 1u)) * L::kHaloPar + lane * 16;
#pragma unroll
            for (int h = 0; h < L::V; ++h)
                *reinterpret_cast<uint4*>(dst + (x * L::V + h) * 512) =
                    make_uint4(v[2 * h].x, v[2 * h].z, v[2 * h + 1].x, v[2 * h + 1].z);
        }
        __syncwarp();
        if (lane == 0) bar_arrive(&sh.full[side][t & 1u]);
    }
}

// Helper warp: the E rounds of one grid, `first` rounds of other grids before
// it.  Lane group gi (8 lanes) takes sweep 4q + gi of round q.
__device__ __forceinline__ void res_rounds(const ResArgs& a, const float* s_wsum, ResShared& sh,
                                           int b, uint32_t first)
{
    const int lane = threadIdx.x & 31, gi = lane >> 3, li = lane & 7;
    const int n = a.n, cta = blockIdx.x, group = cta / n, rank = cta % n;
    const double inv_cells = 1.0 / ((double)a.nx * (double)a.ny * kSumScale);
    for (int q = 0;; ++q) {
        const uint32_t e = first + q, tag = e + 1, slot = e % kResRing;
        // (lanes look at a barrier and at words one by one: every decision
        // about a wait is taken by the warp)
        bool there = __all_sync(
            0xffffffffu, bar_wait(&sh.sums[slot], e / kResRing & 1u, sh.limit));
        const float4 ws = reinterpret_cast<const float4*>(
            s_wsum)[(e * 4 + gi) % kWsumRing * kResWarps + li];
        Pair sum = pair_tree(
            pair_add(pair_add({ws.x * kSumScale, 0.0f}, {ws.y * kSumScale, 0.0f}),
                     pair_add({ws.z * kSumScale, 0.0f}, {ws.w * kSumScale, 0.0f})));
        if (n > 1) {
            if (li == 0)
                st_box(&a.box->part[cta][slot][gi], __float_as_uint(sum.h), __float_as_uint(sum.l),
                       tag);
            if (rank == 0) {
                sum = {0.0f, 0.0f};
                for (int i = li; i < n; i += 32) {  // four loads in flight
                    uint4 v[4];
                    int left = sh.limit;
                    bool ok;
                    do {
                        ok = true;
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int c = i + 8 * u < n ? i + 8 * u : i;
                            v[u] = ld_box(&a.box->part[cta + c][slot][gi]);
                            ok = ok && v[u].y == tag && v[u].w == tag;
                        }
                    } while (!ok && --left > 0);
                    there = there && ok;
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (i + 8 * u < n)
                            sum = pair_add(sum, {__uint_as_float(v[u].x), __uint_as_float(v[u].z)});
                }
                there = __all_sync(0xffffffffu, there);
                sum = pair_tree(sum);
            }
        }
        int code = 0, ks = 0;
        if (rank == 0) {
            // the first lane of each group of eight holds the sum of its sweep
            const int j = 4 * q + gi;
            double ej = 0.0;
            int c = 0;
            if (li == 0 && (!(sum.h > a.sum_near) || !(sum.h <= 3e38f) || j >= a.cap || a.e_hist)) {
                ej = ((double)sum.h + (double)sum.l) * inv_cells;
                if (ej <= a.threshold) c = 1;
                else if (j >= a.cap || !isfinite(ej)) c = 2;
            }
            const uint32_t hit = __ballot_sync(0xffffffffu, c != 0);
            const int from = hit ? __ffs(hit) - 1 : 31;
            if (a.e_hist && li == 0 && lane <= from && j < a.hist_len)
                a.e_hist[(size_t)b * a.hist_len + j] = ej;
            code = there ? __shfl_sync(0xffffffffu, c, from) : 2;  // 2: all leave
            ks = there ? 4 * q + (from >> 3) : 0;
            if (lane == from) sh.estar = ej;
            if (n > 1 && lane == 0)
                st_box(&a.box->dec[group][slot], (uint32_t)code, (uint32_t)ks, tag);
        } else {
            uint4 v;
            int left = sh.limit;
            do {
                v = ld_box(&a.box->dec[group][slot]);
            } while ((v.y != tag || v.w != tag) && --left > 0);
            there = __all_sync(0xffffffffu, there && v.y == tag && v.w == tag);
            code = there ? (int)v.x : 2;
            ks = there ? (int)v.z : 0;
        }
        if (!there) give_up(a, sh.limit);
        __syncwarp();
        if (lane == 0) {
            if (code != 0) {
                sh.kstar = ks;
                sh.code = code;
                sh.stop = q;
            }
            __threadfence_block();
            sh.rounds = q + 1;
        }
        __syncwarp();
        if (code != 0) return;
    }
}

// The copied columns of phi from the CTAs beside (left, right: there is one),
// message m: each warp sends its first and last own columns and waits for its
// neighbours' (the same warp of those CTAs, so message m + 2 cannot overtake
// message m).
template <int R, int WX>
__device__ __forceinline__ void res_columns(const ResArgs& a, uint8_t* sm, float (&phi)[R][8],
                                            int cta, int wid, int lane, bool left, bool right,
                                            uint32_t m, volatile int& limit)
{
    using L = ResLayout<8, R, WX>;
    constexpr int W = R / 8;  // words per lane and side
    float* stage = reinterpret_cast<float*>(sm + L::kGhost) + wid * 2 * R * kResGhost;
    __syncwarp();
    if (lane == 1 || lane == 30) {
        float4* dst = reinterpret_cast<float4*>(stage + (lane == 1 ? 0 : R * kResGhost));
#pragma unroll
        for (int r = 0; r < R; ++r) {
            dst[2 * r] = make_float4(phi[r][0], phi[r][1], phi[r][2], phi[r][3]);
            dst[2 * r + 1] = make_float4(phi[r][4], phi[r][5], phi[r][6], phi[r][7]);
        }
    }
    __syncwarp();
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        if (side ? !right : !left) continue;
        uint4* box = a.cols->w[side ? cta + 1 : cta - 1][side ^ 1][m & 1u][wid][0];
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const float2 v =
                *reinterpret_cast<const float2*>(stage + side * R * kResGhost + (i * 32 + lane) * 2);
            st_box(box + i * 32 + lane, __float_as_uint(v.x), __float_as_uint(v.y), m);
        }
    }
    __syncwarp();
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        if (side ? !right : !left) continue;
        const uint4* box = a.cols->w[cta][side][m & 1u][wid][0];
        uint4 v[W];
        int polls = __shfl_sync(0xffffffffu, limit, 0);  // the warp's
        for (;;) {
            bool ok = true;
#pragma unroll
            for (int i = 0; i < W; ++i) {
                v[i] = ld_box(box + i * 32 + lane);
                ok = ok && v[i].y == m && v[i].w == m;
            }
            if (__all_sync(0xffffffffu, ok)) break;
            if (--polls <= 0) {
                give_up(a, limit);
                break;
            }
        }
#pragma unroll
        for (int i = 0; i < W; ++i)
            *reinterpret_cast<float2*>(stage + side * R * kResGhost + (i * 32 + lane) * 2) =
                make_float2(__uint_as_float(v[i].x), __uint_as_float(v[i].z));
    }
    __syncwarp();
    if ((lane == 0 && left) || (lane == 31 && right)) {
        const float4* src = reinterpret_cast<const float4*>(stage + (lane == 0 ? 0 : R * kResGhost));
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 u = src[2 * r], v = src[2 * r + 1];
            phi[r][0] = u.x; phi[r][1] = u.y; phi[r][2] = u.z; phi[r][3] = u.w;
            phi[r][4] = v.x; phi[r][5] = v.y; phi[r][6] = v.z; phi[r][7] = v.w;
        }
    }
    __syncwarp();
}

// WIDE: the grid is cut into columns too
template <int C, int R, int WX, bool WIDE>
__global__ void __launch_bounds__(kResThreads, 1) sweep_resident_kernel(const ResArgs a)
{
    using L = ResLayout<C, R, WX>;
    using W = ResWarp<C, R, WX>;
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ ResShared sh;
    static_assert(!WIDE || (C == kResGhost && WX == 1), "one lane of copies on each side");
    const int n = a.n, cta = blockIdx.x, group = cta / n, rank = cta % n;
    // strips above one another are ntx CTAs apart
    const int ntx = WIDE ? a.ntx : 1, ty = rank / ntx, tx = rank % ntx, nty = n / ntx;
    float* s_wsum = reinterpret_cast<float*>(sm + L::kWsum);

    W w;
    w.sm = sm;
    w.lane = threadIdx.x & 31;
    w.wid = threadIdx.x >> 5;
    constexpr int kZero = 2 * kResWarps;  // slot of the zero row / column
    if (threadIdx.x < 32) {
        const float z[C] = {};
        for (int p = 0; p < 2; ++p) {
            w.st_row(L::kRow + p * L::kRowPar + kZero * L::kRowSlot + w.lane * 16, z);
            if (threadIdx.x < R)
                *reinterpret_cast<float*>(sm + L::kCol + p * L::kColPar + kZero * R * 4 +
                                          threadIdx.x * 4) = 0.0f;
        }
        if (threadIdx.x < 5) {
            const CellConst k = make_const(0.0f, (1u << threadIdx.x) - 1u);
            *reinterpret_cast<float2*>(sm + L::kLut + 8 * threadIdx.x) = make_float2(k.c, k.inv);
        }
        if (threadIdx.x == 0) {
            for (int i = 0; i < 4; ++i) bar_init(&sh.full[i / 2][i % 2], 1);
            for (int i = 0; i < kResRing; ++i) bar_init(&sh.sums[i], 1);
            sh.end = 0u;
            sh.limit = a.polls;
        }
    }
    __syncthreads();

    if (w.wid >= kResWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kResRegsHelp));
        if (w.wid == kResWarps) {
            int b = group;
            uint32_t first = 0;
            while (b < a.B) {
                sync_grid();  // the sweep warps have set the grid up
                const bool with_e = !a.fixed || a.gs[b].wild == a.epoch;
                if (with_e) res_rounds(a, s_wsum, sh, b, first);
                sync_grid();  // the grid is done
                if (with_e) first += (uint32_t)sh.begun;
                if (a.groups >= a.B) break;
                sync_grid();
                b = sh.grid;
            }
        } else if (w.wid == kResWarps + 1) {
            if (ty > 0) res_receiver<C, R, WX>(a, sm, sh, cta, 0);
        } else if (w.wid == kResWarps + 2) {
            if (ty < nty - 1) res_receiver<C, R, WX>(a, sm, sh, cta, 1);
        }
        return;
    }
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kResRegsSweep));

    w.wx = w.wid % WX;
    w.wy = w.wid / WX;
    w.flip = w.wy >= L::WY / 2;
    const int nx = a.nx, ny = a.ny;
    const bool vec = (nx & 3) == 0;
    const bool top = w.wy == 0, bottom = w.wy == L::WY - 1;
    w.rem = (top && ty > 0) || (bottom && ty < nty - 1);
    {
        // a row goes into the box of the CTA above (from below) or below (from above)
        const int peer = top ? cta - ntx : cta + ntx;
        w.tx = w.rem ? &a.box->row[peer][top ? 1 : 0][0][w.wx * 32 + w.lane] : nullptr;
        const int side = top ? 0 : 1;
        w.full = sh.full[side];
        w.in_h = L::kHalo + side * 2 * L::kHaloPar + w.wx * L::kRowSlot + w.lane * 16;
    }
    w.t = 0;
    w.limit = &sh.limit;
    const bool left = WIDE && tx > 0, right = WIDE && tx < ntx - 1;
    const int x0 = (WIDE ? tx * (32 * C - 2 * kResGhost) - kResGhost : 0) + (w.wx * 32 + w.lane) * C;
    const int y0 = (ty * L::WY + w.wy) * R;
    const bool copy = WIDE && (w.lane == 0 || w.lane == 31);
    w.out = x0 < 0 || x0 >= nx;
    w.mute = w.out || copy;
    auto row_of = [&](int r) { return w.flip ? y0 + R - 1 - r : y0 + r; };

    // where the neighbouring rows and columns of this warp are published
    {
        auto slot_of = [&](int v, int vy, bool low) {  // warp v, its lower (image) row or upper
            const bool vf = vy >= L::WY / 2;
            return 2 * v + (low != vf ? 1 : 0);
        };
        const int above = top ? kZero : slot_of(w.wid - WX, w.wy - 1, true);
        const int below = bottom ? kZero : slot_of(w.wid + WX, w.wy + 1, false);
        w.in_f = L::kRow + (w.flip ? below : above) * L::kRowSlot + w.lane * 16;
        w.in_l = L::kRow + (w.flip ? above : below) * L::kRowSlot + w.lane * 16;
        w.out_r = L::kRow + 2 * w.wid * L::kRowSlot + w.lane * 16;
        const int cl = w.wx > 0 ? 2 * (w.wid - 1) + 1 : kZero;
        const int cr = w.wx < WX - 1 ? 2 * (w.wid + 1) : kZero;
        w.in_c = L::kCol + (w.lane == 31 ? cr : cl) * R * 4;
        w.out_c = L::kCol + (2 * w.wid + (w.lane == 31 ? 1 : 0)) * R * 4;
    }
    // columns an unobstructed inner row has: a wall left of x = 0 and right of nx - 1
    const bool wall0 = x0 == 0, wall3 = x0 + C == nx;
    w.c0 = wall0 ? 1.0f : 0.0f;
    w.c3 = wall3 ? 1.0f : 0.0f;
    w.invm = w.out ? 0.0f : 0.25f;
    w.inv0 = w.out ? 0.0f : wall0 ? 1.0f / 3.0f : 0.25f;
    w.inv3 = w.out ? 0.0f : wall3 ? 1.0f / 3.0f : 0.25f;

    int b = group;
    uint32_t seq = 0;    // grids this group has begun
    uint32_t first = 0;  // E rounds of the grids before this one
    uint32_t fetched = 0;  // messages with copied columns
    float phi[R][C];
    while (b < a.B) {
        ++seq;
        const size_t gbase = (size_t)b * ny * nx;
        // register rows r_lo .. r_hi - 1 are rows of the grid
        const int r_lo = w.flip ? max(0, y0 + R - ny) : 0;
        const int r_hi = w.flip ? R : min(R, ny - y0);
        const size_t first_cell = gbase + (size_t)row_of(0) * nx + x0;
        const ptrdiff_t row_step = w.flip ? -(ptrdiff_t)nx : (ptrdiff_t)nx;
        // (loads and stores of 128 cells, several times in the kernel: written
        // for few instructions, since a call's first sweeps wait for the
        // kernel's code to be fetched)
        auto load_cells = [&](const float* src, bool masked, bool v4) {
            const float* line = src + first_cell;
#pragma unroll
            for (int r = 0; r < R; ++r, line += row_step) {
                const bool in = src && r >= r_lo && r < r_hi;
                if (v4) {
#pragma unroll
                    for (int h = 0; h < C; h += 4) {
                        float4 f = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        if (in && x0 + h >= 0 && x0 + h < nx)
                            f = *reinterpret_cast<const float4*>(line + h);
                        phi[r][h] = f.x; phi[r][h + 1] = f.y;
                        phi[r][h + 2] = f.z; phi[r][h + 3] = f.w;
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < C; ++q)
                        phi[r][q] = in && x0 + q >= 0 && x0 + q < nx ? line[q] : 0.0f;
                }
                if (masked) {
                    const uint32_t code =
                        reinterpret_cast<const uint32_t*>(sm + L::kCode)[(w.wid * R + r) * 32 + w.lane];
#pragma unroll
                    for (int q = 0; q < C; ++q)
                        if (!((code >> (4 * q)) & 15u)) phi[r][q] = 0.0f;
                }
            }
        };
        auto store_cells = [&](float* dst) {
            float* line = dst + first_cell;
#pragma unroll
            for (int r = 0; r < R; ++r, line += row_step) {
                const bool in = !copy && r >= r_lo && r < r_hi;
                if (vec) {
#pragma unroll
                    for (int h = 0; h < C; h += 4)
                        if (in && x0 + h < nx)
                            *reinterpret_cast<float4*>(line + h) = make_float4(
                                phi[r][h], phi[r][h + 1], phi[r][h + 2], phi[r][h + 3]);
                } else {
#pragma unroll
                    for (int q = 0; q < C; ++q)
                        if (in && x0 + q < nx) line[q] = phi[r][q];
                }
            }
        };

        // the copied columns anew; the boundary rows go out again with them
        auto refresh = [&]() {
            if constexpr (WIDE) {
                ++fetched;
                res_columns<R, WX>(a, sm, phi, cta, w.wid, w.lane, left, right, fetched, sh.limit);
                w.publish(phi);
                sync_sweepers();
            }
        };
        // ---- div and the open-face counts on chip, phi_0 in registers
        w.gen = 0u;
        w.skip = (1u << (R / 4)) - 1u;
#pragma unroll 1
        for (int r = 0; r < R; ++r) {
            const int y = row_of(r);
            bool plain = true;
            uint32_t code = 0;
#pragma unroll
            for (int h = 0; h < L::V; ++h) {
                float dr[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                uint32_t m4 = 0;
                if (y < ny) {
                    const size_t o = gbase + (size_t)y * nx;
                    load_row4(a.div + o, x0 + 4 * h, nx, vec, dr);
                    m4 = load_mask4(a.mask + o, x0 + 4 * h, nx, vec);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int cnt = __popc((m4 >> (8 * q)) & 15u);
                    const bool wall = (h == 0 && q == 0 && wall0) ||
                                      (h == L::V - 1 && q == 3 && wall3);
                    plain = plain && cnt == (wall ? 3 : 4);
                    code |= (uint32_t)cnt << (4 * (4 * h + q));
                }
                const int slot = ((w.wid * R + r) * L::V + h) * 32 + w.lane;
                reinterpret_cast<float4*>(sm + L::kDiv)[slot] =
                    make_float4(dr[0], dr[1], dr[2], dr[3]);
            }
            reinterpret_cast<uint32_t*>(sm + L::kCode)[(w.wid * R + r) * 32 + w.lane] = code;
            if (__any_sync(0xffffffffu, !w.out && y < ny)) w.skip &= ~(1u << (r / 4));
            if (!__all_sync(0xffffffffu, w.out || plain)) w.gen |= 1u << (r / 4);
        }
        load_cells(a.phi0, true, vec && a.phi0_vec);
        if (threadIdx.x == 0) {
            sh.act = 0;
            sh.rounds = 0;
            sh.stop = -1;
        }
        float pending = 0.0f;
        int kstar = a.cap, dec = 2;
        double estar = 0.0;
        w.publish(phi);
        sync_grid();

        const bool with_e = !a.fixed || a.gs[b].wild == a.epoch;
        constexpr bool kOneLoop = R * C > 64;
        // sweeps without E: a run of fixed length, or a replay
        int done = 0;
        bool alone = !with_e;
        if (with_e) {
            // Four sweeps at a time; round q needs the sums of sweeps 4q .. 4q+3,
            // the last stored during sweep 4q + 4.  A replay from phi_0 or the
            // checkpoint at or below k* to phi_{k*} takes the same loop where a
            // thread has 128 cells (and leaves its sums unread): the code of the
            // sweeps without E, 94 KB, would have to be fetched first, which took
            // as long as five sweeps (4 x 1024^2, stop at sweep 3: 250 and 200
            // us).  With fewer cells that code is smaller, and the sweeps below
            // are faster (16 x 512^2: 20.0 and 19.9 ms in all).
            int last = 0, before = 0, cb = 1;  // latest checkpoints, buffer of the latest
            bool replay = false;
            for (int k = 0;; k += 4) {
                bool loaded = false;
                if (!replay && sh.act != 0) {
                    kstar = sh.kstar;
                    dec = sh.code;
                    estar = sh.estar;
                    first += (uint32_t)(k / 4 - 1);
                    w.drain(a);
                    if (kstar == a.cap) break;  // phi has been stored
                    const int base = kstar >= last ? last : before;
                    load_cells(base == 0 ? a.phi0 : a.ck[base == last ? cb : cb ^ 1], base == 0,
                               vec && (base != 0 || a.phi0_vec));
                    sync_sweepers();
                    if (!WIDE || base == 0) {
                        w.publish(phi);
                        sync_sweepers();
                    }
                    if (!kOneLoop) {
                        if (WIDE && base > 0) refresh();
                        done = base;
                        alone = true;
                        break;
                    }
                    k = base;
                    replay = loaded = true;
                }
                const int todo = (replay ? kstar : a.cap + 1) - k;
                const int keep_at = replay ? todo : todo - 1;
                if (!replay && k == last + ckpt_step(last) && k <= a.cap) {
                    cb ^= 1;
                    store_cells(a.ck[cb]);
                    before = last;
                    last = k;
                }
                const bool one_thread = threadIdx.x == kResSweepers / 2 && !replay;
                if (WIDE && k > 0 && k % kResGhost == 0 && (todo > 0 || loaded)) {
                    if (!loaded) w.drain(a);
                    refresh();
                }
#pragma unroll 1
                for (int i = 0; i < 4; ++i) {
                    // (behind the barrier that follows the last store of its sums)
                    if (i == 1 && one_thread && k > 0)
                        bar_arrive(&sh.sums[(first + k / 4 - 1) % kResRing]);
                    const int lag = res_lag(k, n);
                    if (i == 3 && one_thread && k + 4 >= 4 * lag) {
                        // the decision of round k / 4 + 1 - lag: mostly there
                        const int q = k / 4 + 1 - lag;
                        int left = sh.limit == 1 ? 1 : a.looks;
                        while (sh.rounds <= q && --left > 0) {
                        }
                        if (sh.rounds <= q) {
                            give_up(a, sh.limit);
                            sh.kstar = 0;
                            sh.code = 2;
                            sh.estar = 0.0;
                            sh.stop = q;
                        }
                        __threadfence_block();
                        if (sh.stop == q) {
                            sh.begun = k / 4;
                            sh.act = 1;
                        }
                    }
                    float* wsum = s_wsum + (((k + i - 1 + 4 * (int)first) & (kWsumRing - 1)) * kResWarps +
                                            w.wid) * kResSums + w.lane;
                    if (i == keep_at) store_cells(a.phi);
                    if (i < todo) {
                        w.template update<true>(phi, pending, wsum, a);
                    } else if (replay) {
                        break;
                    } else if (i == todo) {
                        // past the cap only its sum is left to do
                        float s = pending;
#pragma unroll
                        for (int off = 16; off >= kResSums; off >>= 1)
                            s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, off));
                        if (w.lane < kResSums) *wsum = s;
                    }
                    sync_sweepers();
                }
                if (replay && kstar < k + 4) {
                    w.drain(a);
                    break;
                }
            }
        }
        if (alone) {
            for (int j = done; j < kstar; ++j) {
                if (WIDE && j > done && j % kResGhost == 0) {
                    w.drain(a);
                    refresh();
                }
                w.template update<false>(phi, pending, nullptr, a);
                sync_sweepers();
            }
            store_cells(a.phi);
            w.drain(a);
        }
        if (threadIdx.x == 0 && rank == 0) {
            GridState* gs = a.gs + b;
            gs->active = 0;
            gs->kstar = kstar;
            gs->k0_stop = kstar;
            gs->replay = 0;
            gs->src = 0;
            gs->final_buf = 0;
            gs->converged = dec == 1 ? 1 : 0;
            gs->e_stop = estar;
        }
        // ---- next grid: in turn when every grid takes the same sweeps, else
        // whichever is left (rank 0 asks, the group follows)
        sync_grid();
        if (a.groups >= a.B) break;
        if (threadIdx.x == 0) {
            uint4* nb = &a.box->next[group][seq & 1u];
            if (sh.limit == 1) {  // a wait gave up: the others need not wait for this CTA
                sh.grid = a.B;
                if (!a.fixed && rank == 0 && n > 1) st_box(nb, (uint32_t)a.B, 0u, seq);
            } else if (a.fixed) {
                sh.grid = b + a.groups;
            } else if (rank == 0) {
                sh.grid = a.groups + (int)atomicAdd(&a.box->queue, 1u);
                if (n > 1) st_box(nb, (uint32_t)sh.grid, 0u, seq);
            } else {
                uint4 v;
                int left = sh.limit;
                do {
                    v = ld_box(nb);
                } while (v.y != seq && --left > 0);
                if (v.y != seq) {
                    give_up(a, sh.limit);
                    v.x = (uint32_t)a.B;
                }
                sh.grid = (int)v.x;
            }
        }
        sync_grid();
        b = sh.grid;
    }
    if (threadIdx.x == 0) sh.end = w.t;
}

// An instance: its function, dynamic shared memory and strip height.
struct ResKernel {
    const void* fn;
    int smem;
    int rows;  // of one CTA
};

template <int C, int R, int WX, bool WIDE = false>
ResKernel res_kernel()
{
    using L = ResLayout<C, R, WX>;
    return {(const void*)sweep_resident_kernel<C, R, WX, WIDE>, L::kBytes, L::WY * R};
}

// by width of the grid, with `rows` rows per thread (4, 8 or 16)
ResKernel res_kernel_128(int rows);
ResKernel res_kernel_256(int rows);
ResKernel res_kernel_512(int rows);
ResKernel res_kernel_wide(int rows);  // 8 or 16 rows; columns of 240 cells

}  // namespace hp
