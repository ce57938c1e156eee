// Host side of the grid-resident sweeps (resident_kernel.cuh): the split of a
// grid into strips, the launch, and the query of how many grids fit.
#include "resident_kernel.cuh"

namespace hp {

namespace {

ResKernel res_kernel(int width, int R)
{
    return width == 128   ? res_kernel_128(R)
           : width == 256 ? res_kernel_256(R)
           : width == 512 ? res_kernel_512(R)
                          : res_kernel_wide(R);
}

// How a grid is split: columns of warps, rows per thread, CTAs per grid and
// grids at once.
struct ResPlan {
    int width, R, n, ntx, groups;
};

int width_class(int width) { return width == 128 ? 0 : width == 256 ? 1 : width == 512 ? 2 : 3; }

// CTAs of a cooperative launch that fit on the device: one per SM (every
// instance needs most of an SM's registers)
int res_ctas(const hp_ctx* ctx)
{
    const int ctas = ctx->num_sms < kResMaxCtas ? ctx->num_sms : kResMaxCtas;
    return ctx->res_sms > 0 && ctx->res_sms < ctas ? ctx->res_sms : ctas;
}

// Whether this device runs an instance as it is meant to: its register split
// assumes the registers of the launch, and a CTA has to fit on an SM.  Looked
// up once per context; the blocked kernel serves what does not run here.
bool res_usable(hp_ctx* ctx, int width, int R)
{
    int8_t& known = ctx->res_known[width_class(width)][R / 8];
    if (known == 0) {
        const ResKernel k = res_kernel(width, R);
        cudaFuncAttributes fa;
        int fit = 0;
        cudaError_t e =
            cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, k.smem);
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k.fn);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, k.fn, kResThreads, k.smem);
        if (e != cudaSuccess) cudaGetLastError();
        known = e == cudaSuccess && fa.numRegs == kResRegs && fit >= 1 ? 1 : -1;
    }
    return known > 0;
}

// The split with the least time: waves of groups x time per sweep of a strip,
// measured with all SMs at work and obstacles in every grid (38, 152 and 152
// grids of 128^2; 19, 38 and 64 of 256^2; 16 of 512^2; 4 of 1024^2 and one of
// 2048^2).  More rows per thread make a longer sweep with less of it lost to
// the exchange, fewer rows spread a grid over more SMs: 16 x 512^2 takes 5.3,
// 3.7 and 4.9 us per sweep with 4, 8 and 16 rows (four, two waves and one), one
// 512^2 grid 1.43, 2.0 and 3.4 us.  64 x 256^2 in one wave of 16 rows took 4.5
// us a sweep and all grids as long as the slowest; in two of 8 rows 3.6 us.
bool res_plan(hp_ctx* ctx, hp_shape s, ResPlan* best)
{
    // wider than 512 cells: columns of 240, eight copied on each side
    const int width = s.nx <= 128 ? 128 : s.nx <= 256 ? 256 : s.nx <= 512 ? 512 : 1024;
    const int own = 256 - 2 * kResGhost;
    const int ntx = width == 1024 ? (s.nx + own - 1) / own : 1;
    // us per sweep of a strip with E, R = 4, 8, 16
    static const double us[4][3] = {
        {0.72, 1.03, 1.8}, {1.14, 1.95, 4.5}, {1.35, 1.87, 4.9}, {0.0, 1.95, 3.75}};
    const int ctas = res_ctas(ctx);
    double least = 0.0;
    bool found = false;
    for (int R : {4, 8, 16}) {
        if ((R == 4 && width == 1024) || !res_usable(ctx, width, R)) continue;
        const int rows = res_kernel(width, R).rows, n = (s.ny + rows - 1) / rows * ntx;
        if (n > ctas) continue;
        const int groups = ctas / n < s.batch ? ctas / n : s.batch;
        const int waves = (s.batch + groups - 1) / groups;
        const double t = waves * us[width_class(width)][R / 8];
        if (!found || t < least) {
            least = t;
            *best = {width, R, n, ntx, groups};
            found = true;
        }
    }
    return found;
}

// Per-grid state, the exchange area of `ctas` CTAs in groups (n > 1), and, for
// a fixed number of sweeps, which grids hold values so large that a sum of
// residuals could overflow: those stop at the first non-finite E.
__global__ void resident_prep_kernel(GridState* gs, ResBox* box, ResColumns* cols, int32_t* err,
                                     int B, int ctas, int n,
                                     const float* __restrict__ div,
                                     const float* __restrict__ phi0, size_t cells, uint32_t epoch,
                                     int scan)
{
    const size_t id = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t step = (size_t)gridDim.x * blockDim.x;
    if (id == 0) {
        box->queue = 0u;
        err[1] = 0;
    }
    for (size_t b = id; b < (size_t)B; b += step) gs[b].active = 1;
    if (n > 1) {
        const uint4 z = make_uint4(0, 0, 0, 0);
        uint4* row = &box->row[0][0][0][0];
        for (size_t i = id; i < (size_t)ctas * 2 * 2 * 256; i += step) row[i] = z;
        uint4* part = &box->part[0][0][0];
        for (size_t i = id; i < (size_t)ctas * kResRing * 4; i += step) part[i] = z;
        uint4* dec = &box->dec[0][0];
        for (size_t i = id; i < (size_t)ctas * kResRing; i += step) dec[i] = z;
        uint4* next = &box->next[0][0];
        for (size_t i = id; i < (size_t)ctas * 2; i += step) next[i] = z;
        uint4* col = cols ? &cols->w[0][0][0][0][0][0] : nullptr;
        if (col)
            for (size_t i = id; i < (size_t)ctas * 2 * 2 * kResWarps * 2 * 32; i += step) col[i] = z;
    }
    if (scan) {
        constexpr float kTame = 1e20f;  // |phi| grows by max |div| per sweep at most
        for (size_t i = id; i < cells * B; i += step) {
            const bool ok = fabsf(div[i]) < kTame && (!phi0 || fabsf(phi0[i]) < kTame);
            if (!ok) gs[i / cells].wild = epoch;
        }
    }
}

}  // namespace

size_t resident_box_bytes() { return sizeof(ResBox); }
size_t resident_columns_bytes() { return sizeof(ResColumns); }

// Grids of shape s held on chip at once by a launch; 0 when none is made.
int resident_capacity(hp_ctx* ctx, hp_shape s)
{
    ResPlan p;
    return res_plan(ctx, s, &p) ? res_ctas(ctx) / p.n : 0;
}

hp_status launch_resident(hp_ctx* ctx, hp_shape s, double threshold, int cap, bool fixed,
                          const float* phi0, double* e_hist, int hist_len, cudaStream_t st,
                          bool* launched)
{
    *launched = false;
    ResPlan p;
    if (!res_plan(ctx, s, &p)) return HP_OK;
    if (phi0 == ctx->phi[0]) return HP_ERR_INVALID_ARG;  // see ResArgs::phi
    const ResKernel k = res_kernel(p.width, p.R);
    ResArgs a = {};
    a.phi0 = phi0;
    a.phi0_vec = phi0 && ((uintptr_t)phi0 & 15) == 0;
    a.phi = ctx->phi[0];
    a.ck[0] = ctx->ckpt;
    a.ck[1] = ctx->phi[1];
    a.div = ctx->div;
    a.mask = ctx->mask;
    a.gs = ctx->gs;
    a.box = (ResBox*)ctx->box;
    a.cols = p.ntx > 1 ? (ResColumns*)ctx->cols : nullptr;
    a.ntx = p.ntx;
    a.err = ctx->wait_err;
    a.polls = ctx->wait_limit ? ctx->wait_limit : kResPolls;
    a.looks = ctx->wait_limit ? ctx->wait_limit : kResLooks;
    a.e_hist = e_hist;
    a.hist_len = hist_len;
    a.B = s.batch;
    a.ny = s.ny;
    a.nx = s.nx;
    a.n = p.n;
    a.groups = p.groups;
    a.cap = cap;
    a.fixed = fixed && !e_hist;
    a.epoch = ++ctx->epoch;
    a.threshold = threshold;
    a.sum_near = (float)(threshold * (double)s.ny * s.nx * kSumScale) * (1.0f + 1e-6f);
    const size_t cells = (size_t)s.ny * s.nx;
    const int ctas = p.n * p.groups;
    const size_t work = a.fixed ? cells * s.batch / 8 : p.n > 1 ? (size_t)ctas * 1024 : s.batch;
    const size_t want = work / 256 + 1, most = 8 * (size_t)ctx->num_sms;
    resident_prep_kernel<<<(unsigned)(want < most ? want : most), 256, 0, st>>>(
        ctx->gs, a.box, a.cols, a.err, s.batch, ctas, p.n, ctx->div, phi0, cells, a.epoch, a.fixed);
    hp_status rc = check_launch();
    if (rc != HP_OK) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kResThreads);
    cfg.dynamicSmemBytes = k.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = p.n > 1 ? 1 : 0;  // single CTAs wait for nobody
    void* args[] = {&a};
    cudaError_t e = cudaLaunchKernelExC(&cfg, k.fn, args);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        // fewer SMs for this stream than the device has: the blocked kernel
        cudaGetLastError();
        return HP_OK;
    }
    if (e != cudaSuccess) { set_cuda_error(e); return HP_ERR_CUDA; }
    *launched = true;
    return check_launch();
}

}  // namespace hp

extern "C" {

int32_t hp_resident_grids(hp_ctx* ctx, hp_shape s)
{
    return ctx && hp::shape_ok(s) ? hp::resident_capacity(ctx, s) : 0;
}

int32_t hp_resident_clusters(hp_ctx* ctx, hp_shape s)
{
    if (!ctx || !hp::shape_ok(s)) return 0;
    const int tiles = ((s.nx + 127) / 128) * ((s.ny + 127) / 128);
    return tiles > 16 ? 0 : hp::resident_capacity(ctx, s);
}

hp_status hp_ctx_set_resident_sms(hp_ctx* ctx, int32_t sms)
{
    if (!ctx || sms < 0) return HP_ERR_INVALID_ARG;
    ctx->res_sms = sms;
    return HP_OK;
}

}  // extern "C"
