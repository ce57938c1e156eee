// Adjoint of the fixed-count projection (Sec. 3.2: the gradient of the
// correction of Eq. 2 is known, so the network can be trained through the
// solver).  Forward: div = D(Z u*), phi_k = k masked Jacobi sweeps from
// phi_0, u = Z u* - G phi_k, p = phi_k rho0 / dt.  With W the open-face
// adjacency and n the open-face count, one sweep is phi' = n^-1 (W phi - div);
// its transpose needs no stored iterate (the map is affine):
//   lam_k = D(g_u) + (rho0/dt) g_p            (G^T = -D on open faces)
//   mu_t  = n^-1 lam_t,  lam_{t-1} = W mu_t    for t = k .. 1
//   dL/dphi_0 = lam_0,  dL/ddiv = -sum_{t=1..k} mu_t
//   dL/du* = Z g_u - G dL/ddiv
// and mu_{t-1} = n^-1 W mu_t is the forward sweep with a zero right-hand side.
#include <cuda_runtime.h>

#include "hproj_internal.cuh"

namespace hp {

namespace {

__device__ __forceinline__ float inv_open(uint32_t m)
{
    const int n = __popc(m & 15u);
    return n == 4 ? 0.25f : n == 3 ? (1.0f / 3.0f) : n == 2 ? 0.5f : n == 1 ? 1.0f : 0.0f;
}

// lam_k = D(g) + scale * g_p; mu_k = lam_k / n (k > 0) or g_phi0 = lam_k (k = 0)
__global__ void adj_init_kernel(const float* __restrict__ gu, const float* __restrict__ gv,
                                const float* __restrict__ gp, const uint8_t* __restrict__ mask,
                                float scale, float* __restrict__ mu, float* __restrict__ acc,
                                int k, int ny, int nx)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    const int b = blockIdx.z;
    if (i >= nx) return;
    const size_t q = (size_t)b * ny * nx + (size_t)j * nx + i;
    const uint32_t m = mask[q];
    const float* ub = gu + (size_t)b * ny * (nx + 1) + (size_t)j * (nx + 1);
    const float* vb = gv + (size_t)b * (ny + 1) * nx;
    const float ue = (m & 2u) ? ub[i + 1] : 0.0f;
    const float uw = (m & 1u) ? ub[i] : 0.0f;
    const float vs = (m & 8u) ? vb[(size_t)(j + 1) * nx + i] : 0.0f;
    const float vn = (m & 4u) ? vb[(size_t)j * nx + i] : 0.0f;
    float lam = (ue - uw) + (vs - vn);
    if (gp) lam += scale * gp[q];
    if (!(m & 15u)) lam = 0.0f;
    mu[q] = k > 0 ? lam * inv_open(m) : lam;
    if (k == 0) acc[q] = 0.0f;  // else written by the first block of sweeps
}

// The only sweep of k = 1: acc = mu_1, g_phi0 = W mu_1, a thread per cell.  A
// block of one sweep reads and writes copies besides and runs on fewer CTAs:
// 4096 x 16^2 186 us with its neighbours, 160 us with this one; 2048^2 76 and 71.
// From two sweeps on the blocks are as fast or faster (193 and 197 us, 80 and 89).
__global__ void adj_single_kernel(const float* __restrict__ mu, float* __restrict__ out,
                                  float* __restrict__ acc, const uint8_t* __restrict__ mask, int ny,
                                  int nx)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nx) return;
    const size_t c = ((size_t)blockIdx.z * ny + blockIdx.y) * nx + i;
    const uint32_t m = mask[c];
    acc[c] = 0.0f + mu[c];
    float s = 0.0f;
    if (m & 1u) s += mu[c - 1];
    if (m & 2u) s += mu[c + 1];
    if (m & 4u) s += mu[c - nx];
    if (m & 8u) s += mu[c + nx];
    out[c] = s;
}

// A block of sweeps: acc += mu_t; mu_{t-1} = n^-1 W mu_t, and on the very last
// sweep g_phi0 = W mu_1.
//
// One launch per sweep was bound by the launches; a block of 7 sweeps of
// 8 x 256^2 takes 12.7 us (forward and backward of 20 sweeps, with what the
// host takes for the call: 402 -> 377 us).
// A CTA holds a region of kAdjN x kAdjN cells, each thread 8 rows of a column
// in registers (mu, acc, 1/n, the face bits), so a sweep costs one shared store
// and two shared loads per cell (west and east; north and south are the
// thread's own) and one barrier.  A sweep makes one more ring of the region's
// edge stale: with `sweeps` of them the outer hx columns and hy rows per side
// (= sweeps, or 0 where the region holds the whole side of the grid) are
// copies that other CTAs own.  kAdjSweeps = 8 keeps 48 x 48 of 64 x 64.
constexpr int kAdjN = 64, kAdjRows = 8, kAdjThreads = kAdjN * (kAdjN / kAdjRows);
constexpr int kAdjSweeps = 8;

__global__ void __launch_bounds__(kAdjThreads, 2)
    adj_block_kernel(const float* __restrict__ mu_in, float* __restrict__ out,
                     float* __restrict__ acc, const uint8_t* __restrict__ mask, int sweeps, int hx,
                     int hy, int first, int last, int ny, int nx)
{
    __shared__ float s_mu[2][kAdjN + 2][kAdjN + 2];
    const int lx = threadIdx.x % kAdjN, ly = threadIdx.x / kAdjN * kAdjRows;
    const int x = blockIdx.x * (kAdjN - 2 * hx) - hx + lx;
    const int y = blockIdx.y * (kAdjN - 2 * hy) - hy + ly;
    const size_t base = (size_t)blockIdx.z * ny * nx;
    // the ring around the region is read by its (stale) edge cells only
    for (int i = threadIdx.x; i < 2 * (kAdjN + 2); i += kAdjThreads) {
        const int h = i / (kAdjN + 2), c = i % (kAdjN + 2);
        s_mu[h][0][c] = s_mu[h][kAdjN + 1][c] = s_mu[h][c][0] = s_mu[h][c][kAdjN + 1] = 0.0f;
    }
    const bool xin = x >= 0 && x < nx;
    const bool xown = xin && lx >= hx && lx < kAdjN - hx;
    float mu[kAdjRows], sum[kAdjRows], inv[kAdjRows];
    uint32_t faces = 0u;  // four bits per row
#pragma unroll
    for (int k = 0; k < kAdjRows; ++k) {
        const int j = y + k;
        const bool in = xin && j >= 0 && j < ny;
        const size_t q = base + (size_t)j * nx + x;
        const uint32_t m = in ? mask[q] & 15u : 0u;
        mu[k] = in ? mu_in[q] : 0.0f;
        const bool own = xown && in && ly + k >= hy && ly + k < kAdjN - hy;
        sum[k] = own && !first ? acc[q] : 0.0f;
        inv[k] = inv_open(m);
        faces |= m << (4 * k);
    }
    for (int t = 0; t < sweeps; ++t) {
        // (unpacked in every sweep: hoisted, the face tests spill)
        asm volatile("" : "+r"(faces));
        float(*s)[kAdjN + 2] = s_mu[t & 1];
#pragma unroll
        for (int k = 0; k < kAdjRows; ++k) s[ly + k + 1][lx + 1] = mu[k];
        __syncthreads();
        const bool scaled = !(last && t == sweeps - 1);
        float north = s[ly][lx + 1];
        const float below = s[ly + kAdjRows + 1][lx + 1];
#pragma unroll
        for (int k = 0; k < kAdjRows; ++k) {
            const uint32_t m = faces >> (4 * k);
            const float west = s[ly + k + 1][lx], east = s[ly + k + 1][lx + 2];
            const float south = k + 1 < kAdjRows ? mu[k + 1 < kAdjRows ? k + 1 : k] : below;
            sum[k] += mu[k];
            float w = 0.0f;
            if (m & 1u) w += west;
            if (m & 2u) w += east;
            if (m & 4u) w += north;
            if (m & 8u) w += south;
            north = mu[k];
            mu[k] = scaled ? w * inv[k] : w;
        }
    }
#pragma unroll
    for (int k = 0; k < kAdjRows; ++k) {
        const int j = y + k;
        if (xown && j >= 0 && j < ny && ly + k >= hy && ly + k < kAdjN - hy) {
            const size_t q = base + (size_t)j * nx + x;
            out[q] = mu[k];
            acc[q] = sum[k];
        }
    }
}

// g_u* = g_u + (acc_c - acc_nb) on open faces, 0 on closed faces
__global__ void adj_correct_kernel(const float* __restrict__ gu, const float* __restrict__ gv,
                                   const float* __restrict__ acc, const uint8_t* __restrict__ mask,
                                   float* __restrict__ gus, float* __restrict__ gvs, int ny, int nx)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    const int b = blockIdx.z;
    if (i >= nx) return;
    const size_t base = (size_t)b * ny * nx;
    const size_t c = (size_t)j * nx + i;
    const uint32_t m = mask[base + c];
    const size_t uo = (size_t)b * ny * (nx + 1) + (size_t)j * (nx + 1);
    const size_t vo = (size_t)b * (ny + 1) * nx;
    float uw = 0.0f, vn = 0.0f;
    if (m & 1u) uw = gu[uo + i] + (acc[base + c] - acc[base + c - 1]);
    if (m & 4u) vn = gv[vo + (size_t)j * nx + i] + (acc[base + c] - acc[base + c - nx]);
    gus[uo + i] = uw;
    gvs[vo + (size_t)j * nx + i] = vn;
    if (i == nx - 1) gus[uo + nx] = 0.0f;
    if (j == ny - 1) gvs[vo + (size_t)ny * nx + i] = 0.0f;
}

}  // namespace

}  // namespace hp

using namespace hp;

extern "C" hp_status hp_project_adjoint(hp_ctx* ctx, const float* gu, const float* gv,
                                        const float* gp, const uint8_t* flags, hp_shape s,
                                        int32_t k, float dt, float rho0, float* gu_star,
                                        float* gv_star, float* g_phi0, void* stream)
{
    if (!ctx || !gu || !gv || !flags || !gu_star || !gv_star || !g_phi0 || k < 0 ||
        !shape_ok(s) || s.batch > ctx->max_shape.batch || s.ny > ctx->max_shape.ny ||
        s.nx > ctx->max_shape.nx || !(dt > 0.0f))
        return HP_ERR_INVALID_ARG;
    if (gu_star == gu || gv_star == gv) return HP_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    hp_status rc = launch_mask(flags, ctx->mask, s, st);
    if (rc != HP_OK) return rc;
    dim3 blk(256), grd((s.nx + 255) / 256, s.ny, s.batch);
    float* acc = ctx->div;
    float* bufs[2] = {ctx->phi[0], ctx->phi[1]};
    adj_init_kernel<<<grd, blk, 0, st>>>(gu, gv, gp, ctx->mask, rho0 / dt, k > 0 ? bufs[0] : g_phi0,
                                         acc, k, s.ny, s.nx);
    if ((rc = check_launch()) != HP_OK) return rc;
    // blocks of nearly equal length; a grid that one region holds takes one
    const bool whole = s.nx <= kAdjN && s.ny <= kAdjN;
    int left = k, cur = 0;
    if (k == 1) {
        adj_single_kernel<<<grd, blk, 0, st>>>(bufs[0], g_phi0, acc, ctx->mask, s.ny, s.nx);
        if ((rc = check_launch()) != HP_OK) return rc;
    }
    for (int n = k < 2 ? 0 : whole ? 1 : (k - 1) / kAdjSweeps + 1; n > 0; --n) {
        const int sweeps = (left - 1) / n + 1;
        const int hx = s.nx <= kAdjN ? 0 : sweeps, hy = s.ny <= kAdjN ? 0 : sweeps;
        const int ox = kAdjN - 2 * hx, oy = kAdjN - 2 * hy;
        const dim3 tiles((s.nx + ox - 1) / ox, (s.ny + oy - 1) / oy, s.batch);
        adj_block_kernel<<<tiles, kAdjThreads, 0, st>>>(bufs[cur], n == 1 ? g_phi0 : bufs[cur ^ 1],
                                                        acc, ctx->mask, sweeps, hx, hy, left == k,
                                                        n == 1, s.ny, s.nx);
        if ((rc = check_launch()) != HP_OK) return rc;
        left -= sweeps;
        cur ^= 1;
    }
    adj_correct_kernel<<<grd, blk, 0, st>>>(gu, gv, acc, ctx->mask, gu_star, gv_star, s.ny, s.nx);
    return check_launch();
}
