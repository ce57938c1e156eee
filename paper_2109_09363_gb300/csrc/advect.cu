// Plume driver step for sm_103a: inlet source, semi-Lagrangian advection of
// rho (cell centres) and u, v (faces) with the start-of-step velocity,
// first order or MacCormack, Boussinesq buoyancy on the v faces (forward
// Euler), closed faces zeroed.  This produces u* for the projection
// (Sec. 2.2: advection, then external forces, then the pressure projection).
//
// MacCormack (the scheme Sec. 2.2 names, after Selle et al. 2008): q_f, the
// forward semi-Lagrangian value, q_b, the forward field sampled backwards at
// x + dt vel(x), and q_f + (q - q_b) / 2 clamped to the range of the four
// samples the forward step interpolated.  The forward field is not stored
// in global memory: each CTA evaluates it on a window around its tile in
// shared memory (and evaluates a corner outside the window where it needs
// it), so the step needs no workspace.
//
// Positions: cell (i, j) centred at (i + 1/2, j + 1/2); u face (j, i) at
// (i, j + 1/2); v face (j, i) at (i + 1/2, j); row 0 is the top of the image.
#include <cuda_runtime.h>
#include <math.h>

#include "hproj_internal.cuh"

namespace hp {

namespace {

// The four samples around a position.
struct Corners {
    float q00, q01, q10, q11;
};

// Mx x My samples, sample (0, 0) at (ox, oy).
struct Field {
    const float* q;
    int Mx, My;
    float ox, oy;
    __device__ float at(int i, int j) const { return __ldg(q + (size_t)j * Mx + i); }
    // samples (i, j) and its right and lower neighbours (itself where the
    // field has one column or row)
    __device__ Corners corners(int i, int j) const
    {
        const float* p = q + ((size_t)j * Mx + i);
        const int di = Mx > 1 ? 1 : 0;
        const float* r = p + (My > 1 ? Mx : 0);
        return {__ldg(p), __ldg(p + di), __ldg(r), __ldg(r + di)};
    }
};

// Density with the inlet applied: rho_in on the inlet cells.
struct Rho {
    const float* q;
    int Mx, My;
    float ox, oy;
    int x0, x1;
    float rho_in;
    __device__ bool inlet(int i, int j) const { return j == My - 1 && i >= x0 && i < x1; }
    __device__ float at(int i, int j) const
    {
        return inlet(i, j) ? rho_in : __ldg(q + (size_t)j * Mx + i);
    }
    __device__ Corners corners(int i, int j) const
    {
        Corners c = Field{q, Mx, My, ox, oy}.corners(i, j);
        if (j + 2 >= My) {  // the lower row is the last one
            const int i1 = min(i + 1, Mx - 1), j1 = min(j + 1, My - 1);
            if (inlet(i, j)) c.q00 = rho_in;
            if (inlet(i1, j)) c.q01 = rho_in;
            if (inlet(i, j1)) c.q10 = rho_in;
            if (inlet(i1, j1)) c.q11 = rho_in;
        }
        return c;
    }
};

// Position along one axis: the sample at or below it and the distance to it.
//
// WIDE: fields of 2^22 samples and more along a row.  Else every coordinate
// t and index lies in [0, 2^23), where FP32 addition of 2^23 leaves the whole
// part in the low mantissa bits (rounded down), so that floor and both
// conversions are plain additions.  The conversion instructions issue at an
// eighth of their rate and six per sample held the step back.
constexpr float kTwo23 = 8388608.0f;

template <bool WIDE>
__device__ __forceinline__ float to_float(int i)  // i >= 0
{
    if constexpr (WIDE) return (float)i;
    else return __int_as_float(__float_as_int(kTwo23) + i) - kTwo23;
}

// t in [0, n - 1]; the last sample counts as distance 1 from the one before
template <bool WIDE>
__device__ __forceinline__ int split(float t, int n, float& frac)
{
    const int last = max(n - 2, 0);
    if constexpr (WIDE) {
        const int i = min((int)floorf(t), last);
        frac = t - (float)i;
        return i;
    } else {
        const float r = fminf(__fadd_rd(t, kTwo23), kTwo23 + (float)last);
        frac = t - (r - kTwo23);
        return __float_as_int(r) - __float_as_int(kTwo23);
    }
}

struct Pos {
    int i, j;
    float fx, fy;
};

// (x, y) clamped to the sample span of f
template <bool WIDE, class Q>
__device__ __forceinline__ Pos locate(const Q& f, float x, float y)
{
    const float tx = fminf(fmaxf(x - f.ox, 0.0f), (float)(f.Mx - 1));
    const float ty = fminf(fmaxf(y - f.oy, 0.0f), (float)(f.My - 1));
    Pos p;
    p.i = split<WIDE>(tx, f.Mx, p.fx);
    p.j = split<WIDE>(ty, f.My, p.fy);
    return p;
}

// Which product of a weighted sum goes unrounded into the fused addition, for
// the top, the bottom and the vertical interpolation: written out, so that the
// roundings do not depend on what a compiler makes of the code around them (a
// projection's convergence amplifies the last bit of u* to 5e-6 in E_1).
enum Fuse : bool { kFirst = true, kSecond = false };

template <Fuse F>
__device__ __forceinline__ float mix(float a, float wa, float b, float wb)
{
    return F == kFirst ? __fmaf_rn(a, wa, __fmul_rn(b, wb)) : __fmaf_rn(b, wb, __fmul_rn(a, wa));
}

template <Fuse TOP, Fuse BOT, Fuse VERT>
__device__ __forceinline__ float blend(const Corners& c, const Pos& p)
{
    const float top = mix<TOP>(c.q00, 1.0f - p.fx, c.q01, p.fx);
    const float bot = mix<BOT>(c.q10, 1.0f - p.fx, c.q11, p.fx);
    return mix<VERT>(top, 1.0f - p.fy, bot, p.fy);
}

// The forward value of a quantity: density (kind 0), u (1) or v (2); OWN: as
// a sample's own new value, else as MacCormack's forward field.
template <bool MC, int KIND, bool OWN>
__device__ __forceinline__ float blend_forward(const Corners& c, const Pos& p)
{
    if constexpr (KIND == 0) {
        return MC ? blend<kFirst, kFirst, kFirst>(c, p) : blend<kFirst, kSecond, kFirst>(c, p);
    } else if constexpr (KIND == 1) {
        return MC && OWN ? blend<kSecond, kSecond, kFirst>(c, p)
                         : blend<kSecond, kSecond, kSecond>(c, p);
    } else {
        return blend<kSecond, kSecond, kFirst>(c, p);
    }
}

// Velocity at sample (i, j) of a quantity whose samples sit at (i + ox,
// j + oy): cell centres (1/2, 1/2), u faces (0, 1/2) or v faces (1/2, 0).
// There the bilinear sample of each component has weights 0, 1 or 1/2 on a
// row or column pair (pairs clamped to the field at its borders), so it is a
// copy or the mean of two or four values; for finite inputs the result is
// the same FP32 value as the general bilinear sample of sample_range()
// (products by 1/2 are exact, and the one rounding of each weighted sum is
// the rounding of the plain sum, halved).
__device__ __forceinline__ void vel_at_sample(const Field& fu, const Field& fv, float ox,
                                              float oy, int i, int j, float& vx, float& vy)
{
    const int su = fu.Mx, nx = fv.Mx, ny = fu.My;  // u rows hold nx + 1 faces
    const float* u = fu.q;
    const float* v = fv.q;
    if (ox != 0.0f && oy != 0.0f) {  // cell (i, j)
        const float* ur = u + (size_t)j * su;
        vx = 0.5f * (__ldg(ur + i) + __ldg(ur + i + 1));
        vy = 0.5f * (__ldg(v + (size_t)j * nx + i) + __ldg(v + (size_t)(j + 1) * nx + i));
    } else if (ox == 0.0f) {  // u face (j, i), i in [0, nx]
        vx = __ldg(u + (size_t)j * su + i);
        const int c0 = max(i - 1, 0), c1 = min(i, nx - 1);
        const float* v0 = v + (size_t)j * nx;
        const float* v1 = v0 + nx;
        vy = 0.5f * (0.5f * (__ldg(v0 + c0) + __ldg(v0 + c1)) +
                     0.5f * (__ldg(v1 + c0) + __ldg(v1 + c1)));
    } else {  // v face (j, i), j in [0, ny]
        vy = __ldg(v + (size_t)j * nx + i);
        const int r0 = max(j - 1, 0), r1 = min(j, ny - 1);
        const float* u0 = u + (size_t)r0 * su;
        const float* u1 = u + (size_t)r1 * su;
        vx = 0.5f * (0.5f * (__ldg(u0 + i) + __ldg(u0 + i + 1)) +
                     0.5f * (__ldg(u1 + i) + __ldg(u1 + i + 1)));
    }
}

// Departure point of sample (i, j) of q and the samples around it, with the
// velocity at (i, j).
template <bool WIDE, class Q>
__device__ __forceinline__ Pos departure(const Q& q, const Field& fu, const Field& fv, float dt,
                                         int i, int j, float& vx, float& vy, Corners& c)
{
    const float x = to_float<WIDE>(i) + q.ox, y = to_float<WIDE>(j) + q.oy;
    vel_at_sample(fu, fv, q.ox, q.oy, i, j, vx, vy);
    const Pos p = locate<WIDE>(q, x - dt * vx, y - dt * vy);
    c = q.corners(p.i, p.j);
    return p;
}

__device__ __forceinline__ bool fluid(const uint8_t* fl, int nx, int i, int j)
{
    return fl[(size_t)j * nx + i] == 0;
}

// Tiles of the fused step: a CTA produces the outputs of kAdvTX x adv_ty(MC)
// indices (i, j) of [0, nx] x [0, ny] (cell (i, j) density, u face (j, i),
// v face (j, i)): 16 rows for MacCormack, whose windows (below) then cost
// 1.48 forward values per output, 32 for the first-order scheme, which has
// none.  MacCormack's backward sample reads the forward field at
// four corners within kAdvH samples of its own index whenever the
// displacement dt |vel| is below kAdvH cells; the CTA evaluates the forward
// field of each quantity once on its tile widened by kAdvH (and one row more
// above, for the density of the row above the tile that the buoyancy of the
// tile's top v faces reads) and keeps it in shared memory.  A corner outside
// that window (a faster flow) is evaluated where it is needed, with the same
// arithmetic, so the result does not depend on the window.
constexpr int kAdvTX = 32, kAdvH = 2, kAdvThreads = 256;
__host__ __device__ constexpr int adv_ty(bool mc) { return mc ? 16 : 32; }
constexpr int kFW = kAdvTX + 2 * kAdvH;          // columns of a forward-field window
constexpr int kFH = adv_ty(true) + 2 * kAdvH + 1;  // rows: tile rows - 1 - kAdvH .. + kAdvH

constexpr int kFS = kFH * kFW;
constexpr int kTS = (adv_ty(true) + 1) * kAdvTX;  // the tile and the row above it

// What MacCormack's second half needs of a quantity: the forward field and the
// velocity on the window (sample (ci, cj) at entry 0); on the tile, the value
// itself and the range of the samples that it interpolates.
struct Window {
    float fwd[kFS], vx[kFS], vy[kFS];
    float own[kTS], lo[kTS], hi[kTS];
};

// Samples of the field only: entries outside it are never read (every corner
// of a bilinear sample lies in the field, and so does every output sample).
template <int KIND, bool WIDE, class Q>
__device__ __forceinline__ void fill_entry(Window& w, const Q& q, const Field& fu, const Field& fv,
                                           float dt, int a, int b, int ci, int cj)
{
    const int i = ci + a, j = cj + b;
    if (i < 0 || i >= q.Mx || j < 0 || j >= q.My) return;
    const int t = b * kFW + a;
    float vx, vy;
    Corners c;
    const Pos p = departure<WIDE>(q, fu, fv, dt, i, j, vx, vy, c);
    w.fwd[t] = blend_forward<true, KIND, false>(c, p);
    w.vx[t] = vx;
    w.vy[t] = vy;
    const int ta = a - kAdvH, tb = b - kAdvH;
    if ((unsigned)ta < (unsigned)kAdvTX && (unsigned)tb <= (unsigned)adv_ty(true)) {
        const int tt = tb * kAdvTX + ta;
        w.own[tt] = blend_forward<true, KIND, true>(c, p);
        w.lo[tt] = fminf(fminf(c.q00, c.q01), fminf(c.q10, c.q11));
        w.hi[tt] = fmaxf(fmaxf(c.q00, c.q01), fmaxf(c.q10, c.q11));
    }
}

// New value of sample (i, j) of quantity q, in the first-order scheme the
// forward value; in MacCormack's the backward sample reads the forward field
// in the window, or evaluates the corners there that the window does not hold.
template <bool MC, int KIND, bool WIDE, class Q>
__device__ __forceinline__ float advected(const Window* w, const Q& q, const Field& fu,
                                          const Field& fv, float dt, int ci, int cj, int i, int j)
{
    float vx, vy;
    Corners c;
    if constexpr (!MC) {
        const Pos p = departure<WIDE>(q, fu, fv, dt, i, j, vx, vy, c);
        return blend_forward<false, KIND, true>(c, p);
    } else {
        const int t = (j - cj) * kFW + (i - ci);
        const int tt = (j - cj - kAdvH) * kAdvTX + (i - ci - kAdvH);
        const float x = to_float<WIDE>(i) + q.ox, y = to_float<WIDE>(j) + q.oy;
        const Pos p = locate<WIDE>(q, x + dt * w->vx[t], y + dt * w->vy[t]);
        const int di = q.Mx > 1 ? 1 : 0, dj = q.My > 1 ? 1 : 0;
        const int a = p.i - ci, b = p.j - cj;
        if ((unsigned)a < (unsigned)(kFW - 1) && (unsigned)b < (unsigned)(kFH - 1)) {
            const float* f = w->fwd + b * kFW + a;
            c = {f[0], f[di], f[dj * kFW], f[dj * kFW + di]};
        } else {
#pragma unroll 1
            for (int k = 0; k < 4; ++k) {
                const int ka = a + (k & 1) * di, kb = b + (k >> 1) * dj;
                float val;
                if ((unsigned)ka < (unsigned)kFW && (unsigned)kb < (unsigned)kFH) {
                    val = w->fwd[kb * kFW + ka];
                } else {
                    Corners far;
                    const Pos pf = departure<WIDE>(q, fu, fv, dt, ci + ka, cj + kb, vx, vy, far);
                    val = blend_forward<true, KIND, false>(far, pf);
                }
                if (k == 0) c.q00 = val;
                else if (k == 1) c.q01 = val;
                else if (k == 2) c.q10 = val;
                else c.q11 = val;
            }
        }
        const float qb = blend<kFirst, kFirst, kFirst>(c, p);
        return fminf(fmaxf(w->own[tt] + 0.5f * (q.at(i, j) - qb), w->lo[tt]), w->hi[tt]);
    }
}

// One CTA per tile: (MacCormack) the three windows; the new density of the
// tile's rows and the row above, kept in shared memory for the buoyancy; then
// the u and v faces.
//
// What bounds it: instruction issue.  MacCormack at 16 x 512^2 takes 158 us
// (16 us of memory traffic); 187 us with the corners of every sample addressed
// and clamped one by one, conversion instructions for the whole parts, and the
// tile's own forward values and ranges interpolated a second time.
template <bool MC, bool WIDE>
__global__ void __launch_bounds__(kAdvThreads) advect_kernel(
    const float* __restrict__ u, const float* __restrict__ v, const float* __restrict__ rho,
    const uint8_t* __restrict__ flags, float* __restrict__ u_out, float* __restrict__ v_out,
    float* __restrict__ rho_out, int ny, int nx, hp_plume_params p)
{
    constexpr int kAdvTY = adv_ty(MC);
    __shared__ float s_rho[(kAdvTY + 1) * kAdvTX];  // new rho, rows j0 - 1 ..
    const int i0 = blockIdx.x * kAdvTX, j0 = blockIdx.y * kAdvTY, b = blockIdx.z;
    const size_t cells = (size_t)ny * nx;
    const Field fu = {u + (size_t)b * ny * (nx + 1), nx + 1, ny, 0.0f, 0.5f};
    const Field fv = {v + (size_t)b * (ny + 1) * nx, nx, ny + 1, 0.5f, 0.0f};
    const Rho r = {rho + b * cells, nx, ny, 0.5f, 0.5f, p.inlet_x0, p.inlet_x1, p.rho_in};
    const uint8_t* fl = flags + b * cells;
    const float dt = p.dt;
    const int ci = i0 - kAdvH, cj = j0 - 1 - kAdvH;  // sample at entry 0 of a window
    const Window* win[3] = {nullptr, nullptr, nullptr};

    if constexpr (MC) {
        __shared__ Window s_win[3];  // rho, u, v
        for (int t = threadIdx.x; t < kFS; t += kAdvThreads) {
            const int wb = t / kFW, wa = t - wb * kFW;
            fill_entry<0, WIDE>(s_win[0], r, fu, fv, dt, wa, wb, ci, cj);
            fill_entry<1, WIDE>(s_win[1], fu, fu, fv, dt, wa, wb, ci, cj);
            fill_entry<2, WIDE>(s_win[2], fv, fu, fv, dt, wa, wb, ci, cj);
        }
        for (int k = 0; k < 3; ++k) win[k] = &s_win[k];
        __syncthreads();
    }

    for (int t = threadIdx.x; t < (kAdvTY + 1) * kAdvTX; t += kAdvThreads) {
        const int rr = t / kAdvTX, c = t - rr * kAdvTX;
        const int i = i0 + c, j = j0 - 1 + rr;
        if (i < nx && j >= 0 && j < ny) {
            const float val = advected<MC, 0, WIDE>(win[0], r, fu, fv, dt, ci, cj, i, j);
            s_rho[t] = val;
            if (rr > 0) rho_out[b * cells + (size_t)j * nx + i] = val;
        }
    }
    __syncthreads();

    for (int t = threadIdx.x; t < kAdvTY * kAdvTX; t += kAdvThreads) {
        const int rr = t / kAdvTX, c = t - rr * kAdvTX;
        const int i = i0 + c, j = j0 + rr;
        if (i > nx || j > ny) continue;
        if (j < ny) {
            const bool open = i > 0 && i < nx && fluid(fl, nx, i - 1, j) && fluid(fl, nx, i, j);
            float val = 0.0f;
            if (open) val = advected<MC, 1, WIDE>(win[1], fu, fu, fv, dt, ci, cj, i, j);
            u_out[(size_t)b * ny * (nx + 1) + (size_t)j * (nx + 1) + i] = val;
        }
        if (i < nx) {
            const bool interior = j > 0 && j < ny && fluid(fl, nx, i, j - 1) && fluid(fl, nx, i, j);
            // an open top keeps (advects) its faces; buoyancy acts on interior faces
            const bool top = j == 0 && p.open_top && fluid(fl, nx, i, 0);
            float val = 0.0f;
            if (interior || top) val = advected<MC, 2, WIDE>(win[2], fv, fu, fv, dt, ci, cj, i, j);
            if (interior) {
                // new density of cells (i, j - 1) and (i, j): rows rr and rr + 1
                const float rf = 0.5f * (s_rho[rr * kAdvTX + c] + s_rho[(rr + 1) * kAdvTX + c]);
                val += dt * p.gravity * (rf - p.rho_amb);
            }
            // injection through the inlet faces of the bottom boundary (upwards)
            if (j == ny && i >= p.inlet_x0 && i < p.inlet_x1 && fluid(fl, nx, i, ny - 1))
                val = -p.u_in;
            v_out[(size_t)b * (ny + 1) * nx + (size_t)j * nx + i] = val;
        }
    }
}

__global__ void plume_head_init_kernel(int32_t* __restrict__ out, int B, int ny, int nx)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    out[3 * b + 0] = ny;
    out[3 * b + 1] = nx;
    out[3 * b + 2] = -1;
}

// Smallest row, smallest and largest column of the cells whose density
// contrast reaches the threshold: CTA (slice, grid) reduces its slice of
// rows and merges with atomicMin / atomicMax (integers: order independent).
__global__ void __launch_bounds__(512) plume_head_kernel(const float* __restrict__ rho, int ny,
                                                         int nx, float rho_amb, float contrast,
                                                         int32_t* __restrict__ out)
{
    __shared__ int s_min_row[16], s_min_col[16], s_max_col[16];
    const int b = blockIdx.y;
    const int r0 = (int)((long)ny * blockIdx.x / gridDim.x);
    const int r1 = (int)((long)ny * (blockIdx.x + 1) / gridDim.x);
    const float* r = rho + (size_t)b * ny * nx;
    int min_row = ny, min_col = nx, max_col = -1;
    for (long c = (long)r0 * nx + threadIdx.x; c < (long)r1 * nx; c += blockDim.x) {
        if (fabsf(r[c] - rho_amb) >= contrast) {
            const int j = (int)(c / nx), i = (int)(c - (long)j * nx);
            min_row = min(min_row, j);
            min_col = min(min_col, i);
            max_col = max(max_col, i);
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        min_row = min(min_row, __shfl_down_sync(0xffffffffu, min_row, off));
        min_col = min(min_col, __shfl_down_sync(0xffffffffu, min_col, off));
        max_col = max(max_col, __shfl_down_sync(0xffffffffu, max_col, off));
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        s_min_row[warp] = min_row;
        s_min_col[warp] = min_col;
        s_max_col[warp] = max_col;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
            min_row = min(min_row, s_min_row[w]);
            min_col = min(min_col, s_min_col[w]);
            max_col = max(max_col, s_max_col[w]);
        }
        if (max_col >= 0) {
            atomicMin(&out[3 * b + 0], min_row);
            atomicMin(&out[3 * b + 1], min_col);
            atomicMax(&out[3 * b + 2], max_col);
        }
    }
}

}  // namespace

hp_status launch_advect(const float* u, const float* v, const float* rho, const uint8_t* flags,
                        float* u_out, float* v_out, float* rho_out, hp_shape s,
                        const hp_plume_params& p, cudaStream_t st)
{
    const int ty = adv_ty(p.scheme == 1);
    dim3 blk(kAdvThreads), grd((s.nx + 1 + kAdvTX - 1) / kAdvTX, (s.ny + ty) / ty, s.batch);
    const bool wide = s.nx >= 1 << 22 || s.ny >= 1 << 22;
    auto kernel = p.scheme == 1 ? (wide ? advect_kernel<true, true> : advect_kernel<true, false>)
                                : (wide ? advect_kernel<false, true> : advect_kernel<false, false>);
    kernel<<<grd, blk, 0, st>>>(u, v, rho, flags, u_out, v_out, rho_out, s.ny, s.nx, p);
    return check_launch();
}

}  // namespace hp

extern "C" hp_status hp_advect_step(const float* u, const float* v, const float* rho,
                                    const uint8_t* flags, float* u_out, float* v_out,
                                    float* rho_out, hp_shape s, const hp_plume_params* p,
                                    void* stream)
{
    if (!u || !v || !rho || !flags || !u_out || !v_out || !rho_out || !p || !hp::shape_ok(s))
        return HP_ERR_INVALID_ARG;
    if (u_out == u || v_out == v || rho_out == rho || !(p->dt >= 0.0f)) return HP_ERR_INVALID_ARG;
    if (p->scheme != 0 && p->scheme != 1) return HP_ERR_INVALID_ARG;
    if ((p->open_top != 0 && p->open_top != 1) || !isfinite(p->u_in)) return HP_ERR_INVALID_ARG;
    return hp::launch_advect(u, v, rho, flags, u_out, v_out, rho_out, s, *p, (cudaStream_t)stream);
}

extern "C" hp_status hp_plume_head(const float* rho, hp_shape s, float rho_amb, float contrast,
                                   int32_t* out, void* stream)
{
    if (!rho || !out || !hp::shape_ok(s) || !(contrast >= 0.0f)) return HP_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    hp::plume_head_init_kernel<<<(s.batch + 127) / 128, 128, 0, st>>>(out, s.batch, s.ny, s.nx);
    // about 16 rows per CTA, at most 64 CTAs per grid
    const int slices = s.ny < 16 ? 1 : (s.ny / 16 < 64 ? s.ny / 16 : 64);
    hp::plume_head_kernel<<<dim3(slices, s.batch), 512, 0, st>>>(rho, s.ny, s.nx, rho_amb,
                                                                  contrast, out);
    return hp::check_launch();
}
