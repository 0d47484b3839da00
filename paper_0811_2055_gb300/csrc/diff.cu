// Differentiable float splat: forward image and its adjoint with respect to the points'
// positions, weights and log smoothing lengths, for fitting a node's representatives to the
// full-data image (the paper's goal that the LOD image be indistinguishable from a full render).
//
// Reading (float path, not the exact integer path): fp32 projection as in the renderer,
// sigma = clamp(F exp(l) / zc, sigma_min, sigma_max), kernel
//   K(r) = (exp(-r^2 / 2 sigma^2) - exp(-4.5)) / (2 pi sigma^2 C'),  r < 3 sigma,  C' = 1 - 5.5 e^-4.5
// (unit integral, continuous at the support edge), I = sum_i w_i K_i, fp32 accumulation.
// The forward pass goes by screen tiles, the adjoint point by point over the points' own discs; it recomputes every
// per-pixel term, nothing is stored per pixel.
#include <algorithm>
#include <cmath>
#include <vector>

#include "render.cuh"

namespace gb {
namespace {

constexpr int DRT = 256;          // block size
constexpr int DTW = 64, DTH = 16; // forward tile: eight strips of 8 x 16 pixels, a warp each
constexpr uint32_t DITEM = 1024;  // records per work item, at most
constexpr float E45 = 0.011108996538242306f;   // exp(-4.5)
constexpr float INV_2PI_C = 0.16951204f;       // 1 / (2 pi (1 - 5.5 exp(-4.5)))
constexpr float LOG2E = 1.4426950408889634f;

struct DCam {
    float ex, ey, ez, rx, ry, rz, ux, uy, uz, fx, fy, fz;
    float F, CX, CY, ZN, smin, smax;
    int W, H, tiles_x, tiles_y;
};

__device__ __forceinline__ float ex2(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

struct DProj {
    float u, v, s, xc, yc, zc;
    bool clamped;
};

__device__ __forceinline__ bool dproject(const DCam &c, const float *xyz, const float *logh, uint32_t i, DProj &o)
{
    const float dx = xyz[3 * i] - c.ex, dy = xyz[3 * i + 1] - c.ey, dz = xyz[3 * i + 2] - c.ez;
    o.xc = c.rx * dx + c.ry * dy + c.rz * dz;
    o.yc = c.ux * dx + c.uy * dy + c.uz * dz;
    o.zc = c.fx * dx + c.fy * dy + c.fz * dz;
    if (!(o.zc > c.ZN)) return false;
    const float iz = 1.0f / o.zc;
    o.u = c.CX + c.F * o.xc * iz;
    o.v = c.CY - c.F * o.yc * iz;
    const float s = c.F * expf(logh[i]) * iz;
    o.clamped = !(s >= c.smin && s <= c.smax);
    o.s = s >= c.smin ? (s <= c.smax ? s : c.smax) : c.smin;
    const float R = 3.0f * o.s + 1.0f;
    return o.u + R >= 0.0f && o.u - R <= (float)c.W && o.v + R >= 0.0f && o.v - R <= (float)c.H;
}

__device__ __forceinline__ void dtiles(const DCam &c, const DProj &o, int &tx0, int &tx1, int &ty0, int &ty1)
{
    const float R = 3.0f * o.s + 1.0f;
    const int x0 = max(0, (int)floorf(o.u - R - 0.5f)), x1 = min(c.W - 1, (int)ceilf(o.u + R - 0.5f));
    const int y0 = max(0, (int)floorf(o.v - R - 0.5f)), y1 = min(c.H - 1, (int)ceilf(o.v + R - 0.5f));
    tx0 = x0 / DTW;
    tx1 = x1 / DTW;
    ty0 = y0 / DTH;
    ty1 = y1 / DTH;
    if (x0 > x1 || y0 > y1) tx0 = 1, tx1 = 0;
}

// Forward binning.  blockIdx.y is a view of the chunk, blockIdx.x a part of the points; a CTA counts its
// (tile, point) pairs per tile in shared memory and writes one histogram column, hist[(view, tile)][part];
// the exclusive scan of hist gives every part its base in every tile, and the record pass places
// records {u, v, a = -log2(e) / (2 sigma^2), c = w norm / sigma^2} (c not finite: {u, v, -a, w}) with shared-memory
// atomics.  (Counting
// with warp-aggregated global atomics spent 260 cycles a round in __match_any_sync: 1M points x 16
// views, count + records 4.7 ms; now 0.4 ms.)  With more tiles than a CTA's shared memory holds (SHARED
// false) the counters are global, cnt[(view, tile)], and there is one part.  The scan is modulo 2^32; with
// MANY the counting pass adds the number of records to `pairs` in 64 bits.  It also clears the two counters that the
// next launches use.
template <bool SCATTER, bool SHARED, bool MANY>
__global__ void __launch_bounds__(DRT) k_dbin(const DCam *__restrict__ cams, int v0, const float *__restrict__ xyz,
                                              const float *__restrict__ w, const float *__restrict__ logh, uint32_t n,
                                              uint32_t per_part, uint32_t *__restrict__ hist,
                                              const uint32_t *__restrict__ off, float4 *__restrict__ rec,
                                              unsigned long long *pairs, uint32_t *counters)
{
    extern __shared__ uint32_t dsh[];
    if (!SCATTER && threadIdx.x < 2 && blockIdx.x == 0 && blockIdx.y == 0) counters[threadIdx.x] = 0u;
    const DCam c = cams[v0 + blockIdx.y];
    const uint32_t ntiles = (uint32_t)(c.tiles_x * c.tiles_y), parts = SHARED ? gridDim.x : 1u;
    const size_t row0 = (size_t)blockIdx.y * ntiles;
    uint32_t *cnt = SHARED ? dsh : hist + row0;
    if (SHARED) {
        for (uint32_t t = threadIdx.x; t < ntiles; t += DRT)
            dsh[t] = SCATTER ? off[(row0 + t) * parts + blockIdx.x] : 0u;
        __syncthreads();
    }
    const uint32_t i0 = blockIdx.x * per_part, i1 = min(n, i0 + per_part); // i0 < n; n is at most DPOINTS
    unsigned long long placed = 0;
    for (uint32_t i = i0 + threadIdx.x; i < i1; i += DRT) {
        DProj o;
        if (!dproject(c, xyz, logh, i, o)) continue;
        int tx0, tx1, ty0, ty1;
        dtiles(c, o, tx0, tx1, ty0, ty1);
        if (MANY) placed += (unsigned long long)(max(tx1 - tx0 + 1, 0) * (ty1 - ty0 + 1));
        float4 r;
        if (SCATTER) {
            const float s2 = o.s * o.s;
            r = make_float4(o.u, o.v, -0.5f * LOG2E / s2, w[i] * (INV_2PI_C / s2));
            if (!isfinite(r.w)) r = make_float4(o.u, o.v, -r.z, w[i]);
        }
        for (int ty = ty0; ty <= ty1; ++ty)
            for (int tx = tx0; tx <= tx1; ++tx) {
                const uint32_t t = (uint32_t)(ty * c.tiles_x + tx);
                if (SCATTER) rec[atomicAdd(&cnt[t], 1u)] = r;
                else atomicAdd(&cnt[t], 1u);
            }
    }
    if (SHARED && !SCATTER) {
        __syncthreads();
        for (uint32_t t = threadIdx.x; t < ntiles; t += DRT) hist[(row0 + t) * parts + blockIdx.x] = dsh[t];
    }
    if (MANY) {
        for (int d = 16; d > 0; d >>= 1) placed += __shfl_xor_sync(0xffffffffu, placed, d);
        if ((threadIdx.x & 31) == 0 && placed) atomicAdd(pairs, placed);
    }
}

// Work items {tile, first record, end, 0} of at most per_item records of every (view, tile), from the scanned
// histogram (total = its end).  A block takes room for its 1024 tiles' items at the end of the list, *nitems long (cleared
// before); the list's order is not fixed, nor is that of an image's sums.  (One block over all the tiles in turn: two
// views of 16000 x 16000, 500,000 tiles, 0.7 ms of 1.13; now 0.38 in all.)
__global__ void __launch_bounds__(1024) k_ditems(uint32_t nt, uint32_t parts, uint32_t per_item, const uint32_t *__restrict__ off,
                                                 const uint32_t *total, uint4 *__restrict__ items, uint32_t *nitems)
{
    __shared__ uint32_t wsum[32], first;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t t = blockIdx.x * 1024 + threadIdx.x;
    uint32_t a = 0, b = 0;
    if (t < nt) {
        a = off[(size_t)t * parts];
        b = t + 1 < nt ? off[(size_t)(t + 1) * parts] : *total;
    }
    const uint32_t k = (b - a + per_item - 1) / per_item;
    uint32_t incl = k;
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint32_t before = 0, all = 0;
    for (int q = 0; q < 32; ++q) {
        before += q < warp ? wsum[q] : 0u;
        all += wsum[q];
    }
    if (threadIdx.x == 0) first = all ? atomicAdd(nitems, all) : 0u;
    __syncthreads();
    uint32_t at = first + before + incl - k;
    for (uint32_t s = a; s < b; s += per_item, ++at) items[at] = make_uint4(t, s, min(b, s + per_item), 0u);
}

// Forward.  A unit of work is a strip of 8 x 16 pixels of an item, taken by a warp on its own: one lane
// per pixel of a block of 8 x 4, four blocks.  The warp reads the item's records 32 at a time, one
// per lane, lists those whose disc reaches the upper, the lower or both pairs of blocks, and walks a list of 16 or more
// with the sums in registers.  Per (record, pixel): two products, the exponential, and
// max(e - exp(-4.5), 0) as a saturating addition, which is 0 from the support edge on, so no pixel is
// tested.  (A thread per pixel of 16 x 16 tiles with two divisions a pair: 1M points x 16 views 5.2 ms;
// now 1.6 ms.)  Records whose weight, or its product with the norm, is not finite must not reach
// pixels outside their disc, and inside it the kernel's value scales the weight first: they have a list of their own.
enum { D_BOTH, D_UP, D_LOW, D_ODD, D_LISTS };
constexpr int DLIST_MIN = 16, DLIST = DLIST_MIN - 1 + 32;
struct DSmem {
    uint32_t count[DRT / 32][D_LISTS];
    float4 list[DRT / 32][D_LISTS][DLIST];
};

template <int FIRST, int N, bool TEST>
__device__ __forceinline__ void dwalk(const float4 *__restrict__ list, int n, float px, float py, float (&acc)[4])
{
#pragma unroll 2
    for (int i = 0; i < n; ++i) {
        const float4 A = list[i];
        const float dx = px - A.x, ta = dx * dx * A.z, dy = py + 4 * FIRST - A.y;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const float d = dy + 4 * k, t = fmaf(d * d, A.z, ta), e = ex2(t);
            if (!TEST) acc[FIRST + k] = fmaf(A.w, __saturatef(e - E45), acc[FIRST + k]);
            else if (t > -4.5f * LOG2E) acc[FIRST + k] += A.w * (e - E45) * (A.z * (-2.0f / LOG2E * INV_2PI_C));
        }
    }
}

__global__ void __launch_bounds__(DRT, 4) k_dforward(const DCam *__restrict__ cams, int v0,
                                                     const float4 *__restrict__ rec, const uint4 *__restrict__ items,
                                                     const uint32_t *nitems, uint32_t *next, float *images)
{
    __shared__ DSmem sm;
    const DCam &c = cams[v0]; // one resolution for all views
    const uint32_t ntiles = (uint32_t)(c.tiles_x * c.tiles_y), nunits = *nitems * 8u;
    const int W = c.W, H = c.H, tiles_x = c.tiles_x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = gbd::lanemask_lt();
    float4(*list)[DLIST] = sm.list[warp];
    uint32_t *count = sm.count[warp];
    for (;;) {
        uint32_t unit = 0;
        if (lane == 0) unit = atomicAdd(next, 1u);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        if (unit >= nunits) break;
        const uint4 it = items[unit >> 3];
        const uint32_t vl = it.x / ntiles, t = it.x - vl * ntiles;
        const int xs = (int)(t % tiles_x) * DTW + (int)(unit & 7u) * 8, ys = (int)(t / tiles_x) * DTH;
        if (xs >= W) continue;
        const float px = (float)(xs + (lane & 7)) + 0.5f, py = (float)(ys + (lane >> 3)) + 0.5f;
        // pixel-centre rectangles of the two pairs of blocks
        const float cx0 = xs + 0.5f, cx1 = min(xs + 8, W) - 0.5f, cy0 = ys + 0.5f, cy1 = min(ys + 8, H) - 0.5f;
        const float cy2 = ys + 8.5f, cy3 = min(ys + 16, H) - 0.5f;
        const bool two = ys + 8 < H;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        __syncwarp();
        if (lane < D_LISTS) count[lane] = 0u;
        for (uint32_t base = it.y; base < it.z; base += 32) {
            float4 R = make_float4(0.f, 0.f, -1.f, 0.f);
            bool up = false, low = false, odd = false;
            if (base + lane < it.z) {
                R = __ldg(&rec[base + lane]);
                odd = R.z > 0.0f;
                R.z = -fabsf(R.z);
                const float r9 = __fdividef(-4.5f * LOG2E, R.z) * (1.0f + 0x1p-18f); // 9 sigma^2, rounded up
                const float ex = fmaxf(fmaxf(cx0 - R.x, R.x - cx1), 0.0f), ex2_ = ex * ex;
                const float eu = fmaxf(fmaxf(cy0 - R.y, R.y - cy1), 0.0f);
                const float el = fmaxf(fmaxf(cy2 - R.y, R.y - cy3), 0.0f);
                up = fmaf(eu, eu, ex2_) < r9;
                low = two && fmaf(el, el, ex2_) < r9;
            }
            const bool in = up || low;
            __syncwarp(); // the counters and the walks of the round before
            const int l = odd ? D_ODD : (up && low ? D_BOTH : (up ? D_UP : D_LOW));
#pragma unroll
            for (int q = 0; q < D_LISTS; ++q) {
                const uint32_t m = __ballot_sync(0xffffffffu, in && l == q);
                if (!m) continue;
                const uint32_t at = count[q];
                if (in && l == q) list[q][at + __popc(m & lt)] = R;
                __syncwarp();
                if (lane == 0) count[q] = at + __popc(m);
            }
            __syncwarp();
            const uint32_t cn = lane < D_LISTS ? count[lane] : 0u;
            uint32_t todo = __ballot_sync(0xffffffffu, cn >= (base + 32 >= it.z ? 1u : (uint32_t)DLIST_MIN));
            while (todo) {
                const int q = __ffs(todo) - 1;
                todo &= todo - 1;
                const int m = (int)__shfl_sync(0xffffffffu, cn, q);
                if (q == D_BOTH) dwalk<0, 4, false>(list[q], m, px, py, acc);
                else if (q == D_UP) dwalk<0, 2, false>(list[q], m, px, py, acc);
                else if (q == D_LOW) dwalk<2, 2, false>(list[q], m, px, py, acc);
                else dwalk<0, 4, true>(list[q], m, px, py, acc);
                if (lane == 0) count[q] = 0u;
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = xs + (lane & 7), y = ys + (lane >> 3) + 4 * k;
            if (x < W && y < H && acc[k] != 0.0f) atomicAdd(&images[((size_t)(v0 + vl) * H + y) * W + x], acc[k]);
        }
    }
}

// ------------------------------------------------------------------ adjoint
// Sums over the pixels of one record's disc: g e, g, g e dx, g e dy, g e r^2 (e = exp(-r^2 / 2 sigma^2)).
struct DSums {
    float ge = 0.f, g = 0.f, gex = 0.f, gey = 0.f, ger = 0.f;
    // Column x, rows y0, y0 + step, ... <= y1 of an image (ok false: none, with the same control flow).
    // r^2 is rounded as the sum of two products (no fused operation): the derivative jumps at the support
    // edge, so which pixels are inside is part of the result.  A value outside, finite or not, adds
    // nothing.  ROWS rows' loads are in flight at a time, also where fewer are left (a remainder loop
    // would wait for each); a row past the end reads as 0.
    template <int ROWS>
    __device__ __forceinline__ void column(const float *__restrict__ img, int W, int x, bool ok, int y0, int y1,
                                           int step, float u, float v, float a, float r9)
    {
        const float dx = (float)x + 0.5f - u, dx2 = __fmul_rn(dx, dx), fstep = (float)step;
        const float *p = img + (size_t)y0 * W + x;
        const size_t pitch = (size_t)step * W;
        float fy = (float)y0 + 0.5f, sge = 0.f;
        for (int y = y0; y <= y1; y += ROWS * step) {
            float q[ROWS];
#pragma unroll
            for (int k = 0; k < ROWS; ++k) {
                q[k] = ok && y + k * step <= y1 ? __ldg(p) : 0.0f;
                p += pitch;
            }
#pragma unroll
            for (int k = 0; k < ROWS; ++k) {
                const float dy = fy - v, r2 = __fadd_rn(dx2, __fmul_rn(dy, dy));
                const float in = r2 < r9 ? q[k] : 0.0f, e = in * ex2(r2 * a);
                sge += e;
                g += in;
                gey = fmaf(e, dy, gey);
                ger = fmaf(e, r2, ger);
                fy += fstep;
            }
        }
        ge += sge;
        gex = fmaf(dx, sge, gex);
    }
    template <int FROM> __device__ __forceinline__ void reduce() // over FROM * 2 lanes
    {
#pragma unroll
        for (int d = FROM; d > 0; d >>= 1) {
            ge += __shfl_xor_sync(0xffffffffu, ge, d);
            g += __shfl_xor_sync(0xffffffffu, g, d);
            gex += __shfl_xor_sync(0xffffffffu, gex, d);
            gey += __shfl_xor_sync(0xffffffffu, gey, d);
            ger += __shfl_xor_sync(0xffffffffu, ger, d);
        }
    }
};

// A record's derivatives with respect to its weight, centre and sigma
struct DTerms {
    float w = 0.f, u = 0.f, v = 0.f, s = 0.f;
};

// from the plain sums over its disc
__device__ __forceinline__ DTerms dterms(float s, float wi, const DSums &S)
{
    const float is = 1.0f / s, is2 = is * is, norm = INV_2PI_C * is2, k = S.ge - E45 * S.g, wn = wi * norm;
    DTerms T;
    T.w = norm * k;
    T.u = wn * (S.gex * is2);
    T.v = wn * (S.gey * is2);
    T.s = wn * (is * (S.ger * is2 - 2.0f * k));
    return T;
}

// The same pixel by pixel over every step-th row, by a whole warp: each pixel's terms are scaled before they are added,
// and a pixel without upstream value is left out.  For gradients that the plain sums do not give as finite numbers:
// a weight that is not finite where nothing comes from upstream is 0, not inf 0; one infinite upstream value is
// infinite, not inf - inf; and sums that overflow before they are scaled.
__device__ __forceinline__ DTerms dterms_each(const float *__restrict__ img, int W, int x0, int x1, int y0, int y1,
                                              int step, float u, float v, float s, float wi)
{
    const float s2 = s * s, a = -0.5f * LOG2E / s2, norm = INV_2PI_C / s2, is = 1.0f / s, is2 = is * is;
    const int lane = threadIdx.x & 31, lw = x1 - x0 >= 16 ? 5 : 3, across = 1 << lw; // 32 columns x 1 row, or 8 x 4
    DTerms T;
    for (int y = y0 + (lane >> lw) * step; y <= y1; y += (32 >> lw) * step) {
#pragma unroll 4
        for (int x = x0 + (lane & (across - 1)); x <= x1; x += across) {
            const float g = __ldg(&img[(size_t)y * W + x]), dx = (float)x + 0.5f - u, dy = (float)y + 0.5f - v;
            const float r2 = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
            if (g != 0.0f && r2 < 9.0f * s2) {
                const float e = ex2(r2 * a) * norm, k = e - E45 * norm, gw = g * wi;
                T.w += g * k;
                T.u += gw * e * dx * is2;
                T.v += gw * e * dy * is2;
                T.s += gw * ((e * r2 * is2 - 2.0f * k) * is);
            }
        }
        if (isnan(T.w) && isnan(T.u) && isnan(T.v) && isnan(T.s)) break; // nothing changes them any more
    }
    for (int d = 16; d > 0; d >>= 1) {
        T.w += __shfl_xor_sync(0xffffffffu, T.w, d);
        T.u += __shfl_xor_sync(0xffffffffu, T.u, d);
        T.v += __shfl_xor_sync(0xffffffffu, T.v, d);
        T.s += __shfl_xor_sync(0xffffffffu, T.s, d);
    }
    return T;
}

struct DGrad {
    float x = 0.f, y = 0.f, z = 0.f, w = 0.f, l = 0.f;
    // chains a record's derivatives to its position, weight and log smoothing length
    __device__ __forceinline__ void add(const DCam &c, const DProj &o, const DTerms &T)
    {
        if (T.w == 0.f && T.u == 0.f && T.v == 0.f && T.s == 0.f) return;
        const float iz = 1.0f / o.zc;
        const float dxc = T.u * c.F * iz;
        const float dyc = -T.v * c.F * iz;
        const float ds_dz = o.clamped ? 0.0f : -o.s * iz;
        const float dzc = T.u * (-c.F * o.xc * iz * iz) + T.v * (c.F * o.yc * iz * iz) + T.s * ds_dz;
        x += c.rx * dxc + c.ux * dyc + c.fx * dzc;
        y += c.ry * dxc + c.uy * dyc + c.fy * dzc;
        z += c.rz * dxc + c.uz * dyc + c.fz * dzc;
        w += T.w;
        if (!o.clamped) l += T.s * o.s;
    }
    // false if a term that was added is not finite (or nearly so)
    __device__ __forceinline__ bool finite() const
    {
        return fabsf(x) + fabsf(y) + fabsf(z) + fabsf(w) + fabsf(l) < INFINITY;
    }
    __device__ __forceinline__ void add_to(uint32_t i, float *gxyz, float *gw, float *glogh) const
    {
        atomicAdd(&gxyz[3 * (size_t)i], x);
        atomicAdd(&gxyz[3 * (size_t)i + 1], y);
        atomicAdd(&gxyz[3 * (size_t)i + 2], z);
        atomicAdd(&gw[i], w);
        atomicAdd(&glogh[i], l);
    }
};

// the clipped pixel box of a record's disc
__device__ __forceinline__ void dbox(float u, float v, float s, int W, int H, int &x0, int &x1, int &y0, int &y1)
{
    const float R = 3.0f * s;
    x0 = max(0, (int)floorf(u - R - 0.5f));
    x1 = min(W - 1, (int)ceilf(u + R - 0.5f));
    y0 = max(0, (int)floorf(v - R - 0.5f));
    y1 = min(H - 1, (int)ceilf(v + R - 0.5f));
}

// Adjoint.  A point's gradient only reads dL/dI inside its own disc, so it needs no tiles, no records
// and, with one group of eight lanes summing a point over all views, no atomics.  Lane l projects view
// l of eight; the group walks each visible view's box, a column per lane; the lanes' five sums go
// through shared memory, where lane l adds up and chains view l's (shuffle reductions were the larger
// half of a small disc's cost).  Boxes of more than DSMALL column-rows are walked by the whole warp (8
// columns x 4 rows at a time), one after another, so that a group does not wait for its neighbours'
// larger ones.  The image rows come through L1.  Box areas from DBIG up go to a list that k_dbig
// spreads over the grid (the warp takes them itself when the list is full).  With few points the
// views are split over blockIdx.y (ATOMIC: the outputs were cleared).  Per pixel one exponential and no
// division.  1M points x 16 views of 256 x 256, nine tenths of the discs 5 px wide: by tiles, with
// per-tile records and five atomics each, 10.6 ms + 4.7 ms of binning; with shuffle reductions 4.0
// ms; now 3.0 ms.
constexpr int DSMALL = 12;
constexpr int DROWS = 8;
constexpr int DBIG = 8192;
constexpr uint32_t DBIG_CAP = 1u << 16;
constexpr int DBIG_SLICES = 16; // units of a listed record: every 16th row

template <bool ATOMIC>
__global__ void __launch_bounds__(DRT, 4) k_dgather(const DCam *__restrict__ cams, int nv, int views_per,
                                                 const float *__restrict__ xyz, const float *__restrict__ w,
                                                 const float *__restrict__ logh, uint32_t n,
                                                 const float *__restrict__ grad, float *gxyz, float *gw, float *glogh,
                                                 uint2 *__restrict__ big, uint32_t *nbig,
                                                 uint32_t *__restrict__ oddw, uint32_t *nodd)
{
    __shared__ float part[DRT / 8][8][41]; // per group and view: eight lanes' sums (41: conflict-free reads)
    const int lane = threadIdx.x & 31, l8 = lane & 7, g0 = lane & 24;
    const unsigned long long i64 = (unsigned long long)blockIdx.x * (DRT / 8) + (threadIdx.x >> 3);
    const bool live = i64 < n;
    const uint32_t i = live ? (uint32_t)i64 : 0u;
    const int va = (int)blockIdx.y * views_per, ve = min(nv, va + views_per);
    const int W = cams[0].W, H = cams[0].H;
    const size_t npix = (size_t)W * H;
    const float wi = live ? w[i] : 0.f;
    DGrad G;
    for (int vb = va; vb < ve; vb += 8) {
        DProj o;
        o.u = o.v = 0.f;
        o.s = 1.f;
        int x0 = 0, x1 = -1, y0 = 0, y1 = -1;
        if (live && vb + l8 < ve && dproject(cams[vb + l8], xyz, logh, i, o)) dbox(o.u, o.v, o.s, W, H, x0, x1, y0, y1);
        bool vis = x0 <= x1 && y0 <= y1;
        const bool large = vis && (long long)(x1 - x0 + 1) * (y1 - y0 + 1) >= DBIG;
        if (large) {
            const uint32_t at = atomicAdd(nbig, 1u);
            if (at < DBIG_CAP) {
                big[at] = make_uint2(i, (uint32_t)(vb + l8));
                vis = false;
            }
        }
        const bool small = vis && ((x1 - x0 + 8) >> 3) * (y1 - y0 + 1) <= DSMALL;
        const float s2 = o.s * o.s, a = (-0.5f * LOG2E) / s2, r9 = 9.0f * s2;
        const int xx = x0 | x1 << 16, yy = y0 | y1 << 16; // image coordinates are below 2^14
        const uint32_t groups = __ballot_sync(0xffffffffu, small);
        // small boxes: a group each, the four groups of the warp side by side
        uint32_t todo = (groups | groups >> 8 | groups >> 16 | groups >> 24) & 255u;
        while (todo) {
            const int j = __ffs(todo) - 1, src = g0 + j;
            todo &= todo - 1u;
            const float qu = __shfl_sync(0xffffffffu, o.u, src), qv = __shfl_sync(0xffffffffu, o.v, src);
            const float qa = __shfl_sync(0xffffffffu, a, src), q9 = __shfl_sync(0xffffffffu, r9, src);
            const int qx = __shfl_sync(0xffffffffu, xx, src), qy = __shfl_sync(0xffffffffu, yy, src);
            DSums S;
            if (groups >> src & 1u)
                for (int c = qx & 0xFFFF; c <= qx >> 16; c += 8)
                    S.column<6>(grad + (size_t)(vb + j) * npix, W, c + l8, c + l8 <= qx >> 16, qy & 0xFFFF, qy >> 16, 1, qu,
                                qv, qa, q9);
            float *p = part[threadIdx.x >> 3][j] + l8;
            p[0] = S.ge;
            p[8] = S.g;
            p[16] = S.gex;
            p[24] = S.gey;
            p[32] = S.ger;
        }
        __syncwarp();
        DSums own;
        if (small) {
            const float *p = part[threadIdx.x >> 3][l8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                own.ge += p[q];
                own.g += p[8 + q];
                own.gex += p[16 + q];
                own.gey += p[24 + q];
                own.ger += p[32 + q];
            }
        }
        __syncwarp();
        uint32_t m = __ballot_sync(0xffffffffu, vis && !small);
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1u;
            const float qu = __shfl_sync(0xffffffffu, o.u, src), qv = __shfl_sync(0xffffffffu, o.v, src);
            const float qa = __shfl_sync(0xffffffffu, a, src), q9 = __shfl_sync(0xffffffffu, r9, src);
            const int qx = __shfl_sync(0xffffffffu, xx, src), qy = __shfl_sync(0xffffffffu, yy, src);
            const int lw = (qx >> 16) - (qx & 0xFFFF) >= 16 ? 5 : 4; // 32 columns x 1 row, or 16 x 2
            DSums S;
            const int lx = lane & ((1 << lw) - 1), ly = lane >> lw, step = 32 >> lw;
            for (int c = qx & 0xFFFF; c <= qx >> 16; c += 1 << lw)
                S.column<DROWS>(grad + (size_t)(vb + (src & 7)) * npix, W, c + lx, c + lx <= qx >> 16, (qy & 0xFFFF) + ly,
                                qy >> 16, step, qu, qv, qa, q9);
            S.reduce<16>();
            if (lane == src) own = S;
        }
        if (vis) G.add(cams[vb + l8], o, dterms(o.s, wi, own));
    }
    if (__any_sync(0xffffffffu, !G.finite())) { // left to k_dbig
        if (lane == 0)
            oddw[atomicAdd(nodd, 1u)] = (blockIdx.y * gridDim.x + blockIdx.x) * (DRT / 32) + (threadIdx.x >> 5);
        G = DGrad();
    }
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) {
        G.x += __shfl_xor_sync(0xffffffffu, G.x, d);
        G.y += __shfl_xor_sync(0xffffffffu, G.y, d);
        G.z += __shfl_xor_sync(0xffffffffu, G.z, d);
        G.w += __shfl_xor_sync(0xffffffffu, G.w, d);
        G.l += __shfl_xor_sync(0xffffffffu, G.l, d);
    }
    if (!live || l8) return;
    if (ATOMIC) {
        G.add_to(i, gxyz, gw, glogh);
    } else {
        gxyz[3 * (size_t)i] = G.x;
        gxyz[3 * (size_t)i + 1] = G.y;
        gxyz[3 * (size_t)i + 2] = G.z;
        gw[i] = G.w;
        glogh[i] = G.l;
    }
}

// whether (i, view) is in the list of large records, by a whole warp
__device__ __forceinline__ bool dlisted(const uint2 *__restrict__ big, uint32_t i, uint32_t view)
{
    bool found = false;
    for (uint32_t k = threadIdx.x & 31; k < DBIG_CAP; k += 32) {
        const uint2 b = __ldg(&big[k]);
        found |= b.x == i && b.y == view;
    }
    return __any_sync(0xffffffffu, found);
}

// What k_dgather leaves: the listed large records (a unit is every DBIG_SLICES-th row of one, a warp a row at a
// time), and the warps whose plain sums did not give finite gradients, term by term.  Both here, after the walks, so
// that the second costs k_dgather no registers (with dterms_each inside it: 1M points x 16 views 3.19 -> 3.25 ms).
constexpr uint32_t DBIG_ODD = 2048; // units a block can have
constexpr unsigned DBIG_BLOCKS = DBIG_CAP * DBIG_SLICES / DBIG_ODD; // at least so many blocks
__global__ void __launch_bounds__(DRT) k_dbig(const DCam *__restrict__ cams, const float *__restrict__ xyz,
                                              const float *__restrict__ w, const float *__restrict__ logh,
                                              const float *__restrict__ grad, float *gxyz, float *gw, float *glogh,
                                              const uint2 *__restrict__ big, const uint32_t *nbig, uint32_t n, int nv,
                                              int views_per, uint32_t gather_x, const uint32_t *__restrict__ oddw,
                                              const uint32_t *nodd)
{
    __shared__ DSums part[DRT / 32];
    __shared__ DTerms each[DRT / 32];
    __shared__ uint32_t odd[DBIG_ODD / 32]; // units whose gradient is not finite
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t units = min(*nbig, DBIG_CAP) * DBIG_SLICES, nw = *nodd;
    if (blockIdx.x >= max(units, nw)) return;
    if (threadIdx.x < DBIG_ODD / 32) odd[threadIdx.x] = 0u;
    uint32_t nth = 0; // unit of the block
    for (uint32_t k = blockIdx.x; k < units; k += gridDim.x, ++nth) {
        const uint2 b = big[k / DBIG_SLICES];
        const DCam &c = cams[b.y];
        DProj o;
        (void)dproject(c, xyz, logh, b.x, o);
        int x0, x1, y0, y1;
        dbox(o.u, o.v, o.s, c.W, c.H, x0, x1, y0, y1);
        const float s2 = o.s * o.s, a = -0.5f * LOG2E / s2, r9 = 9.0f * s2;
        DSums S;
        for (int x = x0; x <= x1; x += 32)
            S.column<DROWS>(grad + (size_t)b.y * c.W * c.H, c.W, x + lane, x + lane <= x1, y0 + (int)(k % DBIG_SLICES) + warp * DBIG_SLICES, y1,
                     DBIG_SLICES * (DRT / 32), o.u, o.v, a, r9);
        S.reduce<16>();
        __syncthreads();
        if (lane == 0) part[warp] = S;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 1; q < DRT / 32; ++q) {
                S.ge += part[q].ge;
                S.g += part[q].g;
                S.gex += part[q].gex;
                S.gey += part[q].gey;
                S.ger += part[q].ger;
            }
            DGrad G;
            G.add(c, o, dterms(o.s, w[b.x], S));
            if (G.finite()) G.add_to(b.x, gxyz, gw, glogh);
            else odd[nth >> 5] |= 1u << (nth & 31);
        }
    }
    __syncthreads();
    // those again, term by term
    for (uint32_t q = 0; q < (nth + 31) / 32; ++q)
        for (uint32_t m = odd[q]; m; m &= m - 1u) {
            const uint32_t k = blockIdx.x + (q * 32 + (uint32_t)__ffs((int)m) - 1u) * gridDim.x;
            const uint2 b = big[k / DBIG_SLICES];
            const DCam &c = cams[b.y];
            DProj o;
            (void)dproject(c, xyz, logh, b.x, o);
            int x0, x1, y0, y1;
            dbox(o.u, o.v, o.s, c.W, c.H, x0, x1, y0, y1);
            const DTerms T = dterms_each(grad + (size_t)b.y * c.W * c.H, c.W, x0, x1, y0 + (int)(k % DBIG_SLICES) + warp * DBIG_SLICES, y1,
                                         DBIG_SLICES * (DRT / 32), o.u, o.v, o.s, w[b.x]);
            if (lane == 0) each[warp] = T;
            __syncthreads();
            if (threadIdx.x == 0) {
                DTerms A;
                for (int v = 0; v < DRT / 32; ++v) {
                    A.w += each[v].w;
                    A.u += each[v].u;
                    A.v += each[v].v;
                    A.s += each[v].s;
                }
                DGrad G;
                G.add(c, o, A);
                G.add_to(b.x, gxyz, gw, glogh);
            }
            __syncthreads();
        }
    // a warp of k_dgather each: four points, their views eight at a time
    const int l8 = lane & 7, W = cams[0].W, H = cams[0].H;
    for (uint32_t j = blockIdx.x * (DRT / 32) + warp; j < nw; j += gridDim.x * (DRT / 32)) {
        const uint32_t id = oddw[j], block = id / (DRT / 32);
        const unsigned long long i64 = (unsigned long long)(block % gather_x) * (DRT / 8) + id % (DRT / 32) * 4 + (lane >> 3);
        const bool live = i64 < n;
        const uint32_t i = live ? (uint32_t)i64 : 0u;
        const int va = (int)(block / gather_x) * views_per, ve = min(nv, va + views_per);
        const float wi = w[i];
        DGrad G;
        for (int vb = va; vb < ve; vb += 8) {
            DProj o;
            o.u = o.v = 0.f;
            o.s = 1.f;
            int x0 = 0, x1 = -1, y0 = 0, y1 = -1;
            if (live && vb + l8 < ve && dproject(cams[vb + l8], xyz, logh, i, o)) dbox(o.u, o.v, o.s, W, H, x0, x1, y0, y1);
            const bool vis = x0 <= x1 && y0 <= y1, large = vis && (long long)(x1 - x0 + 1) * (y1 - y0 + 1) >= DBIG;
            for (uint32_t m = __ballot_sync(0xffffffffu, vis && (!large || *nbig > DBIG_CAP)); m; m &= m - 1u) {
                const int src = __ffs(m) - 1;
                const uint32_t view = (uint32_t)(vb + (src & 7)), qi = __shfl_sync(0xffffffffu, i, src);
                if (__shfl_sync(0xffffffffu, large, src) && dlisted(big, qi, view)) continue;
                const int qx0 = __shfl_sync(0xffffffffu, x0, src), qx1 = __shfl_sync(0xffffffffu, x1, src);
                const int qy0 = __shfl_sync(0xffffffffu, y0, src), qy1 = __shfl_sync(0xffffffffu, y1, src);
                const float qu = __shfl_sync(0xffffffffu, o.u, src), qv = __shfl_sync(0xffffffffu, o.v, src);
                const float qs = __shfl_sync(0xffffffffu, o.s, src), qw = __shfl_sync(0xffffffffu, wi, src);
                const DTerms T = dterms_each(grad + (size_t)view * W * H, W, qx0, qx1, qy0, qy1, 1, qu, qv, qs, qw);
                if (lane == src) G.add(cams[view], o, T);
            }
        }
        if (live) G.add_to(i, gxyz, gw, glogh); // zeros so far, or the sums of the point's other views
    }
}

DCam make_dcam(const gblod_camera &c, const gblod_render_params &rp)
{
    DCam d;
    d.ex = (float)c.eye[0]; d.ey = (float)c.eye[1]; d.ez = (float)c.eye[2];
    d.rx = (float)c.right[0]; d.ry = (float)c.right[1]; d.rz = (float)c.right[2];
    d.ux = (float)c.up[0]; d.uy = (float)c.up[1]; d.uz = (float)c.up[2];
    d.fx = (float)c.fwd[0]; d.fy = (float)c.fwd[1]; d.fz = (float)c.fwd[2];
    d.F = (float)c.f_px; d.CX = (float)c.cx; d.CY = (float)c.cy; d.ZN = (float)c.z_near;
    d.smin = (float)rp.sigma_min_px;
    d.smax = (float)rp.sigma_max_px;
    d.W = c.width;
    d.H = c.height;
    d.tiles_x = (c.width + DTW - 1) / DTW;
    d.tiles_y = (c.height + DTH - 1) / DTH;
    return d;
}

// One launch at the head of a pass: the views' constants, from the kernel's parameters (a copy from pageable
// memory costs the host 11 to 18 us, a launch 5), and everything the pass adds to, zeroed.
constexpr int CAMS_PER_LAUNCH = 32;
constexpr unsigned long long DZERO = 1ull << 24; // floats from which a memset's bandwidth pays for its call (2 GB: 0.36, 0.31 ms)
struct DSetup {
    int first, n;
    float *zero[3];
    unsigned long long count[3];
    uint32_t *counter; // two words; may be null
    DCam cam[CAMS_PER_LAUNCH];
};
static_assert(sizeof(DSetup) <= 4096, "kernel parameters");

__global__ void k_dsetup(const __grid_constant__ DSetup S, DCam *__restrict__ cams)
{
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < (size_t)S.n) cams[S.first + t] = S.cam[t];
    if (t < 2 && S.counter) S.counter[t] = 0u;
#pragma unroll
    for (int q = 0; q < 3; ++q)
        for (size_t i = t; i < S.count[q]; i += (size_t)gridDim.x * blockDim.x) S.zero[q][i] = 0.0f;
}

void check_views(uint64_t n, const gblod_camera *cams, int nv)
{
    if (n >= 0xFFFFFFFFull) fail(GBLOD_ERR_INVALID_ARG, "too many points");
    for (int v = 0; v < nv; ++v)
        if (cams[v].width != cams[0].width || cams[v].height != cams[0].height)
            fail(GBLOD_ERR_INVALID_ARG, "all views need one resolution");
}

// S: what to zero
const DCam *setup(gblod_renderer *r, const gblod_camera *cams, int nv, const gblod_render_params &rp, DSetup S,
                  cudaStream_t s)
{
    r->d_cams.ensure(r->A, (size_t)nv * sizeof(DCam), s);
    DCam *dc = reinterpret_cast<DCam *>(r->d_cams.p);
    for (S.first = 0; S.first < nv; S.first += CAMS_PER_LAUNCH) {
        S.n = std::min(CAMS_PER_LAUNCH, nv - S.first);
        for (int v = 0; v < S.n; ++v) S.cam[v] = make_dcam(cams[S.first + v], rp);
        const unsigned long long most = std::max({S.count[0], S.count[1], S.count[2]});
        const unsigned g = (unsigned)std::min<unsigned long long>((unsigned long long)persistent_blocks(8), most / 1024 + 1);
        launch(GBLOD_K_RENDER_OTHER, k_dsetup, dim3(g), dim3(256), 0, s, S, dc);
        S.counter = nullptr;
        for (unsigned long long &c : S.count) c = 0;
    }
    return dc;
}

} // namespace

// A forward pass goes by pieces: views [v0, v0 + nv), points [lo, hi).  The records of a piece are at most
// DRECORDS (16 GiB); a piece of more is counted, halved and counted again.  A piece has at most DPOINTS points, so
// that their numbers and coordinate indices stay below 2^32.
constexpr unsigned long long DRECORDS = 1ull << 30;
constexpr uint64_t DPOINTS = 1ull << 30;
struct DPiece {
    int v0, nv;
    uint64_t lo, hi;
};

void diff_forward(gblod_renderer *r, const float *xyz_all, const float *w_all, const float *logh_all, uint64_t n_all,
                  const gblod_camera *cams, int nv, const gblod_render_params &rp, float *images, cudaStream_t s)
{
    check_views(n_all, cams, nv);
    const Allocator &A = r->A;
    const DCam c0 = make_dcam(cams[0], rp);
    r->d_cnt.ensure(A, 8, s); // counters: work items, next unit, listed large records, listed warps, records (64 bits)
    auto *d_pairs = reinterpret_cast<unsigned long long *>(r->d_cnt.p + 4);
    DSetup S{};
    S.zero[0] = images;
    S.count[0] = (unsigned long long)nv * c0.W * c0.H;
    if (S.count[0] > DZERO) {
        GB_CUDA(cudaMemsetAsync(images, 0, S.count[0] * sizeof(float), s));
        S.count[0] = 0;
    }
    const DCam *dc = setup(r, cams, nv, rp, S, s);
    const uint32_t ntiles = (uint32_t)(c0.tiles_x * c0.tiles_y);
    const bool shared = ntiles <= 12288; // 48 KB of counters
    std::vector<DPiece> todo;
    for (uint64_t lo = 0; lo < n_all; lo += DPOINTS) {
        const uint64_t hi = std::min(n_all, lo + DPOINTS);
        // views per chunk: about 2^26 (view, point) pairs, so records stay near a few GB, 2^24 tiles, a grid's y size
        const int vchunk = (int)std::max<uint64_t>(1, std::min<uint64_t>({(uint64_t)nv, (1ull << 26) / (hi - lo), 32768ull, (1ull << 24) / ntiles}));
        for (int v0 = 0; v0 < nv; v0 += vchunk) todo.push_back(DPiece{v0, std::min(vchunk, nv - v0), lo, hi});
    }
    std::reverse(todo.begin(), todo.end()); // taken from the back
    while (!todo.empty()) {
        const DPiece pc = todo.back();
        todo.pop_back();
        const int v0 = pc.v0, cnv = pc.nv;
        const uint64_t n = pc.hi - pc.lo;
        const float *xyz = xyz_all + 3 * pc.lo, *w = w_all + pc.lo, *logh = logh_all + pc.lo;
        const uint32_t nt = ntiles * (uint32_t)cnv;
        // parts of the points per view: at least 512 points each, about eight CTAs per SM in all, and a
        // histogram of at most 2^22 columns
        const uint64_t want = std::min<uint64_t>((n + 511) / 512, (uint64_t)std::max(1, persistent_blocks(8) / cnv));
        const uint32_t parts0 = shared ? (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(want, (1u << 22) / nt)) : 1u;
        const uint32_t per = (uint32_t)((n + (shared ? parts0 : want) - 1) / (shared ? parts0 : want));
        const uint32_t gx = (uint32_t)((n + per - 1) / per); // CTAs per view; every one has points
        const uint32_t parts = shared ? gx : 1u;
        const size_t nh = (size_t)nt * parts;
        r->d_hist.ensure(A, nh, s);
        r->d_off.ensure(A, nh + 1, s);
        const dim3 grid(gx, (unsigned)cnv);
        // the records are counted in 64 bits where there could be 2^32
        const bool many = (unsigned long long)cnv * n * ntiles >> 32 != 0; // at most 2^30 pairs, 2^18 tiles each
        if (many) GB_CUDA(cudaMemsetAsync(d_pairs, 0, sizeof(*d_pairs), s));
        if (shared) {
            launch(GBLOD_K_RENDER_OTHER, many ? k_dbin<false, true, true> : k_dbin<false, true, false>, grid, dim3(DRT), ntiles * 4, s, dc, v0, xyz, w, logh,
                   (uint32_t)n, per, r->d_hist.p, (const uint32_t *)nullptr, (float4 *)nullptr, d_pairs, r->d_cnt.p);
        } else {
            GB_CUDA(cudaMemsetAsync(r->d_hist.p, 0, nh * 4, s));
            launch(GBLOD_K_RENDER_OTHER, many ? k_dbin<false, false, true> : k_dbin<false, false, false>, grid, dim3(DRT), 0, s, dc, v0, xyz, w, logh,
                   (uint32_t)n, per, r->d_hist.p, (const uint32_t *)nullptr, (float4 *)nullptr, d_pairs, r->d_cnt.p);
        }
        scan_exclusive_u32(A, r->scan, r->d_hist.p, r->d_off.p, nh, r->d_off.p + nh, s);
        auto *h64 = static_cast<unsigned long long *>(r->hs.get(16));
        uint32_t *total = reinterpret_cast<uint32_t *>(h64 + 1);
        if (many) GB_CUDA(cudaMemcpyAsync(h64, d_pairs, sizeof(*d_pairs), cudaMemcpyDeviceToHost, s));
        GB_CUDA(cudaMemcpyAsync(total, r->d_off.p + nh, 4, cudaMemcpyDeviceToHost, s));
        GB_CUDA(cudaStreamSynchronize(s));
        if ((many ? *h64 : *total) > DRECORDS) {
            const int vm = cnv / 2;
            const uint64_t mid = pc.lo + n / 2;
            // one point of one view has at most 2^18 records
            todo.push_back(cnv > 1 ? DPiece{v0 + vm, cnv - vm, pc.lo, pc.hi} : DPiece{v0, 1, mid, pc.hi});
            todo.push_back(cnv > 1 ? DPiece{v0, vm, pc.lo, pc.hi} : DPiece{v0, 1, pc.lo, mid});
            continue;
        }
        if (*total == 0) continue;
        r->d_rec.ensure(A, *total, s);
        // DITEM records an item, fewer if that gives less than four units a warp (16,000 points, 8 views of 128 x 128:
        // 66 us with 1024, 31 with 128; a million points, many items anyway: 1.62 ms, 2.12 with 128)
        const uint32_t even = (*total / ((uint32_t)persistent_blocks(4) * 4u) + 31u) / 32u * 32u;
        const uint32_t per_item = std::max(128u, std::min(DITEM, even));
        r->d_items.ensure(A, (size_t)nt + *total / per_item, s);
        launch(GBLOD_K_RENDER_OTHER, k_ditems, dim3((nt + 1023) / 1024), dim3(1024), 0, s, nt, parts, per_item,
               (const uint32_t *)r->d_off.p, (const uint32_t *)(r->d_off.p + nh), r->d_items.p, r->d_cnt.p);
        if (shared) {
            launch(GBLOD_K_RENDER_OTHER, k_dbin<true, true, false>, grid, dim3(DRT), ntiles * 4, s, dc, v0, xyz, w, logh,
                   (uint32_t)n, per, (uint32_t *)nullptr, (const uint32_t *)r->d_off.p, r->d_rec.p,
                   (unsigned long long *)nullptr, (uint32_t *)nullptr);
        } else { // the offsets themselves are the cursors (k_ditems has read them)
            launch(GBLOD_K_RENDER_OTHER, k_dbin<true, false, false>, grid, dim3(DRT), 0, s, dc, v0, xyz, w, logh,
                   (uint32_t)n, per, r->d_off.p, (const uint32_t *)nullptr, r->d_rec.p, (unsigned long long *)nullptr,
                   (uint32_t *)nullptr);
        }
        launch(GBLOD_K_SPLAT, k_dforward, dim3((unsigned)persistent_blocks(4)), dim3(DRT), 0, s, dc, v0,
               (const float4 *)r->d_rec.p, (const uint4 *)r->d_items.p, (const uint32_t *)r->d_cnt.p, r->d_cnt.p + 1,
               images);
    }
}

void diff_backward(gblod_renderer *r, const float *xyz, const float *w, const float *logh, uint64_t n,
                   const gblod_camera *cams, int nv, const gblod_render_params &rp, const float *grad_img, float *gxyz,
                   float *gw, float *glogh, cudaStream_t s)
{
    check_views(n, cams, nv);
    if (n == 0) return;
    r->d_cnt.ensure(r->A, 8, s);
    r->d_big.ensure(r->A, DBIG_CAP, s);
    uint32_t *nbig = r->d_cnt.p + 2, *nodd = nbig + 1;
    // with few points the views are split over blocks: a warp's four points times its views are walked
    // one after another, so about 256 warps per SM are wanted (16,000 points x 8 views: 154 us unsplit, 75 us split; 128 warps 82)
    const unsigned gx = (unsigned)((n + DRT / 8 - 1) / (DRT / 8));
    const int split = (int)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)nv, (uint64_t)persistent_blocks(32) / gx));
    const int views_per = (nv + split - 1) / split;
    const dim3 grid(gx, (unsigned)((nv + views_per - 1) / views_per));
    DSetup S{};
    S.counter = nbig;
    if (grid.y > 1) { // blocks add up
        float *const g[3] = {gxyz, gw, glogh};
        for (int q = 0; q < 3; ++q) {
            S.zero[q] = g[q];
            S.count[q] = q ? n : 3 * n;
        }
    }
    r->d_odd.ensure(r->A, (size_t)grid.x * grid.y * (DRT / 32), s);
    const DCam *dc = setup(r, cams, nv, rp, S, s);
    launch(GBLOD_K_SPLAT, grid.y > 1 ? k_dgather<true> : k_dgather<false>, grid, dim3(DRT), 0, s, dc, nv, views_per, xyz,
           w, logh, (uint32_t)n, grad_img, gxyz, gw, glogh, r->d_big.p, nbig, r->d_odd.p, nodd);
    launch(GBLOD_K_SPLAT, k_dbig, dim3(std::max((unsigned)persistent_blocks(4), DBIG_BLOCKS)), dim3(DRT), 0, s, dc, xyz, w, logh, grad_img, gxyz,
           gw, glogh, (const uint2 *)r->d_big.p, (const uint32_t *)nbig, (uint32_t)n, nv, views_per, grid.x,
           (const uint32_t *)r->d_odd.p, (const uint32_t *)nodd);
}

} // namespace gb
