// Per-frame path: R1 view-dependent node selection (depth paragraph: near nodes deep, far
// nodes shallow), R2 projection and screen-tile binning, R3 tiled splatting of every point as a
// blob evaluated at every pixel it covers (GPU paragraph) into 64-bit fixed point, R4 log tone
// map.  The brute-force frame runs R2-R4 over the raw particle arrays.
//
// Determinism: the per-point arithmetic is fp32 with one round-to-nearest per operation in a
// fixed order, positions are quantised to 1/256 px, the kernel is a 1024-entry integer table
// and every pixel is an exact 64-bit integer sum, so the image does not depend on launch
// shape, tiling or the order in which splats are added.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <vector>

#include "lodmath.cuh"
#include "render.cuh"

namespace gb {

void check_image(const gblod_camera &c);
void check_format(const gblod_octree *o, const gblod_render_params &rp);

// integer kernel tables (Gaussian, cubic), filled once per device
__device__ int32_t g_ktab[2][1024];

namespace {

constexpr unsigned ST_RANGE = 1u;
constexpr int RT = 256;       // render block size
constexpr int CHUNK = 2048;   // points per block iteration in the projection kernels
constexpr uint32_t ITEM = 2048; // records per splat work item
constexpr float A_GAUSS = 0x1.499c68p+29f; // 2^32 / (2 pi (1 - e^-4.5))
constexpr float A_CUBIC = 0x1.d1a452p+30f; // 2^32 * 10 / (7 pi)
constexpr float B_GAUSS = 0x1.c71c72p+27f; // 2^31 / 9
constexpr float B_CUBIC = 0x1p+29f;        // 2^31 / 4

void kernel_table_host(int kernel, int32_t *K)
{
    const double qmax = kernel == GBLOD_KERNEL_CUBIC ? 4.0 : 9.0;
    for (int i = 0; i < 1024; ++i) {
        const double q = ((double)i + 0.5) * qmax / 1024.0;
        double f;
        if (kernel == GBLOD_KERNEL_CUBIC) {
            const double xi = std::sqrt(q);
            if (xi < 1.0) {
                const double a = 1.0 - 1.5 * q;
                const double b = 0.75 * (q * xi);
                f = a + b;
            } else {
                const double t = 2.0 - xi;
                f = 0.25 * ((t * t) * t);
            }
        } else {
            f = std::exp(-0.5 * q);
        }
        K[i] = (int32_t)std::nearbyint(65536.0 * f);
    }
}

void set_splat_smem();

// once per device: the kernel tables, and the dynamic shared-memory limit of the splat kernels
// (a device setting, so it is made before any launch that a stream capture could record)
void ensure_tables()
{
    static std::mutex mu;
    static std::vector<int> done;
    int dev = 0;
    GB_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> g(mu);
    if ((int)done.size() <= dev) done.resize(dev + 1, 0);
    if (done[dev]) return;
    static int32_t K[2][1024];
    kernel_table_host(GBLOD_KERNEL_GAUSSIAN, K[0]);
    kernel_table_host(GBLOD_KERNEL_CUBIC, K[1]);
    GB_CUDA(cudaMemcpyToSymbol(g_ktab, K, sizeof(K)));
    set_splat_smem();
    done[dev] = 1;
}

struct Proj {
    float ex, ey, ez, rx, ry, rz, ux, uy, uz, fx, fy, fz;
    float F, CX, CY, ZN, smin, smax, A, B, Rk, Wf, Hf;
    int W, H, TW, TH, tiles_x, tiles_y, kernel;
};

Proj make_proj(const gblod_camera &c, const gblod_render_params &rp)
{
    Proj P;
    P.ex = (float)c.eye[0]; P.ey = (float)c.eye[1]; P.ez = (float)c.eye[2];
    P.rx = (float)c.right[0]; P.ry = (float)c.right[1]; P.rz = (float)c.right[2];
    P.ux = (float)c.up[0]; P.uy = (float)c.up[1]; P.uz = (float)c.up[2];
    P.fx = (float)c.fwd[0]; P.fy = (float)c.fwd[1]; P.fz = (float)c.fwd[2];
    P.F = (float)c.f_px;
    P.CX = (float)c.cx;
    P.CY = (float)c.cy;
    P.ZN = (float)c.z_near;
    P.smin = (float)rp.sigma_min_px;
    P.smax = (float)rp.sigma_max_px;
    const bool cubic = rp.kernel == GBLOD_KERNEL_CUBIC;
    P.A = cubic ? A_CUBIC : A_GAUSS;
    P.B = cubic ? B_CUBIC : B_GAUSS;
    P.Rk = cubic ? 2.0f : 3.0f;
    P.Wf = (float)c.width;
    P.Hf = (float)c.height;
    P.W = c.width;
    P.H = c.height;
    P.TW = rp.tile_w > 0 ? rp.tile_w : 64;
    P.TH = rp.tile_h > 0 ? rp.tile_h : 16;
    P.tiles_x = (P.W + P.TW - 1) / P.TW;
    P.tiles_y = (P.H + P.TH - 1) / P.TH;
    P.kernel = cubic ? 1 : 0;
    return P;
}

struct Splat {
    int32_t U, V;
    uint32_t S;
    float Wf; // amplitude before rounding; Wq = rne(Wf)
};

// R2 for one point.  Returns 1 drawn, 0 culled, -1 amplitude out of range.
__device__ __forceinline__ int project(const Proj &P, float x, float y, float z, float w, float h, Splat &s)
{
    const float dx = __fsub_rn(x, P.ex), dy = __fsub_rn(y, P.ey), dz = __fsub_rn(z, P.ez);
    const float xc = __fadd_rn(__fadd_rn(__fmul_rn(P.rx, dx), __fmul_rn(P.ry, dy)), __fmul_rn(P.rz, dz));
    const float yc = __fadd_rn(__fadd_rn(__fmul_rn(P.ux, dx), __fmul_rn(P.uy, dy)), __fmul_rn(P.uz, dz));
    const float zc = __fadd_rn(__fadd_rn(__fmul_rn(P.fx, dx), __fmul_rn(P.fy, dy)), __fmul_rn(P.fz, dz));
    if (!(zc > P.ZN)) return 0;
    const float iz = __fdiv_rn(1.0f, zc);
    const float u = __fadd_rn(P.CX, __fmul_rn(__fmul_rn(P.F, xc), iz));
    const float v = __fsub_rn(P.CY, __fmul_rn(__fmul_rn(P.F, yc), iz));
    const float sg = __fmul_rn(__fmul_rn(P.F, h), iz);
    const float sigma = sg >= P.smin ? (sg <= P.smax ? sg : P.smax) : P.smin;
    const float s2 = __fmul_rn(sigma, sigma);
    const float Wf = __fdiv_rn(__fmul_rn(w, P.A), s2);
    const float Sf = __fdiv_rn(P.B, s2);
    const float R = __fadd_rn(__fmul_rn(P.Rk, sigma), 2.0f);
    if (!(__fadd_rn(u, R) >= 0.0f && __fsub_rn(u, R) <= P.Wf && __fadd_rn(v, R) >= 0.0f &&
          __fsub_rn(v, R) <= P.Hf))
        return 0;
    if (!(Wf >= 0.0f && Wf < 0x1p48f)) return -1;
    s.U = __float2int_rn(__fmul_rn(u, 256.0f));
    s.V = __float2int_rn(__fmul_rn(v, 256.0f));
    s.S = __float2uint_rn(Sf);
    s.Wf = Wf;
    return 1;
}

// Pixel box (inclusive) that contains every pixel where the table index can be below 1024:
// q S < 2^47 needs |d| < sqrt(2^47 / S) in 1/256 px.
// Returns the bounding radius r (1/256 px) the box was cut from: every pixel of the box has |dx| <= r
// and |dy| <= r.
__device__ __forceinline__ int splat_box(int U, int V, uint32_t S, int W, int H, int &x0, int &x1, int &y0, int &y1)
{
    const float ql = __fdiv_rn(140737488355328.0f, __uint2float_rn(S));
    const int r = (int)sqrtf(ql) + 2;
    const int ax = U - 128 - r, bx = U - 128 + r, ay = V - 128 - r, by = V - 128 + r;
    x0 = -((-ax) >> 8);
    x1 = bx >> 8;
    y0 = -((-ay) >> 8);
    y1 = by >> 8;
    x0 = max(x0, 0);
    y0 = max(y0, 0);
    x1 = min(x1, W - 1);
    y1 = min(y1, H - 1);
    return r;
}

// Points whose pixel box is at most DIRECT_BOX pixels on a side are not binned: the scatter pass
// adds their contributions straight to the image, one 64-bit atomic per pixel inside the support.
// The image is a sum of integers, so it is the same whichever pass adds a contribution and in
// whatever order.  Small boxes are most of the drawn points (sigma at or near its minimum) but a
// small share of the pixel work, and each of their (tile, point) records would cost the splat
// kernel a staging slot, a list entry and a test of a 32-pixel block for a few pixels.  Measured
// on the mid fly-through: 8 is faster than 4 and 6.
constexpr int DIRECT_BOX = 8;

__device__ __forceinline__ bool direct_box(int x0, int x1, int y0, int y1)
{
    return x1 - x0 < DIRECT_BOX && y1 - y0 < DIRECT_BOX;
}

// Bounding radius (1/256 px) up to which a box's pixels all have q = dx^2 + dy^2 < 2^32 (2 r^2 <
// 2^32): dx^2 and dy^2 are then signed 32-bit products and the table index (q S) >> 37 is the high
// word of the 32 x 32 product q S shifted by 5.  Wider boxes (the visible sliver of a large blob
// centred off the image) take 64-bit distances.
constexpr int R_NARROW = 46340;

// One point's clipped pixel box for walk_boxes: n pixels (0: none) from origin xy = x0 | y0 << 16,
// meta = ceil(2^8 / bw) | bw << 9 | wide << 13 | Wl << 16 for box width bw <= DIRECT_BOX, and the
// rule's other operands U, V, S and Wh (Wq = Wh 2^16 + Wl).
struct BoxWalk {
    uint32_t n = 0, xy = 0, meta = 0;
    int U = 0, V = 0;
    uint32_t S = 0, Wh = 0;
};

__device__ __forceinline__ BoxWalk box_walk(int U, int V, uint32_t S, unsigned long long Wq, int r, int x0, int x1,
                                            int y0, int y1)
{
    BoxWalk b;
    const uint32_t bw = (uint32_t)(x1 - x0 + 1);
    b.n = bw * (uint32_t)(y1 - y0 + 1);
    b.xy = (uint32_t)x0 | ((uint32_t)y0 << 16);
    b.meta = ((256u + bw - 1u) / bw) | (bw << 9) | (r > R_NARROW ? 1u << 13 : 0u) |
             ((uint32_t)(Wq & 0xFFFFull) << 16);
    b.U = U;
    b.V = V;
    b.S = S;
    b.Wh = (uint32_t)(Wq >> 16);
    return b;
}

// The per-pixel rule over the boxes (at most DIRECT_BOX x DIRECT_BOX pixels) of a warp's points,
// one point per lane: the warp walks the concatenation of all lanes' box pixels (row-major within a
// box) 32 (point, pixel) pairs at a time, pair k on lane k mod 32.  Lanes stay busy whatever the box
// sizes, and neighbouring lanes take neighbouring pixels of one point instead of 32 points' pixels
// at the same offset (in dense regions often the same pixel).  The owner of pair k of a window: each
// lane whose box starts inside the window writes its lane number at its start offset in a per-warp
// table, one OR-reduction gives the mask of start offsets, and pair k belongs to the box with the
// last start at or before k (the highest set bit of the mask up to k), or, if none, to the box that
// owned the previous window's last pair (boxes are contiguous runs of pairs).  Row and column of pixel m of a box:
// m / bw = (m ceil(2^8 / bw)) >> 8, exact for m < 64 and bw <= 8.  tab(meta, idx) reads the table
// entry; add(tag, x, y, c) receives every nonzero contribution with the tag of the point's lane
// (TAGGED: the lane's `tag`, e.g. its view in a batch; else 0).  Returns this lane's pixel updates.
// Every lane of the warp calls it.
template <bool TAGGED, class Tab, class Add>
__device__ __forceinline__ unsigned walk_boxes(const BoxWalk &b, uint32_t tag, Tab tab, Add add)
{
    const int lane = threadIdx.x & 31;
    uint32_t incl = b.n;
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t excl = incl - b.n;
    __shared__ uint8_t owner_at[32][32]; // blocks of up to 1024 threads
    uint8_t *own = owner_at[threadIdx.x >> 5];
    unsigned hits = 0;
    int carry = 0; // owner of the previous window's last pair
    for (uint32_t base = 0; base < total; base += 32) {
        const uint32_t k = base + (uint32_t)lane;
        const bool starts = b.n && excl >= base && excl < base + 32u;
        if (starts) own[excl - base] = (uint8_t)lane;
        const uint32_t smask = __reduce_or_sync(0xffffffffu, starts ? 1u << (excl - base) : 0u);
        __syncwarp();
        const uint32_t upto = smask & (0xffffffffu >> (31 - lane)); // start offsets 0..lane
        const int src = upto ? (int)own[31 - __clz(upto)] : carry;
        carry = __shfl_sync(0xffffffffu, src, 31);
        __syncwarp(); // the table is rewritten in the next window
        const uint32_t m = k - __shfl_sync(0xffffffffu, excl, src);
        const uint32_t meta = __shfl_sync(0xffffffffu, b.meta, src), xy = __shfl_sync(0xffffffffu, b.xy, src);
        const int U = __shfl_sync(0xffffffffu, b.U, src), V = __shfl_sync(0xffffffffu, b.V, src);
        const uint32_t S = __shfl_sync(0xffffffffu, b.S, src), Wh = __shfl_sync(0xffffffffu, b.Wh, src);
        const uint32_t t = TAGGED ? __shfl_sync(0xffffffffu, tag, src) : 0u;
        if (k < total) {
            const uint32_t bw = (meta >> 9) & 15u;
            const uint32_t row = (m * (meta & 0x1FFu)) >> 8, col = m - row * bw;
            const int x = (int)(xy & 0xFFFFu) + (int)col, y = (int)(xy >> 16) + (int)row;
            uint32_t idx;
            if (!(meta & (1u << 13))) {
                const int dx = x * 256 + 128 - U, dy = y * 256 + 128 - V;
                idx = __umulhi((uint32_t)(dx * dx) + (uint32_t)(dy * dy), S) >> 5;
            } else {
                const long long dx = (long long)x * 256 + 128 - U, dy = (long long)y * 256 + 128 - V;
                const unsigned long long i64 = ((unsigned long long)(dx * dx + dy * dy) * S) >> 37;
                idx = i64 < 1024ull ? (uint32_t)i64 : 1024u;
            }
            if (idx < 1024u) {
                const uint32_t kv = (uint32_t)tab(meta, idx);
                const unsigned long long c = (unsigned long long)Wh * kv + (((meta >> 16) * kv) >> 16);
                if (c) add(t, x, y, c);
                ++hits;
            }
        }
    }
    return hits;
}

// The per-pixel rule over boxes of at most 8 x 8 pixels, four points at a time: a group of eight lanes
// takes one point of the warp's (on: this lane has one), a column per lane, row by row.  A round of 32
// (point, pixel) pairs is about 14 instructions, where walk_boxes spends some 66 more on finding each
// pair's point and shuffling its operands; columns and rows a box does not have idle.  With LANES 4, eight
// points of boxes of up to four columns at a time (a 512 x 512 frame's scatter 32 -> 26 us).  Distances in 32
// bits and Wq < 2^32 (group_box decides; walk_boxes takes the rest).  K has a zero entry 1024.  at(t, x, y) gives,
// for a box's column x from row y (t: the point's tag if TAGGED, else 0), the function (j, c) that receives every
// nonzero contribution c < 2^32 to row y + j.  Returns this lane's pixel updates.  Every lane of the warp calls
// it.  LOD scatter of 16.8M particles 0.59 -> 0.43 ms; with a box per lane (BoxQueues) 0.51: a row of a
// group is one transaction of the global additions.
__device__ __forceinline__ bool group_box(int r, float Wf) { return r <= R_NARROW && Wf < 0x1p32f; }

template <int LANES, bool TAGGED, class At>
__device__ __forceinline__ unsigned group_boxes(bool on, int U, int V, uint32_t S, float Wf, int x0, int x1, int y0,
                                                int y1, const int32_t *K, At at, uint32_t tag = 0u)
{
    static_assert(DIRECT_BOX <= 8 && (LANES == 4 || LANES == 8), "a group's lanes are the columns of a box");
    const uint32_t m = __ballot_sync(0xffffffffu, on);
    if (!m) return 0u;
    const int lane = threadIdx.x & 31, col = lane & (LANES - 1);
    __shared__ uint8_t nth[32][32]; // lanes that have a point, in order
    uint8_t *own = nth[threadIdx.x >> 5];
    __syncwarp();
    if (on) own[__popc(m & gbd::lanemask_lt())] = (uint8_t)lane;
    __syncwarp();
    const uint32_t Wq = on ? __float2uint_rn(Wf) : 0u, xy = (uint32_t)x0 | (uint32_t)y0 << 16;
    const uint32_t ext = (uint32_t)(x1 - x0) | (uint32_t)(y1 - y0) << 8;
    const int n = __popc(m);
    unsigned hits = 0;
    for (int r = 0; r < n; r += 32 / LANES) {
        const int k = r + lane / LANES;
        const int src = own[min(k, n - 1)];
        const uint32_t qxy = __shfl_sync(0xffffffffu, xy, src), qext = __shfl_sync(0xffffffffu, ext, src);
        const int qU = __shfl_sync(0xffffffffu, U, src), qV = __shfl_sync(0xffffffffu, V, src);
        const uint32_t qS = __shfl_sync(0xffffffffu, S, src), qW = __shfl_sync(0xffffffffu, Wq, src);
        const uint32_t t = TAGGED ? __shfl_sync(0xffffffffu, tag, src) : 0u;
        const uint32_t Wh = qW >> 16, Wl = qW & 0xFFFFu;
        const auto add = at(t, (int)(qxy & 0xFFFFu) + col, (int)(qxy >> 16));
        const bool act = k < n && col <= (int)(qext & 0xFFu);
        const int rows = act ? (int)(qext >> 8) + 1 : 0;
        const int dx = ((int)(qxy & 0xFFFFu) + col) * 256 + 128 - qU;
        const uint32_t dx2 = (uint32_t)(dx * dx);
        const int dy = (int)(qxy >> 16) * 256 + 128 - qV;
        const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)rows);
        for (int j0 = 0; j0 < most; j0 += 4) { // four rows' lookups in flight, no branch but the additions
            uint32_t c[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int d = dy + (j0 + j) * 256;
                const uint32_t idx = j0 + j < rows ? min(__umulhi(dx2 + (uint32_t)(d * d), qS) >> 5, 1024u) : 1024u;
                const uint32_t kv = (uint32_t)K[idx];
                c[j] = Wh * kv + ((Wl * kv) >> 16);
                hits += idx < 1024u ? 1u : 0u;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (c[j]) add(j0 + j, c[j]);
        }
    }
    return hits;
}

// A warp's queues of small boxes, by size (4, 6 and 8 pixels on a side): a box waits until 32 of its size have
// come, and those are taken one per lane (lane_boxes) -- no operand is shuffled, every lane has a point,
// and the 32 points' table reads and additions go out together.  k_splat_small, 150M particles, the whole box
// in view: 6.6 ms with the smallest boxes one per lane as they came and the rest in groups of eight lanes, 4.7 so
// (sizes 3, 5, 8: 4.7; 4, 5, 8: 4.8; 5, 6, 8: 4.9); bound by the arithmetic of the padded boxes.
constexpr int QUEUES = 3;
struct BoxQueues {
    uint4 rec[QUEUES][64]; // U, V, S, amplitude
    uint2 box[QUEUES][64]; // x0 | y0 << 16, width | height << 8
};

template <int N, bool COUNT, class At>
__device__ __forceinline__ unsigned lane_boxes(bool on, const uint4 R, const uint2 B, const int32_t *K, At at)
{
    const int bw = on ? (int)(B.y & 0xFFu) : 0, bh = on ? (int)(B.y >> 8) : 0;
    const int x0 = (int)(B.x & 0xFFFFu), y0 = (int)(B.x >> 16);
    const int mh = (int)__reduce_max_sync(0xffffffffu, (unsigned)bh);
    const uint32_t Wq = on ? __float2uint_rn(__uint_as_float(R.w)) : 0u, Wh = Wq >> 16, Wl = Wq & 0xFFFFu;
    const auto add = at(x0, y0);
    uint32_t dx2[N];
#pragma unroll
    for (int c = 0; c < N; ++c) {
        const int dx = (x0 + c) * 256 + 128 - (int)R.x;
        dx2[c] = (uint32_t)(dx * dx);
    }
    unsigned hits = 0;
    for (int j = 0; j < mh; ++j) {
        const int dy = (y0 + j) * 256 + 128 - (int)R.y;
        const uint32_t dy2 = (uint32_t)(dy * dy);
        const int w = j < bh ? bw : 0;
        uint32_t v[N];
#pragma unroll
        for (int c = 0; c < N; ++c) {
            const uint32_t idx = min(__umulhi(dx2[c] + dy2, R.z) >> 5, 1024u);
            const uint32_t kv = (uint32_t)K[idx];
            v[c] = Wh * kv + ((Wl * kv) >> 16);
            if (COUNT) hits += c < w && idx < 1024u ? 1u : 0u;
        }
#pragma unroll
        for (int c = 0; c < N; ++c)
            if (c < w) add(c, j, v[c]);
    }
    return hits;
}

// Takes queue q's last boxes, 32 of them or (fewer) all n
template <bool COUNT, class At>
__device__ __forceinline__ unsigned take_boxes(const BoxQueues &Q, int q, int n, const int32_t *K, At at)
{
    const int lane = threadIdx.x & 31, first = max(n - 32, 0);
    const bool on = first + lane < n;
    const uint4 R = on ? Q.rec[q][first + lane] : make_uint4(0u, 0u, 0u, 0u);
    const uint2 B = on ? Q.box[q][first + lane] : make_uint2(0u, 0u);
    switch (q) {
    case 0: return lane_boxes<4, COUNT>(on, R, B, K, at);
    case 1: return lane_boxes<6, COUNT>(on, R, B, K, at);
    default: return lane_boxes<8, COUNT>(on, R, B, K, at);
    }
}

// Adds the lanes' boxes to the queues (on: this lane has one; n: boxes in each queue, the same in all lanes),
// takes what has become full.  Every lane of the warp calls it.
template <bool COUNT, class At>
__device__ __forceinline__ unsigned queue_boxes(BoxQueues &Q, int (&n)[QUEUES], bool on, const uint4 R, int x0, int x1,
                                                int y0, int y1, const int32_t *K, At at)
{
    const int side = on ? max(x1 - x0, y1 - y0) + 1 : 0;
    const int mine = on ? (side <= 4 ? 0 : (side <= 6 ? 1 : 2)) : -1;
    unsigned hits = 0;
#pragma unroll
    for (int q = 0; q < QUEUES; ++q) {
        const uint32_t m = __ballot_sync(0xffffffffu, mine == q);
        if (!m) continue;
        if (mine == q) {
            const int to = n[q] + __popc(m & gbd::lanemask_lt());
            Q.rec[q][to] = R;
            Q.box[q][to] = make_uint2((uint32_t)x0 | (uint32_t)y0 << 16, (uint32_t)(x1 - x0 + 1) | (uint32_t)(y1 - y0 + 1) << 8);
        }
        n[q] += __popc(m);
        __syncwarp();
        if (n[q] >= 32) {
            hits += take_boxes<COUNT>(Q, q, n[q], K, at);
            n[q] -= 32;
            __syncwarp();
        }
    }
    return hits;
}

// Adds a warp's pixel updates to the frame counters (every lane of the warp calls it)
__device__ __forceinline__ void count_hits(unsigned hits, FrameStatsDev *stats)
{
    unsigned long long h64 = hits;
    for (int d = 16; d > 0; d >>= 1) h64 += __shfl_xor_sync(0xffffffffu, h64, d);
    if ((threadIdx.x & 31) == 0 && h64) {
        atomicAdd(&stats->pixel_updates, h64);
        atomicAdd(&stats->pixel_updates_total, h64);
    }
}

// ------------------------------------------------------------------ R1
struct Frustum {
    double n[5][3];
    double off[5];
    double E[3];
    double lo[3];
    double F, side, lam2, zn2, rk;
};

Frustum make_frustum(const gblod_camera &c, const gblod_render_params &rp, const gblod_octree *o)
{
    // host FP64, every product and sum rounded on its own (built with -ffp-contract=off)
    Frustum f;
    const double rk = rp.kernel == GBLOD_KERNEL_CUBIC ? 2.0 : 3.0;
    const double M = rk * rp.sigma_min_px + 2.0;
    const double F = c.f_px;
    const double cl = c.cx + M;
    const double cr = ((double)c.width + M) - c.cx;
    const double ct = c.cy + M;
    const double cb = ((double)c.height + M) - c.cy;
    for (int a = 0; a < 3; ++a) {
        f.n[0][a] = c.fwd[a];
        double t1, t2;
        t1 = F * c.right[a]; t2 = cl * c.fwd[a]; f.n[1][a] = t1 + t2;
        t1 = -(F * c.right[a]); t2 = cr * c.fwd[a]; f.n[2][a] = t1 + t2;
        t1 = -(F * c.up[a]); t2 = ct * c.fwd[a]; f.n[3][a] = t1 + t2;
        t1 = F * c.up[a]; t2 = cb * c.fwd[a]; f.n[4][a] = t1 + t2;
        f.E[a] = c.eye[a];
        f.lo[a] = o->lo[a];
    }
    f.off[0] = -c.z_near;
    f.off[1] = f.off[2] = f.off[3] = f.off[4] = 0.0;
    f.F = F;
    f.side = o->side;
    const double lam = rp.lambda_px < 0.0 ? std::sqrt((double)o->n_max) : rp.lambda_px;
    f.lam2 = lam * lam;
    f.zn2 = c.z_near * c.z_near;
    f.rk = rk;
    return f;
}

// How many of a tree's nodes a view can reach, and the depths they have (nodes are numbered by depth, so they are the
// first ones): where not even a node at the root cube's distance from the eye is refined, nothing deeper is reached.
// With 1e-9 to spare on either side, far above what the rule rounds off.  (A view from far away, of a tree of
// 300,000 nodes: the frame 0.22 ms with all of them classified, 0.18 level by level, now 0.11.)
uint64_t reached_nodes(const gblod_octree *o, const Frustum &f, int &levels)
{
    levels = o->depth_max + 1;
    if (o->n_nodes == 0) return 0;
    double d2 = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double out = std::max(f.lo[a] - f.E[a], f.E[a] - (f.lo[a] + f.side));
        const double da = std::max(0.0, out - 1e-9 * (std::fabs(f.E[a]) + std::fabs(f.lo[a]) + f.side));
        d2 += da * da;
    }
    const double rhs = f.lam2 * std::max(d2, f.zn2) * (1.0 - 1e-9);
    for (int d = 0; d < levels; ++d) {
        const double fe = f.F * std::ldexp(f.side, -d);
        if (!(fe * fe > rhs)) levels = d + 1;
    }
    return o->level_first[levels];
}

// 0 cull, 1 emit, 2 refine
__device__ __forceinline__ int classify(const gblod_node &g, const Frustum &fr)
{
    const double rho = __dmul_rn(fr.rk, (double)g.h_cull);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        double s = fr.off[k];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double na = fr.n[k][a];
            const double pa = na > 0.0 ? __dsub_rn(__dadd_rn((double)g.bmax[a], rho), fr.E[a])
                                       : __dsub_rn(__dsub_rn((double)g.bmin[a], rho), fr.E[a]);
            s = __dadd_rn(s, __dmul_rn(na, pa));
        }
        if (s < 0.0) return 0;
    }
    if (!(g.flags & GBLOD_NODE_INTERNAL)) return 1;
    const int d = g.depth;
    const uint64_t pfx = g.code ^ (1ull << (3 * d));
    const uint32_t q[3] = {gbd::compact3(pfx >> 2), gbd::compact3(pfx >> 1), gbd::compact3(pfx)};
    const double e = ldexp(fr.side, -d);
    double d2 = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double blo = __dadd_rn(fr.lo[a], __dmul_rn(e, (double)q[a]));
        const double bhi = __dadd_rn(blo, e);
        const double E = fr.E[a];
        const double da = E < blo ? __dsub_rn(blo, E) : (E > bhi ? __dsub_rn(E, bhi) : 0.0);
        d2 = __dadd_rn(d2, __dmul_rn(da, da));
    }
    const double fe = __dmul_rn(fr.F, e);
    const double lhs = __dmul_rn(fe, fe);
    const double rhs = __dmul_rn(fr.lam2, d2 > fr.zn2 ? d2 : fr.zn2);
    return lhs > rhs ? 2 : 1;
}

// A node is drawn if the rule emits it and refines all its ancestors.  Up to SELECT_FLAT reached nodes: classify
// every node and look at the ancestors' classes, in two launches (up to SELECT_ONE nodes: in one block that
// also does k_sel_prefix's work); larger trees are walked level by level, which reads only the nodes that are
// reached.  A level costs a launch of 5 to 6 us whatever its size: 64 nodes, 4 levels 29 us with first and
// prefix launch, now 8 us; 1M particles, 11 levels 63 us, now 12 us.  What bounds the flat form is the FP64
// of the rule, some 80 operations a node at two a clock and SM: 2^19 nodes take as long as ten levels.
constexpr uint64_t SELECT_ONE = 256, SELECT_FLAT = 1u << 19;

__global__ void __launch_bounds__(128) k_classify(const gblod_node *__restrict__ nodes, uint32_t nn, Frustum fr,
                                                  uint8_t *__restrict__ cls)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nn) cls[i] = (uint8_t)classify(nodes[i], fr);
}

// appends the warp's nodes with `take` set to sel
template <class T> __device__ __forceinline__ void append_nodes(bool take, T node, T *__restrict__ sel, uint32_t *nsel)
{
    const uint32_t em = __ballot_sync(0xffffffffu, take);
    if (!em) return;
    const int leader = __ffs(em) - 1;
    uint32_t b = 0;
    if ((int)(threadIdx.x & 31) == leader) b = atomicAdd(nsel, (uint32_t)__popc(em));
    b = __shfl_sync(0xffffffffu, b, leader);
    if (take) sel[b + __popc(em & gbd::lanemask_lt())] = node;
}

// Emitted nodes are kept only if they belong to this part of a split frame (node index mod n_parts ==
// part; n_parts = 1 keeps every one).
__global__ void __launch_bounds__(RT) k_select_flat(const gblod_node *__restrict__ nodes, uint32_t nn,
                                                    const uint8_t *__restrict__ cls, uint32_t *__restrict__ sel,
                                                    uint32_t *nsel, uint32_t part, uint32_t n_parts)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    bool take = i < nn && cls[i] == 1 && (n_parts <= 1 || i % n_parts == part);
    if (take)
        for (int p = nodes[i].parent; p >= 0 && take; p = nodes[p].parent) take = cls[p] == 2;
    append_nodes(take, i, sel, nsel);
}

__global__ void k_select_init(uint32_t *front, uint32_t *cnt)
{
    front[0] = 0u;
    cnt[0] = 1u;
}

// One level of the walk.  Emitted nodes are kept only if they belong to this part of a split frame
// (node index mod n_parts == part; n_parts = 1 keeps every one); refined nodes are walked either way.
__global__ void __launch_bounds__(RT) k_select_level(const gblod_node *__restrict__ nodes, Frustum fr,
                                                     const uint32_t *__restrict__ fin, const uint32_t *nin,
                                                     uint32_t *__restrict__ fout, uint32_t *nout,
                                                     uint32_t *__restrict__ sel, uint32_t *nsel, uint32_t part,
                                                     uint32_t n_parts)
{
    const uint32_t n = *nin;
    const int lane = threadIdx.x & 31;
    for (uint32_t base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {
        const uint32_t i = base + threadIdx.x;
        int cls = 0;
        uint32_t node = 0, ccount = 0, cfirst = 0;
        if (i < n) {
            node = fin[i];
            const gblod_node g = nodes[node];
            cls = classify(g, fr);
            ccount = g.child_count;
            cfirst = g.child_first;
            if (cls == 1 && n_parts > 1 && node % n_parts != part) cls = 0;
        }
        append_nodes(cls == 1, node, sel, nsel);
        uint32_t want = cls == 2 ? ccount : 0u, incl = want;
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        if (total) {
            uint32_t b = 0;
            if (lane == 31) b = atomicAdd(nout, total);
            b = __shfl_sync(0xffffffffu, b, 31);
            const uint32_t at = b + incl - want;
            for (uint32_t k = 0; k < want; ++k) fout[at + k] = cfirst + k;
        }
    }
}

// exclusive prefix of the selected nodes' point counts; base[j] maps a flat index to a point
__global__ void __launch_bounds__(1024) k_sel_prefix(const gblod_node *__restrict__ nodes,
                                                     const uint32_t *__restrict__ sel, const uint32_t *nsel,
                                                     uint64_t *__restrict__ pfx, int64_t *__restrict__ base,
                                                     FrameStatsDev *stats)
{
    __shared__ unsigned long long wsum[32];
    const uint32_t n = *nsel;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long run = 0;
    for (uint32_t start = 0; start < n; start += 1024) {
        const uint32_t i = start + threadIdx.x;
        unsigned long long c = 0, pf = 0;
        if (i < n) {
            const gblod_node &g = nodes[sel[i]];
            c = g.point_count;
            pf = g.point_first;
        }
        unsigned long long incl = c;
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        unsigned long long before = 0, all = 0;
        for (int w = 0; w < 32; ++w) {
            before += w < warp ? wsum[w] : 0ull;
            all += wsum[w];
        }
        const unsigned long long ex = run + before + incl - c;
        if (i < n) {
            pfx[i] = ex;
            base[i] = (int64_t)pf - (int64_t)ex;
        }
        run += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        pfx[n] = run;
        stats->points = run;
        stats->nodes_selected = n;
    }
}

// R1 of a tree of at most SELECT_ONE nodes: a node per thread, classes and parents in shared memory
__global__ void __launch_bounds__(SELECT_ONE) k_select_one(const gblod_node *__restrict__ nodes, uint32_t nn, Frustum fr,
                                                           uint32_t part, uint32_t n_parts, uint32_t *__restrict__ sel,
                                                           uint32_t *nsel, uint64_t *__restrict__ pfx,
                                                           int64_t *__restrict__ base, FrameStatsDev *stats)
{
    __shared__ uint8_t cls[SELECT_ONE];
    __shared__ int16_t parent[SELECT_ONE];
    __shared__ unsigned long long points[SELECT_ONE / 32];
    __shared__ uint32_t taken[SELECT_ONE / 32];
    const uint32_t i = threadIdx.x;
    const int lane = i & 31, warp = i >> 5;
    unsigned long long c = 0, pf = 0;
    if (i < nn) {
        const gblod_node g = nodes[i];
        parent[i] = (int16_t)g.parent;
        cls[i] = (uint8_t)classify(g, fr);
        c = g.point_count;
        pf = g.point_first;
    }
    __syncthreads();
    bool take = i < nn && cls[i] == 1 && (n_parts <= 1 || i % n_parts == part);
    if (take)
        for (int p = parent[i]; p >= 0 && take; p = parent[p]) take = cls[p] == 2;
    const uint32_t em = __ballot_sync(0xffffffffu, take);
    if (!take) c = 0;
    unsigned long long incl = c;
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) {
        points[warp] = incl;
        taken[warp] = (uint32_t)__popc(em);
    }
    __syncthreads();
    unsigned long long ex = incl - c, all = 0;
    uint32_t at = (uint32_t)__popc(em & gbd::lanemask_lt()), n = 0;
    for (int w = 0; w < (int)(SELECT_ONE / 32); ++w) {
        ex += w < warp ? points[w] : 0ull;
        at += w < warp ? taken[w] : 0u;
        all += points[w];
        n += taken[w];
    }
    if (take) {
        sel[at] = i;
        pfx[at] = ex;
        base[at] = (int64_t)pf - (int64_t)ex;
    }
    if (i == 0) {
        *nsel = n;
        pfx[n] = all;
        stats->points = all;
        stats->nodes_selected = n;
    }
}

// The largest j < n with pfx[j] <= v (pfx[0] = 0), by a whole warp: 33 parts a step, where one thread's
// bisection waits for log2(n) reads one after another (at the head of every chunk of points).
__device__ __forceinline__ uint32_t warp_find(const uint64_t *__restrict__ pfx, uint32_t n, unsigned long long v)
{
    const uint32_t lane = threadIdx.x & 31;
    uint32_t lo = 0, hi = n; // pfx[lo] <= v, and pfx[hi] > v or hi = n
    while (hi - lo > 1) {
        const uint32_t step = (hi - lo + 32) / 33, at = lo + step * (lane + 1);
        const uint32_t m = __ballot_sync(0xffffffffu, at < hi && pfx[at] <= v);
        const uint32_t k = (uint32_t)__popc(m); // the lanes below the first that is past v
        hi = min(hi, lo + step * (k + 1));
        lo += step * k;
    }
    return lo;
}

// ------------------------------------------------------------------ R2
struct SrcLOD {
    const float4 *pts4;
    const float *hs;
    const uint64_t *pfx;  // n_sel + 1 entries
    const int64_t *base;
    const uint32_t *nsel;
    const unsigned long long *total;
    unsigned long long bound; // host: at least the number of points
};

// selected nodes' 16-bit block codes (decoded on load)
struct SrcLODQ : SrcLOD {
    const ushort4 *q4;
    const uint16_t *qw;
    const float4 *qa;
    const uint32_t *sel; // node index per selected entry
};

struct SrcFlat {
    const float *xyz, *mass, *h;
    unsigned long long n, bound;
};

__device__ __forceinline__ unsigned long long src_total(const SrcLOD &s) { return *s.total; }
__device__ __forceinline__ unsigned long long src_total(const SrcFlat &s) { return s.n; }

// per block iteration: locate the selected nodes covering [a, b)
__device__ __forceinline__ void src_range(const SrcLOD &s, unsigned long long a, unsigned long long b, uint32_t &j0,
                                          uint32_t &j1)
{
    __shared__ uint32_t sj[2];
    if (threadIdx.x < 64) {
        const uint32_t j = warp_find(s.pfx, *s.nsel, threadIdx.x < 32 ? a : b - 1);
        if ((threadIdx.x & 31) == 0) sj[threadIdx.x >> 5] = j;
    }
    __syncthreads();
    j0 = sj[0];
    j1 = sj[1];
    __syncthreads();
}
__device__ __forceinline__ void src_range(const SrcFlat &, unsigned long long, unsigned long long, uint32_t &j0,
                                          uint32_t &j1)
{
    j0 = j1 = 0;
}

__device__ __forceinline__ void src_load(const SrcLOD &s, unsigned long long e, uint32_t j0, uint32_t j1, float &x,
                                         float &y, float &z, float &w, float &h)
{
    uint32_t lo = j0, hi = j1 + 1;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (s.pfx[mid] <= e)
            lo = mid;
        else
            hi = mid;
    }
    const unsigned long long p = (unsigned long long)((long long)e + s.base[lo]);
    const float4 q = s.pts4[p];
    x = q.x; y = q.y; z = q.z; w = q.w;
    h = s.hs[p];
}
__device__ __forceinline__ void src_load(const SrcLODQ &s, unsigned long long e, uint32_t j0, uint32_t j1, float &x,
                                         float &y, float &z, float &w, float &h)
{
    uint32_t lo = j0, hi = j1 + 1;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (s.pfx[mid] <= e)
            lo = mid;
        else
            hi = mid;
    }
    const unsigned long long p = (unsigned long long)((long long)e + s.base[lo]);
    const uint32_t node = s.sel[lo];
    block_decode(s.q4[p], s.qw[p], s.qa[2 * node], s.qa[2 * node + 1], x, y, z, w, h);
}
__device__ __forceinline__ void src_load(const SrcFlat &s, unsigned long long e, uint32_t, uint32_t, float &x,
                                         float &y, float &z, float &w, float &h)
{
    x = s.xyz[3 * e];
    y = s.xyz[3 * e + 1];
    z = s.xyz[3 * e + 2];
    w = s.mass[e];
    h = s.h[e];
}

// Sum of drawn amplitudes as 128 bits per thread; one atomic pair per warp at the end (the sum
// must stay below 2^64, reading R-19)
struct AmpSum {
    unsigned long long lo = 0, hi = 0;
    __device__ __forceinline__ void add(unsigned long long v)
    {
        lo += v;
        hi += lo < v ? 1ull : 0ull;
    }
    __device__ __forceinline__ void flush(FrameStatsDev *stats)
    {
        for (int d = 16; d > 0; d >>= 1) {
            const unsigned long long ol = __shfl_xor_sync(0xffffffffu, lo, d), oh = __shfl_xor_sync(0xffffffffu, hi, d);
            lo += ol;
            hi += oh + (lo < ol ? 1ull : 0ull);
        }
        if ((threadIdx.x & 31) == 0 && (lo | hi)) {
            const unsigned long long old = lo ? atomicAdd(&stats->amp_lo, lo) : 0ull;
            const unsigned long long carry = lo && old + lo < old ? 1ull : 0ull;
            if (hi + carry) atomicAdd(&stats->amp_hi, hi + carry);
        }
    }
};

// Warp-cooperative scatter of (splat, tile) records.  Lane l contributes n_l pairs: the tiles
// t00_l + row * tiles_x_l + col of its box, row < n_l / tw_l, col < tw_l (n_l = 0: none).  The warp
// walks the concatenation of all lanes' pairs 32 at a time, so one lane with many tiles does not
// hold the others idle; pairs of one round that share a tile reserve their slots from cursor[t]
// with one atomic (match_any) and write the source lane's record r (slots at or past rec_cap are
// dropped).
__device__ __forceinline__ void scatter_pairs(uint32_t n, uint32_t t00, int tw, int tiles_x, const uint4 r,
                                              uint32_t *__restrict__ cursor, uint4 *__restrict__ rec,
                                              unsigned long long rec_cap)
{
    const int lane = threadIdx.x & 31;
    const uint32_t lt = gbd::lanemask_lt();
    uint32_t incl = n;
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t excl = incl - n;
    for (uint32_t base = 0; base < total; base += 32) {
        const uint32_t k = base + (uint32_t)lane;
        int src = 0; // the last lane whose pairs start at or before k
        for (int step = 16; step > 0; step >>= 1) {
            const uint32_t ex = __shfl_sync(0xffffffffu, excl, src + step);
            if (ex <= k) src += step;
        }
        const uint32_t m = k - __shfl_sync(0xffffffffu, excl, src);
        const uint32_t st00 = __shfl_sync(0xffffffffu, t00, src);
        const int stw = __shfl_sync(0xffffffffu, tw, src), stx = __shfl_sync(0xffffffffu, tiles_x, src);
        uint4 sr;
        sr.x = __shfl_sync(0xffffffffu, r.x, src);
        sr.y = __shfl_sync(0xffffffffu, r.y, src);
        sr.z = __shfl_sync(0xffffffffu, r.z, src);
        sr.w = __shfl_sync(0xffffffffu, r.w, src);
        const bool act = k < total;
        const uint32_t amask = __ballot_sync(0xffffffffu, act);
        if (act) {
            const uint32_t row = m / (uint32_t)stw, col = m - row * (uint32_t)stw;
            const uint32_t t = st00 + row * (uint32_t)stx + col;
            const uint32_t peers = __match_any_sync(amask, t);
            const int leader = __ffs(peers) - 1;
            uint32_t b = 0;
            if (lane == leader) b = atomicAdd(&cursor[t], (uint32_t)__popc(peers));
            b = __shfl_sync(peers, b, leader);
            const unsigned long long pos = (unsigned long long)b + __popc(peers & lt);
            if (pos < rec_cap) rec[pos] = sr;
        }
    }
}

template <class Src>
__global__ void __launch_bounds__(RT, 4) k_project_count(Src src, Proj P, unsigned long long e_lo,
                                                      unsigned long long e_hi, uint32_t *__restrict__ tile_cnt,
                                                      unsigned *status, FrameStatsDev *stats)
{
    const unsigned long long total = min(src_total(src), e_hi);
    const int lane = threadIdx.x & 31;
    unsigned long long splats = 0, pairs = 0;
    AmpSum amp;
    for (unsigned long long a = e_lo + (unsigned long long)blockIdx.x * CHUNK; a < total;
         a += (unsigned long long)gridDim.x * CHUNK) {
        const unsigned long long b = min(total, a + CHUNK);
        uint32_t j0, j1;
        src_range(src, a, b, j0, j1);
        for (unsigned long long e0 = a; e0 < b; e0 += RT) {
            const unsigned long long e = e0 + threadIdx.x;
            int res = 0;
            Splat s;
            if (e < b) {
                float x, y, z, w, h;
                src_load(src, e, j0, j1, x, y, z, w, h);
                res = project(P, x, y, z, w, h, s);
            }
            if (__any_sync(0xffffffffu, res < 0) && lane == 0) atomicOr(status, ST_RANGE);
            if (res == 1) {
                amp.add(__float2ull_rn(s.Wf));
                ++splats;
                int x0, x1, y0, y1;
                splat_box(s.U, s.V, s.S, P.W, P.H, x0, x1, y0, y1);
                if (x0 <= x1 && y0 <= y1 && !direct_box(x0, x1, y0, y1)) {
                    const int tx0 = x0 / P.TW, tx1 = x1 / P.TW, ty0 = y0 / P.TH, ty1 = y1 / P.TH;
                    pairs += (unsigned long long)(tx1 - tx0 + 1) * (unsigned long long)(ty1 - ty0 + 1);
                    for (int ty = ty0; ty <= ty1; ++ty)
                        for (int tx = tx0; tx <= tx1; ++tx) {
                            const uint32_t t = (uint32_t)(ty * P.tiles_x + tx);
                            const uint32_t mask = __activemask();
                            const uint32_t peers = __match_any_sync(mask, t);
                            const int leader = __ffs(peers) - 1;
                            if (lane == leader) atomicAdd(&tile_cnt[t], (uint32_t)__popc(peers));
                        }
                }
            }
        }
    }
    for (int d = 16; d > 0; d >>= 1) {
        splats += __shfl_xor_sync(0xffffffffu, splats, d);
        pairs += __shfl_xor_sync(0xffffffffu, pairs, d);
    }
    if (lane == 0 && splats) atomicAdd(&stats->splats, splats);
    if (lane == 0 && pairs) atomicAdd(&stats->pairs, pairs);
    amp.flush(stats);
}

// Writes the (tile, point) records of the binned points and splats the points with small boxes
// into img; cstats (null: not counted) receives the pixel updates of the latter.
template <class Src>
__global__ void __launch_bounds__(RT, 4) k_project_scatter(Src src, Proj P, unsigned long long e_lo,
                                                           unsigned long long e_hi, uint32_t *__restrict__ cursor,
                                                           uint4 *__restrict__ rec, unsigned long long *img,
                                                           FrameStatsDev *cstats)
{
    const unsigned long long total = min(src_total(src), e_hi);
    const int32_t *K = g_ktab[P.kernel];
    unsigned hits = 0;
    for (unsigned long long a = e_lo + (unsigned long long)blockIdx.x * CHUNK; a < total;
         a += (unsigned long long)gridDim.x * CHUNK) {
        const unsigned long long b = min(total, a + CHUNK);
        uint32_t j0, j1;
        src_range(src, a, b, j0, j1);
        for (unsigned long long e0 = a; e0 < b; e0 += RT) {
            const unsigned long long e = e0 + threadIdx.x;
            int res = 0;
            Splat s;
            if (e < b) {
                float x, y, z, w, h;
                src_load(src, e, j0, j1, x, y, z, w, h);
                res = project(P, x, y, z, w, h, s);
            }
            uint32_t n = 0, t00 = 0;
            int tw = 1;
            uint4 r = make_uint4(0u, 0u, 0u, 0u);
            BoxWalk direct;
            if (res == 1) {
                int x0, x1, y0, y1;
                const int rad = splat_box(s.U, s.V, s.S, P.W, P.H, x0, x1, y0, y1);
                if (x0 <= x1 && y0 <= y1) {
                    if (direct_box(x0, x1, y0, y1)) {
                        direct = box_walk(s.U, s.V, s.S, __float2ull_rn(s.Wf), rad, x0, x1, y0, y1);
                    } else {
                        r = make_uint4((uint32_t)s.U, (uint32_t)s.V, s.S, __float_as_uint(s.Wf));
                        const int tx0 = x0 / P.TW, tx1 = x1 / P.TW, ty0 = y0 / P.TH, ty1 = y1 / P.TH;
                        tw = tx1 - tx0 + 1;
                        n = (uint32_t)(tw * (ty1 - ty0 + 1));
                        t00 = (uint32_t)(ty0 * P.tiles_x + tx0);
                    }
                }
            }
            scatter_pairs(n, t00, tw, P.tiles_x, r, cursor, rec, ~0ull);
            hits += walk_boxes<false>(
                direct, 0u, [&](uint32_t, uint32_t i) { return K[i]; },
                [&](uint32_t, int x, int y, unsigned long long c) { atomicAdd(&img[(size_t)y * P.W + x], c); });
        }
    }
    if (cstats) count_hits(hits, cstats);
}

// Partitioned binning.  Each CTA of the grid counts its own points per tile in shared memory and writes
// one histogram, tile-major: hist[t * G + cta].  An exclusive scan of the histograms gives every CTA
// its own base in every tile, so the scatter pass places records with shared-memory atomics only.  The CTAs
// may be split in groups of gs, each with its own tile-major histogram and so its own region of the
// records, where a tile has one run per group (see binning).  Both passes walk the same chunks (the same
// grid G and chunk stride), so they see the same points.  (Global counters need the pairs of a warp
// grouped by tile: __match_any_sync loops over the distinct tiles, up to 260 cycles a round.  LOD frames,
// count + scatter: 16.8M particles 1080p 2.07 ms with it, 0.58 ms so; 150M near view 5.4, 2.1 ms.)
//
// Points whose pixel box is at most DIRECT_BOX on a side: of an octree's nodes (SMALL false), the scatter
// pass adds their contributions straight to the image (neighbours in the order are neighbours in
// space); of a caller's arrays in no spatial order (SMALL true) they are binned too, into a second
// record stream (their own histograms, after the binned points' in the same scan), and splatted by
// k_splat_small into a shared-memory tile image: added straight to the image, every pixel would be a
// global atomic at a random address.
// One CTA of 1024 threads per SM for unordered points: every CTA writes into all tiles' records, and a
// quarter of the CTAs leaves a quarter of the half-written lines open in L2 (16.8M particles, scatter 1.00 ->
// 0.64 ms); an octree's points reach few tiles at a time, and four CTAs of 256 overlap better (0.59
// against 0.66).
template <bool SMALL> constexpr int PART_THREADS = SMALL ? 1024 : 256;
constexpr size_t PART_MAX_SMEM = 200 * 1024; // shared-memory histograms: frames of more tiles take the global counters
constexpr uint32_t ITEM_SMALL = 4096;        // small records per k_splat_small work item

// where CTA `cta` keeps tile t's count
__device__ __forceinline__ size_t hist_at(uint32_t t, uint32_t ntiles, uint32_t cta, uint32_t gs)
{
    return ((size_t)(cta / gs) * ntiles + t) * gs + cta % gs;
}

struct PointIn {
    float x, y, z, w, h;
};

template <class Src, bool SMALL>
__global__ void __launch_bounds__(PART_THREADS<SMALL>, 1024 / PART_THREADS<SMALL>) k_project_hist(Src src, Proj P, unsigned long long e_lo,
                                                     unsigned long long e_hi, uint32_t chunk, uint32_t gs,
                                                     uint32_t *__restrict__ hist, unsigned *status, FrameStatsDev *stats)
{
    constexpr int NT = PART_THREADS<SMALL>;
    extern __shared__ uint32_t sh_cnt[]; // [ntiles] binned points, then (SMALL) [ntiles] small boxes
    const uint32_t ntiles = (uint32_t)(P.tiles_x * P.tiles_y), ncnt = SMALL ? 2 * ntiles : ntiles;
    for (uint32_t t = threadIdx.x; t < ncnt; t += NT) sh_cnt[t] = 0u;
    __syncthreads();
    const unsigned long long total = min(src_total(src), e_hi);
    const int lane = threadIdx.x & 31;
    unsigned long long splats = 0, pairs = 0;
    AmpSum amp;
    PointIn ahead; // SMALL: the thread's next point, read before this one's arithmetic
    if constexpr (SMALL) {
        const unsigned long long e = e_lo + (unsigned long long)blockIdx.x * chunk + threadIdx.x;
        if (e < total) src_load(src, e, 0u, 0u, ahead.x, ahead.y, ahead.z, ahead.w, ahead.h);
    }
    for (unsigned long long a = e_lo + (unsigned long long)blockIdx.x * chunk; a < total;
         a += (unsigned long long)gridDim.x * chunk) {
        const unsigned long long b = min(total, a + chunk);
        uint32_t j0, j1;
        src_range(src, a, b, j0, j1);
        for (unsigned long long e0 = a; e0 < b; e0 += NT) {
            const unsigned long long e = e0 + threadIdx.x;
            int res = 0;
            Splat s;
            if constexpr (SMALL) {
                const PointIn q = ahead;
                const unsigned long long en = e0 + NT < b ? e + NT : a + (unsigned long long)gridDim.x * chunk + threadIdx.x;
                if (en < total) src_load(src, en, 0u, 0u, ahead.x, ahead.y, ahead.z, ahead.w, ahead.h);
                if (e < b) res = project(P, q.x, q.y, q.z, q.w, q.h, s);
            } else if (e < b) {
                float x, y, z, w, h;
                src_load(src, e, j0, j1, x, y, z, w, h);
                res = project(P, x, y, z, w, h, s);
            }
            if (__any_sync(0xffffffffu, res < 0) && lane == 0) atomicOr(status, ST_RANGE);
            if (res == 1) {
                amp.add(__float2ull_rn(s.Wf));
                ++splats;
                int x0, x1, y0, y1;
                splat_box(s.U, s.V, s.S, P.W, P.H, x0, x1, y0, y1);
                const bool small = direct_box(x0, x1, y0, y1);
                if (x0 <= x1 && y0 <= y1 && (SMALL || !small)) {
                    uint32_t *cnt = small ? sh_cnt + ntiles : sh_cnt;
                    const int tx0 = x0 / P.TW, tx1 = x1 / P.TW, ty0 = y0 / P.TH, ty1 = y1 / P.TH;
                    if (!small) pairs += (unsigned long long)(tx1 - tx0 + 1) * (unsigned long long)(ty1 - ty0 + 1);
                    for (int ty = ty0; ty <= ty1; ++ty)
                        for (int tx = tx0; tx <= tx1; ++tx) atomicAdd(&cnt[ty * P.tiles_x + tx], 1u);
                }
            }
        }
    }
    for (int d = 16; d > 0; d >>= 1) {
        splats += __shfl_xor_sync(0xffffffffu, splats, d);
        pairs += __shfl_xor_sync(0xffffffffu, pairs, d);
    }
    if (lane == 0 && splats) atomicAdd(&stats->splats, splats);
    if (lane == 0 && pairs) atomicAdd(&stats->pairs, pairs);
    amp.flush(stats);
    __syncthreads();
    unsigned long long smalls = 0;
    for (uint32_t t = threadIdx.x; t < ntiles; t += NT) {
        const size_t at = hist_at(t, ntiles, blockIdx.x, gs);
        hist[at] = sh_cnt[t];
        if (SMALL) {
            hist[(size_t)ntiles * gridDim.x + at] = sh_cnt[ntiles + t];
            smalls += sh_cnt[ntiles + t];
        }
    }
    if (SMALL) {
        for (int d = 16; d > 0; d >>= 1) smalls += __shfl_xor_sync(0xffffffffu, smalls, d);
        if (lane == 0 && smalls) atomicAdd(&stats->small_pairs, smalls);
    }
}

// Records per work item of `total` records: ITEM, less if that makes fewer than `want` items, so that a small
// frame's work spreads over the grid and ends together (a million particles, 640 x 360: 275 -> 125 us; 262k, 512 x
// 512: 46 -> 13 us, with 256 at least 25).
constexpr uint32_t ITEM_MIN = 64;
__host__ __device__ __forceinline__ uint32_t item_size(uint32_t total, uint32_t want)
{
    const uint32_t each = total / want + (total % want != 0u); // rounded up: no more than `want` full items
    const uint32_t per = each < ITEM ? (each + 31u) / 32u * 32u : ITEM;
    return per < ITEM_MIN ? ITEM_MIN : (per < ITEM ? per : ITEM);
}
// wanted items: four units a warp of the splat kernel's grid (a unit is a strip of up to eight)
uint32_t items_wanted() { return (uint32_t)persistent_blocks(4) * 4u; }

// counts, offsets and work items (of per_item records; 0: by item_size) of the tiles' runs from the scanned
// (tile, CTA) histogram of CTA groups of G
__global__ void k_tiles_from_hist(uint32_t ntiles, uint32_t G, uint32_t per_item, uint32_t want,
                                  const uint32_t *__restrict__ off, const uint32_t *total, uint32_t *tile_cnt, uint32_t *tile_off, uint32_t *item_cnt,
                                  unsigned long long *frame_tiles, uint32_t in_frame)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0 && frame_tiles) *frame_tiles = in_frame;
    if (t >= ntiles) return;
    const uint32_t a = off[(size_t)t * G], b = t + 1 < ntiles ? off[(size_t)(t + 1) * G] : *total;
    tile_off[t] = a;
    tile_cnt[t] = b - a;
    if (!per_item) per_item = item_size(*total, want);
    item_cnt[t] = (b - a + per_item - 1) / per_item;
}

// Writes the (tile, point) records of the binned points (SMALL: and of the small boxes) at this CTA's
// bases; without SMALL the points with small boxes are splatted into img (cstats, if not null,
// receives their pixel updates).
template <class Src, bool SMALL>
__global__ void __launch_bounds__(PART_THREADS<SMALL>, 1024 / PART_THREADS<SMALL>) k_project_scatter_part(Src src, Proj P, unsigned long long e_lo,
                                                             unsigned long long e_hi, uint32_t chunk, uint32_t gs,
                                                             const uint32_t *__restrict__ off,
                                                             uint4 *__restrict__ rec, unsigned long long *img,
                                                             FrameStatsDev *cstats)
{
    constexpr int NT = PART_THREADS<SMALL>;
    __shared__ int32_t K[SMALL ? 1 : 1025];
    extern __shared__ uint32_t sh_cur[]; // [ntiles] binned points, then (SMALL) [ntiles] small boxes
    const uint32_t ntiles = (uint32_t)(P.tiles_x * P.tiles_y);
    const unsigned long long total = min(src_total(src), e_hi);
    unsigned hits = 0;
    if (e_lo + (unsigned long long)blockIdx.x * chunk < total)
        for (uint32_t t = threadIdx.x; t < ntiles; t += NT) {
            const size_t at = hist_at(t, ntiles, blockIdx.x, gs);
            sh_cur[t] = off[at];
            if (SMALL) sh_cur[ntiles + t] = off[(size_t)ntiles * gridDim.x + at];
        }
    if (!SMALL)
        for (int t = threadIdx.x; t <= 1024; t += NT) K[t] = t < 1024 ? g_ktab[P.kernel][t] : 0;
    __syncthreads();
    PointIn ahead; // SMALL: the thread's next point, read before this one's arithmetic
    if constexpr (SMALL) {
        const unsigned long long e = e_lo + (unsigned long long)blockIdx.x * chunk + threadIdx.x;
        if (e < total) src_load(src, e, 0u, 0u, ahead.x, ahead.y, ahead.z, ahead.w, ahead.h);
    }
    for (unsigned long long a = e_lo + (unsigned long long)blockIdx.x * chunk; a < total;
         a += (unsigned long long)gridDim.x * chunk) {
        const unsigned long long b = min(total, a + chunk);
        uint32_t j0, j1;
        src_range(src, a, b, j0, j1);
        for (unsigned long long e0 = a; e0 < b; e0 += NT) {
            const unsigned long long e = e0 + threadIdx.x;
            int res = 0;
            Splat s;
            if constexpr (SMALL) {
                const PointIn q = ahead;
                const unsigned long long en = e0 + NT < b ? e + NT : a + (unsigned long long)gridDim.x * chunk + threadIdx.x;
                if (en < total) src_load(src, en, 0u, 0u, ahead.x, ahead.y, ahead.z, ahead.w, ahead.h);
                if (e < b) res = project(P, q.x, q.y, q.z, q.w, q.h, s);
            } else if (e < b) {
                float x, y, z, w, h;
                src_load(src, e, j0, j1, x, y, z, w, h);
                res = project(P, x, y, z, w, h, s);
            }
            BoxWalk direct;
            int x0 = 0, x1 = -1, y0 = 0, y1 = -1;
            bool mine = false;
            if (res == 1) {
                const int rad = splat_box(s.U, s.V, s.S, P.W, P.H, x0, x1, y0, y1);
                if (x0 <= x1 && y0 <= y1) {
                    const bool small = direct_box(x0, x1, y0, y1);
                    if (!SMALL && small) {
                        mine = group_box(rad, s.Wf);
                        if (!mine) direct = box_walk(s.U, s.V, s.S, __float2ull_rn(s.Wf), rad, x0, x1, y0, y1);
                    } else {
                        uint32_t *cur = small ? sh_cur + ntiles : sh_cur;
                        const uint4 r = make_uint4((uint32_t)s.U, (uint32_t)s.V, s.S, __float_as_uint(s.Wf));
                        const int tx0 = x0 / P.TW, tx1 = x1 / P.TW, ty0 = y0 / P.TH, ty1 = y1 / P.TH;
                        for (int ty = ty0; ty <= ty1; ++ty)
                            for (int tx = tx0; tx <= tx1; ++tx) rec[atomicAdd(&cur[ty * P.tiles_x + tx], 1u)] = r;
                    }
                }
            }
            if (!SMALL) {
                auto at = [&](uint32_t, int x, int y) {
                    unsigned long long *p = img + (size_t)y * P.W + x;
                    return [p, &P](int j, uint32_t c) { atomicAdd(&p[(size_t)j * P.W], (unsigned long long)c); };
                };
                const bool four = x1 - x0 < 4;
                hits += group_boxes<4, false>(mine && four, s.U, s.V, s.S, s.Wf, x0, x1, y0, y1, K, at);
                hits += group_boxes<8, false>(mine && !four, s.U, s.V, s.S, s.Wf, x0, x1, y0, y1, K, at);
                hits += walk_boxes<false>(
                    direct, 0u, [&](uint32_t, uint32_t i) { return K[i]; },
                    [&](uint32_t, int x, int y, unsigned long long c) { atomicAdd(&img[(size_t)y * P.W + x], c); });
            }
        }
    }
    if (!SMALL && cstats) count_hits(hits, cstats);
}

// Small-box records of one work item (a tile and up to ITEM_SMALL of its records): each warp takes
// 32 records at a time and takes their pixel boxes, clipped to the tile, by size (BoxQueues) or, for
// wide supports and the largest amplitudes, together (walk_boxes), adding the
// per-pixel rule's contributions to a shared tile image.  A contribution c < 2^49 is added as three
// fields, c = lo + mid 2^16 + hi 2^32 with lo, mid < 2^16, to 32-bit words by fire-and-forget
// 32-bit shared atomics (hi, rarely nonzero, only when it is): a pixel receives at most one
// contribution per record, so at most ITEM_SMALL = 2^12 per item, and no word can overflow
// (mid sums < 2^28, lo sums < 2^32, hi sums < 2^29).  The fields are then recombined in 64 bits and added
// to the image once per pixel.  One copy of the tile: with four for the warps of a CTA (44 KB more with the
// queues) two CTAs fit an SM instead of four, and 150M particles take 6.6 ms instead of 4.7.  A box is small once clipped to the image, so its pixels can lie far from a
// centre outside the image (the visible sliver of a large blob): walk_boxes takes 64-bit distances
// for those.
static_assert(ITEM_SMALL <= (1u << 12), "32-bit field sums of the small-box tile image");
struct SmallSmem {
    uint32_t lo[1024], mid[1024], hi[1024]; // TW x TH <= 1024 (checked on the host)
    int32_t K[1025];
    BoxQueues queue[RT / 32];
};

template <bool COUNT>
__global__ void __launch_bounds__(RT) k_splat_small(const uint4 *__restrict__ rec, const uint4 *__restrict__ items,
                                                      Proj P, unsigned long long *__restrict__ img, FrameStatsDev *stats)
{
    extern __shared__ __align__(16) unsigned char small_smem[];
    SmallSmem &sm = *reinterpret_cast<SmallSmem *>(small_smem);
    const int32_t *K = sm.K;
    if (threadIdx.x == 0) sm.K[1024] = 0;
    for (int i = threadIdx.x; i < 1024; i += RT) {
        sm.K[i] = g_ktab[P.kernel][i];
        sm.lo[i] = sm.mid[i] = sm.hi[i] = 0u;
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    uint32_t *lo = sm.lo, *mid = sm.mid;
    const uint4 it = items[blockIdx.x];
    const int tx = (int)(it.x % (uint32_t)P.tiles_x), ty = (int)(it.x / (uint32_t)P.tiles_x);
    const int X0 = tx * P.TW, Y0 = ty * P.TH;
    const int X1 = min(X0 + P.TW, P.W) - 1, Y1 = min(Y0 + P.TH, P.H) - 1;
    const int TW = P.TW;
    unsigned hits = 0;
    int nq[QUEUES] = {0, 0, 0};
    // a contribution below 2^32 as 20 low bits and the rest in the middle word (2^12 contributions of less than
    // 2^20 stay below 2^32)
    auto at = [&](int x, int y) {
        const int p = (y - Y0) * TW + (x - X0);
        return [=](int c, int j, uint32_t v) {
            atomicAdd(&lo[p + j * TW + c], v & 0xFFFFFu);
            atomicAdd(&mid[p + j * TW + c], (v >> 20) << 4);
        };
    };
    for (uint32_t base = it.y + (threadIdx.x & ~31u); base < it.z; base += RT) { // uniform per warp
        const uint32_t r = base + (threadIdx.x & 31u);
        BoxWalk b;
        uint4 R = make_uint4(0u, 0u, 0u, 0u);
        int x0 = 0, x1 = -1, y0 = 0, y1 = -1;
        bool mine = false;
        if (r < it.z) {
            R = rec[r];
            const int U = (int)R.x, V = (int)R.y;
            const int rad = splat_box(U, V, R.z, P.W, P.H, x0, x1, y0, y1);
            x0 = max(x0, X0);
            x1 = min(x1, X1);
            y0 = max(y0, Y0);
            y1 = min(y1, Y1);
            if (x0 <= x1 && y0 <= y1) {
                mine = group_box(rad, __uint_as_float(R.w));
                if (!mine) b = box_walk(U, V, R.z, __float2ull_rn(__uint_as_float(R.w)), rad, x0, x1, y0, y1);
            }
        }
        hits += queue_boxes<COUNT>(sm.queue[warp], nq, mine, R, x0, x1, y0, y1, K, at);
        hits += walk_boxes<false>(b, 0u, [&](uint32_t, uint32_t i) { return K[i]; },
                                  [&](uint32_t, int x, int y, unsigned long long c) {
            const int p = (y - Y0) * TW + (x - X0);
            atomicAdd(&lo[p], (uint32_t)c & 0xFFFFu);
            atomicAdd(&mid[p], ((uint32_t)c >> 16));
            const uint32_t h = (uint32_t)(c >> 32);
            if (h) atomicAdd(&sm.hi[p], h);
        });
    }
#pragma unroll
    for (int q = 0; q < QUEUES; ++q)
        if (nq[q]) hits += take_boxes<COUNT>(sm.queue[warp], q, nq[q], K, at);
    __syncthreads();
    const int tw = X1 - X0 + 1, th = Y1 - Y0 + 1;
    for (int i = threadIdx.x; i < tw * th; i += RT) {
        const int y = i / tw, x = i - y * tw, k = y * P.TW + x;
        const unsigned long long v =
            sm.lo[k] + ((unsigned long long)sm.mid[k] << 16) + ((unsigned long long)sm.hi[k] << 32);
        if (v) atomicAdd(&img[(size_t)(Y0 + y) * P.W + (X0 + x)], v);
    }
    if (COUNT) count_hits(hits, stats);
}

__global__ void k_tile_items(uint32_t ntiles, const uint32_t *tile_cnt, uint32_t *item_cnt,
                             unsigned long long *frame_tiles)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0 && frame_tiles) *frame_tiles = ntiles;
    if (t < ntiles) item_cnt[t] = (tile_cnt[t] + ITEM - 1) / ITEM;
}

// Work items of nruns runs: run t belongs to tile t mod ntiles.  Also clears the unit counter of the splat launch that
// follows and the frame's maximum (either may be null)
__global__ void k_fill_items(uint32_t nruns, uint32_t ntiles, const uint32_t *tile_cnt, const uint32_t *tile_off,
                             const uint32_t *item_off, uint32_t per_item, uint4 *items, unsigned *next,
                             unsigned long long *maxv)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0 && next) *next = 0u;
    if (t == 0 && maxv) *maxv = 0ull;
    if (t >= nruns) return;
    const uint32_t c = tile_cnt[t], o = tile_off[t];
    uint32_t k = item_off[t];
    for (uint32_t s = 0; s < c; s += per_item, ++k) items[k] = make_uint4(t % ntiles, o + s, o + min(c, s + per_item), 0u);
}

// ------------------------------------------------------------------ R3
// The tile is cut into 8 x 4 pixel blocks, one lane per pixel; a warp owns up to SPLAT_SLOTS blocks of
// one block column (see strip_height) and works on its own: a unit of work is (item, strip), an item
// a tile and up to ITEM of its records, and the warps of a persistent grid take units from a
// counter.  No barrier, no staging by other warps: a warp reads its item's records 32 at a time, one
// per lane, tests each against its two pairs of blocks, and compacts the ones that reach them into
// lists of its own in shared memory, by the arithmetic they need; a list of 16 or more is walked with one
// pixel per lane and block, without branches, the sums in registers.  Each pixel's sum is added to
// the image once per unit.
//
// What bounds the walk: a (record, pixel) pair takes one table read (about 2.6 shared-memory
// wavefronts for 32 lanes, of one a cycle for the four schedulers: 10.6 cycles), one high-word
// multiply (4.2 cycles of the multiplier) and about seven other instructions, 12.8 cycles in all for
// 32 pairs of a faint record, 15 of a light one.  Measured (GB300): 16.8M particles at 1080p, 8.4e9
// pairs, 4.37 ms (6.74 with block-wide staging, barriers and a 64-bit sum per pair); 150M particles,
// 4.7e10 pairs, 28.4 ms (41.1).  Reading and listing the records, walks skipped, is 0.9 and 6.2 ms of
// that.  The forms used, all identities of the rule:
//   index  (q S) >> 37, q < 2^32: the high word of q S, shifted by 5; q of the warp's blocks from one
//          square each in x and y and one three-input addition a block; indices from 1024 on (outside
//          the support) are clamped to a zero entry, so no pixel is tested.
//   amplitude, Wq < 2^23 (most of the pixel work: wide blobs are faint): floor(Wq K / 2^16) + 2^23 is one
//          fp32 multiply-add rounded towards zero (exact product, unit spacing in [2^23, 2^24)); its
//          bits are summed as integers, the constant taken off once per list.
//   amplitude, Wq < 2^32: Wh K + floor(Wl K / 2^16), Wq = Wh 2^16 + Wl, both below 2^16 (Wh + 1), in one
//          32-bit sum that is emptied after every `chunk` records, chunk (largest Wh + 1) <= 2^16.
constexpr int SPLAT_SLOTS = 4; // 8 warps x 4 blocks of 32 pixels: tiles up to 1024 pixels
constexpr int LIST_MIN = 16;   // a list is walked when it holds this many records
constexpr int LIST = LIST_MIN - 1 + 32;

// A warp's lists.  FAINT: Wq < 2^23; LIGHT: Wq < 2^32; either with a narrow support (QL = 2^47 / S <= 2^30:
// every pixel of a strip the support reaches lies within 2^15 + 32 px, in 1/256 px, of the centre, so
// q < 2^32), by the pairs of blocks reached: both, only the upper, only the lower.  WIDE: Wq < 2^23 with a
// wider support.  HEAVY: the rest.
enum { L_FAINT, L_FAINT_UP, L_FAINT_LOW, L_LIGHT, L_LIGHT_UP, L_LIGHT_LOW, L_WIDE, L_HEAVY, L_COUNT };

struct SplatSmem {
    uint32_t K[1025];                   // the kernel table and a zero entry
    float Kf[1025];                     // K 2^-16
    uint32_t count[RT / 32][L_COUNT];   // records in each list
    uint4 list[RT / 32][L_COUNT][LIST]; // {U, V, S, Wq}; Wq as a float in FAINT, WIDE and HEAVY
};
// dynamic shared memory: four CTAs per SM fit in its 228 KB with the 1 KB each CTA reserves
static_assert(4 * (sizeof(SplatSmem) + 1024) <= 228 * 1024, "four splat CTAs per SM");

// Each warp owns up to SPLAT_SLOTS blocks of 8 x 4 pixels in one block column: with the tile's
// nbx x nby blocks, sh = the smallest count with nbx ceil(nby / sh) <= 8 strips, strip w takes column
// w % nbx and the sh consecutive block rows from (w / nbx) sh on.
__host__ __device__ __forceinline__ int strip_height(int nbx, int nby)
{
    int sh = 1;
    while (sh < SPLAT_SLOTS && nbx * ((nby + sh - 1) / sh) > RT / 32) ++sh;
    return sh;
}

// strips of a TW x TH tile (at most 8)
__host__ __device__ __forceinline__ uint32_t strips_of(int TW, int TH)
{
    const int nbx = (TW + 7) >> 3, nby = (TH + 3) >> 2, sh = strip_height(nbx, nby);
    return (uint32_t)(nbx * ((nby + sh - 1) / sh));
}

constexpr int BLOCK_DY = 4 * 256; // y offset between consecutive blocks, 1/256 px

// Table indices (1024: outside) of blocks FIRST .. FIRST + N - 1 at this lane's pixel (px, py)
template <int FIRST, int N> __device__ __forceinline__ void block_idx(const uint4 &A, int px, int py, uint32_t (&idx)[N])
{
    const uint32_t dx = (uint32_t)px - A.x, dy = (uint32_t)(py + FIRST * BLOCK_DY) - A.y;
    const uint32_t g = 2u * BLOCK_DY * dy; // (dy + BLOCK_DY)^2 = dy^2 + g + BLOCK_DY^2
    uint32_t q = dx * dx + dy * dy;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        idx[k] = min(__umulhi(q, A.z) >> 5, 1024u);
        q += g + (uint32_t)((2 * k + 1) * BLOCK_DY * BLOCK_DY);
    }
}

// The same for any support: q in 64 bits, (q S) >> 32 = S (q >> 32) + the high word of S and q's low word
// (a pixel of a strip the support reaches has q S < 2^52, so nothing is lost)
__device__ __forceinline__ void block_idx_wide(const uint4 &A, int px, int py, uint32_t (&idx)[SPLAT_SLOTS])
{
    const int dx = px - (int)A.x, dy = py - (int)A.y;
    const long long g = 2ll * BLOCK_DY * dy;
    unsigned long long q = (unsigned long long)((long long)dx * dx + (long long)dy * dy);
#pragma unroll
    for (int k = 0; k < SPLAT_SLOTS; ++k) {
        idx[k] = min((__umulhi((uint32_t)q, A.z) + (uint32_t)(q >> 32) * A.z) >> 5, 1024u);
        q += (unsigned long long)(g + (2 * k + 1) * BLOCK_DY * BLOCK_DY);
    }
}

struct StripSums {
    unsigned long long acc[SPLAT_SLOTS] = {0ull, 0ull, 0ull, 0ull};
    unsigned hits[SPLAT_SLOTS] = {0u, 0u, 0u, 0u};
};

// Walks a list of n faint records over blocks FIRST .. FIRST + N - 1 (N even)
template <int FIRST, int N, bool WIDE, bool COUNT>
__device__ __forceinline__ void walk_faint(const uint4 *__restrict__ list, int n, int px, int py, const float *Kf,
                                           StripSums &a)
{
    uint32_t sum[N];
#pragma unroll
    for (int k = 0; k < N; ++k) sum[k] = 0u - (uint32_t)n * 0x4B000000u; // n times the bits of 2^23
#pragma unroll 2
    for (int i = 0; i < n; ++i) {
        const uint4 A = list[i];
        uint32_t idx[N];
        if constexpr (WIDE) block_idx_wide(A, px, py, idx);
        else block_idx<FIRST, N>(A, px, py, idx);
        float k[N];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            k[j] = Kf[idx[j]];
            if (COUNT) a.hits[FIRST + j] += idx[j] < 1024u ? 1u : 0u;
        }
#pragma unroll
        for (int j = 0; j < N; j += 2) // two products an instruction
            asm("{.reg .b64 w, k, c, r;\n\tmov.b64 w, {%4, %4};\n\tmov.b64 k, {%2, %3};\n\tmov.b64 c, {%5, %5};\n\t"
                "fma.rz.f32x2 r, w, k, c;\n\tmov.b64 {%0, %1}, r;}"
                : "=f"(k[j]), "=f"(k[j + 1])
                : "f"(k[j]), "f"(k[j + 1]), "f"(__uint_as_float(A.w)), "f"(0x1p23f));
#pragma unroll
        for (int j = 0; j < N; ++j) sum[j] += __float_as_uint(k[j]);
    }
#pragma unroll
    for (int k = 0; k < N; ++k) a.acc[FIRST + k] += sum[k]; // below 2^23 LIST
}

// records a 32-bit sum takes between flushes: a power of two with chunk (Wh + 1) <= 2^16 for Wh <= wmax < 2^16
__device__ __forceinline__ int flush_chunk(uint32_t wmax) { return 1 << (16 - (32 - __clz((int)wmax))); }

// Walks a list of n light records
template <int FIRST, int N, bool COUNT>
__device__ __forceinline__ void walk_light(const uint4 *__restrict__ list, int n, int px, int py, const uint32_t *K,
                                           StripSums &a)
{
    const int lane = threadIdx.x & 31;
    uint32_t wmax = lane < n ? list[lane].w >> 16 : 0u;
    if (32 + lane < n) wmax = max(wmax, list[32 + lane].w >> 16);
    const int chunk = flush_chunk(__reduce_max_sync(0xffffffffu, wmax));
    for (int i0 = 0; i0 < n; i0 += chunk) {
        const int i1 = min(n, i0 + chunk);
        uint32_t sum[N];
#pragma unroll
        for (int k = 0; k < N; ++k) sum[k] = 0u;
#pragma unroll 2
        for (int i = i0; i < i1; ++i) {
            const uint4 A = list[i];
            const uint32_t Wh = A.w >> 16, Wl = A.w & 0xFFFFu;
            uint32_t idx[N];
            block_idx<FIRST, N>(A, px, py, idx);
#pragma unroll
            for (int k = 0; k < N; ++k) {
                const uint32_t kv = K[idx[k]];
                sum[k] += Wh * kv;
                sum[k] += (Wl * kv) >> 16;
                if (COUNT) a.hits[FIRST + k] += idx[k] < 1024u ? 1u : 0u;
            }
        }
#pragma unroll
        for (int k = 0; k < N; ++k) a.acc[FIRST + k] += sum[k];
    }
}

template <bool COUNT>
__device__ __forceinline__ void walk_heavy(const uint4 *__restrict__ list, int n, int px, int py, const uint32_t *K,
                                           StripSums &a)
{
    for (int i = 0; i < n; ++i) {
        const uint4 A = list[i];
        const unsigned long long Wq = __float2ull_rn(__uint_as_float(A.w));
        const uint32_t Wh = (uint32_t)(Wq >> 16), Wl = (uint32_t)Wq & 0xFFFFu;
        uint32_t idx[SPLAT_SLOTS];
        block_idx_wide(A, px, py, idx);
#pragma unroll
        for (int k = 0; k < SPLAT_SLOTS; ++k) {
            const uint32_t kv = K[idx[k]];
            a.acc[k] += (unsigned long long)Wh * kv + ((Wl * kv) >> 16);
            if (COUNT) a.hits[k] += idx[k] < 1024u ? 1u : 0u;
        }
    }
}

// Splats records [it.y, it.z) of tile it.x (index inside the view) of view P into the pixels of strip
// `strip`; COUNT adds the pixel updates to `hits`.  Every lane of the warp calls it.
template <bool COUNT>
__device__ __forceinline__ void splat_unit(const uint4 *__restrict__ rec, const uint4 it, const int strip,
                                           const Proj &P, unsigned long long *__restrict__ img, SplatSmem &sm,
                                           unsigned &hits)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = gbd::lanemask_lt();
    const int nbx = (P.TW + 7) >> 3, nby = (P.TH + 3) >> 2;
    const int sh = strip_height(nbx, nby);
    const int tx = (int)(it.x % (uint32_t)P.tiles_x), ty = (int)(it.x / (uint32_t)P.tiles_x);
    const int X1 = min((tx + 1) * P.TW, P.W), Y1 = min((ty + 1) * P.TH, P.H); // tile clipped to the image
    const int xs = tx * P.TW + (strip % nbx) * 8, ys = ty * P.TH + (strip / nbx) * sh * 4; // the strip's first pixel
    if (xs >= X1 || ys >= Y1) return;
    const int ye = min(ys + sh * 4, Y1); // its end
    const int px = (xs + (lane & 7)) * 256 + 128, py = (ys + (lane >> 3)) * 256 + 128;
    // pixel-centre rectangles of the two pairs of blocks (there may be no lower pair)
    const float cx0 = (float)(xs * 256 + 128), cx1 = (float)((min(xs + 8, X1) - 1) * 256 + 128);
    const float cy0 = (float)(ys * 256 + 128), cy1 = (float)((min(ys + 8, ye) - 1) * 256 + 128);
    const float cy2 = (float)((ys + 8) * 256 + 128), cy3 = (float)((ye - 1) * 256 + 128);
    const bool two = ys + 8 < ye;
    StripSums a;
    uint4(*list)[LIST] = sm.list[warp];
    uint32_t *count = sm.count[warp];
    if (lane < L_COUNT) count[lane] = 0u;
    for (uint32_t base = it.y; base < it.z; base += 32) {
        uint4 R = make_uint4(0u, 0u, 1u, 0u);
        bool up = false, low = false;
        float ql = 0.0f;
        if (base + lane < it.z) {
            R = __ldg(&rec[base + lane]);
            // the next 32, read after this round's walks (eight views 12.86 -> 12.42 ms, a 512 x 512 frame 50 -> 46 us)
            if (base + 32 + lane < it.z) asm volatile("prefetch.global.L1 [%0];" ::"l"(&rec[base + 32 + lane]));
            // Pairs the support may reach: |centre - pixel-centre rectangle|^2 < QL, QL rounded up (2^-18
            // covers the reciprocal's and the sums' rounding); a pair more only costs time, the clamped
            // table index decides every pixel.
            ql = __fdividef(0x1p47f, __uint2float_rn(R.z)) * (1.0f + 0x1p-18f) + 2.0f;
            const float u = (float)(int)R.x, v = (float)(int)R.y;
            const float ex = fmaxf(fmaxf(cx0 - u, u - cx1), 0.0f), ex2 = ex * ex;
            const float eu = fmaxf(fmaxf(cy0 - v, v - cy1), 0.0f), el = fmaxf(fmaxf(cy2 - v, v - cy3), 0.0f);
            up = fmaf(eu, eu, ex2) < ql;
            low = two && fmaf(el, el, ex2) < ql;
        }
        const bool in = up || low;
        const uint32_t any = __ballot_sync(0xffffffffu, in);
        __syncwarp(); // the counters and the walks of the round before
        if (in) {
            const float W = __uint_as_float(R.w);
            const bool narrow = ql < 0x1p30f * 0.999f, faint = W < 0x1p23f - 1.0f;
            int l = up && low ? 0 : (up ? 1 : 2);
            if (!faint) l += L_LIGHT;
            if (!narrow) l = L_WIDE;
            if (!(W < 0x1p32f) || (!narrow && !faint)) l = L_HEAVY;
            R.w = l >= L_LIGHT && l <= L_LIGHT_LOW ? __float2uint_rn(W) : __float_as_uint(rintf(W));
            const uint32_t peers = __match_any_sync(any, l), rank = __popc(peers & lt);
            const uint32_t at = count[l] + rank;
            list[l][at] = R;
            __syncwarp(any);
            if (rank == 0) count[l] = at + __popc(peers);
        }
        __syncwarp();
        // lists to walk: the full ones, and after the last round every one that holds a record
        const uint32_t n = lane < L_COUNT ? count[lane] : 0u;
        uint32_t todo = __ballot_sync(0xffffffffu, n >= (base + 32 >= it.z ? 1u : (uint32_t)LIST_MIN));
        while (todo) {
            const int l = __ffs(todo) - 1;
            todo &= todo - 1;
            const int m = (int)__shfl_sync(0xffffffffu, n, l);
            const uint4 *t = list[l];
            switch (l) {
            case L_FAINT: walk_faint<0, 4, false, COUNT>(t, m, px, py, sm.Kf, a); break;
            case L_FAINT_UP: walk_faint<0, 2, false, COUNT>(t, m, px, py, sm.Kf, a); break;
            case L_FAINT_LOW: walk_faint<2, 2, false, COUNT>(t, m, px, py, sm.Kf, a); break;
            case L_LIGHT: walk_light<0, 4, COUNT>(t, m, px, py, sm.K, a); break;
            case L_LIGHT_UP: walk_light<0, 2, COUNT>(t, m, px, py, sm.K, a); break;
            case L_LIGHT_LOW: walk_light<2, 2, COUNT>(t, m, px, py, sm.K, a); break;
            case L_WIDE: walk_faint<0, 4, true, COUNT>(t, m, px, py, sm.Kf, a); break;
            default: walk_heavy<COUNT>(t, m, px, py, sm.K, a); break;
            }
            if (lane == 0) count[l] = 0u;
        }
    }
#pragma unroll
    for (int k = 0; k < SPLAT_SLOTS; ++k) {
        const int x = xs + (lane & 7), y = ys + (lane >> 3) + 4 * k;
        if (x >= X1 || y >= ye) continue;
        if (COUNT) hits += a.hits[k];
        if (a.acc[k]) atomicAdd(&img[(size_t)y * P.W + x], a.acc[k]);
    }
}

__device__ __forceinline__ void splat_table(SplatSmem &sm, int kernel)
{
    for (int i = threadIdx.x; i <= 1024; i += RT) {
        sm.K[i] = i < 1024 ? (uint32_t)g_ktab[kernel][i] : 0u;
        sm.Kf[i] = (float)sm.K[i] * 0x1p-16f;
    }
    __syncthreads();
}

// the next unit of a persistent grid's warp
__device__ __forceinline__ uint32_t next_unit(unsigned *counter)
{
    uint32_t u = 0;
    if ((threadIdx.x & 31) == 0) u = atomicAdd(counter, 1u);
    return __shfl_sync(0xffffffffu, u, 0);
}

template <bool COUNT>
__global__ void __launch_bounds__(RT, 4) k_splat_tiles(const uint4 *__restrict__ rec, const uint4 *__restrict__ items,
                                                       uint32_t nunits, uint32_t strips, unsigned *next, Proj P,
                                                       unsigned long long *__restrict__ img, FrameStatsDev *stats)
{
    extern __shared__ __align__(16) unsigned char splat_smem[];
    SplatSmem &sm = *reinterpret_cast<SplatSmem *>(splat_smem);
    splat_table(sm, P.kernel);
    unsigned hits = 0;
    for (uint32_t u = next_unit(next); u < nunits; u = next_unit(next))
        splat_unit<COUNT>(rec, items[u / strips], (int)(u % strips), P, img, sm, hits);
    if (COUNT) count_hits(hits, stats);
}

// ------------------------------------------------------------------ R4
// Both passes over an image keep eight pixels' loads in flight per thread; they read 8 bytes a pixel, and with
// one load a thread they waited for memory (eight views, 20.7M pixels: maximum 0.193 -> 0.036 ms, tone map
// 0.249 -> 0.054 ms).
constexpr int PX = 8;

__device__ __forceinline__ unsigned long long pixels_max(const unsigned long long *__restrict__ img, size_t n)
{
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    unsigned long long m = 0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += PX * stride) {
        unsigned long long a[PX];
#pragma unroll
        for (int k = 0; k < PX; ++k) a[k] = i + k * stride < n ? __ldg(&img[i + k * stride]) : 0ull;
#pragma unroll
        for (int k = 0; k < PX; ++k) m = a[k] > m ? a[k] : m;
    }
    for (int d = 16; d > 0; d >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, d);
        m = o > m ? o : m;
    }
    return m;
}

// out = 0 if I <= lo, else min(255, rne(255 ln(I/lo) / ln(hi/lo))), I = acc 2^-32
__device__ __forceinline__ void pixels_tone(const unsigned long long *__restrict__ img, size_t n, double lo, double hi,
                                            uint8_t *__restrict__ out)
{
    __shared__ unsigned long long s_low;
    __shared__ float s_l2lo, s_scale;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long a[PX];
    auto load = [&] {
#pragma unroll
        for (int k = 0; k < PX; ++k) a[k] = i + k * stride < n ? __ldg(&img[i + k * stride]) : 0ull;
    };
    load(); // under the range's logarithms
    if (threadIdx.x == 0) {
        const bool ok = hi > 0.0 && lo > 0.0 && hi > lo;
        // the largest accumulator a with !((double)a > lo): a compare of integers per pixel, where FP64
        // runs at 1/64 of the integer rate.  From 2^53 on, (double)a rounds to nearest even.
        unsigned long long low = ~0ull;
        if (ok && lo < 0x1p64) {
            low = (unsigned long long)lo;
            if (lo >= 0x1p53) {
                low += (1ull << (63 - __clzll((long long)low) - 52)) / 2; // half a step above
                if ((double)low > lo) --low;
            }
        }
        s_low = low;
        s_l2lo = ok ? (float)log2(lo) : 0.0f;
        s_scale = ok ? (float)(255.0 / log2(hi / lo)) : 0.0f;
    }
    __syncthreads();
    const unsigned long long low = s_low;
    const float l2lo = s_l2lo, scale = s_scale;
    while (i < n) {
#pragma unroll
        for (int k = 0; k < PX; ++k) {
            const float t = rintf((log2f((float)a[k]) - l2lo) * scale);
            const uint8_t o = a[k] > low ? (uint8_t)(t > 255.0f ? 255.0f : (t < 0.0f ? 0.0f : t)) : (uint8_t)0;
            if (i + k * stride < n) out[i + k * stride] = o;
        }
        i += PX * stride;
        load();
    }
}

__global__ void __launch_bounds__(256) k_image_max(const unsigned long long *img, size_t n, unsigned long long *out)
{
    const unsigned long long m = pixels_max(img, n);
    if ((threadIdx.x & 31) == 0 && m) atomicMax(out, m);
}

__global__ void __launch_bounds__(256) k_tonemap(const unsigned long long *img, size_t n, const unsigned long long *maxv,
                                                 int auto_range, double lo_acc_fixed, double hi_acc_fixed, uint8_t *out)
{
    double hi = hi_acc_fixed, lo = lo_acc_fixed;
    if (auto_range) {
        hi = (double)*maxv;
        lo = hi * 1e-4;
    }
    pixels_tone(img, n, lo, hi, out);
}

// blocks for R4 over npix pixels in all: a thread's eight pixels or more
unsigned tone_blocks(unsigned long long npix)
{
    return (unsigned)std::max<unsigned long long>(1, std::min<unsigned long long>((unsigned long long)persistent_blocks(8), npix / (256 * PX)));
}

__global__ void k_project_debug(const float4 *pts4, const float *h, size_t n, Proj P, long long *out)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float4 q = pts4[i];
        Splat s;
        const int r = project(P, q.x, q.y, q.z, q.w, h[i], s);
        out[5 * i + 0] = r;
        out[5 * i + 1] = r == 1 ? s.U : 0;
        out[5 * i + 2] = r == 1 ? s.V : 0;
        out[5 * i + 3] = r == 1 ? (long long)s.S : 0;
        out[5 * i + 4] = r == 1 ? (long long)__float2ull_rn(s.Wf) : 0;
    }
}

__global__ void k_morton_plain(const float *xyz, size_t n, double lx, double ly, double lz, double scale,
                               uint64_t *keys)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        keys[i] = gbd::morton_key(xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], lx, ly, lz, scale);
}

// ------------------------------------------------------------------ frame driver
// A frame is binned and splatted in one pass when its (tile, splat) records fit the record
// budget; otherwise the projected points are split into ranges whose records fit, each range is
// binned and splatted on its own, and the integer partial images add up to the same image.
constexpr unsigned long long RECORD_BUDGET_DEFAULT = 1ull << 28; // 4 GiB of records
constexpr unsigned long long RECORD_BUDGET_MAX = 1ull << 31;     // offsets stay 32-bit

struct PassCounts {
    unsigned long long pairs, points; // records of the pass (both streams when partitioned), points
    unsigned long long binned;        // records of the tile stream alone
    uint32_t items, small_items;      // splat work items, small-box work items (partitioned only)
};

// The caller's particle arrays are in no spatial order (a stream of its own for small boxes).
template <class Src> constexpr bool unordered_source() { return false; }
template <> constexpr bool unordered_source<SrcFlat>() { return true; }

// How a frame is binned: in parts (shared-memory histograms) whenever they fit, with `grid` CTAs over
// chunks of `chunk` points -- about four CTAs per SM, fewer when the points or the histograms do not
// allow -- or through the global tile counters.
struct Binning {
    bool part;
    unsigned grid, groups; // CTAs; groups of grid / groups CTAs
    uint32_t chunk;
    size_t smem;
};

template <class Src> Binning binning(const Src &src, const Proj &P)
{
    Binning b;
    b.smem = (size_t)P.tiles_x * P.tiles_y * (unordered_source<Src>() ? 8 : 4);
    b.part = b.smem <= PART_MAX_SMEM;
    const unsigned nt = (unsigned)PART_THREADS<unordered_source<Src>()>;
    const unsigned full = (unsigned)persistent_blocks(
        b.part ? (int)std::min<size_t>(1024 / nt, std::max<size_t>(1, 216 * 1024 / (b.smem + 6 * 1024))) : 4);
    // at least one point a thread; the bound is all that is known here of an octree frame's points
    const unsigned long long per = (src.bound + full - 1) / full;
    b.chunk = b.part ? (uint32_t)std::min<unsigned long long>(CHUNK, std::max<unsigned long long>(nt, (per + nt - 1) / nt * nt))
                     : CHUNK;
    b.grid = b.part ? (unsigned)std::max<unsigned long long>(1, std::min<unsigned long long>(full, (src.bound + b.chunk - 1) / b.chunk))
                    : full;
    // Records go to one place per (CTA, tile).  Of points in no order every CTA writes to all of them all the
    // time, and stores spread over gigabytes miss the address-translation caches: a group's region is
    // kept to some 128 MB (24 bytes of records a point).  150M points: scatter 5.37 ms in one region of 3.7 GB,
    // 3.8 in 8, 3.0 in 19 and in 152; 16.8M: 0.66 in one, 0.57 in 3.  More runs are more work items with fewer records.
    b.groups = 1;
    if (b.part && unordered_source<Src>()) {
        const unsigned want = (unsigned)std::min<unsigned long long>(b.grid / 8, src.bound * 24 >> 27);
        b.groups = std::max(1u, want);
        b.grid = b.grid / b.groups * b.groups;
    }
    return b;
}

template <class Src>
PassCounts bin_count(gblod_renderer *r, const Src &src, const Proj &P, unsigned long long lo, unsigned long long hi,
                     FrameStatsDev *stats, cudaStream_t s)
{
    const Allocator &A = r->A;
    const uint32_t ntiles = (uint32_t)(P.tiles_x * P.tiles_y);
    const Binning bn = binning(src, P);
    constexpr bool SMALL = unordered_source<Src>();
    const size_t nh = (size_t)ntiles * bn.grid, nall = SMALL ? 2 * nh : nh;
    const uint32_t nruns = ntiles * bn.groups, gs = bn.grid / bn.groups;
    r->tile_cnt.ensure(A, nruns, s);
    r->tile_off.ensure(A, nruns + 1, s);
    r->item_cnt.ensure(A, nruns, s);
    r->item_off.ensure(A, nruns + 1, s);
    if (bn.part) {
        r->cta_hist.ensure(A, nall, s);
        r->cta_off.ensure(A, nall, s);
        launch(GBLOD_K_PROJECT_COUNT, k_project_hist<Src, SMALL>, dim3(bn.grid), dim3(PART_THREADS<SMALL>), bn.smem, s, src, P, lo, hi,
               bn.chunk, gs, r->cta_hist.p, r->status, stats);
        scan_exclusive_u32(A, r->scan, r->cta_hist.p, r->cta_off.p, nall, &stats->records, s);
        const dim3 tg((nruns + 255) / 256);
        launch(GBLOD_K_RENDER_OTHER, k_tiles_from_hist, tg, dim3(256), 0, s, nruns, gs, 0u, items_wanted(),
               (const uint32_t *)r->cta_off.p, SMALL ? (const uint32_t *)(r->cta_off.p + nh) : &stats->records,
               r->tile_cnt.p, r->tile_off.p, r->item_cnt.p, &stats->tiles, ntiles);
        if (SMALL) {
            r->tile_cnt_s.ensure(A, nruns, s);
            r->tile_off_s.ensure(A, nruns, s);
            r->item_cnt_s.ensure(A, nruns, s);
            r->item_off_s.ensure(A, nruns, s);
            launch(GBLOD_K_RENDER_OTHER, k_tiles_from_hist, tg, dim3(256), 0, s, nruns, gs, ITEM_SMALL, 0u,
                   (const uint32_t *)(r->cta_off.p + nh), &stats->records, r->tile_cnt_s.p, r->tile_off_s.p,
                   r->item_cnt_s.p, (unsigned long long *)nullptr, 0u);
            scan_exclusive_u32(A, r->scan, r->item_cnt_s.p, r->item_off_s.p, nruns, &stats->small_items, s);
        }
    } else {
        r->tile_cur.ensure(A, ntiles, s);
        GB_CUDA(cudaMemsetAsync(r->tile_cnt.p, 0, (size_t)ntiles * 4, s));
        launch(GBLOD_K_PROJECT_COUNT, k_project_count<Src>, dim3(bn.grid), dim3(RT), 0, s, src, P, lo, hi, r->tile_cnt.p,
               r->status, stats);
        scan_exclusive_u32(A, r->scan, r->tile_cnt.p, r->tile_off.p, ntiles, r->tile_off.p + ntiles, s);
        launch(GBLOD_K_RENDER_OTHER, k_tile_items, dim3((ntiles + 255) / 256), dim3(256), 0, s, ntiles,
               (const uint32_t *)r->tile_cnt.p, r->item_cnt.p, &stats->tiles);
    }
    scan_exclusive_u32(A, r->scan, r->item_cnt.p, r->item_off.p, nruns, &stats->items, s);
    FrameStatsDev *h = static_cast<FrameStatsDev *>(r->hs.get(sizeof(FrameStatsDev)));
    GB_CUDA(cudaMemcpyAsync(h, stats, sizeof(FrameStatsDev), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    // the scanned offsets, and with them the item counts, are modulo 2^32: the pass is sized by the 64-bit counts, and
    // one whose records do not fit the budget is split before anything is placed
    return PassCounts{h->pairs + h->small_pairs, h->points, h->pairs, h->items, bn.part && SMALL ? h->small_items : 0u};
}

// R3 over `items` work items: a persistent grid, no more CTAs than the units need
void launch_splat(bool count, const uint4 *rec, const uint4 *items, uint32_t nitems, unsigned *next, const Proj &P,
                  unsigned long long *img, FrameStatsDev *stats, cudaStream_t s)
{
    const uint32_t strips = strips_of(P.TW, P.TH);
    const unsigned long long units = (unsigned long long)nitems * strips;
    if (units > 0xFFFF0000ull) fail(GBLOD_ERR_RANGE, "too many splat work units");
    const unsigned grid = (unsigned)std::min<unsigned long long>((units + RT / 32 - 1) / (RT / 32),
                                                                (unsigned long long)persistent_blocks(4));
    launch(GBLOD_K_SPLAT, count ? k_splat_tiles<true> : k_splat_tiles<false>, dim3(grid), dim3(RT), sizeof(SplatSmem), s, rec,
           items, (uint32_t)units, strips, next, P, img, stats);
}

template <class Src>
void bin_splat(gblod_renderer *r, const Src &src, const Proj &P, unsigned long long lo, unsigned long long hi,
               const PassCounts &pc, unsigned long long *img, cudaStream_t s)
{
    const Allocator &A = r->A;
    const uint32_t ntiles = (uint32_t)(P.tiles_x * P.tiles_y);
    const Binning bn = binning(src, P);
    constexpr bool SMALL = unordered_source<Src>();
    const uint32_t nruns = ntiles * bn.groups;
    const dim3 tg((nruns + 255) / 256);
    FrameStatsDev *cstats = r->count_updates ? r->stats : (FrameStatsDev *)nullptr;
    r->records.ensure(A, pc.pairs, s);
    r->items.ensure(A, (size_t)pc.items + pc.small_items, s);
    if (bn.part) {
        launch(GBLOD_K_PROJECT_SCATTER, k_project_scatter_part<Src, SMALL>, dim3(bn.grid), dim3(PART_THREADS<SMALL>), bn.smem, s,
               src, P, lo, hi, bn.chunk, bn.grid / bn.groups, (const uint32_t *)r->cta_off.p, r->records.p, img, cstats);
        if (SMALL) {
            launch(GBLOD_K_RENDER_OTHER, k_fill_items, tg, dim3(256), 0, s, nruns, ntiles,
                   (const uint32_t *)r->tile_cnt_s.p, (const uint32_t *)r->tile_off_s.p,
                   (const uint32_t *)r->item_off_s.p, ITEM_SMALL, r->items.p + pc.items, (unsigned *)nullptr,
                   (unsigned long long *)nullptr);
            launch(GBLOD_K_SPLAT, r->count_updates ? k_splat_small<true> : k_splat_small<false>, dim3(pc.small_items),
                   dim3(RT), sizeof(SmallSmem), s, (const uint4 *)r->records.p, (const uint4 *)(r->items.p + pc.items), P, img, r->stats);
        }
    } else {
        GB_CUDA(cudaMemcpyAsync(r->tile_cur.p, r->tile_off.p, (size_t)ntiles * 4, cudaMemcpyDeviceToDevice, s));
        launch(GBLOD_K_PROJECT_SCATTER, k_project_scatter<Src>, dim3(bn.grid), dim3(RT), 0, s, src, P, lo, hi,
               r->tile_cur.p, r->records.p, img, cstats);
    }
    launch(GBLOD_K_RENDER_OTHER, k_fill_items, tg, dim3(256), 0, s, nruns, ntiles,
           (const uint32_t *)r->tile_cnt.p, (const uint32_t *)r->tile_off.p, (const uint32_t *)r->item_off.p,
           bn.part ? item_size((uint32_t)pc.binned, items_wanted()) : ITEM, r->items.p, r->status + 1, r->maxv.p);
    launch_splat(r->count_updates, r->records.p, r->items.p, pc.items, r->status + 1, P, img, r->stats, s);
}

template <class Src>
void frame_common(gblod_renderer *r, const Src &src, const Proj &P, const gblod_render_params &rp, uint8_t *image,
                  uint64_t *accum, cudaStream_t s)
{
    const Allocator &A = r->A;
    const uint32_t ntiles = (uint32_t)(P.tiles_x * P.tiles_y);
    r->count_updates = (rp.flags & GBLOD_RENDER_COUNT_UPDATES) != 0;
    r->pass_stats.ensure(A, 1, s);
    const size_t npix = (size_t)P.W * P.H;
    unsigned long long *img = reinterpret_cast<unsigned long long *>(accum);
    if (!img) {
        r->accum.ensure(A, npix, s);
        img = r->accum.p;
    }
    r->maxv.ensure(A, 1, s);
    GB_CUDA(cudaMemsetAsync(img, 0, npix * 8, s));
    const unsigned long long RECORD_BUDGET =
        rp.record_budget ? std::min<unsigned long long>(rp.record_budget, RECORD_BUDGET_MAX) : RECORD_BUDGET_DEFAULT;
    // whole frame first; its counts also give the frame statistics
    const PassCounts all = bin_count(r, src, P, 0ull, ~0ull, r->stats, s);
    if (all.pairs <= RECORD_BUDGET) {
        bin_splat(r, src, P, 0ull, ~0ull, all, img, s);
    } else {
        // split the point range until every piece's records fit the budget (a single point
        // may exceed it; its records always fit the 2^31 maximum)
        const unsigned long long pieces =
            std::max(1ull, std::min(all.points, (all.pairs + RECORD_BUDGET - 1) / RECORD_BUDGET * 2));
        std::vector<std::pair<unsigned long long, unsigned long long>> todo;
        for (unsigned long long k = pieces; k-- > 0;) {
            const unsigned long long lo = all.points * k / pieces, hi = all.points * (k + 1) / pieces;
            if (hi > lo) todo.emplace_back(lo, hi);
        }
        while (!todo.empty()) {
            const auto [lo, hi] = todo.back();
            todo.pop_back();
            GB_CUDA(cudaMemsetAsync(r->pass_stats.p, 0, sizeof(FrameStatsDev), s));
            const PassCounts pc = bin_count(r, src, P, lo, hi, r->pass_stats.p, s);
            if (pc.pairs > RECORD_BUDGET && hi - lo > 1) {
                const unsigned long long mid = lo + (hi - lo) / 2;
                todo.emplace_back(mid, hi);
                todo.emplace_back(lo, mid);
                continue;
            }
            if (pc.pairs > RECORD_BUDGET_MAX) fail(GBLOD_ERR_RANGE, "one point needs more than 2^31 tile records");
            bin_splat(r, src, P, lo, hi, pc, img, s);
        }
    }
    if (image) {
        double lo = 0.0, hi = 0.0;
        if (rp.tone_auto) {
            launch(GBLOD_K_TONEMAP, k_image_max, dim3(tone_blocks(npix)), dim3(256), 0, s,
                   (const unsigned long long *)img, npix, r->maxv.p);
        } else {
            lo = std::ldexp(rp.tone_lo, 32);
            hi = std::ldexp(rp.tone_hi, 32);
        }
        launch(GBLOD_K_TONEMAP, k_tonemap, dim3(tone_blocks(npix)), dim3(256), 0, s,
               (const unsigned long long *)img, npix, (const unsigned long long *)r->maxv.p, rp.tone_auto ? 1 : 0,
               lo, hi, image);
    }
}


// ------------------------------------------------------------------ batched views (no host waits)
// Many views -- each with its own camera, resolution and octree -- rendered by one set of
// launches: R1 walks (view, node) pairs, the points of all selected nodes of all views form one
// flat index space, screen tiles of all views one global tile space, and persistent kernels read
// every data-dependent count from device memory.  Nothing waits on the host, so the sequence can
// be captured in a CUDA graph.  Scratch has a reserved capacity; a batch that needs more sets the
// sticky capacity bit of the renderer's status instead of growing it.
constexpr unsigned ST_CAPACITY = 4u;
constexpr int VIEWS_PER_CHUNK = 40;

struct ViewDev {
    Proj P;
    Frustum F;
    const gblod_node *nodes;
    const float4 *pts4;
    const float *hs;
    const ushort4 *q4;   // non-null: draw the 16-bit block codes
    const uint16_t *qw;
    const float4 *qa;
    unsigned long long *accum;
    uint8_t *image;
    unsigned long long pix_base;
    uint32_t tile_base, n_nodes, node_base;
    double lo_acc, hi_acc; // fixed tone range in accumulator units (unused when automatic)
};

struct ViewChunk {
    int first, n;
    ViewDev v[VIEWS_PER_CHUNK];
};
static_assert(sizeof(ViewChunk) < 30000, "kernel parameter block too large");

__global__ void k_set_views(ViewChunk c, ViewDev *dst)
{
    for (int i = threadIdx.x; i < c.n; i += blockDim.x) dst[c.first + i] = c.v[i];
}

__global__ void k_bzero(const ViewDev *__restrict__ views)
{
    const ViewDev &V = views[blockIdx.y];
    const size_t n = (size_t)V.P.W * V.P.H;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        V.accum[i] = 0ull;
}

// The flat form of the selection over the nodes that the views can reach (up to SELECT_FLAT in all)
__device__ __forceinline__ int view_of_node(const ViewDev *__restrict__ views, int n, uint32_t e)
{
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (views[mid].node_base <= e) lo = mid; else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(128) k_bclassify(const ViewDev *__restrict__ views, int n, uint32_t total,
                                                   uint8_t *__restrict__ cls)
{
    const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    const ViewDev &V = views[view_of_node(views, n, e)];
    cls[e] = (uint8_t)classify(V.nodes[e - V.node_base], V.F);
}

__global__ void __launch_bounds__(RT) k_bselect_flat(const ViewDev *__restrict__ views, int n, uint32_t total,
                                                     const uint8_t *__restrict__ cls,
                                                     unsigned long long *__restrict__ sel, uint32_t *nsel)
{
    const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
    int v = 0;
    uint32_t node = 0;
    bool take = e < total && cls[e] == 1;
    if (take) {
        v = view_of_node(views, n, e);
        const uint32_t b = views[v].node_base;
        const gblod_node *nodes = views[v].nodes;
        node = e - b;
        for (int p = nodes[node].parent; p >= 0 && take; p = nodes[p].parent) take = cls[b + (uint32_t)p] == 2;
    }
    append_nodes(take, (unsigned long long)v << 32 | node, sel, nsel);
}

__global__ void k_bselect_init(const ViewDev *__restrict__ views, int n, unsigned long long *front, uint32_t *cnt)
{
    for (int v = threadIdx.x; v < n; v += blockDim.x)
        if (views[v].n_nodes) front[atomicAdd(cnt, 1u)] = (unsigned long long)v << 32;
}

__global__ void __launch_bounds__(RT) k_bselect_level(const ViewDev *__restrict__ views,
                                                      const unsigned long long *__restrict__ fin, const uint32_t *nin,
                                                      unsigned long long *__restrict__ fout, uint32_t *nout,
                                                      unsigned long long *__restrict__ sel, uint32_t *nsel)
{
    const uint32_t n = *nin;
    const int lane = threadIdx.x & 31;
    for (uint32_t base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {
        const uint32_t i = base + threadIdx.x;
        int cls = 0;
        unsigned long long ent = 0;
        uint32_t ccount = 0, cfirst = 0;
        if (i < n) {
            ent = fin[i];
            const int v = (int)(ent >> 32);
            const gblod_node g = views[v].nodes[(uint32_t)ent];
            cls = classify(g, views[v].F);
            ccount = g.child_count;
            cfirst = g.child_first;
        }
        append_nodes(cls == 1, ent, sel, nsel);
        uint32_t want = cls == 2 ? ccount : 0u, incl = want;
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        if (total) {
            uint32_t b = 0;
            if (lane == 31) b = atomicAdd(nout, total);
            b = __shfl_sync(0xffffffffu, b, 31);
            const uint32_t at = b + incl - want;
            const unsigned long long hiv = ent & 0xFFFFFFFF00000000ull;
            for (uint32_t k = 0; k < want; ++k) fout[at + k] = hiv | (cfirst + k);
        }
    }
}

__global__ void k_bsel_counts(const ViewDev *__restrict__ views, const unsigned long long *__restrict__ sel,
                              const uint32_t *nsel, uint32_t cap, unsigned long long *counts)
{
    const uint32_t n = *nsel;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cap; i += gridDim.x * blockDim.x) {
        unsigned long long c = 0;
        if (i < n) {
            const unsigned long long e = sel[i];
            c = views[e >> 32].nodes[(uint32_t)e].point_count;
        }
        counts[i] = c;
    }
}

__global__ void k_bsel_base(const ViewDev *__restrict__ views, const unsigned long long *__restrict__ sel,
                            const uint32_t *nsel, const unsigned long long *__restrict__ pfx, long long *base,
                            FrameStatsDev *stats)
{
    const uint32_t n = *nsel;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const unsigned long long e = sel[i];
        base[i] = (long long)views[e >> 32].nodes[(uint32_t)e].point_first - (long long)pfx[i];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) stats->nodes_selected = n;
}

struct SrcBatch {
    const ViewDev *views;
    const unsigned long long *sel;
    const unsigned long long *pfx;
    const long long *base;
    const uint32_t *nsel;
    const unsigned long long *total;
};

__device__ __forceinline__ void bsrc_range(const SrcBatch &s, unsigned long long a, unsigned long long b,
                                           uint32_t &j0, uint32_t &j1)
{
    __shared__ uint32_t sj[2];
    if (threadIdx.x < 64) {
        const uint32_t j = warp_find(reinterpret_cast<const uint64_t *>(s.pfx), *s.nsel, threadIdx.x < 32 ? a : b - 1);
        if ((threadIdx.x & 31) == 0) sj[threadIdx.x >> 5] = j;
    }
    __syncthreads();
    j0 = sj[0];
    j1 = sj[1];
    __syncthreads();
}

// point e of the flat space: its view and its data
__device__ __forceinline__ int bsrc_load(const SrcBatch &s, unsigned long long e, uint32_t j0, uint32_t j1, float &x,
                                         float &y, float &z, float &w, float &h)
{
    uint32_t lo = j0, hi = j1 + 1;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (s.pfx[mid] <= e) lo = mid; else hi = mid;
    }
    const unsigned long long ent = s.sel[lo];
    const int v = (int)(ent >> 32);
    const unsigned long long p = (unsigned long long)((long long)e + s.base[lo]);
    const ViewDev &V = s.views[v];
    if (V.q4) {
        const uint32_t node = (uint32_t)ent;
        block_decode(V.q4[p], V.qw[p], V.qa[2 * node], V.qa[2 * node + 1], x, y, z, w, h);
    } else {
        const float4 q = V.pts4[p];
        x = q.x; y = q.y; z = q.z; w = q.w;
        h = V.hs[p];
    }
    return v;
}

// Counting pass (SCATTER false) or record pass (true) over the flat point space of a batch; the
// record pass also splats the points with small boxes into their view's image, and counts their
// pixel updates when count_updates is set.  PART: binned in parts like an octree frame, the tiles of all
// views in one shared-memory histogram; `tiles` is the (tile, CTA) histogram (counting) or its scan (records).
// Else it is the tiles' counts or cursors.  (Eight views, 1080p, count + records: 4.5 ms with global counters
// and walked boxes, 2.3 ms in parts and with group_boxes.)
template <bool SCATTER, bool PART>
__global__ void __launch_bounds__(RT, 4) k_bproject(SrcBatch src, uint32_t *__restrict__ tiles,
                                                 uint32_t ntiles, int kernel, uint4 *__restrict__ rec,
                                                 unsigned long long rec_cap, unsigned *status, FrameStatsDev *stats,
                                                 int count_updates)
{
    extern __shared__ uint32_t sh_tiles[]; // PART: [ntiles] counts or next record positions
    __shared__ int32_t K[SCATTER ? 1025 : 1];
    if (PART)
        for (uint32_t t = threadIdx.x; t < ntiles; t += RT)
            sh_tiles[t] = SCATTER ? tiles[(size_t)t * gridDim.x + blockIdx.x] : 0u;
    if (SCATTER)
        for (int t = threadIdx.x; t <= 1024; t += RT) K[t] = t < 1024 ? g_ktab[kernel][t] : 0;
    __syncthreads();
    const unsigned long long total = *src.total;
    unsigned hits = 0;
    const int lane = threadIdx.x & 31;
    unsigned long long splats = 0, pairs = 0;
    AmpSum amp;
    __shared__ Proj sP[2];
    __shared__ int sV[2];
    for (unsigned long long a = (unsigned long long)blockIdx.x * CHUNK; a < total;
         a += (unsigned long long)gridDim.x * CHUNK) {
        const unsigned long long b = min(total, a + CHUNK);
        uint32_t j0, j1;
        bsrc_range(src, a, b, j0, j1);
        // the chunk's points belong to the views of its first and last nodes, or rarely in between
        if (threadIdx.x < 2) {
            const int vv = (int)(src.sel[threadIdx.x == 0 ? j0 : j1] >> 32);
            sV[threadIdx.x] = vv;
            sP[threadIdx.x] = src.views[vv].P;
        }
        __syncthreads();
        for (unsigned long long e0 = a; e0 < b; e0 += RT) {
            const unsigned long long e = e0 + threadIdx.x;
            int res = 0, v = 0;
            Splat s;
            if (e < b) {
                float x, y, z, w, h;
                v = bsrc_load(src, e, j0, j1, x, y, z, w, h);
                const Proj &Pv = v == sV[0] ? sP[0] : (v == sV[1] ? sP[1] : src.views[v].P);
                res = project(Pv, x, y, z, w, h, s);
            }
            if (!SCATTER) {
                if (__any_sync(0xffffffffu, res < 0) && lane == 0) atomicOr(status, ST_RANGE);
                if (res == 1) amp.add(__float2ull_rn(s.Wf));
            }
            uint32_t n = 0, t00 = 0;
            int tw = 1, tiles_x = 1;
            uint4 r = make_uint4(0u, 0u, 0u, 0u);
            BoxWalk direct;
            bool mine = false;
            int x0 = 0, x1 = -1, y0 = 0, y1 = -1;
            if (res == 1) {
                const Proj &P = v == sV[0] ? sP[0] : (v == sV[1] ? sP[1] : src.views[v].P);
                const uint32_t tb = src.views[v].tile_base;
                if (!SCATTER) ++splats;
                const int rad = splat_box(s.U, s.V, s.S, P.W, P.H, x0, x1, y0, y1);
                if (x0 <= x1 && y0 <= y1) {
                    if (direct_box(x0, x1, y0, y1)) {
                        if (SCATTER) {
                            mine = group_box(rad, s.Wf);
                            if (!mine) direct = box_walk(s.U, s.V, s.S, __float2ull_rn(s.Wf), rad, x0, x1, y0, y1);
                        }
                    } else {
                        const int tx0 = x0 / P.TW, tx1 = x1 / P.TW, ty0 = y0 / P.TH, ty1 = y1 / P.TH;
                        tw = tx1 - tx0 + 1;
                        n = (uint32_t)(tw * (ty1 - ty0 + 1));
                        t00 = tb + (uint32_t)(ty0 * P.tiles_x + tx0);
                        tiles_x = P.tiles_x;
                        if (!SCATTER) pairs += n;
                        r = make_uint4((uint32_t)s.U, (uint32_t)s.V, s.S, __float_as_uint(s.Wf));
                    }
                }
            }
            if (SCATTER) {
                if (PART) {
                    const uint32_t th = n / (uint32_t)tw;
                    for (uint32_t ty = 0; ty < th; ++ty)
                        for (uint32_t tx = 0; tx < (uint32_t)tw; ++tx) {
                            const uint32_t pos = atomicAdd(&sh_tiles[t00 + ty * (uint32_t)tiles_x + tx], 1u);
                            if (pos < rec_cap) rec[pos] = r;
                        }
                } else {
                    scatter_pairs(n, t00, tw, tiles_x, r, tiles, rec, rec_cap);
                }
                auto at = [&](uint32_t t, int x, int y) {
                    const ViewDev &V = src.views[t];
                    const int W = V.P.W;
                    unsigned long long *p = V.accum + (size_t)y * W + x;
                    return [p, W](int j, unsigned long long c) { atomicAdd(&p[(size_t)j * W], c); };
                };
                const bool four = x1 - x0 < 4;
                hits += group_boxes<4, true>(mine && four, s.U, s.V, s.S, s.Wf, x0, x1, y0, y1, K, at, (uint32_t)v);
                hits += group_boxes<8, true>(mine && !four, s.U, s.V, s.S, s.Wf, x0, x1, y0, y1, K, at, (uint32_t)v);
                hits += walk_boxes<true>(direct, (uint32_t)v, [&](uint32_t, uint32_t i) { return K[i]; },
                                         [&](uint32_t t, int x, int y, unsigned long long c) { at(t, x, y)(0, c); });
            } else if (n) {
                const uint32_t th = n / (uint32_t)tw;
                for (uint32_t ty = 0; ty < th; ++ty)
                    for (uint32_t tx = 0; tx < (uint32_t)tw; ++tx) {
                        const uint32_t t = t00 + ty * (uint32_t)tiles_x + tx;
                        if (PART) {
                            atomicAdd(&sh_tiles[t], 1u);
                        } else {
                            const uint32_t peers = __match_any_sync(__activemask(), t);
                            if (lane == __ffs(peers) - 1) atomicAdd(&tiles[t], (uint32_t)__popc(peers));
                        }
                    }
            }
        }
        __syncthreads();
    }
    if (!SCATTER) {
        if (PART) // the loop ends in a barrier, or has not run
            for (uint32_t t = threadIdx.x; t < ntiles; t += RT) tiles[(size_t)t * gridDim.x + blockIdx.x] = sh_tiles[t];
        for (int d = 16; d > 0; d >>= 1) {
            splats += __shfl_xor_sync(0xffffffffu, splats, d);
            pairs += __shfl_xor_sync(0xffffffffu, pairs, d);
        }
        if (lane == 0 && splats) atomicAdd(&stats->splats, splats);
        if (lane == 0 && pairs) atomicAdd(&stats->pairs, pairs);
        amp.flush(stats);
    } else if (count_updates) {
        count_hits(hits, stats);
    }
}

// items of every tile of every view; a tile's view comes from the tile bases
__global__ void k_bfill_items(uint32_t ntiles, const ViewDev *__restrict__ views, int nviews,
                              const uint32_t *tile_cnt, const uint32_t *tile_off, const uint32_t *item_off,
                              uint4 *items, uint32_t items_cap, unsigned long long rec_cap,
                              const FrameStatsDev *stats, unsigned *status, uint32_t want)
{
    const uint32_t per_item = want ? item_size((uint32_t)stats->pairs, want) : ITEM;
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0 && (stats->pairs > rec_cap || item_off[ntiles] > items_cap)) atomicOr(status, ST_CAPACITY);
    if (t >= ntiles) return;
    int lo = 0, hi = nviews;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (views[mid].tile_base <= t) lo = mid; else hi = mid;
    }
    const uint32_t c = tile_cnt[t], o = tile_off[t], local = t - views[lo].tile_base;
    uint32_t k = item_off[t];
    for (uint32_t s = 0; s < c && k < items_cap; s += per_item, ++k) {
        const uint32_t b = o + s, e = o + min(c, s + per_item);
        // records beyond the capacity were never written: clip (the batch is flagged)
        const uint32_t bc = (uint32_t)min((unsigned long long)b, rec_cap), ec = (uint32_t)min((unsigned long long)e, rec_cap);
        items[k] = make_uint4(local, bc, ec, (uint32_t)lo);
    }
}

template <bool COUNT>
__global__ void __launch_bounds__(RT, 4) k_bsplat(const uint4 *__restrict__ rec, const uint4 *__restrict__ items,
                                                  const uint32_t *nitems_p, uint32_t items_cap, uint32_t strips,
                                                  int kernel, const ViewDev *__restrict__ views, unsigned *next,
                                                  FrameStatsDev *stats)
{
    extern __shared__ __align__(16) unsigned char splat_smem[];
    SplatSmem &sm = *reinterpret_cast<SplatSmem *>(splat_smem);
    splat_table(sm, kernel);
    unsigned hits = 0;
    const uint32_t nunits = min(*nitems_p, items_cap) * strips;
    for (uint32_t u = next_unit(next); u < nunits; u = next_unit(next)) {
        const uint4 it = items[u / strips];
        splat_unit<COUNT>(rec, it, (int)(u % strips), views[it.w].P, views[it.w].accum, sm, hits);
    }
    if (COUNT) count_hits(hits, stats);
}

// R4 over the views of a batch: blockIdx.y = view
__global__ void __launch_bounds__(256) k_bmax(const ViewDev *__restrict__ views, unsigned long long *maxv)
{
    const ViewDev &V = views[blockIdx.y];
    const unsigned long long m = pixels_max(V.accum, (size_t)V.P.W * V.P.H);
    if ((threadIdx.x & 31) == 0 && m) atomicMax(&maxv[blockIdx.y], m);
}

__global__ void __launch_bounds__(256) k_btonemap(const ViewDev *__restrict__ views, const unsigned long long *maxv,
                                                  int auto_range)
{
    const ViewDev &V = views[blockIdx.y];
    if (!V.image) return;
    double hi = V.hi_acc, lo = V.lo_acc;
    if (auto_range) {
        hi = (double)maxv[blockIdx.y];
        lo = hi * 1e-4;
    }
    pixels_tone(V.accum, (size_t)V.P.W * V.P.H, lo, hi, V.image);
}

// A batch is binned in parts if its tiles fit a shared-memory histogram: CTAs per SM, 0 if not
int batch_part(uint32_t ntiles)
{
    const size_t smem = (size_t)ntiles * 4;
    if (smem > PART_MAX_SMEM) return 0;
    return (int)std::min<size_t>(4, std::max<size_t>(1, 216 * 1024 / (smem + 6 * 1024)));
}

// work items of a batch, at most: one begun item a tile, and full ones, of which there are no more than are
// wanted, or than ITEM records each give
uint64_t batch_items(uint32_t ntiles, uint64_t records) { return ntiles + std::max<uint64_t>(records / ITEM, items_wanted()) + 1; }

// histogram entries of a batch of up to ntiles tiles
size_t batch_hist(uint32_t ntiles)
{
    size_t m = 0;
    for (int k = 1; k <= 4; ++k) { // the most tiles with k CTAs per SM
        const size_t most = std::min<size_t>(PART_MAX_SMEM / 4, (216 * 1024 / (size_t)k - 6 * 1024) / 4);
        m = std::max(m, std::min<size_t>(ntiles, most) * (size_t)persistent_blocks(k));
    }
    return m;
}

struct BatchPlan {
    std::vector<ViewDev> host;
    uint32_t ntiles = 0, max_levels = 0;
    unsigned long long npix = 0;
    uint64_t nodes = 0;     // of all views' trees (sizes the scratch)
    uint64_t reached = 0;   // of them, those the views can reach,
    uint32_t deep = 0;      // and the depths these have
};

BatchPlan plan_batch(const gblod_view *views, int n, const gblod_render_params &rp)
{
    if (n > 65535) fail(GBLOD_ERR_INVALID_ARG, "a batch holds at most 65535 views");
    BatchPlan b;
    b.host.resize(n);
    for (int v = 0; v < n; ++v) {
        const gblod_view &V = views[v];
        if (!V.octree) fail(GBLOD_ERR_INVALID_ARG, "batch view has no octree");
        if (!V.d_accum) fail(GBLOD_ERR_INVALID_ARG, "batch views need d_accum");
        check_image(V.camera);
        check_format(V.octree, rp);
        ViewDev &d = b.host[v];
        std::memset(&d, 0, sizeof(d));
        d.P = make_proj(V.camera, rp);
        d.F = make_frustum(V.camera, rp, V.octree);
        if (rp.point_format == GBLOD_POINTS_BLOCK16) {
            d.nodes = V.octree->qnodes;
            d.q4 = V.octree->q4;
            d.qw = V.octree->qw;
            d.qa = V.octree->qa;
        } else {
            d.nodes = V.octree->nodes;
            d.pts4 = V.octree->pts4;
            d.hs = V.octree->hs;
        }
        d.accum = reinterpret_cast<unsigned long long *>(V.d_accum);
        d.image = V.d_image;
        d.pix_base = b.npix;
        d.tile_base = b.ntiles;
        d.n_nodes = (uint32_t)V.octree->n_nodes;
        d.node_base = (uint32_t)b.reached;
        d.lo_acc = std::ldexp(rp.tone_lo, 32);
        d.hi_acc = std::ldexp(rp.tone_hi, 32);
        const unsigned long long tiles = (unsigned long long)d.P.tiles_x * d.P.tiles_y;
        if ((unsigned long long)b.ntiles + tiles > 0x7FFFFFFFull) fail(GBLOD_ERR_INVALID_ARG, "too many tiles in batch");
        b.ntiles += (uint32_t)tiles;
        b.npix += (unsigned long long)d.P.W * d.P.H;
        b.nodes += V.octree->n_nodes;
        int deep = 0;
        b.reached += reached_nodes(V.octree, d.F, deep);
        b.deep = std::max(b.deep, (uint32_t)deep);
        b.max_levels = std::max<uint32_t>(b.max_levels, (uint32_t)V.octree->depth_max + 1);
    }
    if (b.nodes >= 0xFFFFFFFFull) fail(GBLOD_ERR_INVALID_ARG, "too many nodes in batch");
    return b;
}

// the splat kernels' SplatSmem and the binning histograms of frames with many tiles are above the 48 KB
// a launch may take without opting in
void set_splat_smem()
{
    const void *part[] = {(const void *)k_project_hist<SrcLOD, false>, (const void *)k_project_hist<SrcLODQ, false>,
                          (const void *)k_project_hist<SrcFlat, true>, (const void *)k_project_scatter_part<SrcLOD, false>,
                          (const void *)k_project_scatter_part<SrcLODQ, false>,
                          (const void *)k_project_scatter_part<SrcFlat, true>, (const void *)k_bproject<false, true>,
                          (const void *)k_bproject<true, true>};
    for (const void *f : part)
        GB_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PART_MAX_SMEM));
    GB_CUDA(cudaFuncSetAttribute(k_splat_small<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem)));
    GB_CUDA(cudaFuncSetAttribute(k_splat_small<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem)));
    const int bytes = (int)sizeof(SplatSmem);
    GB_CUDA(cudaFuncSetAttribute(k_splat_tiles<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    GB_CUDA(cudaFuncSetAttribute(k_splat_tiles<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    GB_CUDA(cudaFuncSetAttribute(k_bsplat<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    GB_CUDA(cudaFuncSetAttribute(k_bsplat<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
}

} // namespace

void reserve_batch(gblod_renderer *r, const gblod_view *views, int n, const gblod_render_params &rp,
                   uint64_t record_capacity, cudaStream_t s)
{
    if (n < 1) fail(GBLOD_ERR_INVALID_ARG, "batch needs at least one view");
    const BatchPlan b = plan_batch(views, n, rp);
    const Allocator &A = r->A;
    const uint64_t rec_cap = record_capacity ? record_capacity : RECORD_BUDGET_DEFAULT;
    if (rec_cap > 0xFFFFFFFFull) fail(GBLOD_ERR_INVALID_ARG, "record capacity must stay below 2^32");
    r->b_views.ensure(A, (size_t)n * sizeof(ViewDev), s);
    r->b_frontA.ensure(A, b.nodes + 1, s);
    r->b_frontB.ensure(A, b.nodes + 1, s);
    r->b_sel.ensure(A, b.nodes + 1, s);
    r->b_counts.ensure(A, b.nodes + 1, s);
    r->b_pfx.ensure(A, b.nodes + 2, s);
    r->b_base.ensure(A, b.nodes + 1, s);
    r->b_lvl_cnt.ensure(A, b.max_levels + 3, s);
    r->b_tile_cnt.ensure(A, b.ntiles, s);
    r->b_tile_off.ensure(A, b.ntiles + 1, s);
    r->b_tile_cur.ensure(A, b.ntiles, s);
    r->b_item_cnt.ensure(A, b.ntiles, s);
    r->b_item_off.ensure(A, b.ntiles + 1, s);
    r->records.ensure(A, rec_cap, s);
    r->b_items.ensure(A, batch_items(b.ntiles, rec_cap), s);
    r->maxv.ensure(A, n, s);
    r->b_hist.ensure(A, batch_hist(b.ntiles) + 1, s);
    // scan temp for the largest scans of this batch
    scan_exclusive_u64(A, r->b_scan, reinterpret_cast<const uint64_t *>(r->b_counts.p),
                       reinterpret_cast<uint64_t *>(r->b_pfx.p), b.nodes + 1, nullptr, s);
    scan_exclusive_u32(A, r->b_scan, r->b_tile_cnt.p, r->b_tile_off.p, b.ntiles, nullptr, s);
    scan_exclusive_u32(A, r->b_scan, r->b_hist.p, r->b_hist.p, batch_hist(b.ntiles), nullptr, s);
    r->b_rec_cap = rec_cap;
    GB_CUDA(cudaStreamSynchronize(s));
}

void render_batch(gblod_renderer *r, const gblod_view *views, int n, const gblod_render_params &rp, cudaStream_t s)
{
    if (n < 1) fail(GBLOD_ERR_INVALID_ARG, "batch needs at least one view");
    BatchPlan b = plan_batch(views, n, rp);
    const Allocator &A = r->A;
    // scratch must have been reserved (no allocation here, so the call can be graph-captured)
    const uint64_t items_cap = batch_items(b.ntiles, r->b_rec_cap);
    // every buffer the call uses is looked at: one buffer's size says nothing of another's
    if (r->b_views.cap < (size_t)n * sizeof(ViewDev) || r->b_frontA.cap < b.nodes + 1 || r->b_frontB.cap < b.nodes + 1 ||
        r->b_sel.cap < b.nodes + 1 || r->b_counts.cap < b.nodes + 1 || r->b_pfx.cap < b.nodes + 2 ||
        r->b_base.cap < b.nodes + 1 || r->b_lvl_cnt.cap < b.max_levels + 3 || r->b_tile_cnt.cap < b.ntiles ||
        r->b_tile_off.cap < b.ntiles + 1 || r->b_tile_cur.cap < b.ntiles || r->b_item_cnt.cap < b.ntiles ||
        r->b_item_off.cap < b.ntiles + 1 || r->records.cap < r->b_rec_cap || r->b_items.cap < items_cap ||
        r->maxv.cap < (size_t)n || r->b_hist.cap < batch_hist(b.ntiles) + 1 || r->b_rec_cap == 0)
        fail(GBLOD_ERR_INVALID_ARG, "gblod_render_batch: call gblod_renderer_reserve_batch for this batch first");
    r->last_stream = s;
    r->last_was_lod = false;
    ViewDev *dv = reinterpret_cast<ViewDev *>(r->b_views.p);
    for (int c0 = 0; c0 < n; c0 += VIEWS_PER_CHUNK) {
        ViewChunk ch;
        ch.first = c0;
        ch.n = std::min(VIEWS_PER_CHUNK, n - c0);
        for (int i = 0; i < ch.n; ++i) ch.v[i] = b.host[c0 + i];
        launch(GBLOD_K_RENDER_OTHER, k_set_views, dim3(1), dim3(64), 0, s, ch, dv);
    }
    const unsigned G = (unsigned)persistent_blocks(4);
    GB_CUDA(cudaMemsetAsync(r->stats, 0, offsetof(FrameStatsDev, pixel_updates_total), s));
    GB_CUDA(cudaMemsetAsync(r->b_lvl_cnt.p, 0, (size_t)(b.max_levels + 3) * 4, s));
    const dim3 GV((unsigned)std::max(1, (int)G / n), (unsigned)n); // (blocks per view, views)
    launch(GBLOD_K_RENDER_OTHER, k_bzero, GV, dim3(256), 0, s, (const ViewDev *)dv);
    // R1 over (view, node) pairs
    uint32_t *nsel = r->b_lvl_cnt.p + b.max_levels + 1;
    if (b.reached <= SELECT_FLAT) {
        uint8_t *cls = reinterpret_cast<uint8_t *>(r->b_frontA.p);
        const uint32_t total = (uint32_t)b.reached;
        launch(GBLOD_K_SELECT_NODES, k_bclassify, dim3((total + 127) / 128), dim3(128), 0, s, (const ViewDev *)dv, n, total,
               cls);
        launch(GBLOD_K_SELECT_NODES, k_bselect_flat, dim3((total + RT - 1) / RT), dim3(RT), 0, s, (const ViewDev *)dv, n,
               total, (const uint8_t *)cls, r->b_sel.p, nsel);
    } else {
        unsigned long long *fin = r->b_frontA.p, *fout = r->b_frontB.p;
        launch(GBLOD_K_SELECT_NODES, k_bselect_init, dim3(1), dim3(256), 0, s, (const ViewDev *)dv, n, fin, r->b_lvl_cnt.p);
        for (uint32_t d = 0; d < b.deep; ++d) {
            launch(GBLOD_K_SELECT_NODES, k_bselect_level, dim3((unsigned)persistent_blocks(2)), dim3(RT), 0, s,
                   (const ViewDev *)dv, (const unsigned long long *)fin, (const uint32_t *)(r->b_lvl_cnt.p + d), fout,
                   r->b_lvl_cnt.p + d + 1, r->b_sel.p, nsel);
            std::swap(fin, fout);
        }
    }
    const uint32_t cap = (uint32_t)(b.nodes + 1);
    launch(GBLOD_K_SELECT_NODES, k_bsel_counts, dim3(G), dim3(256), 0, s, (const ViewDev *)dv,
           (const unsigned long long *)r->b_sel.p, (const uint32_t *)nsel, cap, r->b_counts.p);
    scan_exclusive_u64(A, r->b_scan, reinterpret_cast<const uint64_t *>(r->b_counts.p),
                       reinterpret_cast<uint64_t *>(r->b_pfx.p), cap, reinterpret_cast<uint64_t *>(&r->stats->points),
                       s);
    launch(GBLOD_K_SELECT_NODES, k_bsel_base, dim3(G), dim3(256), 0, s, (const ViewDev *)dv,
           (const unsigned long long *)r->b_sel.p, (const uint32_t *)nsel, (const unsigned long long *)r->b_pfx.p,
           r->b_base.p, r->stats);
    // R2: count, offsets, scatter
    const SrcBatch src{dv, r->b_sel.p, r->b_pfx.p, r->b_base.p, nsel, &r->stats->points};
    const int per_sm = batch_part(b.ntiles), kernel = b.host[0].P.kernel, count = (rp.flags & GBLOD_RENDER_COUNT_UPDATES) ? 1 : 0;
    const unsigned long long rec_cap = r->b_rec_cap;
    const dim3 tg((b.ntiles + 255) / 256);
    if (per_sm) {
        const unsigned GP = (unsigned)persistent_blocks(per_sm);
        const size_t smem = (size_t)b.ntiles * 4, nh = (size_t)b.ntiles * GP;
        launch(GBLOD_K_PROJECT_COUNT, k_bproject<false, true>, dim3(GP), dim3(RT), smem, s, src, r->b_hist.p, b.ntiles, kernel,
               (uint4 *)nullptr, 0ull, r->status, r->stats, 0);
        scan_exclusive_u32(A, r->b_scan, r->b_hist.p, r->b_hist.p, nh, r->b_hist.p + nh, s);
        launch(GBLOD_K_RENDER_OTHER, k_tiles_from_hist, tg, dim3(256), 0, s, b.ntiles, (uint32_t)GP, 0u, items_wanted(),
               (const uint32_t *)r->b_hist.p, (const uint32_t *)(r->b_hist.p + nh), r->b_tile_cnt.p, r->b_tile_off.p,
               r->b_item_cnt.p, (unsigned long long *)nullptr, 0u);
        launch(GBLOD_K_PROJECT_SCATTER, k_bproject<true, true>, dim3(GP), dim3(RT), smem, s, src, r->b_hist.p, b.ntiles, kernel,
               r->records.p, rec_cap, r->status, r->stats, count);
    } else {
        GB_CUDA(cudaMemsetAsync(r->b_tile_cnt.p, 0, (size_t)b.ntiles * 4, s));
        launch(GBLOD_K_PROJECT_COUNT, k_bproject<false, false>, dim3(G), dim3(RT), 0, s, src, r->b_tile_cnt.p, b.ntiles, kernel,
               (uint4 *)nullptr, 0ull, r->status, r->stats, 0);
        scan_exclusive_u32(A, r->b_scan, r->b_tile_cnt.p, r->b_tile_off.p, b.ntiles, r->b_tile_off.p + b.ntiles, s);
        launch(GBLOD_K_RENDER_OTHER, k_tile_items, tg, dim3(256), 0, s, b.ntiles, (const uint32_t *)r->b_tile_cnt.p,
               r->b_item_cnt.p, (unsigned long long *)nullptr);
        GB_CUDA(cudaMemcpyAsync(r->b_tile_cur.p, r->b_tile_off.p, (size_t)b.ntiles * 4, cudaMemcpyDeviceToDevice, s));
        launch(GBLOD_K_PROJECT_SCATTER, k_bproject<true, false>, dim3(G), dim3(RT), 0, s, src, r->b_tile_cur.p, b.ntiles, kernel,
               r->records.p, rec_cap, r->status, r->stats, count);
    }
    scan_exclusive_u32(A, r->b_scan, r->b_item_cnt.p, r->b_item_off.p, b.ntiles, r->b_item_off.p + b.ntiles, s);
    launch(GBLOD_K_RENDER_OTHER, k_bfill_items, dim3((b.ntiles + 255) / 256), dim3(256), 0, s, b.ntiles,
           (const ViewDev *)dv, n, (const uint32_t *)r->b_tile_cnt.p, (const uint32_t *)r->b_tile_off.p,
           (const uint32_t *)r->b_item_off.p, r->b_items.p, (uint32_t)items_cap, (unsigned long long)r->b_rec_cap,
           (const FrameStatsDev *)r->stats, r->status, per_sm ? items_wanted() : 0u);
    // R3: persistent over the items of all views
    launch(GBLOD_K_SPLAT, (rp.flags & GBLOD_RENDER_COUNT_UPDATES) ? k_bsplat<true> : k_bsplat<false>, dim3(G), dim3(RT),
           sizeof(SplatSmem), s, (const uint4 *)r->records.p, (const uint4 *)r->b_items.p,
           (const uint32_t *)(r->b_item_off.p + b.ntiles),
           (uint32_t)items_cap, strips_of(b.host[0].P.TW, b.host[0].P.TH), b.host[0].P.kernel, (const ViewDev *)dv,
           r->b_lvl_cnt.p + b.max_levels + 2, r->stats);
    // R4
    const dim3 GT((tone_blocks(b.npix) + (unsigned)n - 1) / (unsigned)n, (unsigned)n);
    if (rp.tone_auto) {
        GB_CUDA(cudaMemsetAsync(r->maxv.p, 0, (size_t)n * 8, s));
        launch(GBLOD_K_TONEMAP, k_bmax, GT, dim3(256), 0, s, (const ViewDev *)dv, r->maxv.p);
    }
    launch(GBLOD_K_TONEMAP, k_btonemap, GT, dim3(256), 0, s, (const ViewDev *)dv,
           (const unsigned long long *)r->maxv.p, rp.tone_auto ? 1 : 0);
}

void renderer_init(gblod_renderer *r, cudaStream_t s)
{
    ensure_tables();
    r->status = static_cast<unsigned *>(r->A.get(2 * sizeof(unsigned), s)); // and the splat's unit counter
    r->stats = static_cast<FrameStatsDev *>(r->A.get(sizeof(FrameStatsDev), s));
    GB_CUDA(cudaMemsetAsync(r->status, 0, 2 * sizeof(unsigned), s));
    GB_CUDA(cudaMemsetAsync(r->stats, 0, sizeof(FrameStatsDev), s));
    GB_CUDA(cudaStreamSynchronize(s));
}

void renderer_release(gblod_renderer *r)
{
    cudaStream_t s = r->last_stream;
    const Allocator &A = r->A;
    if (s) (void)cudaStreamSynchronize(s);
    A.put(r->status, 2 * sizeof(unsigned), s);
    A.put(r->stats, sizeof(FrameStatsDev), s);
    r->frontA.release(A, s); r->frontB.release(A, s); r->sel.release(A, s); r->lvl_cnt.release(A, s);
    r->sel_pfx.release(A, s); r->sel_base.release(A, s);
    r->tile_cnt.release(A, s); r->tile_off.release(A, s); r->tile_cur.release(A, s);
    r->cta_hist.release(A, s); r->cta_off.release(A, s);
    r->tile_cnt_s.release(A, s); r->tile_off_s.release(A, s); r->item_cnt_s.release(A, s); r->item_off_s.release(A, s);
    r->item_cnt.release(A, s); r->item_off.release(A, s);
    r->records.release(A, s); r->items.release(A, s); r->accum.release(A, s); r->maxv.release(A, s);
    r->pass_stats.release(A, s);
    r->b_views.release(A, s); r->b_frontA.release(A, s); r->b_frontB.release(A, s); r->b_sel.release(A, s);
    r->b_counts.release(A, s); r->b_pfx.release(A, s); r->b_base.release(A, s);
    r->b_lvl_cnt.release(A, s); r->b_tile_cnt.release(A, s); r->b_tile_off.release(A, s); r->b_tile_cur.release(A, s);
    r->b_item_cnt.release(A, s); r->b_item_off.release(A, s); r->b_hist.release(A, s); r->b_items.release(A, s);
    r->b_scan.buf.release(A, s);
    r->d_cams.release(A, s); r->d_rec.release(A, s); r->d_hist.release(A, s); r->d_off.release(A, s);
    r->d_cnt.release(A, s); r->d_items.release(A, s); r->d_big.release(A, s); r->d_odd.release(A, s);
    r->scan.buf.release(A, s);
}

void check_format(const gblod_octree *o, const gblod_render_params &rp)
{
    if (rp.point_format == GBLOD_POINTS_BLOCK16 ? !o->has_block16 : !o->has_float)
        fail(GBLOD_ERR_INVALID_ARG, rp.point_format == GBLOD_POINTS_BLOCK16
                                        ? "octree holds no 16-bit block codes (gblod_octree_quantize)"
                                        : "octree holds no fp32 points (dropped after quantisation)");
}

void check_image(const gblod_camera &c)
{
    if (c.width < 1 || c.height < 1 || c.width > 16384 || c.height > 16384)
        fail(GBLOD_ERR_INVALID_ARG, "camera width/height must be in 1..16384");
}

void render_lod(gblod_renderer *r, const gblod_octree *o, const gblod_camera &cam, const gblod_render_params &rp,
                uint8_t *image, uint64_t *accum, cudaStream_t s, uint32_t part, uint32_t n_parts)
{
    check_image(cam);
    check_format(o, rp);
    r->last_stream = s;
    r->last_was_lod = true;
    const Allocator &A = r->A;
    const Proj P = make_proj(cam, rp);
    GB_CUDA(cudaMemsetAsync(r->stats, 0, offsetof(FrameStatsDev, pixel_updates_total), s));
    const uint64_t nn = o->n_nodes;
    const int levels = o->depth_max + 1;
    r->sel.ensure(A, nn + 1, s);
    r->lvl_cnt.ensure(A, levels + 2, s);
    r->sel_pfx.ensure(A, nn + 2, s);
    r->sel_base.ensure(A, nn + 1, s);
    uint32_t *nsel = r->lvl_cnt.p + levels + 1;
    const bool q = rp.point_format == GBLOD_POINTS_BLOCK16;
    const gblod_node *nodes = q ? o->qnodes : o->nodes;
    const Frustum fr = make_frustum(cam, rp, o);
    int deep = 0;
    const uint64_t nr = reached_nodes(o, fr, deep);
    if (nr <= SELECT_ONE) {
        launch(GBLOD_K_SELECT_NODES, k_select_one, dim3(1), dim3((unsigned)SELECT_ONE), 0, s, nodes, (uint32_t)nr, fr, part,
               n_parts, r->sel.p, nsel, r->sel_pfx.p, r->sel_base.p, r->stats);
    } else {
        GB_CUDA(cudaMemsetAsync(r->lvl_cnt.p, 0, (size_t)(levels + 2) * 4, s));
        r->frontA.ensure(A, nn + 1, s);
        if (nr <= SELECT_FLAT) {
            uint8_t *cls = reinterpret_cast<uint8_t *>(r->frontA.p);
            launch(GBLOD_K_SELECT_NODES, k_classify, dim3((unsigned)((nr + 127) / 128)), dim3(128), 0, s, nodes, (uint32_t)nr,
                   fr, cls);
            launch(GBLOD_K_SELECT_NODES, k_select_flat, dim3((unsigned)((nr + RT - 1) / RT)), dim3(RT), 0, s, nodes,
                   (uint32_t)nr, (const uint8_t *)cls, r->sel.p, nsel, part, n_parts);
        } else {
            r->frontB.ensure(A, nn + 1, s);
            launch(GBLOD_K_SELECT_NODES, k_select_init, dim3(1), dim3(1), 0, s, r->frontA.p, r->lvl_cnt.p);
            uint32_t *fin = r->frontA.p, *fout = r->frontB.p;
            const unsigned G = (unsigned)persistent_blocks(2);
            for (int d = 0; d < deep; ++d) {
                launch(GBLOD_K_SELECT_NODES, k_select_level, dim3(G), dim3(RT), 0, s, nodes, fr,
                       (const uint32_t *)fin, (const uint32_t *)(r->lvl_cnt.p + d), fout, r->lvl_cnt.p + d + 1,
                       r->sel.p, nsel, part, n_parts);
                std::swap(fin, fout);
            }
        }
        launch(GBLOD_K_SELECT_NODES, k_sel_prefix, dim3(1), dim3(1024), 0, s, nodes, (const uint32_t *)r->sel.p,
               (const uint32_t *)nsel, r->sel_pfx.p, r->sel_base.p, r->stats);
    }
    SrcLOD src{o->pts4, o->hs, r->sel_pfx.p, r->sel_base.p, nsel, &r->stats->points, o->n_points};
    if (q) {
        SrcLODQ sq;
        static_cast<SrcLOD &>(sq) = src;
        sq.q4 = o->q4;
        sq.qw = o->qw;
        sq.qa = o->qa;
        sq.sel = r->sel.p;
        frame_common(r, sq, P, rp, image, accum, s);
    } else {
        frame_common(r, src, P, rp, image, accum, s);
    }
}

// R4 alone on a caller's accumulation image (e.g. the sum of the parts of a split frame).
void tonemap_image(gblod_renderer *r, const uint64_t *accum, int W, int H, const gblod_render_params &rp,
                   uint8_t *image, cudaStream_t s)
{
    const size_t npix = (size_t)W * H;
    r->maxv.ensure(r->A, 1, s);
    double lo = 0.0, hi = 0.0;
    if (rp.tone_auto) {
        GB_CUDA(cudaMemsetAsync(r->maxv.p, 0, 8, s));
        launch(GBLOD_K_TONEMAP, k_image_max, dim3(tone_blocks(npix)), dim3(256), 0, s,
               (const unsigned long long *)accum, npix, r->maxv.p);
    } else {
        lo = std::ldexp(rp.tone_lo, 32);
        hi = std::ldexp(rp.tone_hi, 32);
    }
    launch(GBLOD_K_TONEMAP, k_tonemap, dim3(tone_blocks(npix)), dim3(256), 0, s, (const unsigned long long *)accum,
           npix, (const unsigned long long *)r->maxv.p, rp.tone_auto ? 1 : 0, lo, hi, image);
}

void render_brute(gblod_renderer *r, const float *xyz, const float *mass, const float *h, uint64_t n,
                  const gblod_camera &cam, const gblod_render_params &rp, uint8_t *image, uint64_t *accum,
                  cudaStream_t s)
{
    check_image(cam);
    r->last_stream = s;
    r->last_was_lod = false;
    const Proj P = make_proj(cam, rp);
    GB_CUDA(cudaMemsetAsync(r->stats, 0, offsetof(FrameStatsDev, pixel_updates_total), s));
    const unsigned long long pts[1] = {n};
    GB_CUDA(cudaMemcpyAsync(&r->stats->points, pts, 8, cudaMemcpyHostToDevice, s));
    SrcFlat src{xyz, mass, h, n, n};
    frame_common(r, src, P, rp, image, accum, s);
}

void project_points(const float4 *pts4, const float *h, uint64_t n, const gblod_camera &cam,
                    const gblod_render_params &rp, int64_t *out, cudaStream_t s)
{
    const Proj P = make_proj(cam, rp);
    launch(GBLOD_K_RENDER_OTHER, k_project_debug, dim3(persistent_blocks(4)), dim3(256), 0, s, pts4, h, (size_t)n, P,
           reinterpret_cast<long long *>(out));
}

void morton_keys(const float *xyz, uint64_t n, const double lo[3], double side, uint64_t *keys, cudaStream_t s)
{
    launch(GBLOD_K_MORTON, k_morton_plain, dim3(persistent_blocks(4)), dim3(256), 0, s, xyz, (size_t)n, lo[0], lo[1],
           lo[2], 2097152.0 / side, keys);
}

} // namespace gb

// ------------------------------------------------------------------ fixed-scratch brute-force frame
// For callers that cannot allocate device memory: the scratch of a brute-force frame lives in one
// file-scope device array of fixed size, and nothing is allocated per call.  Host code must not
// pass g_noalloc_scratch itself to a kernel (in host code the name is only a stand-in for the
// device object); its device address is looked up with cudaGetSymbolAddress in the current device's
// context on every call.
namespace gb {
namespace {

constexpr size_t na_align(size_t b) { return (b + 255) / 256 * 256; }
constexpr size_t NA_TILES = GBLOD_NOALLOC_MAX_TILES;
constexpr size_t NA_RECORDS = GBLOD_NOALLOC_MAX_RECORDS;
constexpr size_t NA_ITEMS = NA_TILES + NA_RECORDS / ITEM;
constexpr size_t NA_SCAN_BYTES = 65536;
constexpr size_t NA_OFF_RECORDS = 0;
constexpr size_t NA_OFF_ITEMS = NA_OFF_RECORDS + na_align(NA_RECORDS * sizeof(uint4));
constexpr size_t NA_OFF_TILE_CNT = NA_OFF_ITEMS + na_align(NA_ITEMS * sizeof(uint4));
constexpr size_t NA_OFF_TILE_OFF = NA_OFF_TILE_CNT + na_align(NA_TILES * 4);
constexpr size_t NA_OFF_TILE_CUR = NA_OFF_TILE_OFF + na_align((NA_TILES + 1) * 4);
constexpr size_t NA_OFF_ITEM_CNT = NA_OFF_TILE_CUR + na_align(NA_TILES * 4);
constexpr size_t NA_OFF_ITEM_OFF = NA_OFF_ITEM_CNT + na_align(NA_TILES * 4);
constexpr size_t NA_OFF_SCAN = NA_OFF_ITEM_OFF + na_align((NA_TILES + 1) * 4);
constexpr size_t NA_OFF_STATS = NA_OFF_SCAN + na_align(NA_SCAN_BYTES);
constexpr size_t NA_OFF_STATUS = NA_OFF_STATS + na_align(sizeof(FrameStatsDev));
constexpr size_t NA_OFF_MAXV = NA_OFF_STATUS + na_align(2 * sizeof(unsigned)); // status, the splat's unit counter
constexpr size_t NA_BYTES = NA_OFF_MAXV + na_align(sizeof(unsigned long long));
static_assert(NA_BYTES == GBLOD_NOALLOC_SCRATCH_BYTES, "GBLOD_NOALLOC_SCRATCH_BYTES must match the layout");
// the two scans of NA_TILES counts find their temp space large enough and never allocate
static_assert(scan_temp_bytes(NA_TILES, sizeof(uint32_t)) <= NA_SCAN_BYTES, "scan temp exceeds its fixed region");

} // namespace
} // namespace gb

static __device__ __align__(256) unsigned char g_noalloc_scratch[gb::NA_BYTES];

namespace gb {
namespace {

// Device address of g_noalloc_scratch in the current device's context, looked up on every call
// (a lookup is cheap next to a frame, and a cached address would go stale if the context were
// torn down and created again).
unsigned char *noalloc_scratch()
{
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    check_cuda(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
    if (!p) fail(GBLOD_ERR_CUDA, "cudaGetSymbolAddress returned NULL");
    return static_cast<unsigned char *>(p);
}

} // namespace

gblod_status render_brute_noalloc(const float *xyz, const float *mass, const float *h, uint64_t n,
                                  const gblod_camera &cam, const gblod_render_params &rp, uint8_t *image,
                                  uint64_t *accum, cudaStream_t s)
{
    check_image(cam);
    if (!accum) fail(GBLOD_ERR_INVALID_ARG, "gblod_render_bruteforce_noalloc needs d_accum (caller-owned output)");
    const Proj P = make_proj(cam, rp);
    const size_t ntiles = (size_t)P.tiles_x * P.tiles_y;
    if (ntiles > NA_TILES)
        fail(GBLOD_ERR_INVALID_ARG, "gblod_render_bruteforce_noalloc: " + std::to_string(ntiles) +
                                        " screen tiles exceed the fixed maximum of " + std::to_string(NA_TILES));
    ensure_tables();
    unsigned char *base = noalloc_scratch();
    uint4 *records = reinterpret_cast<uint4 *>(base + NA_OFF_RECORDS);
    uint4 *items = reinterpret_cast<uint4 *>(base + NA_OFF_ITEMS);
    uint32_t *tile_cnt = reinterpret_cast<uint32_t *>(base + NA_OFF_TILE_CNT);
    uint32_t *tile_off = reinterpret_cast<uint32_t *>(base + NA_OFF_TILE_OFF);
    uint32_t *tile_cur = reinterpret_cast<uint32_t *>(base + NA_OFF_TILE_CUR);
    uint32_t *item_cnt = reinterpret_cast<uint32_t *>(base + NA_OFF_ITEM_CNT);
    uint32_t *item_off = reinterpret_cast<uint32_t *>(base + NA_OFF_ITEM_OFF);
    FrameStatsDev *stats = reinterpret_cast<FrameStatsDev *>(base + NA_OFF_STATS);
    unsigned *status = reinterpret_cast<unsigned *>(base + NA_OFF_STATUS);
    unsigned long long *maxv = reinterpret_cast<unsigned long long *>(base + NA_OFF_MAXV);
    // the scan helper finds its temp space already large enough and never allocates
    const Allocator none;
    ScanTmp scan;
    scan.buf.p = base + NA_OFF_SCAN;
    scan.buf.cap = NA_SCAN_BYTES;

    // the array keeps the previous call's contents: clear everything that must start at zero
    GB_CUDA(cudaMemsetAsync(tile_cnt, 0, ntiles * 4, s));
    GB_CUDA(cudaMemsetAsync(stats, 0, sizeof(FrameStatsDev), s));
    GB_CUDA(cudaMemsetAsync(status, 0, sizeof(unsigned), s));
    const SrcFlat src{xyz, mass, h, n, n};
    const unsigned G = (unsigned)persistent_blocks(4);
    const uint32_t nt = (uint32_t)ntiles;
    launch(GBLOD_K_PROJECT_COUNT, k_project_count<SrcFlat>, dim3(G), dim3(RT), 0, s, src, P, 0ull, ~0ull, tile_cnt,
           status, stats);
    scan_exclusive_u32(none, scan, tile_cnt, tile_off, ntiles, tile_off + ntiles, s);
    launch(GBLOD_K_RENDER_OTHER, k_tile_items, dim3((nt + 255) / 256), dim3(256), 0, s, nt,
           (const uint32_t *)tile_cnt, item_cnt, (unsigned long long *)nullptr);
    scan_exclusive_u32(none, scan, item_cnt, item_off, ntiles, item_off + ntiles, s);
    if (scan.buf.p != base + NA_OFF_SCAN) fail(GBLOD_ERR_CUDA, "scan temp left the fixed scratch");

    // one read-back into host stack memory (no pinned staging buffer is allocated)
    uint32_t counts[2] = {0, 0};
    unsigned long long amp_hi = 0, pairs64 = 0;
    unsigned st_bits = 0;
    GB_CUDA(cudaMemcpyAsync(&pairs64, &stats->pairs, 8, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaMemcpyAsync(&counts[0], tile_off + ntiles, 4, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaMemcpyAsync(&counts[1], item_off + ntiles, 4, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaMemcpyAsync(&amp_hi, &stats->amp_hi, 8, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaMemcpyAsync(&st_bits, status, 4, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    const uint32_t nitems = counts[1];
    if (pairs64 > NA_RECORDS || nitems > NA_ITEMS)
        fail(GBLOD_ERR_RANGE, "gblod_render_bruteforce_noalloc: the frame needs " + std::to_string(pairs64) +
                                  " (tile, splat) records, more than the fixed maximum of " +
                                  std::to_string(NA_RECORDS));
    const size_t npix = (size_t)P.W * P.H;
    unsigned long long *img = reinterpret_cast<unsigned long long *>(accum);
    GB_CUDA(cudaMemsetAsync(img, 0, npix * 8, s)); // before the scatter, which adds the small boxes
    GB_CUDA(cudaMemcpyAsync(tile_cur, tile_off, ntiles * 4, cudaMemcpyDeviceToDevice, s));
    launch(GBLOD_K_PROJECT_SCATTER, k_project_scatter<SrcFlat>, dim3(G), dim3(RT), 0, s, src, P, 0ull, ~0ull,
           tile_cur, records, img,
           (rp.flags & GBLOD_RENDER_COUNT_UPDATES) ? stats : (FrameStatsDev *)nullptr);
    launch(GBLOD_K_RENDER_OTHER, k_fill_items, dim3((nt + 255) / 256), dim3(256), 0, s, nt, nt,
           (const uint32_t *)tile_cnt, (const uint32_t *)tile_off, (const uint32_t *)item_off, ITEM, items, status + 1,
           (unsigned long long *)nullptr);
    launch_splat((rp.flags & GBLOD_RENDER_COUNT_UPDATES) != 0, records, items, nitems, status + 1, P, img, stats, s);
    if (image) {
        double lo = 0.0, hi = 0.0;
        if (rp.tone_auto) {
            GB_CUDA(cudaMemsetAsync(maxv, 0, 8, s));
            launch(GBLOD_K_TONEMAP, k_image_max, dim3(tone_blocks(npix)), dim3(256), 0, s,
                   (const unsigned long long *)img, npix, maxv);
        } else {
            lo = std::ldexp(rp.tone_lo, 32);
            hi = std::ldexp(rp.tone_hi, 32);
        }
        launch(GBLOD_K_TONEMAP, k_tonemap, dim3(tone_blocks(npix)), dim3(256), 0, s,
               (const unsigned long long *)img, npix, (const unsigned long long *)maxv, rp.tone_auto ? 1 : 0, lo, hi,
               image);
    }
    return (st_bits & ST_RANGE) || amp_hi ? GBLOD_ERR_RANGE : GBLOD_OK;
}

} // namespace gb
