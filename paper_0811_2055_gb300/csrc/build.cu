// Octree build on the device (octree paragraph of the paper): A1 Morton keys, A2 radix sort,
// A3 the nodes of all levels from one pass over the sorted keys, exact node masses, leaf blocks and
// the cull data, from the leaves up.  The subselection (A4/A5) lives in select.cu.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "lodmath.cuh"
#include "octree.cuh"

namespace gb {
namespace {

constexpr uint32_t FL_LEAF = GBLOD_NODE_LEAF, FL_INTERNAL = GBLOD_NODE_INTERNAL, FL_LOSSY = GBLOD_NODE_LOSSY,
                   FL_REPS = GBLOD_NODE_REPS;

inline unsigned blocks_for(size_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// ------------------------------------------------------------------ A1 and input checks
// out (zeroed before): the complement of the smallest mass's bits, the largest one's bits, 1 if a mass is not allowed
__global__ void k_mass_check(const float *mass, size_t n, unsigned *out)
{
    unsigned lo = 0xFFFFFFFFu, hi = 0u, nbad = 0u;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float m = mass[i];
        if (!(m >= 0x1p-24f && m <= 0x1p+24f)) {
            nbad = 1u;
            continue;
        }
        const unsigned b = __float_as_uint(m);
        lo = b < lo ? b : lo;
        hi = b > hi ? b : hi;
    }
    for (int d = 16; d > 0; d >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, d));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, d));
        nbad |= __shfl_xor_sync(0xffffffffu, nbad, d);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(out, ~lo);
        atomicMax(out + 1, hi);
        if (nbad) atomicOr(out + 2, 1u);
    }
}

// Keys, the particles packed for the gather by sorted position (one aligned 16-byte read each instead
// of 12 + 4 bytes from two arrays), and the OR of every key's difference from particle 0's (which
// digits the sort must pass over).  pow2: the root cube starts at 0 and scale is a power of two in fp32
// range (the fp32 product is exact)
__global__ void k_morton(const float *__restrict__ xyz, const float *__restrict__ h,
                         const uint32_t *__restrict__ order, size_t n, double lx, double ly, double lz, double scale,
                         uint64_t *__restrict__ keys, uint32_t *__restrict__ vals, float4 *__restrict__ pack,
                         unsigned long long *diff, int pow2)
{
    const float sf = (float)scale;
    const uint64_t key0 = pow2 ? gbd::morton_key_pow2(xyz[0], xyz[1], xyz[2], sf)
                               : gbd::morton_key(xyz[0], xyz[1], xyz[2], lx, ly, lz, scale);
    uint64_t acc = 0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const size_t src = order ? (size_t)order[i] : i;
        const float x = xyz[3 * src], y = xyz[3 * src + 1], z = xyz[3 * src + 2];
        const uint64_t key = pow2 ? gbd::morton_key_pow2(x, y, z, sf) : gbd::morton_key(x, y, z, lx, ly, lz, scale);
        keys[i] = key;
        acc |= key ^ key0;
        if (!order) vals[i] = (uint32_t)i;
        pack[src] = make_float4(x, y, z, h[src]);
    }
    for (int d = 16; d > 0; d >>= 1) acc |= __shfl_xor_sync(0xffffffffu, acc, d);
    if ((threadIdx.x & 31) == 0 && acc) atomicOr(diff, (unsigned long long)acc);
}

__global__ void k_id_keys(const uint32_t *ids, size_t n, uint64_t *keys, uint32_t *vals)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        keys[i] = ids[i];
        vals[i] = (uint32_t)i;
    }
}

// Particles in sorted order: s4 = (x, y, z, h), sm = mass (written only for unequal masses: with one
// mass m0 for all the mass array is not read), sid = the caller's id (written only when the caller gave
// ids: otherwise it equals perm), mfix = the fixed-point mass (unequal masses only: else a node's
// exact mass is its count times m0's).  Bound by random 16-byte reads (150M: 7.2 ms from the
// caller's arrays, 36 ms of build + frame; 3.6 ms from the packed ones).
__global__ void k_gather_sorted(const float4 *__restrict__ pack, const float *__restrict__ mass,
                                const uint32_t *__restrict__ ids, const uint32_t *__restrict__ perm, size_t n,
                                float4 *__restrict__ s4, float *__restrict__ sm, uint32_t *__restrict__ sid,
                                U128 *__restrict__ mfix)
{
    // four independent elements per thread and iteration (each a coalesced sweep of the sorted
    // order), so that four random reads of the particle arrays are in flight at a time
    constexpr int GU = 4;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t j0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x; j0 < n; j0 += stride * GU) {
        uint32_t i[GU];
        float4 p[GU];
#pragma unroll
        for (int u = 0; u < GU; ++u) i[u] = j0 + u * stride < n ? perm[j0 + u * stride] : 0u;
#pragma unroll
        for (int u = 0; u < GU; ++u) p[u] = pack[i[u]];
#pragma unroll
        for (int u = 0; u < GU; ++u) {
            const size_t j = j0 + u * stride;
            if (j < n) {
                s4[j] = p[u];
                if (sid) sid[j] = ids[i[u]];
                if (mfix) {
                    const float m = mass[i[u]];
                    sm[j] = m;
                    mfix[j] = gbd::mass_fixed(m);
                }
            }
        }
    }
}

// ------------------------------------------------------------------ A3 levels
__device__ __forceinline__ uint32_t lower_bound_u64(const uint64_t *a, uint32_t lo, uint32_t hi, uint64_t v)
{
    while (lo < hi) {
        const uint32_t mid = lo + ((hi - lo) >> 1);
        if (a[mid] < v)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

struct NodeSoA {
    uint64_t *code;
    uint32_t *first, *count, *child_first, *child_count;
    int32_t *depth, *parent;
};

// The refined nodes of all levels come from one pass over the sorted keys: particle j is the first of a
// depth-d cell if it shares fewer than d octal digits with particle j - 1, and that cell holds more than
// n_max particles if j shares d digits or more with particle j + n_max.  Numbered by (depth, j) they are in the
// order of their nodes; their children (eight searches each, all levels at once) in that order are the
// nodes in level order.  A level at a time cost two launches, a scan and a wait for its node count: 1M
// particles, 11 levels 0.65 ms from the sorted particles to the node table, now 0.21.  Bound by the launches and
// two waits; 150M particles: by the pass over the keys, 0.28 ms.
constexpr int DEPTHS = GBLOD_MAX_DEPTH; // a refined node's depth is below this
constexpr uint32_t RB = 4096;           // positions per block
constexpr int RT_REF = 256;

// octal digits two keys that differ by the bits x share, of 21
__device__ __forceinline__ int shared_digits(uint64_t x) { return x ? (__clzll((long long)x) - 1) / 3 : 21; }

// depths (lo, hi] at which position j starts a refined node
__device__ __forceinline__ void refined_depths(const uint64_t *__restrict__ skey, size_t n, uint64_t n_max, size_t j,
                                               int &lo, int &hi)
{
    lo = hi = 0;
    if (j + n_max >= n) return; // every cell that starts here is small enough
    const uint64_t k = skey[j];
    // more digits shared with the later particle than with the one before: the differing bits are a smaller
    // number (nearly all positions end here)
    const uint64_t before = j ? k ^ skey[j - 1] : ~0ull, after = k ^ skey[j + n_max];
    if (after >= before) return;
    lo = j ? shared_digits(before) : -1;
    hi = max(lo, min(shared_digits(after), DEPTHS - 1));
}

// refined nodes by depth and block: hist[d * gridDim.x + block]
__global__ void __launch_bounds__(RT_REF) k_count_refined(const uint64_t *__restrict__ skey, size_t n, uint64_t n_max,
                                                          uint32_t *__restrict__ hist)
{
    __shared__ uint32_t cnt[DEPTHS];
    if (threadIdx.x < DEPTHS) cnt[threadIdx.x] = 0u;
    __syncthreads();
    const size_t base = (size_t)blockIdx.x * RB;
#pragma unroll 8
    for (uint32_t q = threadIdx.x; q < RB; q += RT_REF) {
        int lo, hi;
        refined_depths(skey, n, n_max, base + q, lo, hi);
        for (int d = lo + 1; d <= hi; ++d) atomicAdd(&cnt[d], 1u);
    }
    __syncthreads();
    if (threadIdx.x < DEPTHS) hist[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = cnt[threadIdx.x];
}

// first[i] = particle of refined node i; dfirst[d] = the first refined node of depth d (DEPTHS + 1 entries)
__global__ void __launch_bounds__(RT_REF) k_list_refined(const uint64_t *__restrict__ skey, size_t n, uint64_t n_max,
                                                         const uint32_t *__restrict__ off, uint32_t *__restrict__ first,
                                                         uint32_t *__restrict__ dfirst)
{
    __shared__ uint32_t bits[DEPTHS][RB / 32];   // positions of the block that start a refined node
    __shared__ uint16_t before[DEPTHS][RB / 32]; // those in the words before
    const uint32_t G = gridDim.x, total = off[(size_t)DEPTHS * G];
    if (blockIdx.x == 0 && threadIdx.x <= DEPTHS)
        dfirst[threadIdx.x] = threadIdx.x < DEPTHS ? off[(size_t)threadIdx.x * G] : total;
    uint32_t mine = 0;
    if (threadIdx.x < DEPTHS) {
        const size_t at = (size_t)threadIdx.x * G + blockIdx.x;
        mine = off[at + 1] - off[at];
    }
    if (!__syncthreads_or((int)mine)) return;
    for (int i = threadIdx.x; i < DEPTHS * (int)(RB / 32); i += RT_REF) (&bits[0][0])[i] = 0u;
    __syncthreads();
    const size_t base = (size_t)blockIdx.x * RB;
    for (uint32_t q = threadIdx.x; q < RB; q += RT_REF) {
        int lo, hi;
        refined_depths(skey, n, n_max, base + q, lo, hi);
        for (int d = lo + 1; d <= hi; ++d) atomicOr(&bits[d][q >> 5], 1u << (q & 31));
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int d = threadIdx.x >> 5; d < DEPTHS; d += RT_REF / 32) {
        uint32_t c[RB / 1024], sum = 0; // a lane's consecutive words
#pragma unroll
        for (int k = 0; k < (int)(RB / 1024); ++k) {
            c[k] = sum;
            sum += __popc(bits[d][lane * (RB / 1024) + k]);
        }
        uint32_t incl = sum;
        for (int s = 1; s < 32; s <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += o;
        }
#pragma unroll
        for (int k = 0; k < (int)(RB / 1024); ++k) before[d][lane * (RB / 1024) + k] = (uint16_t)(incl - sum + c[k]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < DEPTHS * (int)(RB / 32); i += RT_REF) {
        const int d = i / (int)(RB / 32), w = i % (int)(RB / 32);
        uint32_t m = bits[d][w], at = m ? off[(size_t)d * G + blockIdx.x] + before[d][w] : 0u;
        while (m) {
            first[at++] = (uint32_t)(base + (size_t)w * 32 + (uint32_t)(__ffs((int)m) - 1));
            m &= m - 1u;
        }
    }
}

__device__ __forceinline__ int depth_of(const uint32_t *__restrict__ dfirst, uint32_t i)
{
    int lo = 0, hi = DEPTHS;
    while (hi - lo > 1) { // the last depth whose first refined node is at or before i
        const int mid = (lo + hi) >> 1;
        if (dfirst[mid] <= i) lo = mid; else hi = mid;
    }
    return lo;
}

// Child t & 7 of refined node t >> 3: its particles [cf, cf + cc), and the flags to be scanned: 1 if there
// is one, 2^32 if it is refined itself
__global__ void k_children(uint32_t n_ref, const uint32_t *__restrict__ ref_first, const uint32_t *__restrict__ dfirst,
                           const uint64_t *__restrict__ skey, uint32_t n, uint32_t n_max, uint32_t *__restrict__ cc,
                           uint32_t *__restrict__ cf, uint64_t *__restrict__ flag)
{
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool on = t < (size_t)n_ref * 8; // whole groups of eight lanes
    const uint32_t i = on ? (uint32_t)(t >> 3) : 0u, o = (uint32_t)(t & 7), j = ref_first[i];
    const int d = depth_of(dfirst, i), sh = 60 - 3 * d;
    const uint64_t cp = ((skey[j] >> (63 - 3 * d)) << 3) | o;
    const uint32_t lo = o ? lower_bound_u64(skey, j, n, cp << sh) : j;
    uint32_t hi = __shfl_down_sync(0xffffffffu, lo, 1);
    if (o == 7) hi = lower_bound_u64(skey, lo, n, (cp + 1) << sh);
    if (!on) return;
    const uint32_t c = hi - lo;
    cc[t] = c;
    cf[t] = lo;
    flag[t] = (c ? 1ull : 0ull) | (c > n_max && d + 1 < DEPTHS ? 1ull << 32 : 0ull);
}

// Numbers from the scanned flags (pos): the node of child t is 1 + its low word, the refined node (if it is
// one) 1 + its high word.  node[i] = node of refined node i; level[d] = first node of depth d, level[DEPTHS + 2]
// entries from depth 0 on.
__global__ void k_number_nodes(uint32_t n_ref, const uint64_t *__restrict__ flag, const uint64_t *__restrict__ pos,
                               const uint32_t *__restrict__ dfirst, uint32_t *__restrict__ node,
                               unsigned long long *__restrict__ level)
{
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x, m = (size_t)n_ref * 8;
    if (t < m && flag[t] >> 32) node[1 + (uint32_t)(pos[t] >> 32)] = 1u + (uint32_t)pos[t];
    if (t == 0) node[0] = 0u;
    if (t <= DEPTHS) { // pos[m] is the total
        if (t == 0) level[0] = 0ull;
        level[t + 1] = 1ull + (uint32_t)pos[(size_t)dfirst[t] * 8];
    }
}

__global__ void k_emit_nodes(NodeSoA N, uint32_t n, uint32_t n_ref, const uint32_t *__restrict__ ref_first,
                             const uint32_t *__restrict__ dfirst, const uint64_t *__restrict__ skey,
                             const uint32_t *__restrict__ cc, const uint32_t *__restrict__ cf,
                             const uint64_t *__restrict__ flag, const uint64_t *__restrict__ pos,
                             const uint32_t *__restrict__ node)
{
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x, m = (size_t)n_ref * 8;
    auto children = [&](size_t x, bool refined, uint32_t i) {
        const uint32_t a = refined ? (uint32_t)pos[(size_t)i * 8] : 0u, b = refined ? (uint32_t)pos[(size_t)i * 8 + 8] : 0u;
        N.child_first[x] = refined ? 1u + a : 0u;
        N.child_count[x] = b - a;
    };
    if (t == 0) {
        N.code[0] = 1ull;
        N.first[0] = 0u;
        N.count[0] = n;
        N.depth[0] = 0;
        N.parent[0] = -1;
        children(0, n_ref > 0, 0u);
    }
    if (t >= m || !cc[t]) return;
    const uint32_t i = (uint32_t)(t >> 3), x = 1u + (uint32_t)pos[t];
    const int d = depth_of(dfirst, i);
    N.code[x] = (1ull << (3 * (d + 1))) | ((skey[ref_first[i]] >> (63 - 3 * d)) << 3) | (t & 7);
    N.first[x] = cf[t];
    N.count[x] = cc[t];
    N.depth[x] = d + 1;
    N.parent[x] = (int32_t)node[i];
    children(x, flag[t] >> 32 != 0, 1u + (uint32_t)(pos[t] >> 32));
}

// ------------------------------------------------------------------ node table
__global__ void k_node_classify(size_t nn, const uint32_t *count, const int32_t *depth, uint32_t n_max,
                                uint32_t *flags, uint64_t *pcount, uint32_t *isrep)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nn) return;
    const uint32_t c = count[i];
    uint32_t f;
    if (c > n_max)
        f = depth[i] < GBLOD_MAX_DEPTH ? (FL_INTERNAL | FL_REPS) : (FL_LOSSY | FL_REPS);
    else
        f = FL_LEAF;
    flags[i] = f;
    pcount[i] = (f & FL_REPS) ? n_max : c;
    isrep[i] = (f & FL_REPS) ? 1u : 0u;
}

__global__ void k_compact_reps(size_t nn, const uint32_t *isrep, const uint32_t *pos, uint32_t *out)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nn && isrep[i]) out[pos[i]] = (uint32_t)i;
}

// Node mass from the exclusive prefix of mass * 2^47; representative weight and h scale.
// Exact node masses: prefix differences of the fixed-point masses, or (prefix null: one mass m0
// for every particle) count times m0's fixed-point value.
__global__ void k_node_mass(size_t nn, size_t n, const uint32_t *first, const uint32_t *count, const uint32_t *flags,
                            const U128 *prefix, const U128 *total, float m0, uint32_t n_max, uint64_t *mlo,
                            uint64_t *mhi, float *w, float *s)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nn) return;
    U128 M;
    if (prefix) {
        const size_t b = first[i], e = b + count[i];
        const U128 a = prefix[b];
        const U128 z = e < n ? prefix[e] : *total;
        M = gbd::sub128(z, a);
    } else {
        const U128 f = gbd::mass_fixed(m0); // < 2^71, times a count < 2^32
        M.lo = f.lo * count[i];
        M.hi = f.hi * count[i] + __umul64hi(f.lo, (uint64_t)count[i]);
    }
    mlo[i] = M.lo;
    mhi[i] = M.hi;
    if (flags[i] & FL_REPS) {
        const double Md =
            __dmul_rn(__dadd_rn(__dmul_rn(__ull2double_rn(M.hi), 0x1p64), __ull2double_rn(M.lo)), 0x1p-47);
        w[i] = __double2float_rn(__ddiv_rn(Md, (double)n_max));
        const double t = __ddiv_rn((double)count[i], (double)n_max);
        s[i] = __double2float_rn(gbd::cube_root_ge1(t));
    } else {
        w[i] = 0.0f;
        s[i] = 1.0f;
    }
}

// Leaves: copy the sorted particles into the node block; every non-internal node: particle
// bounds; leaves: largest h.  One block per node (grid-stride), NaN coordinates are skipped.
__global__ void k_leaf_nodes(size_t nn, const uint32_t *__restrict__ flags, const uint32_t *__restrict__ first,
                             const uint32_t *__restrict__ count, const uint64_t *__restrict__ pfirst,
                             const float4 *__restrict__ s4, const float *__restrict__ sm, float m0, float4 *__restrict__ pts4,
                             float *__restrict__ hs, uint32_t *__restrict__ pt_src, float *__restrict__ bmin,
                             float *__restrict__ bmax, unsigned *__restrict__ hmax_bits)
{
    __shared__ float red[7][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (size_t node = blockIdx.x; node < nn; node += gridDim.x) {
        const uint32_t f = flags[node];
        if (f & FL_INTERNAL) continue;
        const uint32_t b = first[node], c = count[node];
        const uint64_t pf = pfirst[node];
        float mn0 = INFINITY, mn1 = INFINITY, mn2 = INFINITY, mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY;
        float hm = 0.0f;
        const bool leaf = (f & FL_LEAF) != 0;
        for (uint32_t k = threadIdx.x; k < c; k += blockDim.x) {
            const float4 p = s4[b + k];
            mn0 = fminf(mn0, p.x);
            mn1 = fminf(mn1, p.y);
            mn2 = fminf(mn2, p.z);
            mx0 = fmaxf(mx0, p.x);
            mx1 = fmaxf(mx1, p.y);
            mx2 = fmaxf(mx2, p.z);
            if (leaf) {
                const float h = p.w;
                pts4[pf + k] = make_float4(p.x, p.y, p.z, sm ? sm[b + k] : m0);
                hs[pf + k] = h;
                pt_src[pf + k] = b + k;
                hm = h > hm ? h : hm;
            }
        }
        for (int d = 16; d > 0; d >>= 1) {
            mn0 = fminf(mn0, __shfl_xor_sync(0xffffffffu, mn0, d));
            mn1 = fminf(mn1, __shfl_xor_sync(0xffffffffu, mn1, d));
            mn2 = fminf(mn2, __shfl_xor_sync(0xffffffffu, mn2, d));
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, d));
            mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, d));
            mx2 = fmaxf(mx2, __shfl_xor_sync(0xffffffffu, mx2, d));
            const float o = __shfl_xor_sync(0xffffffffu, hm, d);
            hm = o > hm ? o : hm;
        }
        if (lane == 0) {
            red[0][warp] = mn0; red[1][warp] = mn1; red[2][warp] = mn2;
            red[3][warp] = mx0; red[4][warp] = mx1; red[5][warp] = mx2;
            red[6][warp] = hm;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < nw; ++w) {
                mn0 = fminf(mn0, red[0][w]); mn1 = fminf(mn1, red[1][w]); mn2 = fminf(mn2, red[2][w]);
                mx0 = fmaxf(mx0, red[3][w]); mx1 = fmaxf(mx1, red[4][w]); mx2 = fmaxf(mx2, red[5][w]);
                hm = red[6][w] > hm ? red[6][w] : hm;
            }
            bmin[3 * node] = mn0; bmin[3 * node + 1] = mn1; bmin[3 * node + 2] = mn2;
            bmax[3 * node] = mx0; bmax[3 * node + 1] = mx1; bmax[3 * node + 2] = mx2;
            if (leaf) hmax_bits[node] = __float_as_uint(hm);
        }
        __syncthreads();
    }
}

// Cull radius and bounds of every node, from the leaves up: a thread per node that is not refined climbs as
// long as it is the last of a node's children to arrive, and takes that node's.  (A launch per level
// before: the same 37 us for 11 levels on the device, but the host had 11 launches to make.)  Children are read past L1, where a line may be older
// than their values.
__global__ void k_bottom_up(size_t nn, const uint32_t *__restrict__ flags, const uint32_t *__restrict__ child_first,
                            const uint32_t *__restrict__ child_count, const int32_t *__restrict__ parent, float *bmin,
                            float *bmax, const unsigned *__restrict__ hmax_bits, float *hcull, uint32_t *arrived)
{
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nn || (flags[t] & FL_INTERNAL)) return;
    hcull[t] = __uint_as_float(hmax_bits[t]);
    for (int i = parent[t], next; i >= 0; i = next) {
        const uint32_t k0 = child_first[i], kc = child_count[i];
        next = parent[i];
        __threadfence();
        if (atomicAdd(&arrived[i], 1u) + 1u < kc) return;
        __threadfence();
        float h = __uint_as_float(hmax_bits[i]);
        float mn0 = INFINITY, mn1 = INFINITY, mn2 = INFINITY, mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY;
#pragma unroll
        for (uint32_t q = 0; q < 8; ++q) { // all children's reads in flight (past the last: the last again)
            const uint32_t k = k0 + min(q, kc - 1u);
            mn0 = fminf(mn0, __ldcg(&bmin[3 * k])); mn1 = fminf(mn1, __ldcg(&bmin[3 * k + 1])); mn2 = fminf(mn2, __ldcg(&bmin[3 * k + 2]));
            mx0 = fmaxf(mx0, __ldcg(&bmax[3 * k])); mx1 = fmaxf(mx1, __ldcg(&bmax[3 * k + 1])); mx2 = fmaxf(mx2, __ldcg(&bmax[3 * k + 2]));
            const float hc = __ldcg(&hcull[k]);
            h = hc > h ? hc : h;
        }
        bmin[3 * i] = mn0; bmin[3 * i + 1] = mn1; bmin[3 * i + 2] = mn2;
        bmax[3 * i] = mx0; bmax[3 * i + 1] = mx1; bmax[3 * i + 2] = mx2;
        hcull[i] = h;
    }
}

struct PackIn {
    const uint64_t *code, *pfirst, *mlo, *mhi;
    const uint32_t *first, *count, *child_first, *child_count, *flags;
    const int32_t *depth, *parent;
    const float *hcull, *w, *s, *bmin, *bmax;
    uint32_t n_max;
};

__global__ void k_pack_nodes(size_t nn, PackIn P, gblod_node *out)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nn) return;
    gblod_node g;
    g.code = P.code[i];
    g.seg_first = P.first[i];
    g.point_first = P.pfirst[i];
    g.mass_lo = P.mlo[i];
    g.mass_hi = P.mhi[i];
    g.seg_count = P.count[i];
    g.point_count = (P.flags[i] & FL_REPS) ? P.n_max : P.count[i];
    g.child_first = P.child_first[i];
    g.child_count = P.child_count[i];
    g.depth = P.depth[i];
    g.flags = (int32_t)P.flags[i];
    g.parent = P.parent[i];
    g.pad = 0;
    g.h_cull = P.hcull[i];
    g.w_rep = P.w[i];
    g.s_rep = P.s[i];
    g.pad2 = 0.0f;
    for (int a = 0; a < 3; ++a) {
        g.bmin[a] = P.bmin[3 * i + a];
        g.bmax[a] = P.bmax[3 * i + a];
    }
    out[i] = g;
}

template <class T> T read1(const T *d, cudaStream_t s, HostStage &hs)
{
    T *h = static_cast<T *>(hs.get(sizeof(T)));
    GB_CUDA(cudaMemcpyAsync(h, d, sizeof(T), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    return *h;
}

} // namespace

void free_octree(gblod_octree *o)
{
    if (!o) return;
    cudaStream_t s = o->stream;
    o->A.put(o->nodes, o->n_nodes * sizeof(gblod_node), s);
    o->A.put(o->pts4, o->n_points * sizeof(float4), s);
    o->A.put(o->hs, o->n_points * sizeof(float), s);
    o->A.put(o->pt_src, o->n_points * sizeof(uint32_t), s);
    o->A.put(o->skey, o->n * sizeof(uint64_t), s);
    o->A.put(o->sidx, o->n * sizeof(uint32_t), s);
    o->A.put(o->q4, o->n_points * sizeof(ushort4), s);
    o->A.put(o->qw, o->n_points * sizeof(uint16_t), s);
    o->A.put(o->qa, 2 * o->n_nodes * sizeof(float4), s);
    o->A.put(o->qnodes, o->n_nodes * sizeof(gblod_node), s);
    delete o;
}

namespace {
struct BuildTemps {
    const Allocator &A;
    cudaStream_t s;
    ScanTmp scan;
    SortTmp sort;
    BuildTemps(const Allocator &a, cudaStream_t st) : A(a), s(st) {}
    ~BuildTemps()
    {
        scan.buf.release(A, s);
        sort.buf.release(A, s);
        sort.scan.buf.release(A, s);
    }
};
} // namespace

static void build_octree_impl(gblod_octree *o, const float *xyz, const float *mass, const float *h,
                                       const uint32_t *ids, uint64_t n, const gblod_build_params &p,
                                       const Allocator &A, cudaStream_t s, HostStage &hs, bool roomy);

gblod_octree *build_octree(const float *xyz, const float *mass, const float *h, const uint32_t *ids, uint64_t n,
                           const gblod_build_params &p, const Allocator &A, cudaStream_t s)
{
    // A roomy build takes up to about 94 bytes a particle with the octree, a lean one 66, and the library's pool keeps
    // what a build has taken.  Memory from a caller's allocator is spent leanly; from the pool leanly when roomy does
    // not fit, and above ROOMY_MAX particles, so that the pool never keeps more than 8 GB that a lean build would not
    // have taken (leanly the pool maps memory anew in every build: 181M particles 24.3 ms roomy, 31.8 lean).
    constexpr uint64_t ROOMY_MAX = 1ull << 28;
    HostStage hs;
    for (bool roomy = !A.has_hook && n <= ROOMY_MAX;; roomy = false) {
        gblod_octree *o = new gblod_octree();
        try {
            // the work arrays are given back, in stream order, under the last kernels
            build_octree_impl(o, xyz, mass, h, ids, n, p, A, s, hs, roomy);
            GB_CUDA(cudaStreamSynchronize(s));
            return o;
        } catch (const Error &e) {
            (void)cudaStreamSynchronize(s);
            free_octree(o);
            if (e.st != GBLOD_ERR_OOM || !roomy) throw;
        } catch (...) {
            (void)cudaStreamSynchronize(s);
            free_octree(o);
            throw;
        }
    }
}

static void build_octree_impl(gblod_octree *o, const float *xyz, const float *mass, const float *h,
                                       const uint32_t *ids, uint64_t n, const gblod_build_params &p,
                                       const Allocator &A, cudaStream_t s, HostStage &hs, bool roomy)
{
    BuildTemps tmp(A, s);
    ScanTmp &scan = tmp.scan;
    SortTmp &sort = tmp.sort;
    o->A = A;
    o->stream = s;
    o->n = n;
    o->n_max = p.n_max;
    o->seed = p.seed;
    for (int a = 0; a < 3; ++a) o->lo[a] = p.root_lo[a];
    o->side = p.root_side;
    if (n == 0) {
        o->level_first = {0};
        return;
    }
    const int T = 256;
    const unsigned G = (unsigned)persistent_blocks(8);
    float m0 = 0.0f; // the common mass when all are equal

    // masses: range and whether they are all equal; read with the sort's first counts (the sort's own read
    // uses the stage's first bytes)
    unsigned long long *diff;
    unsigned *mm;
    const Scratch<unsigned char> checks = carve(A, s, {part(diff, 1), part(mm, 3)});
    GB_CUDA(cudaMemsetAsync(checks.p, 0, checks.n, s));
    launch(GBLOD_K_BUILD_OTHER, k_mass_check, dim3(G), dim3(T), 0, s, mass, (size_t)n, mm);
    const unsigned *hm = static_cast<unsigned *>(hs.get(256)) + 16;
    GB_CUDA(cudaMemcpyAsync(const_cast<unsigned *>(hm), mm, 3 * sizeof(unsigned), cudaMemcpyDeviceToHost, s));

    // A1 + A2: keys in (key, id) order.  Roomy builds hold all work arrays of the sort and the sorted
    // particles in one block: the pool then finds the same few sizes free in every build (with an array
    // each, the next build's requests split the freed blocks and the pool maps memory anew: 5 ms at 150M).
    const size_t n16 = (n + 3) / 4 * 4; // keeps the parts of the block 16-byte aligned
    Scratch<float4> block(A, roomy ? 2 * n16 + n16 / 2 + n16 / 4 : 0, s);
    Scratch<uint64_t> keyA(A, n, s), keyB(A, roomy ? 0 : n, s);
    Scratch<uint32_t> valA(A, n, s), valB(A, roomy ? 0 : n, s);
    Scratch<float4> own_pack(A, roomy ? 0 : n, s);
    float4 *pack = roomy ? block.p + n16 : own_pack.p;
    uint64_t *kalt = roomy ? reinterpret_cast<uint64_t *>(block.p + 2 * n16) : keyB.p;
    uint32_t *valt = roomy ? reinterpret_cast<uint32_t *>(block.p + 2 * n16 + n16 / 2) : valB.p;
    uint64_t *keys = keyA.p;
    uint32_t *vals = valA.p;
    auto other_key = [&] { return keys == keyA.p ? kalt : keyA.p; };
    auto other_val = [&] { return vals == valA.p ? valt : valA.p; };
    const double scale = 2097152.0 / p.root_side;
    int sexp = 0;
    const int pow2 = p.root_lo[0] == 0.0 && p.root_lo[1] == 0.0 && p.root_lo[2] == 0.0 &&
                     std::frexp(scale, &sexp) == 0.5 && sexp > -120 && sexp < 120 ? 1 : 0;
    if (ids) {
        launch(GBLOD_K_BUILD_OTHER, k_id_keys, dim3(G), dim3(T), 0, s, ids, (size_t)n, keys, vals);
        radix_sort_pairs(A, sort, &keys, &vals, other_key(), other_val(), n, 32, s, hs);
        // vals = input indices in id order; keys in that order
        uint64_t *kdst = other_key();
        launch(GBLOD_K_MORTON, k_morton, dim3(G), dim3(T), 0, s, xyz, h, (const uint32_t *)vals, (size_t)n,
               p.root_lo[0], p.root_lo[1], p.root_lo[2], scale, kdst, (uint32_t *)nullptr, pack, diff, pow2);
        keys = kdst;
    } else {
        launch(GBLOD_K_MORTON, k_morton, dim3(G), dim3(T), 0, s, xyz, h, (const uint32_t *)nullptr, (size_t)n,
               p.root_lo[0], p.root_lo[1], p.root_lo[2], scale, keys, vals, pack, diff, pow2);
    }
    radix_sort_pairs(A, sort, &keys, &vals, other_key(), other_val(), n, 63, s, hs, diff);
    if (n == 1) GB_CUDA(cudaStreamSynchronize(s)); // nothing to sort, no count read
    if (hm[2]) fail(GBLOD_ERR_RANGE, "gblod_build_lod: every mass must be finite and in [2^-24, 2^24]");
    const unsigned lightest = ~hm[0];
    o->equal_mass = lightest == hm[1] ? 1 : 0;
    std::memcpy(&m0, &lightest, sizeof(float));
    // keep the sorted keys and permutation in the octree
    if (keys == kalt && roomy) {
        GB_CUDA(cudaMemcpyAsync(keyA.p, keys, n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
        keys = keyA.p;
    }
    if (vals == valt && roomy) {
        GB_CUDA(cudaMemcpyAsync(valA.p, vals, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
        vals = valA.p;
    }
    uint64_t *skey = keys;
    uint32_t *sidx = vals;
    if (skey == keyA.p) keyA.release_ptr(); else keyB.release_ptr();
    if (sidx == valA.p) valA.release_ptr(); else valB.release_ptr();
    o->skey = skey;
    o->sidx = sidx;
    keyA.reset(); keyB.reset(); valA.reset(); valB.reset();

    // sorted particle arrays and fixed-point masses (with no caller ids the sorted ids are sidx;
    // with equal masses no sorted masses and no prefix of them are needed)
    Scratch<float4> own_s4(A, roomy ? 0 : n, s);
    float4 *s4 = roomy ? block.p : own_s4.p;
    Scratch<float> sm(A, o->equal_mass ? 1 : n, s);
    Scratch<uint32_t> sid(A, ids ? n : 1, s);
    Scratch<U128> mpre(A, o->equal_mass ? 1 : n, s), mtot(A, 1, s);
    launch(GBLOD_K_BUILD_OTHER, k_gather_sorted, dim3(G), dim3(T), 0, s, (const float4 *)pack, mass, ids,
           (const uint32_t *)sidx, (size_t)n, s4, sm.p, ids ? sid.p : (uint32_t *)nullptr,
           o->equal_mass ? (U128 *)nullptr : mpre.p);
    own_pack.reset();
    if (!o->equal_mass) scan_exclusive_u128(A, scan, mpre.p, mpre.p, n, mtot.p, s);
    const uint32_t *sorted_ids = ids ? sid.p : sidx;

    // A3: refined nodes, their children, the nodes in level order
    NodeSoA N;
    uint32_t *flags, *isrep, *reppos, *total;
    uint64_t *pcount, *pfirst, *ptotal, *mlo, *mhi;
    float *w, *sc, *hcull, *bmin, *bmax;
    unsigned *hmax; // largest h, then k_bottom_up's arrivals
    Scratch<unsigned char> node_mem;
    const uint32_t nb = (uint32_t)((n + RB - 1) / RB);
    uint32_t n_ref = 0;
    std::vector<uint64_t> level_first = {0, 1};
    {
        Scratch<uint32_t> roff(A, (size_t)DEPTHS * nb + 1, s), dfirst(A, DEPTHS + 1, s);
        if (n > p.n_max) {
            launch(GBLOD_K_BUILD_OTHER, k_count_refined, dim3(nb), dim3(RT_REF), 0, s, (const uint64_t *)skey, (size_t)n,
                   (uint64_t)p.n_max, roff.p);
            scan_exclusive_u32(A, scan, roff.p, roff.p, (size_t)DEPTHS * nb, roff.p + (size_t)DEPTHS * nb, s);
            n_ref = read1(roff.p + (size_t)DEPTHS * nb, s, hs);
        }
        const size_t m = (size_t)n_ref * 8;
        const unsigned mg = blocks_for(std::max<size_t>(m, DEPTHS + 1), T);
        uint32_t *rfirst, *node, *cc, *cf;
        uint64_t *flag, *pos;
        unsigned long long *level;
        const Scratch<unsigned char> ref_mem = carve(A, s, {part(rfirst, n_ref), part(node, n_ref), part(cc, m), part(cf, m),
                                                            part(flag, m), part(pos, m + 1), part(level, DEPTHS + 2)});
        if (n_ref) {
            launch(GBLOD_K_BUILD_OTHER, k_list_refined, dim3(nb), dim3(RT_REF), 0, s, (const uint64_t *)skey, (size_t)n,
                   (uint64_t)p.n_max, (const uint32_t *)roff.p, rfirst, dfirst.p);
            launch(GBLOD_K_BUILD_OTHER, k_children, dim3(blocks_for(m, T)), dim3(T), 0, s, n_ref,
                   (const uint32_t *)rfirst, (const uint32_t *)dfirst.p, (const uint64_t *)skey, (uint32_t)n, p.n_max,
                   cc, cf, flag);
            scan_exclusive_u64(A, scan, flag, pos, m, pos + m, s);
            launch(GBLOD_K_BUILD_OTHER, k_number_nodes, dim3(mg), dim3(T), 0, s, n_ref, (const uint64_t *)flag,
                   (const uint64_t *)pos, (const uint32_t *)dfirst.p, node, level);
            auto *hl = static_cast<unsigned long long *>(hs.get((DEPTHS + 2) * sizeof(unsigned long long)));
            GB_CUDA(cudaMemcpyAsync(hl, level, (DEPTHS + 2) * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
            GB_CUDA(cudaStreamSynchronize(s));
            // level[d + 1] = the first node of depth d + 1, up to the depth with no nodes left
            for (int d = 2; d < DEPTHS + 2 && hl[d] > level_first.back(); ++d) level_first.push_back(hl[d]);
        }
        const size_t nn = level_first.back();
        node_mem = carve(A, s, {part(N.code, nn), part(N.first, nn), part(N.count, nn), part(N.child_first, nn),
                                part(N.child_count, nn), part(N.depth, nn), part(N.parent, nn), part(flags, nn),
                                part(isrep, nn), part(reppos, nn), part(total, 1), part(pcount, nn), part(pfirst, nn),
                                part(ptotal, 1), part(mlo, nn), part(mhi, nn), part(w, nn), part(sc, nn), part(hcull, nn),
                                part(bmin, 3 * nn), part(bmax, 3 * nn), part(hmax, 2 * nn)});
        launch(GBLOD_K_BUILD_OTHER, k_emit_nodes, dim3(mg), dim3(T), 0, s, N, (uint32_t)n, n_ref,
               (const uint32_t *)rfirst, (const uint32_t *)dfirst.p, (const uint64_t *)skey, (const uint32_t *)cc,
               (const uint32_t *)cf, (const uint64_t *)flag, (const uint64_t *)pos, (const uint32_t *)node);
    }
    const size_t nn = level_first.back();
    o->n_nodes = nn;
    o->depth_max = (int)level_first.size() - 2;
    o->level_first = level_first;

    // classify, number the stored points, masses and representative parameters
    launch(GBLOD_K_BUILD_OTHER, k_node_classify, dim3(blocks_for(nn, T)), dim3(T), 0, s, nn,
           (const uint32_t *)N.count, (const int32_t *)N.depth, p.n_max, flags, pcount, isrep);
    scan_exclusive_u64(A, scan, pcount, pfirst, nn, ptotal, s);
    scan_exclusive_u32(A, scan, isrep, reppos, nn, total, s);
    uint64_t *hp = static_cast<uint64_t *>(hs.get(16));
    uint32_t *hr = reinterpret_cast<uint32_t *>(hp + 1);
    GB_CUDA(cudaMemcpyAsync(hp, ptotal, 8, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaMemcpyAsync(hr, total, 4, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    const uint64_t npts = *hp;
    const uint32_t n_rep = *hr;
    o->n_points = npts;
    launch(GBLOD_K_BUILD_OTHER, k_node_mass, dim3(blocks_for(nn, T)), dim3(T), 0, s, nn, (size_t)n,
           (const uint32_t *)N.first, (const uint32_t *)N.count, (const uint32_t *)flags,
           o->equal_mass ? (const U128 *)nullptr : (const U128 *)mpre.p, (const U128 *)mtot.p, m0, p.n_max, mlo,
           mhi, w, sc);
    mpre.reset();
    GB_CUDA(cudaMemsetAsync(hmax, 0, 2 * nn * sizeof(unsigned), s));

    o->pts4 = static_cast<float4 *>(A.get(npts * sizeof(float4), s));
    o->hs = static_cast<float *>(A.get(npts * sizeof(float), s));
    o->pt_src = static_cast<uint32_t *>(A.get(npts * sizeof(uint32_t), s));
    o->nodes = static_cast<gblod_node *>(A.get(nn * sizeof(gblod_node), s));

    // A4 + A5: representatives of every over-full node
    if (n_rep) {
        Scratch<uint32_t> reps(A, n_rep, s);
        launch(GBLOD_K_BUILD_OTHER, k_compact_reps, dim3(blocks_for(nn, T)), dim3(T), 0, s, nn,
               (const uint32_t *)isrep, (const uint32_t *)reppos, reps.p);
        SelectIn in{s4, sm.p, sorted_ids, N.code, N.first, N.count, pfirst, w, sc, hmax,
                    o->pts4, o->hs, o->pt_src, p.n_max};
        // the packed particles and the sort's buffers are done with: 28 bytes a particle for the codes
        select_representatives(A, s, hs, scan, in, reps.p, n_rep, p.n_max, p.seed, o->equal_mass,
                               roomy ? block.p + n16 : nullptr, roomy ? (n16 + n16 / 2 + n16 / 4) * sizeof(float4) : 0);
    }

    // leaves, bounds, cull radii
    launch(GBLOD_K_BUILD_OTHER, k_leaf_nodes, dim3((unsigned)std::min<size_t>(nn, 65535 * 4)), dim3(T), 0, s, nn,
           (const uint32_t *)flags, (const uint32_t *)N.first, (const uint32_t *)N.count,
           (const uint64_t *)pfirst, (const float4 *)s4, o->equal_mass ? (const float *)nullptr : (const float *)sm.p,
           m0, o->pts4, o->hs, o->pt_src, bmin, bmax, hmax);
    launch(GBLOD_K_BUILD_OTHER, k_bottom_up, dim3(blocks_for(nn, T)), dim3(T), 0, s, nn, (const uint32_t *)flags,
           (const uint32_t *)N.child_first, (const uint32_t *)N.child_count, (const int32_t *)N.parent, bmin, bmax,
           (const unsigned *)hmax, hcull, hmax + nn);
    PackIn P{N.code, pfirst, mlo, mhi, N.first, N.count, N.child_first, N.child_count, flags,
             N.depth, N.parent, hcull, w, sc, bmin, bmax, p.n_max};
    launch(GBLOD_K_BUILD_OTHER, k_pack_nodes, dim3(blocks_for(nn, T)), dim3(T), 0, s, nn, P, o->nodes);
    o->bytes = nn * sizeof(gblod_node) + npts * (sizeof(float4) + sizeof(float) + sizeof(uint32_t)) +
               n * (sizeof(uint64_t) + sizeof(uint32_t));
}

} // namespace gb
