// A4 + A5: density-weighted random subselection of every over-full node (octree paragraph:
// "simplified using a density-weighted random subselection ... until the same data is
// represented by only n points"), and the representatives' blocks.
//
// Every particle i of node c gets the key k_i = u_i (all masses equal) or the bits of
// E(u_i)/m_i (exponential race), u_i = Philox(seed; id_i, code_c); the node keeps the n_max
// smallest (k_i, id_i).  Per node this is a segmented radix select, all nodes at once:
//   hist     4096-element chunks histogram the elements' bins (shared memory); equal masses: the top
//            log2(B) key bits (B ~ count/128 bins, at most 4096).  Unequal masses: B logarithmic bins
//            around the expected threshold, of the key computed in fp32 -- FP64 runs at 1/64 of the fp32
//            rate, and the key's series takes some 50 FP64 operations.  Each element's bin goes to a
//            16-bit code, with a mark if the key's error could put it into the next bin.
//   find     per node, the bin b that holds rank n_max (an fp32 key errs by a factor below 1 + 2^-16, and so
//            does the threshold: an element whose bins, error included, all lie below b is kept, above b
//            dropped)
//   mark     from the codes alone: elements below set their bit in a per-node bitmap, the others of bin b
//            become candidates, with their exact key
//   resolve  per node, 8-bit radix rounds over the candidates' remaining (k, id) bits decide the last
//            n_max - kept members
//   write    a stable compaction of the bitmap writes the representatives in ascending (Morton
//            key, id) order.
// Keys are recomputed from the ids (counter-based generator) instead of being stored; where there is no
// memory for the codes, mark recomputes them too (Philox is the cost of either pass: 150M equal masses, mark
// 3.4 ms recomputed, 0.72 ms from codes; 1M unequal masses, hist + mark + resolve 1.73 ms in
// FP64, now 0.11).
#include <algorithm>

#include "lodmath.cuh"
#include "octree.cuh"

namespace gb {
namespace {

constexpr int ST = 256;          // threads per selection block
constexpr uint32_t CH = 4096;    // elements per chunk (multiple of 32 * 8 warps)
constexpr int ROUNDS = CH / ST;  // 16 words of 32 per warp

struct Cand {
    uint64_t key;
    uint32_t id;
    uint32_t rel;
};

struct RepInfo {
    const uint32_t *nodes;     // node index per rep slot
    const uint32_t *chunk_off; // first chunk of each rep slot (n_rep + 1 entries)
    const uint32_t *hoff;      // first histogram bin of each rep slot
    const uint8_t *logb;       // log2 bins
    const int16_t *bin0;       // unequal masses: the bits above bin_shift of the first bin's lower edge
    const float *rmean;        // unequal masses: 1 / mean mass
    const uint64_t *woff;      // first bitmap word of each rep slot
};

// key bits below a fine bin's, of 2^logb bins: 2^(logb - 4) of them an octave
__device__ __forceinline__ int bin_shift(int logb) { return 23 - (logb - 4); }

__global__ void k_sel_setup(uint32_t n_rep, const uint32_t *nodes, const uint32_t *ncount, const float *nw,
                            uint32_t n_max, int equal_mass, uint32_t *nchunks, uint32_t *nbins, uint8_t *logb,
                            int16_t *bin0, float *rmean, uint64_t *nwords)
{
    const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_rep) return;
    const uint32_t c = ncount[nodes[r]];
    nchunks[r] = (c + CH - 1) / CH;
    uint32_t lb = 0;
    if (equal_mass) {
        const uint32_t want = (c + 127) / 128;
        while (lb < 12 && (1u << lb) < want) ++lb; // at most 4096 bins: the chunk histogram stays in shared memory
    } else {
        // 16, 4 or 1 bins an octave of E m_mean / m_i around the expected threshold (see log_bin).  That of equal
        // masses, x, has n_max / c = 1 - exp(-x); unequal masses move it up (1 - exp(-x m) is concave in m): a little
        // as a rule, far where a few particles hold most of the mass.
        lb = c >= 4096 ? 8 : (c >= 64 ? 6 : 4);
        const float part = (float)n_max / (float)c;
        rmean[r] = 1.0f / (nw[nodes[r]] * part);
        bin0[r] = (int16_t)((int)(__float_as_uint(-log1pf(-fminf(part, 0.9999f))) >> bin_shift((int)lb)) - (1 << (lb - 2)));
    }
    logb[r] = (uint8_t)lb;
    nbins[r] = 1u << lb;
    nwords[r] = (c + 31) / 32;
}

__device__ __forceinline__ uint32_t find_slot(const uint32_t *chunk_off, uint32_t n_rep, uint32_t c)
{
    // largest r with chunk_off[r] <= c
    uint32_t lo = 0, hi = n_rep;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (chunk_off[mid] <= c)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

// What a block needs to know of its chunk, laid out once (blocks that looked it up through the node arrays,
// four dependent loads: 150M, mark 0.93 -> 0.72 ms, write 1.52 -> 1.43, and 1.28 with the warps' lists)
struct __align__(16) Chunk {
    uint32_t j0, len, start, r; // first element; elements; the first one's position in the node; rep slot
    uint64_t code, words;       // node code; first bitmap word
    int logb, bin0;
    float rmean;
    uint32_t node;
};

__global__ void k_sel_chunks(uint32_t n_chunks, uint32_t n_rep, SelectIn in, RepInfo R, Chunk *__restrict__ chunks)
{
    const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n_chunks) return;
    const uint32_t r = find_slot(R.chunk_off, n_rep, c), node = R.nodes[r], start = (c - R.chunk_off[r]) * CH;
    Chunk C;
    C.j0 = in.nfirst[node] + start;
    C.len = min(CH, in.ncount[node] - start);
    C.start = start;
    C.r = r;
    C.code = in.ncode[node];
    C.words = R.woff[r] + start / 32;
    C.logb = R.logb[r];
    C.bin0 = R.bin0[r];
    C.rmean = R.rmean[r];
    C.node = node;
    chunks[c] = C;
}

__device__ __forceinline__ Chunk load_chunk(const Chunk *chunks)
{
    static_assert(sizeof(Chunk) == 48, "three 16-byte loads");
    const uint4 *p = reinterpret_cast<const uint4 *>(chunks + blockIdx.x);
    union {
        uint4 q[3];
        Chunk c;
    } u;
#pragma unroll
    for (int i = 0; i < 3; ++i) u.q[i] = __ldg(p + i);
    return u.c;
}

__device__ __forceinline__ uint64_t sel_key(const SelectIn &in, uint32_t j, uint64_t code, uint64_t seed,
                                            int equal_mass, uint32_t &id)
{
    id = in.sid[j];
    const uint64_t u = gbd::node_draw(seed, code, id);
    if (equal_mass) return u;
    const double k = __ddiv_rn(gbd::neg_log_unit(u), (double)in.sm[j]);
    return (uint64_t)__double_as_longlong(k);
}

// An element's code: its bin, and bit 15 if the exact key may lie in the next one.  `mid` is the bin that
// counts it in the histogram.
constexpr uint32_t CODE_NEXT = 0x8000u, CODE_NONE = 0x7FFFu; // CODE_NONE: past the node's end, above every bin

// E(u) / m in fp32, m the mass over the node's mean, within a factor 1 + 2^-18 of the exact key: 1 - U is
// exact where U is near 1 (the smallest keys), so both forms keep their relative error (logf, log1pf: 2 ulp;
// four roundings more).  Masses lie in [2^-24, 2^24], so m and E / m are normal numbers, and __fdividef is
// good to 2 ulp.
__device__ __forceinline__ float fast_key(uint64_t u, float m)
{
    const uint64_t v = u >> 12;                                                   // U = (v + 1/2) 2^-52
    const float U = __ull2float_rn(2 * v + 1) * 0x1p-53f, V = __ull2float_rn((1ull << 53) - (2 * v + 1)) * 0x1p-53f;
    const float E = v >= (1ull << 51) ? -log1pf(-V) : -logf(U);
    return __fdividef(E, m);
}

// The bin of a scaled key, n = 2^logb of them from four octaves below the expected threshold on: 5 n / 8 fine ones (ten
// octaves), 3 n / 16 four times as wide (twelve), 3 n / 16 sixteen times as wide (48); the first and the last take
// what lies outside.  (Sixteen octaves of fine bins only: 10M particles of which 1,000 hold 2^24 of the others' mass
// each had their threshold past the last bin, so that every particle became a candidate, for one block to sort out:
// 78 ms, now 3.1.  From the next width on v grows faster than the line of that width, so the smallest is the bin.)
__device__ __forceinline__ uint32_t log_bin(float a, const Chunk &C)
{
    const int v = max((int)(__float_as_uint(a) >> bin_shift(C.logb)) - C.bin0, 0), n = 1 << C.logb;
    const int f = n / 8 * 5, w = n / 16 * 3;
    return (uint32_t)min(min(v, f + ((v - f) >> 2)), min(f + w + ((v - f - 4 * w) >> 4), n - 1));
}

__device__ __forceinline__ uint32_t sel_code(const SelectIn &in, uint32_t j, const Chunk &C, uint64_t seed,
                                             int equal_mass, uint32_t &mid)
{
    const uint64_t u = gbd::node_draw(seed, C.code, in.sid[j]);
    if (equal_mass) {
        mid = C.logb ? (uint32_t)(u >> (64 - C.logb)) : 0u;
        return mid;
    }
    const float a = fast_key(u, in.sm[j] * C.rmean);
    mid = log_bin(a, C);
    const uint32_t low = log_bin(a * (1.0f - 0x1p-16f), C), high = log_bin(a * (1.0f + 0x1p-16f), C);
    return low | (high != low ? CODE_NEXT : 0u);
}

// codes (may be null): n_chunks x CH
__global__ void __launch_bounds__(ST) k_sel_hist(SelectIn in, RepInfo R, const Chunk *chunks, uint64_t seed,
                                                 int equal_mass, uint32_t *hist, uint16_t *__restrict__ codes)
{
    __shared__ uint32_t sh[4096];
    const Chunk C = load_chunk(chunks);
    const int nb = 1 << C.logb; // <= 4096
    for (int i = threadIdx.x; i < nb; i += ST) sh[i] = 0u;
    __syncthreads();
    uint32_t *gh = hist + R.hoff[C.r];
    uint16_t *co = codes ? codes + (size_t)blockIdx.x * CH : nullptr;
    for (int k = 0; k < ROUNDS; ++k) {
        const uint32_t at = (uint32_t)k * ST + threadIdx.x;
        uint32_t code = CODE_NONE;
        if (at < C.len) {
            uint32_t mid;
            code = sel_code(in, C.j0 + at, C, seed, equal_mass, mid);
            atomicAdd(&sh[mid], 1u);
        }
        if (co) co[at] = (uint16_t)code;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += ST)
        if (sh[i]) atomicAdd(&gh[i], sh[i]);
}

// block exclusive scan of one u32 per thread; every thread gets the total
__device__ __forceinline__ uint32_t block_scan_u32(uint32_t v, uint32_t &tot)
{
    __shared__ uint32_t wsum[ST / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < ST / 32; ++w) {
        const uint32_t x = wsum[w];
        before += w < warp ? x : 0u;
        all += x;
    }
    __syncthreads();
    tot = all;
    return before + incl - v;
}

// the threshold's bin, and at most how many candidates there are: its elements, and with fp32 keys those
// of the two bins beside it whose error reaches it
__global__ void __launch_bounds__(ST) k_sel_find(RepInfo R, uint32_t n_max, int equal_mass, const uint32_t *hist,
                                                 uint32_t *tb, uint64_t *ccap)
{
    const uint32_t r = blockIdx.x;
    const uint32_t nb = 1u << R.logb[r];
    const uint32_t *h = hist + R.hoff[r];
    uint32_t run = 0;
    for (uint32_t base = 0; base < nb; base += ST) {
        const uint32_t i = base + threadIdx.x;
        const uint32_t hv = i < nb ? h[i] : 0u;
        uint32_t tot;
        const uint32_t ex = block_scan_u32(hv, tot);
        const uint32_t cum = run + ex;
        if (cum < n_max && n_max <= cum + hv) {
            tb[r] = i;
            ccap[r] = (uint64_t)hv + (equal_mass || i == 0 ? 0u : h[i - 1]) + (equal_mass || i + 1 >= nb ? 0u : h[i + 1]);
        }
        run += tot;
    }
}

// A thread takes 16 consecutive elements of the chunk: from their codes (two 16-byte loads), or computed
// (CODES false).  kept[r] counts a node's elements below the threshold's bin, chunk_sel a chunk's.
template <bool CODES>
__global__ void __launch_bounds__(ST) k_sel_mark(SelectIn in, const Chunk *chunks, uint64_t seed, int equal_mass,
                                                 const uint16_t *__restrict__ codes, const uint32_t *tb,
                                                 const uint64_t *cand_off, uint32_t *cursor, uint32_t *kept,
                                                 uint32_t *chunk_sel, Cand *cand, uint32_t *bitmap)
{
    static_assert(CH == ST * 16, "16 elements a thread");
    __shared__ uint32_t sum;
    if (threadIdx.x == 0) sum = 0u;
    const Chunk C = load_chunk(chunks);
    __syncthreads();
    const uint32_t b = tb[C.r], at = threadIdx.x * 16;
    uint32_t code[16];
    if (CODES) {
        const uint4 *p = reinterpret_cast<const uint4 *>(codes + (size_t)blockIdx.x * CH + at);
        const uint4 q0 = __ldg(p), q1 = __ldg(p + 1);
        const uint32_t w[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
#pragma unroll
        for (int k = 0; k < 16; ++k) code[k] = k & 1 ? w[k >> 1] >> 16 : w[k >> 1] & 0xFFFFu;
    } else {
#pragma unroll 4
        for (int k = 0; k < 16; ++k) {
            uint32_t mid;
            code[k] = at + k < C.len ? sel_code(in, C.j0 + at + k, C, seed, equal_mass, mid) : CODE_NONE;
        }
    }
    uint32_t below = 0, eq = 0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const uint32_t low = code[k] & CODE_NONE, high = low + (code[k] >> 15);
        below |= high < b ? 1u << k : 0u;
        eq |= low <= b && b <= high ? 1u << k : 0u;
    }
    // two threads' 16 bits are a bitmap word (the last may lie past the node's words)
    const uint32_t other = __shfl_down_sync(0xffffffffu, below, 1);
    if (!(threadIdx.x & 1) && at < C.len) bitmap[C.words + (at >> 5)] = below | other << 16;
    const uint32_t nk = __reduce_add_sync(0xffffffffu, __popc(below));
    if ((threadIdx.x & 31) == 0 && nk) atomicAdd(&sum, nk);
    if (eq) {
        Cand *cb = cand + cand_off[C.r];
        uint32_t to = atomicAdd(&cursor[C.r], (uint32_t)__popc(eq));
        while (eq) {
            const uint32_t i = at + (uint32_t)(__ffs(eq) - 1);
            eq &= eq - 1u;
            uint32_t id;
            const uint64_t key = sel_key(in, C.j0 + i, C.code, seed, equal_mass, id);
            cb[to++] = Cand{key, id, C.start + i};
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        chunk_sel[blockIdx.x] = sum;
        if (sum) atomicAdd(&kept[C.r], sum);
    }
}

// bits [sh, sh + nbits) of the 96-bit value (key << 32) | id
__device__ __forceinline__ uint32_t digit96(const Cand &c, int sh, int nbits)
{
    uint64_t v;
    if (sh >= 32)
        v = c.key >> (sh - 32);
    else
        v = (c.key << (32 - sh)) | (uint64_t)(c.id >> sh);
    return (uint32_t)(v & ((1ull << nbits) - 1ull));
}

// The candidates' members: their n_max - kept smallest (key, id).  Equal-mass candidates share their top
// logb key bits; keys of unequal masses start at the sign bit.
__global__ void __launch_bounds__(ST) k_sel_resolve(RepInfo R, uint32_t n_max, int equal_mass, const uint32_t *kept,
                                                    const uint32_t *ncand, const uint64_t *cand_off,
                                                    uint64_t cand_total, Cand *cand, uint32_t *bitmap,
                                                    uint32_t *chunk_sel)
{
    __shared__ uint32_t hist[256];
    __shared__ uint32_t s_b, s_cum, s_hb, s_cnt;
    const uint32_t r = blockIdx.x;
    uint32_t m = ncand[r], need = n_max - kept[r];
    Cand *A = cand + cand_off[r];
    Cand *B = cand + cand_total + cand_off[r];
    uint32_t *words = bitmap + R.woff[r], *sel = chunk_sel + R.chunk_off[r];
    auto keep = [&](uint32_t rel) {
        atomicOr(&words[rel >> 5], 1u << (rel & 31));
        atomicAdd(&sel[rel / CH], 1u);
    };
    int top = 96 - (equal_mass ? R.logb[r] : 0);
    while (need < m && top > 0) {
        const int nbits = top < 8 ? top : 8;
        const int sh = top - nbits;
        for (int i = threadIdx.x; i < 256; i += ST) hist[i] = 0u;
        if (threadIdx.x == 0) s_cnt = 0u;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < m; i += ST) atomicAdd(&hist[digit96(A[i], sh, nbits)], 1u);
        __syncthreads();
        // the digit that holds rank `need`
        uint32_t tot;
        const uint32_t hv = hist[threadIdx.x], cum = block_scan_u32(hv, tot);
        if (cum < need && need <= cum + hv) {
            s_b = threadIdx.x;
            s_cum = cum;
            s_hb = hv;
        }
        __syncthreads();
        const uint32_t b = s_b;
        if (s_hb < m) { // else every candidate has this digit
            for (uint32_t i = threadIdx.x; i < m; i += ST) {
                const Cand c = A[i];
                const uint32_t d = digit96(c, sh, nbits);
                if (d < b)
                    keep(c.rel);
                else if (d == b)
                    B[atomicAdd(&s_cnt, 1u)] = c;
            }
            Cand *t = A;
            A = B;
            B = t;
        }
        __syncthreads();
        need -= s_cum;
        m = s_hb;
        top = sh;
        __syncthreads();
    }
    // the remaining candidates are all kept (need == m), or, only possible with duplicate ids,
    // the first `need` of them
    for (uint32_t i = threadIdx.x; i < m && i < need; i += ST) keep(A[i].rel);
}
static_assert(ST == 256, "one thread per digit");

__global__ void __launch_bounds__(ST) k_sel_write(SelectIn in, const Chunk *chunks, const uint32_t *bitmap,
                                                  const uint32_t *chunk_pos)
{
    __shared__ uint32_t woff[ST / 32];
    __shared__ uint16_t kept[ST / 32][ROUNDS * 32];
    const Chunk C = load_chunk(chunks);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t nw = (C.len + 31) / 32;
    const uint32_t *words = bitmap + C.words;
    const uint32_t w0 = (uint32_t)warp * ROUNDS;
    const uint32_t mw = lane < ROUNDS && w0 + lane < nw ? words[w0 + lane] : 0u; // the warp's words, one a lane
    const uint32_t mine = __reduce_add_sync(0xffffffffu, __popc(mw));
    if (lane == 0) woff[warp] = mine;
    __syncthreads();
    uint32_t base = chunk_pos[blockIdx.x] - C.r * in.n_max; // every node before it keeps n_max
    for (int w = 0; w < warp; ++w) base += woff[w];
    if (!mine) return;
    const uint64_t pf = in.npfirst[C.node];
    const float wr = in.nw[C.node], sr = in.ns[C.node];
    // the warp's kept elements, in order, so that every lane of the copy has one and its stores are contiguous
    const uint32_t lt = gbd::lanemask_lt();
    uint16_t *list = kept[warp];
    uint32_t n = 0;
#pragma unroll
    for (int q = 0; q < ROUNDS; ++q) {
        const uint32_t W = __shfl_sync(0xffffffffu, mw, q);
        if ((W >> lane) & 1u) list[n + __popc(W & lt)] = (uint16_t)(q * 32 + lane);
        n += __popc(W);
    }
    __syncwarp();
    float hm = 0.0f;
    const uint32_t j0 = C.j0 + w0 * 32, end = base < in.n_max ? min(mine, in.n_max - base) : 0u;
#pragma unroll 4
    for (uint32_t k = lane; k < end; k += 32) {
        const uint64_t idx = pf + base + k;
        const uint32_t j = j0 + list[k];
        const float4 p = __ldg(&in.s4[j]);
        const float h = __fmul_rn(p.w, sr);
        in.pts4[idx] = make_float4(p.x, p.y, p.z, wr);
        in.hs[idx] = h;
        in.pt_src[idx] = j;
        hm = h > hm ? h : hm;
    }
    for (int d = 16; d > 0; d >>= 1) {
        const float o = __shfl_xor_sync(0xffffffffu, hm, d);
        hm = o > hm ? o : hm;
    }
    if (lane == 0 && hm > 0.0f) atomicMax(&in.nhmax[C.node], __float_as_uint(hm));
}

template <class T> T readback(const T *d, cudaStream_t s, HostStage &hs)
{
    T *h = static_cast<T *>(hs.get(sizeof(T)));
    GB_CUDA(cudaMemcpyAsync(h, d, sizeof(T), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    return *h;
}

} // namespace

void select_representatives(const Allocator &A, cudaStream_t s, HostStage &hs, ScanTmp &scan, const SelectIn &in,
                            const uint32_t *rep_nodes, uint32_t n_rep, uint32_t n_max, uint64_t seed,
                            int equal_mass, void *spare, size_t spare_bytes)
{
    uint32_t *nchunks, *chunk_off, *nbins, *hoff, *tot32;
    uint64_t *nwords, *woff, *tot64;
    uint8_t *logb;
    int16_t *bin0;
    float *rmean;
    const Scratch<unsigned char> per_rep =
        carve(A, s, {part(nchunks, n_rep), part(chunk_off, n_rep + 1), part(nbins, n_rep), part(hoff, n_rep), part(tot32, 2),
                     part(nwords, n_rep), part(woff, n_rep), part(tot64, 1), part(logb, n_rep), part(bin0, n_rep),
                     part(rmean, n_rep)});
    launch(GBLOD_K_BUILD_OTHER, k_sel_setup, dim3((n_rep + 255) / 256), dim3(256), 0, s, n_rep, rep_nodes, in.ncount,
           in.nw, n_max, equal_mass, nchunks, nbins, logb, bin0, rmean,
           nwords);
    scan_exclusive_u32(A, scan, nchunks, chunk_off, n_rep, chunk_off + n_rep, s);
    scan_exclusive_u32(A, scan, nbins, hoff, n_rep, tot32, s);
    scan_exclusive_u64(A, scan, nwords, woff, n_rep, tot64, s);
    uint32_t *h32 = static_cast<uint32_t *>(hs.get(16));
    uint64_t *h64 = reinterpret_cast<uint64_t *>(h32 + 2);
    GB_CUDA(cudaMemcpyAsync(h32, chunk_off + n_rep, 4, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaMemcpyAsync(h32 + 1, tot32, 4, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaMemcpyAsync(h64, tot64, 8, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    const uint32_t n_chunks = h32[0], n_bins = h32[1];
    const uint64_t total_words = *h64;

    RepInfo R{rep_nodes, chunk_off, hoff, logb, bin0, rmean, woff};
    Chunk *chunks;
    uint32_t *hist, *tb, *cursor, *kept, *bitmap, *chunk_sel, *chunk_pos;
    uint64_t *ccap, *cand_off;
    const Scratch<unsigned char> work =
        carve(A, s, {part(chunks, n_chunks), part(hist, n_bins), part(tb, n_rep), part(cursor, 2 * (size_t)n_rep),
                     part(ccap, n_rep), part(cand_off, n_rep), part(bitmap, total_words), part(chunk_sel, n_chunks),
                     part(chunk_pos, n_chunks)});
    kept = cursor + n_rep;
    launch(GBLOD_K_BUILD_OTHER, k_sel_chunks, dim3((n_chunks + 255) / 256), dim3(256), 0, s, n_chunks, n_rep, in, R,
           chunks);
    uint16_t *codes = (size_t)n_chunks * CH * sizeof(uint16_t) <= spare_bytes ? static_cast<uint16_t *>(spare) : nullptr;
    GB_CUDA(cudaMemsetAsync(hist, 0, (size_t)n_bins * 4, s));
    GB_CUDA(cudaMemsetAsync(cursor, 0, 2 * (size_t)n_rep * 4, s));
    launch(GBLOD_K_SEL_HIST, k_sel_hist, dim3(n_chunks), dim3(ST), 0, s, in, R, (const Chunk *)chunks, seed,
           equal_mass, hist, codes);
    launch(GBLOD_K_BUILD_OTHER, k_sel_find, dim3(n_rep), dim3(ST), 0, s, R, n_max, equal_mass, (const uint32_t *)hist,
           tb, ccap);
    scan_exclusive_u64(A, scan, ccap, cand_off, n_rep, tot64, s);
    const uint64_t cand_total = readback(tot64, s, hs);
    Scratch<Cand> cand(A, 2 * (size_t)cand_total + 2, s);
    launch(GBLOD_K_SEL_MARK, codes ? k_sel_mark<true> : k_sel_mark<false>, dim3(n_chunks), dim3(ST), 0, s, in,
           (const Chunk *)chunks, seed, equal_mass, (const uint16_t *)codes, (const uint32_t *)tb, (const uint64_t *)cand_off, cursor, kept,
           chunk_sel, cand.p, bitmap);
    launch(GBLOD_K_BUILD_OTHER, k_sel_resolve, dim3(n_rep), dim3(ST), 0, s, R, n_max, equal_mass, (const uint32_t *)kept,
           (const uint32_t *)cursor, (const uint64_t *)cand_off, cand_total, cand.p, bitmap, chunk_sel);
    scan_exclusive_u32(A, scan, chunk_sel, chunk_pos, n_chunks, tot32, s);
    launch(GBLOD_K_SEL_WRITE, k_sel_write, dim3(n_chunks), dim3(ST), 0, s, in, (const Chunk *)chunks, (const uint32_t *)bitmap,
           (const uint32_t *)chunk_pos);
    const uint32_t n_kept = readback(tot32, s, hs); // modulo 2^32, like the positions it sums
    if (n_kept != (uint32_t)((uint64_t)n_rep * n_max))
        fail(GBLOD_ERR_CUDA, "subselection kept " + std::to_string(n_kept) + " points, expected " +
                                 std::to_string((uint64_t)n_rep * n_max));
}

} // namespace gb
