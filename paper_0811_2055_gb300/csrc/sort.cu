// A2: stable LSD radix sort of (64-bit key, 32-bit value) pairs, 8-bit digits.
//
// Each pass is reduce-then-scan with no inter-CTA waiting: an upsweep writes one 256-bin
// digit histogram per 4096-key tile (digit-major), a device scan turns them into global
// offsets, and the scatter kernel re-reads its tile, ranks every key stably inside the tile
// (warp-striped rounds of 32 keys; per-warp running counters carry ranks across rounds, warps are
// ordered by a prefix over the tile) and writes it to its final place.  Digits that are the same for every key are skipped.
#include <mutex>
#include <vector>

#include "common.cuh"

namespace gb {
namespace {

constexpr int RS_THREADS = 512;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_ROUNDS = 8;
constexpr int RS_CTAS = 2; // resident scatter CTAs per SM
constexpr int RS_TILE = RS_THREADS * RS_ROUNDS; // 4096 keys

__global__ void k_diff_or(const uint64_t *keys, size_t n, unsigned long long *out)
{
    const uint64_t k0 = keys[0];
    uint64_t acc = 0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        acc |= keys[i] ^ k0;
    for (int d = 16; d > 0; d >>= 1) acc |= __shfl_xor_sync(0xffffffffu, acc, d);
    if ((threadIdx.x & 31) == 0 && acc) atomicOr(out, (unsigned long long)acc);
}

// One tile's digit histogram, in four copies (warps add to different ones)
constexpr int US_THREADS = 256;
__global__ void __launch_bounds__(US_THREADS) k_upsweep(const uint64_t *__restrict__ keys, size_t n, int shift,
                                                        uint32_t *__restrict__ hist, uint32_t ntiles)
{
    __shared__ uint32_t wh[4][256];
    for (int i = threadIdx.x; i < 4 * 256; i += US_THREADS) (&wh[0][0])[i] = 0u;
    const size_t base = (size_t)blockIdx.x * RS_TILE;
    uint64_t k[RS_TILE / US_THREADS];
#pragma unroll
    for (int r = 0; r < RS_TILE / US_THREADS; ++r) {
        const size_t i = base + (size_t)r * US_THREADS + threadIdx.x;
        k[r] = i < n ? keys[i] : 0ull;
    }
    __syncthreads();
    uint32_t *w = wh[(threadIdx.x >> 5) & 3];
#pragma unroll
    for (int r = 0; r < RS_TILE / US_THREADS; ++r)
        if (base + (size_t)r * US_THREADS + threadIdx.x < n) atomicAdd(&w[(uint32_t)(k[r] >> shift) & 255u], 1u);
    __syncthreads();
    const uint32_t d = threadIdx.x;
    hist[(size_t)d * ntiles + blockIdx.x] = wh[0][d] + wh[1][d] + wh[2][d] + wh[3][d];
}
static_assert(US_THREADS == 256 && RS_TILE % US_THREADS == 0, "one upsweep thread per digit");

// Scatter of one tile: keys are ranked stably inside the tile, placed with their values in shared
// memory in the tile's digit order, and written out by consecutive threads, so that each digit's run
// of keys (about 16 per tile and digit) goes to consecutive addresses.
//
// Ranking, one round of 32 keys of a warp: eight votes, one per bit, give every lane the lanes with the same
// digit, and a table of the warp's counts the keys before them.  All rounds' votes come first: they need
// no memory and run under the loads and the table reads of other warps.  (A mask table in shared memory
// instead of the votes: 30 cycles a round of the one shared-memory port, and the ranking bound the kernel;
// __match_any_sync loops over the distinct values, 260 cycles.)  512 threads x 8 keys, two CTAs per SM:
// 150M pairs, 3.6 GB moved, 1.84 ms a pass with match_any, 1.06 with the mask table, now 0.96 (a copy of the pairs
// 0.54; without ranking 0.67, three CTAs at 42 registers 1.19).
struct ScatterSmem {
    uint64_t k[RS_TILE];
    uint32_t v[RS_TILE];
    uint32_t wh[RS_WARPS][256]; // keys of each digit in this warp so far, then in the warps before
    uint32_t to[256];           // global position of a digit's first key, less its tile-local one
    uint32_t tstart[256];       // first tile-local position of each digit
    uint32_t wsum[RS_WARPS];
};

__global__ void __launch_bounds__(RS_THREADS, RS_CTAS)
    k_scatter(const uint64_t *__restrict__ kin, const uint32_t *__restrict__ vin, uint64_t *__restrict__ kout,
              uint32_t *__restrict__ vout, size_t n, int shift, const uint32_t *__restrict__ offs, uint32_t ntiles)
{
    extern __shared__ __align__(16) unsigned char sort_smem[];
    ScatterSmem &sm = *reinterpret_cast<ScatterSmem *>(sort_smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = gbd::lanemask_lt();
    const size_t tile0 = (size_t)blockIdx.x * RS_TILE;
    const size_t base = tile0 + (size_t)warp * (RS_ROUNDS * 32);
    const uint32_t nt = (uint32_t)min((size_t)RS_TILE, n - tile0); // keys in this tile
    const uint32_t off = threadIdx.x < 256 ? offs[(size_t)threadIdx.x * ntiles + blockIdx.x] : 0u;
    uint64_t k[RS_ROUNDS];
    uint32_t v[RS_ROUNDS];
    uint32_t rk[RS_ROUNDS];
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const size_t i = base + (size_t)r * 32 + lane;
        k[r] = i < n ? kin[i] : 0ull;
    }
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const size_t i = base + (size_t)r * 32 + lane;
        v[r] = i < n ? vin[i] : 0u;
    }
    for (int i = lane; i < 256; i += 32) sm.wh[warp][i] = 0u;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const uint32_t d = (uint32_t)(k[r] >> shift) & 255u;
        uint32_t peers = __ballot_sync(0xffffffffu, base + (size_t)r * 32 + lane < n);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const bool bit = (d >> b) & 1u;
            const uint32_t m = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? m : ~m;
        }
        rk[r] = peers;
    }
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const bool ok = base + (size_t)r * 32 + lane < n;
        const uint32_t d = (uint32_t)(k[r] >> shift) & 255u;
        const uint32_t peers = rk[r], cur = sm.wh[warp][d], before = __popc(peers & lt);
        rk[r] = cur + before;
        __syncwarp();
        if (ok && before == 0) sm.wh[warp][d] = cur + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // thread d < 256: exclusive prefix of digit d over the warps, and its keys in the tile; then the
    // exclusive scan of those over the digits
    uint32_t total = 0, incl = 0;
    if (threadIdx.x < 256) {
#pragma unroll
        for (int w = 0; w < RS_WARPS; ++w) {
            const uint32_t c = sm.wh[w][threadIdx.x];
            sm.wh[w][threadIdx.x] = total;
            total += c;
        }
        incl = total;
        for (int dd = 1; dd < 32; dd <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, incl, dd);
            if (lane >= dd) incl += o;
        }
        if (lane == 31) sm.wsum[warp] = incl;
    }
    __syncthreads();
    if (threadIdx.x < 256) {
        uint32_t start = incl - total;
        for (int w = 0; w < warp; ++w) start += sm.wsum[w];
        sm.tstart[threadIdx.x] = start;
        sm.to[threadIdx.x] = off - start; // modulo 2^32
    }
    __syncthreads();
    // keys and values in tile-local digit order
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
        if (base + (size_t)r * 32 + lane < n) {
            const uint32_t d = (uint32_t)(k[r] >> shift) & 255u;
            const uint32_t L = sm.tstart[d] + sm.wh[warp][d] + rk[r];
            sm.k[L] = k[r];
            sm.v[L] = v[r];
        }
    }
    __syncthreads();
#pragma unroll 4
    for (uint32_t L = threadIdx.x; L < nt; L += RS_THREADS) {
        const uint64_t key = sm.k[L];
        const uint32_t to = sm.to[(uint32_t)(key >> shift) & 255u] + L;
        kout[to] = key;
        vout[to] = sm.v[L];
    }
}

// the scatter's shared memory is above the 48 KB a launch may take without opting in (a device setting)
void set_scatter_smem()
{
    static std::mutex mu;
    static std::vector<int> done;
    int dev = 0;
    GB_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> g(mu);
    if ((int)done.size() <= dev) done.resize(dev + 1, 0);
    if (done[dev]) return;
    GB_CUDA(cudaFuncSetAttribute(k_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ScatterSmem)));
    done[dev] = 1;
}

} // namespace

void radix_sort_pairs(const Allocator &A, SortTmp &t, uint64_t **keys, uint32_t **vals, uint64_t *keys_alt,
                      uint32_t *vals_alt, size_t n, int key_bits, cudaStream_t s, HostStage &hs,
                      const unsigned long long *varying_bits)
{
    if (n <= 1) return;
    if (n >= (1ull << 32)) fail(GBLOD_ERR_INVALID_ARG, "radix sort: n must be below 2^32");
    const uint32_t ntiles = (uint32_t)((n + RS_TILE - 1) / RS_TILE);
    const size_t hist_n = (size_t)256 * ntiles;
    t.buf.ensure(A, hist_n * sizeof(uint32_t) + 256, s);
    uint32_t *hist = reinterpret_cast<uint32_t *>(t.buf.p);

    // which digits vary at all
    Scratch<unsigned long long> diff(A, varying_bits ? 0 : 1, s);
    if (!varying_bits) {
        GB_CUDA(cudaMemsetAsync(diff.p, 0, sizeof(unsigned long long), s));
        launch(GBLOD_K_SORT_UPSWEEP, k_diff_or, dim3(persistent_blocks(4)), dim3(256), 0, s, (const uint64_t *)*keys, n,
               diff.p);
        varying_bits = diff.p;
    }
    auto *hdiff = static_cast<unsigned long long *>(hs.get(sizeof(unsigned long long)));
    GB_CUDA(cudaMemcpyAsync(hdiff, varying_bits, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    const unsigned long long varying = *hdiff;

    set_scatter_smem();
    uint64_t *kin = *keys, *kout = keys_alt;
    uint32_t *vin = *vals, *vout = vals_alt;
    for (int shift = 0; shift < key_bits; shift += 8) {
        if (((varying >> shift) & 255ull) == 0ull) continue;
        launch(GBLOD_K_SORT_UPSWEEP, k_upsweep, dim3(ntiles), dim3(US_THREADS), 0, s, (const uint64_t *)kin, n, shift,
               hist, ntiles);
        scan_exclusive_u32(A, t.scan, hist, hist, hist_n, (uint32_t *)nullptr, s);
        launch(GBLOD_K_SORT_SCATTER, k_scatter, dim3(ntiles), dim3(RS_THREADS), sizeof(ScatterSmem), s, (const uint64_t *)kin,
               (const uint32_t *)vin, kout, vout, n, shift, (const uint32_t *)hist, ntiles);
        std::swap(kin, kout);
        std::swap(vin, vout);
    }
    *keys = kin;
    *vals = vin;
}

} // namespace gb
