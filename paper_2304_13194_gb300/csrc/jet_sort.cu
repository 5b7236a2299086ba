// Stable LSD radix sort of (64-bit key, int32 value) pairs, device-wide: per
// digit a histogram of every tile of kSortTile elements, then a scatter that keeps
// the input order among equal digits.  A warp takes consecutive elements of the
// tile and counts them digit by digit in its own counters, so that a tile has four
// block barriers, not five per 256 elements.  Up to kSortDirect tiles every tile
// adds the histograms up itself: two launches per digit; more tiles take an
// exclusive scan of all counts in digit-major order between them.  A digit of
// 131,072 pairs: 37 us in five launches before, 12 us in two now.
// Used where the method orders vertices by a key with ties broken by vertex id:
// the values enter in id order.
#include "jet_internal.cuh"

#include <algorithm>

namespace jet {

namespace {

constexpr int kSortItems = 8;                     // elements per thread and tile
constexpr int kSortTile = kTB * kSortItems;       // elements per tile
constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;

constexpr int kSortWarps = kTB / 32;
constexpr int64_t kSortDirect = 128;              // tiles up to which the scatter adds the histograms up
static_assert(kTB == kRadix, "one thread per digit");

// Digit histogram of each tile: hist[tile * kRadix + d] (DIRECT) or hist[d * ntiles + tile].
template <bool DIRECT>
__global__ void __launch_bounds__(kTB) k_sort_hist(const uint64_t *key, int64_t n, int shift, int64_t ntiles,
                                                   int64_t *hist) {
    __shared__ int32_t h[kRadix];
    h[threadIdx.x] = 0;
    __syncthreads();
    pdl_enter();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    uint64_t k[kSortItems];
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const int64_t e = base + (int64_t)i * kTB + threadIdx.x;
        k[i] = e < n ? key[e] : 0;
    }
#pragma unroll
    for (int i = 0; i < kSortItems; ++i)
        if (base + (int64_t)i * kTB + threadIdx.x < n) atomicAdd(&h[(int)((k[i] >> shift) & (kRadix - 1))], 1);
    __syncthreads();
    if (DIRECT) reinterpret_cast<int32_t *>(hist)[(int64_t)blockIdx.x * kRadix + threadIdx.x] = h[threadIdx.x];
    else hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

struct HistVal {
    const int64_t *hist;
    __device__ int64_t operator()(int64_t i) const { return hist[i]; }
};

// Scatter of one tile.  Warp w takes the elements base + w * 32 kSortItems + 32 i + lane:
// the rank of an element among the tile's equal digits keeps the input order.
template <bool DIRECT>
__global__ void __launch_bounds__(kTB) k_sort_scatter(const uint64_t *key_in, const int32_t *val_in, uint64_t *key_out,
                                                      int32_t *val_out, int64_t n, int shift, int64_t ntiles,
                                                      const int64_t *off) {
    __shared__ int32_t wcnt[kSortWarps][kRadix];   // per-warp digit counts, then the warps' offsets in the tile's digit
    __shared__ int64_t run[kRadix];                // first position of the tile's digit
    __shared__ long long sh[40];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) wcnt[w][threadIdx.x] = 0;
    __syncthreads();
    pdl_enter();
    const int64_t base = (int64_t)blockIdx.x * kSortTile + (int64_t)warp * 32 * kSortItems + lane;
    uint64_t k[kSortItems];
    int32_t v[kSortItems], pos[kSortItems];
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const int64_t e = base + 32 * i;
        k[i] = e < n ? key_in[e] : 0;
        v[i] = e < n ? val_in[e] : 0;
    }
    int64_t first = 0;                             // of digit threadIdx.x
    if (DIRECT) {
        const int32_t *hist = reinterpret_cast<const int32_t *>(off);
        int32_t before = 0, all = 0;
#pragma unroll 16
        for (int t = 0; t < (int)ntiles; ++t) {
            const int32_t x = hist[t * kRadix + threadIdx.x];
            all += x;
            before += t < (int)blockIdx.x ? x : 0;
        }
        first = block_exscan_i64(all, sh, nullptr) + before;
    } else {
        first = off[(int64_t)threadIdx.x * ntiles + blockIdx.x];
    }
    run[threadIdx.x] = first;
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const int d = base + 32 * i < n ? (int)((k[i] >> shift) & (kRadix - 1)) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int leader = __ffs(peers) - 1;
        int32_t c = 0;
        if (d >= 0 && (int)lane == leader) {
            c = wcnt[warp][d];
            wcnt[warp][d] = c + __popc(peers);
        }
        pos[i] = __shfl_sync(0xffffffffu, c, leader) + __popc(peers & lt);
        __syncwarp();
    }
    __syncthreads();
    {
        int32_t acc = 0;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) {
            const int32_t c = wcnt[w][threadIdx.x];
            wcnt[w][threadIdx.x] = acc;
            acc += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        if (base + 32 * i >= n) continue;
        const int d = (int)((k[i] >> shift) & (kRadix - 1));
        const int64_t p = run[d] + wcnt[warp][d] + pos[i];
        key_out[p] = k[i];
        val_out[p] = v[i];
    }
}

}  // namespace

int bits_for(int64_t x) {
    int b = 0;
    while (b < 63 && (x >> b) != 0) ++b;
    return b;
}

size_t sort_scratch_bytes(int64_t n) {
    const size_t nn = (size_t)std::max<int64_t>(n, 1);
    const int64_t ntiles = (n + kSortTile - 1) / kSortTile;
    const int64_t nhist = std::max<int64_t>(ntiles, 1) * kRadix;
    auto a256 = [](size_t x) { return (x + 255) & ~size_t(255); };
    return 2 * a256(nn * 8) + 2 * a256(nn * 4) + 2 * a256((size_t)nhist * 8) +
           a256((size_t)(scan_tiles_for(nhist) + 1) * 8) + a256(16);
}

void sort_scratch_carve(char *p, int64_t n, SortScratch &s) {
    const size_t nn = (size_t)std::max<int64_t>(n, 1);
    const int64_t ntiles = (n + kSortTile - 1) / kSortTile;
    const int64_t nhist = std::max<int64_t>(ntiles, 1) * kRadix;
    auto a256 = [](size_t x) { return (x + 255) & ~size_t(255); };
    auto take = [&](size_t b) { char *r = p; p += a256(b); return r; };
    s.key[0] = reinterpret_cast<uint64_t *>(take(nn * 8));
    s.key[1] = reinterpret_cast<uint64_t *>(take(nn * 8));
    s.val[0] = reinterpret_cast<int32_t *>(take(nn * 4));
    s.val[1] = reinterpret_cast<int32_t *>(take(nn * 4));
    s.hist = reinterpret_cast<int64_t *>(take((size_t)nhist * 8));
    s.off = reinterpret_cast<int64_t *>(take((size_t)nhist * 8));
    s.scan = reinterpret_cast<int64_t *>(take((size_t)(scan_tiles_for(nhist) + 1) * 8));
    s.total = reinterpret_cast<int64_t *>(take(16));
}

int sort_pairs(Ctx &c, SortScratch &sc, int64_t n, int kbits, int *which) {
    cudaStream_t s = c.stream;
    *which = 0;
    if (n <= 0) return JET_OK;
    const int64_t ntiles = (n + kSortTile - 1) / kSortTile;
    const int64_t nhist = ntiles * kRadix;
    int cur = 0;
    for (int shift = 0; shift < kbits; shift += kRadixBits) {
        const uint64_t *kin = sc.key[cur];
        const int32_t *vin = sc.val[cur];
        if (ntiles <= kSortDirect) {
            JET_CUDA_TRY(launch_pdl(k_sort_hist<true>, (int)ntiles, kTB, 0, s, true, kin, n, shift, ntiles, sc.hist));
            JET_CUDA_TRY(launch_pdl(k_sort_scatter<true>, (int)ntiles, kTB, 0, s, true, kin, vin, sc.key[cur ^ 1], sc.val[cur ^ 1],
                                    n, shift, ntiles, (const int64_t *)sc.hist));
            c.launches += 2;
        } else {
            JET_CUDA_TRY(launch_pdl(k_sort_hist<false>, (int)ntiles, kTB, 0, s, true, kin, n, shift, ntiles, sc.hist));
            JET_TRY(device_exscan(HistVal{sc.hist}, nhist, sc.off, sc.total, sc.scan, s));
            JET_CUDA_TRY(launch_pdl(k_sort_scatter<false>, (int)ntiles, kTB, 0, s, true, kin, vin, sc.key[cur ^ 1],
                                    sc.val[cur ^ 1], n, shift, ntiles, (const int64_t *)sc.off));
            c.launches += 2 + scan_launches(nhist);
        }
        cur ^= 1;
    }
    *which = cur;
    return JET_OK;
}

}  // namespace jet
