// Coarsening (Sec. 3.1): heavy-edge matching, coarse mapping, edge
// contraction (Alg. 2), projection (Alg. 1 ProjectPartition) and the greedy
// initial partition of the coarsest graph (Alg. 1 InitialPartition).
//
// Matching is a deterministic handshake: every unmatched vertex proposes its
// heaviest unmatched neighbour (ties: smaller splitmix64 hash of the
// neighbour, then smaller id) and mutual proposals match, round after round.
// Contraction merges each coarse vertex's (at most two) fine rows, sorts the
// mapped neighbour ids and sums duplicate entries: rows of <= 32 entries in
// one thread (register bitonic network), up to 256 in one warp (bitonic sort in
// shared memory), up to 4,096 in one block (radix sort in shared memory) and longer
// rows together in one device-wide radix sort.
#include "jet_internal.cuh"

#include <algorithm>
#include <cstring>
#include <mutex>

namespace jet {

template <bool EW>
__device__ __forceinline__ int32_t cw(const DGraph &g, int64_t j) {
    if constexpr (EW) return __ldg(g.ew + j);
    else return 1;
}

// device_exscan over many tiles: exclusive scan of the tile sums (one block).
__global__ void __launch_bounds__(1024) k_scan_sums(int64_t *tile_sums, int64_t ntiles) {
    __shared__ long long sh[40];
    pdl_enter();
    long long carry = 0;
    for (int64_t t0 = 0; t0 < ntiles; t0 += blockDim.x) {
        int64_t t = t0 + threadIdx.x;
        long long x = t < ntiles ? tile_sums[t] : 0;
        long long tot = 0;
        long long ex = block_exscan_i64(x, sh, &tot);
        if (t < ntiles) tile_sums[t] = carry + ex;
        carry += tot;
    }
}

// Matching state between the rounds of the launched form.
struct HemCtl {
    int32_t stop;
    int32_t nbig, nhuge;     // rows in the lists of k_hem_start
    int32_t pad;
    int64_t added[64];
};

__device__ __forceinline__ uint64_t hem_hash(uint64_t seed, uint64_t salt, int32_t u) {
    return splitmix64(seed ^ salt ^ (uint64_t)(uint32_t)u);
}

__device__ __forceinline__ bool hem_skip(const HemCtl *hc, int r) {
    return r > 0 && (hc->stop || hc->added[r - 1] == 0);
}

// The best proposal so far of a lane, a group of lanes or a block: larger
// weight, then smaller hash (splitmix64 is one to one, so that no two neighbours
// tie and their ids need no look).
struct HemBest {
    int32_t u = -1, w = INT32_MIN;
    uint64_t h = ~0ull;
    __device__ __forceinline__ void take(bool ok, int32_t ou, int32_t ow, uint64_t oh) {   // ou >= 0 where ok; no branch
        const bool better = ok & ((ow > w) | ((ow == w) & (oh < h)) | (u < 0));
        u = better ? ou : u;
        w = better ? ow : w;
        h = better ? oh : h;
    }
    // over lanes that differ in the bits below `lanes` (a power of two); the whole warp calls it
    __device__ __forceinline__ void reduce(int lanes) {
        for (int o = lanes >> 1; o > 0; o >>= 1) {
            const int32_t ou = __shfl_xor_sync(0xffffffffu, u, o);
            const int32_t ow = __shfl_xor_sync(0xffffffffu, w, o);
            const uint64_t oh = __shfl_xor_sync(0xffffffffu, h, o);
            take(ou >= 0, ou, ow, oh);
        }
    }
};

// The heaviest unmatched neighbour over the entries first, first + step, ...
// < end of a row, U at a time (ids and weights, then their matched bits, in
// flight together); folds into best.  A bit per vertex instead of its mate: the
// gathers of a whole mesh level fit in L1, and a hub-heavy graph's mostly do.
template <bool EW, int U = 4>
__device__ __forceinline__ void hem_row(const DGraph &g, const uint32_t *matched, uint64_t seed, uint64_t salt,
                                        int64_t first, int64_t end, int64_t step, HemBest &best) {
    for (int64_t j0 = first; j0 < end; j0 += U * step) {
        int32_t u[U], w[U];
        bool open[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int64_t j = j0 + q * step;
            u[q] = j < end ? __ldg(g.adj + j) : -1;
            w[q] = j < end ? cw<EW>(g, j) : 0;
        }
#pragma unroll
        for (int q = 0; q < U; ++q) open[q] = u[q] >= 0 && !(matched[u[q] >> 5] >> (u[q] & 31) & 1u);
#pragma unroll
        for (int q = 0; q < U; ++q) best.take(open[q], u[q], w[q], hem_hash(seed, salt, u[q]));
    }
}

// The whole block's best (blockDim.x <= 1024); valid in thread 0.
__device__ __forceinline__ void hem_block_best(HemBest &best, HemBest *sh) {
    best.reduce(32);
    if (lane_id() == 0) sh[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x < 32) {
        best = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : HemBest{};
        best.reduce(32);
    }
    __syncthreads();
}

// ---- one cluster, all rounds in one launch ----
//
// Small levels are bound by launches (three per round) and by dependent trips to
// L2.  Here a cluster keeps a matched bit of every vertex in each block's shared
// memory; a round is: the block's unmatched vertices are listed, groups of lanes
// scan their rows against the local bits, one cluster barrier, mutual proposals
// match, one cluster barrier, and every block copies the other blocks' bits.
// Ends with the first round that matches nothing, as the launched form does.  Whole
// calls, launched form against this one: 4,096 vertices of degree 6 100 -> 79 us,
// 15,625 107 -> 87, 32,768 111 -> 105, 40,000 no gain; 4,000 of degree 32 125 -> 155,
// hence kHemClusterN and kHemClusterDeg.  A lane group takes a row whole, so that one
// long row holds a round up: R-MAT of two entries per vertex, scale 12 (longest row
// 367) 228 -> 516, scale 15 (1,431) 281 -> 708 against the rounds before both forms;
// with rows of up to 127 entries nothing lost (R-MAT s11, 2,048 vertices 1.29 times as
// fast), hence kHemClusterRow; and 32,768 vertices with 459,000 entries 253 -> 261,
// with 328,000 1.1 times as fast, hence kHemClusterNnz.
constexpr int kHemThreads = 1024;
constexpr int kHemSlice = 2048;             // vertices per block at most
constexpr int kHemCluster = 16;
constexpr int kHemClusterDeg = 16;          // entries per vertex at most, on average
constexpr int kHemClusterRow = 128;         // entries of a row at most
constexpr int64_t kHemClusterNnz = 400000;  // entries at most
static_assert(kHemClusterN == kHemSlice * kHemCluster, "slices cover the largest level");

__device__ __forceinline__ void hem_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <bool EW>
__global__ void __launch_bounds__(kHemThreads) k_hem_cluster(DGraph g, int32_t per, int lanes, int rounds, uint64_t seed,
                                                             uint64_t salt0, int32_t *mate, int32_t *prop) {
    __shared__ uint32_t bits[kHemClusterN / 32];     // matched, all vertices
    __shared__ uint32_t own[kHemSlice / 32];         // matched, this block's slice (read by the others)
    __shared__ int32_t act[kHemSlice];               // unmatched vertices
    __shared__ int s_act;
    pdl_enter();
    const int tid = threadIdx.x, n = g.n;
    const int v0 = (int)blockIdx.x * per, nv = max(0, min(per, n - v0));
    const int words = (n + 31) >> 5, wper = per >> 5;
    for (int i = tid; i < words; i += kHemThreads) bits[i] = 0;
    for (int i = tid; i < wper; i += kHemThreads) own[i] = 0;
    for (int i = tid; i < nv; i += kHemThreads) mate[v0 + i] = -1;
    if (tid == 0) s_act = 0;
    __syncthreads();
    const int groups = kHemThreads / lanes, gi = tid / lanes, gl = tid & (lanes - 1);
    for (int r = 0; r < rounds; ++r) {
        const uint64_t salt = salt0 + 0xD1B54A32D192ED03ULL * (uint64_t)(r + 1);
        for (int i0 = 0; i0 < nv; i0 += kHemThreads) {
            const int i = i0 + tid;
            const bool active = i < nv && !(own[i >> 5] >> (i & 31) & 1u);
            const int slot = warp_append(&s_act, active);
            if (active) act[slot] = v0 + i;
        }
        __syncthreads();
        const int ns = s_act;
        for (int a0 = 0; a0 < ns; a0 += groups) {
            const int a = a0 + gi;
            const int32_t v = a < ns ? act[a] : -1;
            HemBest best;
            if (v >= 0) hem_row<EW>(g, bits, seed, salt, g.xadj[v] + gl, g.xadj[v + 1], lanes, best);
            best.reduce(lanes);
            if (v >= 0 && gl == 0) prop[v] = best.u;
        }
        hem_cluster_sync();
        // every proposal names a vertex that was unmatched, so whose proposal is this round's
        for (int a = tid; a < ns; a += kHemThreads) {
            const int32_t v = act[a];
            const int32_t u = __ldcg(prop + v);
            if (u >= 0 && __ldcg(prop + u) == v) {
                mate[v] = u;
                atomicOr(&own[(v - v0) >> 5], 1u << ((v - v0) & 31));
            }
        }
        if (tid == 0) s_act = 0;
        hem_cluster_sync();
        int changed = 0;
        for (int i = tid; i < words; i += kHemThreads) {
            uint32_t a, x;
            asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(&own[i % wper])), "r"(i / wper));
            asm volatile("ld.shared::cluster.b32 %0, [%1];" : "=r"(x) : "r"(a) : "memory");
            changed |= x != bits[i];
            bits[i] = x;
        }
        if (!__syncthreads_or(changed)) break;   // the same outcome in every block
    }
    hem_cluster_sync();   // the others may still read this block's bits
}

// Blocks of the cluster form on this device (0: not available).
static int hem_cluster_blocks(int device) {
    static std::mutex mu;
    static int cache[256];   // blocks + 1
    if (device < 0 || device >= 256) return 0;
    std::lock_guard<std::mutex> lock(mu);
    if (cache[device]) return cache[device] - 1;
    int best = 0;
    if (cudaFuncSetAttribute(k_hem_cluster<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaFuncSetAttribute(k_hem_cluster<false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        for (int cs = kHemCluster; cs >= 4 && !best; cs /= 2) {
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3(cs);
            cfg.blockDim = dim3(kHemThreads);
            cudaLaunchAttribute la{};
            la.id = cudaLaunchAttributeClusterDimension;
            la.val.clusterDim.x = cs; la.val.clusterDim.y = 1; la.val.clusterDim.z = 1;
            cfg.attrs = &la;
            cfg.numAttrs = 1;
            int a = 0, b = 0;
            if (cudaOccupancyMaxActiveClusters(&a, k_hem_cluster<true>, &cfg) == cudaSuccess &&
                cudaOccupancyMaxActiveClusters(&b, k_hem_cluster<false>, &cfg) == cudaSuccess && a >= 1 && b >= 1)
                best = cs;
        }
    }
    cudaGetLastError();   // a refused query only closes this form
    cache[device] = best + 1;
    return best;
}

// ---- the launched form: two kernels per round over the whole GPU ----

// Unmatched everywhere; rows longer than kSmallDeg are listed: warp rows (up to
// kHugeDeg entries) in list, hub rows in hlist, one reservation per block each.
__global__ void __launch_bounds__(kTB) k_hem_start(DGraph g, int32_t *mate, uint32_t *matched, uint32_t *done, int32_t *list,
                                                   int32_t *hlist, HemCtl *hc) {
    __shared__ int cnt[2], base[2];
    const int32_t v = blockIdx.x * kTB + threadIdx.x;
    const int64_t d = v < g.n ? ld_xadj(g.xadj, (int64_t)v + 1) - ld_xadj(g.xadj, v) : 0;
    if (v < g.n) mate[v] = -1;
    if (v < g.n && (v & 31) == 0) { matched[v >> 5] = 0; done[v >> 5] = 0; }
    if (threadIdx.x < 2) cnt[threadIdx.x] = 0;
    __syncthreads();
    const bool big = d > kSmallDeg && d <= kHugeDeg, huge = d > kHugeDeg;
    const int s0 = warp_append(&cnt[0], big), s1 = warp_append(&cnt[1], huge);
    __syncthreads();
    if (threadIdx.x < 2) base[threadIdx.x] = cnt[threadIdx.x] ? atomicAdd(threadIdx.x ? &hc->nhuge : &hc->nbig, cnt[threadIdx.x]) : 0;
    __syncthreads();
    if (big) list[base[0] + s0] = v;
    if (huge) hlist[base[1] + s1] = v;
}

// One proposal round: prop[v] = the chosen neighbour or -1 for the vertices not
// done (matched, or without an unmatched neighbour in an earlier round, which stays
// so).  The first long_blocks blocks take the hub rows, one at a time, then the warp
// rows, one per warp; the others the short rows, one per thread: one launch instead
// of three, so that the kinds of row fill the GPU together.  Bound by the gathers and
// the hashes; the eight rounds on R-MAT s15 459 -> 195 us a call, s18 1309 -> 565.
template <bool EW>
__global__ void __launch_bounds__(kTB) k_hem_propose(DGraph g, const int32_t *bigv, const int32_t *hugev,
                                                     const uint32_t *matched, const uint32_t *done, int32_t *prop, uint64_t seed,
                                                     uint64_t salt, int r, int long_blocks, HemCtl *hc) {
    __shared__ HemBest sh[kTB / 32];
    pdl_enter();
    if (hem_skip(hc, r)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) hc->stop = 1;
        return;
    }
    if ((int)blockIdx.x >= long_blocks) {
        const int64_t v = (int64_t)((int)blockIdx.x - long_blocks) * kTB + threadIdx.x;
        if (v >= g.n) return;
        if (done[v >> 5] >> (v & 31) & 1u) return;
        const int64_t beg = ld_xadj(g.xadj, v), end = ld_xadj(g.xadj, v + 1);
        if (end - beg > kSmallDeg) return;
        HemBest best;
        hem_row<EW>(g, matched, seed, salt, beg, end, 1, best);
        prop[v] = best.u;
        return;
    }
    const int32_t nhuge = hc->nhuge, nbig = hc->nbig;
    for (int64_t t = blockIdx.x; t < nhuge; t += long_blocks) {
        const int32_t v = hugev[t];
        if (done[v >> 5] >> (v & 31) & 1u) continue;
        HemBest best;
        hem_row<EW, 8>(g, matched, seed, salt, ld_xadj(g.xadj, v) + threadIdx.x, ld_xadj(g.xadj, (int64_t)v + 1), kTB, best);
        hem_block_best(best, sh);
        if (threadIdx.x == 0) prop[v] = best.u;
    }
    const unsigned lane = lane_id();
    for (int64_t w = (int64_t)blockIdx.x * (kTB / 32) + (threadIdx.x >> 5); w < nbig; w += (int64_t)long_blocks * (kTB / 32)) {
        const int32_t v = bigv[w];
        if (done[v >> 5] >> (v & 31) & 1u) continue;
        HemBest best;
        hem_row<EW>(g, matched, seed, salt, ld_xadj(g.xadj, v) + lane, ld_xadj(g.xadj, (int64_t)v + 1), 32, best);
        best.reduce(32);
        if (lane == 0) prop[v] = best.u;
    }
}

// Mutual proposals match; a warp owns its 32 vertices' words.  A proposal names a
// vertex that was unmatched when the round began; that one's own is this round's, or
// -1 from an earlier one.
__global__ void __launch_bounds__(kTB) k_hem_match(int32_t n, int32_t *mate, uint32_t *matched, uint32_t *done,
                                                   const int32_t *prop, int r, HemCtl *hc) {
    __shared__ long long red[40];
    pdl_enter();
    if (hc->stop) return;
    long long c = 0;
    const int64_t n32 = ((int64_t)n + 31) / 32 * 32;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n32; v += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t before = done[v >> 5];
        const bool open = v < n && !(before >> (v & 31) & 1u);
        const int32_t u = open ? prop[v] : -1;
        const bool ok = u >= 0 && prop[u] == (int32_t)v;
        if (ok) { mate[v] = u; ++c; }
        const uint32_t now = __ballot_sync(0xffffffffu, ok), end = __ballot_sync(0xffffffffu, ok || (open && u < 0));
        if (end && lane_id() == 0) {
            if (now) matched[v >> 5] |= now;
            done[v >> 5] = before | end;
        }
    }
    c = block_sum_i64(c, red);
    if (threadIdx.x == 0 && c) atomic_add_i64(&hc->added[r], c);
}

int hem(Ctx &c, const DGraph &g, int64_t longest, uint64_t seed, int32_t level, int32_t rounds, int32_t *mate) {
    cudaStream_t s = c.stream;
    if (g.n == 0) return JET_OK;
    rounds = std::min(rounds, 64);
    const bool pdl = !(c.opt.flags & JET_FLAG_NO_PDL);
    const uint64_t salt0 = 0xD1B54A32D192ED03ULL * (uint64_t)(64 * (int64_t)level);
    DevBuf buf;
    const bool small = g.n <= kHemClusterN && g.nnz <= std::min(kHemClusterNnz, (int64_t)kHemClusterDeg * g.n) &&
                       longest >= 0 && longest <= kHemClusterRow;
    const int cs = small ? hem_cluster_blocks(c.device) : 0;
    if (cs > 0 && g.n <= cs * kHemSlice) {
        JET_TRY(dev_alloc(buf, (size_t)g.n * 4, s));
        int32_t *prop = buf.as<int32_t>();
        const int32_t per = ((g.n + cs - 1) / cs + 31) / 32 * 32;
        int lanes = 1;   // four entries in flight per lane
        while (lanes < 32 && (int64_t)lanes * 4 * g.n < g.nnz) lanes *= 2;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)cs);
        cfg.blockDim = dim3(kHemThreads);
        cfg.stream = s;
        cudaLaunchAttribute la{};
        la.id = cudaLaunchAttributeClusterDimension;
        la.val.clusterDim.x = cs; la.val.clusterDim.y = 1; la.val.clusterDim.z = 1;
        cfg.attrs = &la;
        cfg.numAttrs = 1;
        if (g.ew) JET_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_hem_cluster<true>, g, per, lanes, (int)rounds, seed, salt0, mate, prop));
        else JET_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_hem_cluster<false>, g, per, lanes, (int)rounds, seed, salt0, mate, prop));
        c.launches += 1;
        return JET_OK;   // mate is final once the stream passes here (the scratch is freed in stream order)
    }
    auto a256 = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t nb = a256((size_t)g.n * 4), mb = a256(((size_t)g.n + 31) / 32 * 4);
    JET_TRY(dev_alloc(buf, 3 * nb + 2 * mb + sizeof(HemCtl), s));
    int32_t *prop = buf.as<int32_t>();
    int32_t *bigv = reinterpret_cast<int32_t *>(buf.as<char>() + nb);
    int32_t *hugev = reinterpret_cast<int32_t *>(buf.as<char>() + 2 * nb);
    uint32_t *matched = reinterpret_cast<uint32_t *>(buf.as<char>() + 3 * nb);
    uint32_t *done = reinterpret_cast<uint32_t *>(buf.as<char>() + 3 * nb + mb);
    HemCtl *hc = reinterpret_cast<HemCtl *>(buf.as<char>() + 3 * nb + 2 * mb);
    JET_CUDA_TRY(cudaMemsetAsync(hc, 0, sizeof(HemCtl), s));
    const int gs = grid_for(g.n, kTB);
    k_hem_start<<<gs, kTB, 0, s>>>(g, mate, matched, done, bigv, hugev, hc);
    c.launches += 1;
    JET_CUDA_TRY(cudaGetLastError());
    // the rounds follow one another by programmatic launch (each kernel waits
    // for the previous one on the device before it reads anything)
    const int lb = std::min(num_sms() * 8, grid_for(g.n, kTB / 32));
    const int gm = std::min(num_sms() * 8, gs);
    for (int r = 0; r < rounds; ++r) {
        const uint64_t salt = salt0 + 0xD1B54A32D192ED03ULL * (uint64_t)(r + 1);
        auto kern = g.ew ? k_hem_propose<true> : k_hem_propose<false>;
        JET_CUDA_TRY(launch_pdl(kern, lb + gs, kTB, 0, s, pdl, g, (const int32_t *)bigv, (const int32_t *)hugev,
                                (const uint32_t *)matched, (const uint32_t *)done, prop, seed, salt, r, lb, hc));
        JET_CUDA_TRY(launch_pdl(k_hem_match, gm, kTB, 0, s, pdl, g.n, mate, matched, done, (const int32_t *)prop, r, hc));
        c.launches += 2;
    }
    return JET_OK;
}

// ---------------------------------------------------------------------------
// coarse mapping: representatives are unmatched vertices and the smaller id
// of each pair; C[v] = rank of v's representative
// ---------------------------------------------------------------------------
struct RepFlag {
    const int32_t *mate;
    __device__ int64_t operator()(int64_t v) const {
        int32_t m = mate[v];
        return (m < 0 || v < m) ? 1 : 0;
    }
};

__global__ void k_cmap(int32_t n, const int32_t *mate, const int64_t *cidx, int32_t *cmap, int32_t *crep) {
    pdl_enter();
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        int32_t m = mate[v];
        int64_t r = (m >= 0 && m < v) ? m : v;
        cmap[v] = (int32_t)cidx[r];
        if (r == v) crep[cidx[v]] = (int32_t)v;
    }
}

// Entries of coarse row c before merging; 0 past the last row, whose number only
// the device knows when the scan is launched.
struct RowBound {
    const int64_t *xadj;
    const int32_t *crep, *mate;
    const int64_t *nc;
    __device__ int64_t operator()(int64_t c) const {
        if (c >= *nc) return 0;
        int32_t r = crep[c];
        int32_t m = mate[r];
        int64_t b = xadj[r + 1] - xadj[r];
        if (m >= 0) b += xadj[(int64_t)m + 1] - xadj[m];
        return b;
    }
};

// Longest merged row sorted in shared memory by one block; longer rows go
// through the device-wide radix sort (a launch-shape choice).
#ifndef JET_SORT_SMEM
#define JET_SORT_SMEM 4096
#endif
constexpr int kSortSmem = JET_SORT_SMEM;

__host__ __device__ inline int64_t pow2ceil(int64_t x) {
    int64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

// Hub rows (bound > kSortSmem) are contracted through one device-wide radix
// sort of all their entries: HubBound gives each hub row's segment length
// (0 for the others), HubFlag its rank among the hub rows.
struct HubBound {
    const int32_t *crep, *mate;
    const int64_t *xadj;
    __device__ int64_t operator()(int64_t c) const {
        int32_t r = crep[c];
        int32_t m = mate[r];
        int64_t b = xadj[r + 1] - xadj[r];
        if (m >= 0) b += xadj[(int64_t)m + 1] - xadj[m];
        return b > kSortSmem ? b : 0;
    }
};
struct HubFlag {
    HubBound hb;
    __device__ int64_t operator()(int64_t c) const { return hb(c) > 0 ? 1 : 0; }
};

// What the host learns about a coarse level in one read.
struct LevelCount {
    int64_t nc;            // coarse vertices
    int64_t btotal;        // entries of all rows before merging
    int64_t htotal, nhub;  // entries and number of the hub rows
    int32_t rows[4];       // {warp rows, block rows, 16-entry thread rows, 32-entry thread rows}
    int32_t longest, pad;  // entries of the longest row before merging (up to kHemClusterN rows)
};

// The coarse rows sorted into classes by their bound (entries of the merged fine
// rows): <= 16 and <= 32 (one thread), <= kWarpSort (one warp), longer (one block,
// hub rows among them).  boff has an entry past the last row (nc < n for every
// level that is built; a level without a match is dropped).
constexpr int kWarpSort = 256;
__global__ void __launch_bounds__(kTB) k_row_classes(int32_t n, const int64_t *boff, LevelCount *lc, int32_t *warp_list,
                                                     int32_t *large_list, int32_t *t16_list, int32_t *t32_list) {
    __shared__ int cnt[4], base[4];
    pdl_enter();
    const int64_t nc = lc->nc;
    if (nc >= n) return;
    const int64_t rounded = (nc + kTB - 1) / kTB * kTB;
    for (int64_t c = (int64_t)blockIdx.x * kTB + threadIdx.x; c < rounded; c += (int64_t)gridDim.x * kTB) {
        if (threadIdx.x < 4) cnt[threadIdx.x] = 0;
        __syncthreads();
        const int64_t b = c < nc ? boff[c + 1] - boff[c] : -1;
        if (nc <= kHemClusterN) {   // the next level's matching asks for it
            const int32_t most = __reduce_max_sync(0xffffffffu, (int32_t)b);
            if (lane_id() == 0 && most > 0) atomicMax(&lc->longest, most);
        }
        const int cls = b < 0 ? -1 : b <= 16 ? 2 : b <= 32 ? 3 : b <= kWarpSort ? 0 : 1;
        int slot[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) slot[q] = warp_append(&cnt[q], cls == q);
        if (b > kSortSmem) {
            atomic_add_i64(&lc->htotal, b);
            atomic_add_i64(&lc->nhub, 1);
        }
        __syncthreads();
        if (threadIdx.x < 4) base[threadIdx.x] = cnt[threadIdx.x] ? atomicAdd(&lc->rows[threadIdx.x], cnt[threadIdx.x]) : 0;
        __syncthreads();
        if (cls == 0) warp_list[base[0] + slot[0]] = (int32_t)c;
        if (cls == 1) large_list[base[1] + slot[1]] = (int32_t)c;
        if (cls == 2) t16_list[base[2] + slot[2]] = (int32_t)c;
        if (cls == 3) t32_list[base[3] + slot[3]] = (int32_t)c;
        __syncthreads();
    }
}

// Gathers entry i (0 <= i < bound) of coarse row c: (C[u] << 32) | w.
template <bool EW>
__device__ __forceinline__ unsigned long long row_entry(const DGraph &g, const int32_t *cmap, int32_t r, int32_t m,
                                                        int64_t degr, int64_t i) {
    int64_t j = i < degr ? ld_xadj(g.xadj, r) + i : ld_xadj(g.xadj, m) + (i - degr);
    int32_t cu = cmap[__ldg(g.adj + j)];
    return ((unsigned long long)(uint32_t)cu << 32) | (uint32_t)cw<EW>(g, j);
}

// Rows of <= N entries (N = 16 or 32): one thread each (32 rows of a warp in
// flight together), the keys (C[u] << 32 | w) sorted by a bitonic network
// over registers, then one pass that adds up equal coarse neighbours and
// drops the row's own vertex.  Same output as the warp and block forms.
// counts[slot] rows in list.
template <bool EW, int N>
__global__ void __launch_bounds__(kTB) k_contract_thread(DGraph g, const int32_t *cmap, const int32_t *mate,
                                                       const int32_t *crep, const int32_t *list, const int32_t *counts,
                                                       const int64_t *boff, int32_t *tadj, int32_t *tw, int32_t *rowcnt) {
    pdl_enter();
    const int32_t nrows = counts[N == 16 ? 2 : 3];
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < nrows; w += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = list[w];
        const int32_t r = crep[c], m = mate[r];
        const int64_t r0 = ld_xadj(g.xadj, r), degr = ld_xadj(g.xadj, (int64_t)r + 1) - r0;
        int64_t m0 = 0, degm = 0;
        if (m >= 0) {
            m0 = ld_xadj(g.xadj, m);
            degm = ld_xadj(g.xadj, (int64_t)m + 1) - m0;
        }
        const int64_t bound = degr + degm;
        unsigned long long key[N];
#pragma unroll
        for (int t = 0; t < N; ++t) {
            key[t] = ~0ull;
            if (t < bound) {
                const int64_t j = t < degr ? r0 + t : m0 + (t - degr);
                key[t] = ((unsigned long long)(uint32_t)cmap[__ldg(g.adj + j)] << 32) | (uint32_t)cw<EW>(g, j);
            }
        }
#pragma unroll
        for (int kk = 2; kk <= N; kk <<= 1) {
#pragma unroll
            for (int j = kk >> 1; j > 0; j >>= 1) {
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const int l = i ^ j;
                    if (l > i) {
                        const unsigned long long a = key[i], b = key[l];
                        const bool swap = ((i & kk) == 0) ? (a > b) : (a < b);
                        key[i] = swap ? b : a;
                        key[l] = swap ? a : b;
                    }
                }
            }
        }
        const int64_t base = boff[c];
        int32_t cnt = 0;
        uint32_t cur = 0xFFFFFFFFu;
        long long sum = 0;
#pragma unroll
        for (int t = 0; t < N; ++t) {
            const unsigned long long kt = key[t];
            const uint32_t ck = (uint32_t)(kt >> 32);
            if (kt != ~0ull && ck != (uint32_t)c) {
                if (ck != cur) {
                    if (cur != 0xFFFFFFFFu) {
                        tadj[base + cnt] = (int32_t)cur;
                        tw[base + cnt] = (int32_t)sum;
                        ++cnt;
                    }
                    cur = ck;
                    sum = 0;
                }
                sum += (long long)(uint32_t)(kt & 0xFFFFFFFFull);
            }
        }
        if (cur != 0xFFFFFFFFu) {
            tadj[base + cnt] = (int32_t)cur;
            tw[base + cnt] = (int32_t)sum;
            ++cnt;
        }
        rowcnt[c] = cnt;
    }
}

// Rows of 33..kWarpSort entries: one warp each, bitonic sort over the warp's
// shared-memory segment (pairs of a stage split over the lanes, __syncwarp
// between stages), then heads of equal-id runs summed and written in order.
template <bool EW>
__global__ void __launch_bounds__(kTB) k_contract_warp(DGraph g, const int32_t *cmap, const int32_t *mate,
                                                       const int32_t *crep, const int32_t *list, const int32_t *counts,
                                                       const int64_t *boff, int32_t *tadj, int32_t *tw, int32_t *rowcnt) {
    __shared__ unsigned long long sk[kTB / 32][kWarpSort];
    pdl_enter();
    const int warps = blockDim.x >> 5;
    const unsigned lane = lane_id();
    unsigned long long *keys = sk[threadIdx.x >> 5];
    const int32_t nrows = counts[0];
    for (int64_t w = (int64_t)blockIdx.x * warps + (threadIdx.x >> 5); w < nrows; w += (int64_t)gridDim.x * warps) {
        const int32_t c = list[w];
        const int32_t r = crep[c], m = mate[r];
        const int64_t degr = ld_xadj(g.xadj, (int64_t)r + 1) - ld_xadj(g.xadj, r);
        const int64_t bound = degr + (m >= 0 ? ld_xadj(g.xadj, (int64_t)m + 1) - ld_xadj(g.xadj, m) : 0);
        const int P = (int)pow2ceil(bound);   // <= kWarpSort by the class
        for (int i = lane; i < P; i += 32) keys[i] = i < bound ? row_entry<EW>(g, cmap, r, m, degr, i) : ~0ull;
        __syncwarp();
        for (int kk = 2; kk <= P; kk <<= 1) {
            for (int j = kk >> 1; j > 0; j >>= 1) {
                for (int i = lane; i < P; i += 32) {
                    const int l = i ^ j;
                    if (l > i) {
                        const unsigned long long a = keys[i], b = keys[l];
                        const bool up = (i & kk) == 0;
                        if ((a > b) == up) { keys[i] = b; keys[l] = a; }
                    }
                }
                __syncwarp();
            }
        }
        const int64_t base = boff[c];
        int32_t written = 0;
        for (int i0 = 0; i0 < bound; i0 += 32) {
            const int i = i0 + (int)lane;
            bool head = false;
            uint32_t ck = 0;
            long long sum = 0;
            if (i < bound) {
                ck = (uint32_t)(keys[i] >> 32);
                head = (i == 0 || (uint32_t)(keys[i - 1] >> 32) != ck) && ck != (uint32_t)c;
                if (head)
                    for (int t = i; t < bound && (uint32_t)(keys[t] >> 32) == ck; ++t)
                        sum += (long long)(uint32_t)(keys[t] & 0xFFFFFFFFull);
            }
            const unsigned hm = __ballot_sync(0xffffffffu, head);
            const int pos = __popc(hm & ((1u << lane) - 1u));
            if (head) {
                tadj[base + written + pos] = (int32_t)ck;
                tw[base + written + pos] = (int32_t)sum;
            }
            written += __popc(hm);
        }
        if (lane == 0) rowcnt[c] = written;
        __syncwarp();
    }
}

// Rows of kWarpSort..kSortSmem entries: one block per row, stable LSD radix sort
// of (coarse id, weight) by the id's bits.  A warp holds consecutive entries in
// registers and ranks them digit by digit with its own counters, so that a row
// takes five barriers per 8 bits of id, two or three digits for most levels, where a
// bitonic network of 4,096 entries took 78 barriers.  Bound by the gathers and the
// digit ranks; first level of R-MAT s17 458 -> 121 us, its 16 levels 3.75 -> 0.76 ms.
constexpr int kLargeThreads = 512;
constexpr int kLargeWarps = kLargeThreads / 32;
constexpr int kLargeItems = kSortSmem / kLargeThreads;
static_assert(kLargeItems * kLargeThreads == kSortSmem, "a row fits the block's registers");

template <bool EW>
__global__ void __launch_bounds__(kLargeThreads, 2) k_contract_large(DGraph g, const int32_t *cmap, const int32_t *mate,
                                                                     const int32_t *crep, const int32_t *list,
                                                                     const int32_t *counts, const int64_t *boff,
                                                                     int32_t *tadj, int32_t *tw, int32_t *rowcnt, int idbits) {
    __shared__ uint32_t skey[kSortSmem];
    __shared__ int32_t sval[kSortSmem];
    __shared__ uint16_t wcnt[kLargeWarps][256];   // per-warp digit counts, then the warps' offsets in the digit
    __shared__ int32_t first[256];                // first position of a digit
    __shared__ int32_t wsum[kLargeWarps];
    pdl_enter();
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int32_t nrows = counts[1];
    for (int64_t w = blockIdx.x; w < nrows; w += gridDim.x) {
        const int32_t c = list[w];
        const int32_t r = crep[c], m = mate[r];
        const int64_t r0 = ld_xadj(g.xadj, r), degr = ld_xadj(g.xadj, (int64_t)r + 1) - r0;
        int64_t m0 = 0, degm = 0;
        if (m >= 0) {
            m0 = ld_xadj(g.xadj, m);
            degm = ld_xadj(g.xadj, (int64_t)m + 1) - m0;
        }
        if (degr + degm > kSortSmem) continue;   // hub row: the device-wide sort (uniform over the block)
        const int bound = (int)(degr + degm);
        const int per = (bound + kLargeThreads - 1) / kLargeThreads;   // entries per lane (<= kLargeItems)
        const int e0 = (int)warp * per * 32 + (int)lane;               // entry i of a lane: e0 + 32 i
        uint32_t key[kLargeItems];
        int32_t val[kLargeItems], pos[kLargeItems];
#pragma unroll
        for (int i = 0; i < kLargeItems; ++i) {
            const int e = e0 + 32 * i;
            key[i] = 0;
            val[i] = 0;
            if (i < per && e < bound) {
                const int64_t j = e < degr ? r0 + e : m0 + (e - degr);
                key[i] = (uint32_t)__ldg(g.adj + j);
                val[i] = cw<EW>(g, j);
            }
        }
#pragma unroll
        for (int i = 0; i < kLargeItems; ++i)
            if (i < per && e0 + 32 * i < bound) key[i] = (uint32_t)cmap[key[i]];
        for (int shift = 0; shift < idbits; shift += 8) {
            if (shift > 0) {
#pragma unroll
                for (int i = 0; i < kLargeItems; ++i)
                    if (i < per && e0 + 32 * i < bound) {
                        key[i] = skey[e0 + 32 * i];
                        val[i] = sval[e0 + 32 * i];
                    }
            }
            for (int t = threadIdx.x; t < kLargeWarps * 128; t += kLargeThreads) reinterpret_cast<uint32_t *>(&wcnt[0][0])[t] = 0;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kLargeItems; ++i) {
                if (i >= per) continue;
                const int d = e0 + 32 * i < bound ? (int)(key[i] >> shift & 255u) : -1;
                const unsigned peers = __match_any_sync(0xffffffffu, d);
                const int leader = __ffs(peers) - 1;
                int k0 = 0;
                if (d >= 0 && (int)lane == leader) {
                    k0 = wcnt[warp][d];
                    wcnt[warp][d] = (uint16_t)(k0 + __popc(peers));
                }
                pos[i] = __shfl_sync(0xffffffffu, k0, leader) + __popc(peers & lt);
                __syncwarp();
            }
            __syncthreads();
            int total = 0, x = 0;
            if (threadIdx.x < 256) {
#pragma unroll
                for (int q = 0; q < kLargeWarps; ++q) {
                    const int k0 = wcnt[q][threadIdx.x];
                    wcnt[q][threadIdx.x] = (uint16_t)total;
                    total += k0;
                }
                x = total;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if ((int)lane >= o) x += y;
                }
                if (lane == 31) wsum[warp] = x;
            }
            __syncthreads();
            if (threadIdx.x < 256) {
                int before = 0;
                for (unsigned q = 0; q < warp; ++q) before += wsum[q];
                first[threadIdx.x] = before + x - total;
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kLargeItems; ++i) {
                if (i >= per || e0 + 32 * i >= bound) continue;
                const int d = (int)(key[i] >> shift & 255u);
                const int p = first[d] + wcnt[warp][d] + pos[i];
                skey[p] = key[i];
                sval[p] = val[i];
            }
            __syncthreads();
        }
        // heads of runs with equal coarse id, summed, the row's own vertex dropped; written in order.
        // bit i of heads: entry e0 + 32 i is one
        unsigned heads = 0;
        int mine = 0;
        for (int i = 0; i < per; ++i) {
            const int e = e0 + 32 * i;
            const bool head = e < bound && skey[e] != (uint32_t)c && (e == 0 || skey[e - 1] != skey[e]);
            mine += __popc(__ballot_sync(0xffffffffu, head));
            heads |= (head ? 1u : 0u) << i;
        }
        if (lane == 0) wsum[warp] = mine;
        __syncthreads();
        int written = 0, all = 0;
#pragma unroll
        for (int q = 0; q < kLargeWarps; ++q) {
            if (q < (int)warp) written += wsum[q];
            all += wsum[q];
        }
        const int64_t base = boff[c];
        for (int i = 0; i < per; ++i) {
            const bool head = heads >> i & 1u;
            const unsigned hm = __ballot_sync(0xffffffffu, head);
            if (head) {
                const int e = e0 + 32 * i;
                const uint32_t ck = skey[e];
                int32_t sum = 0;
                for (int t = e; t < bound && skey[t] == ck; ++t) sum += sval[t];
                const int64_t q = base + written + __popc(hm & lt);
                tadj[q] = (int32_t)ck;
                tw[q] = sum;
            }
            written += __popc(hm);
        }
        if (threadIdx.x == 0) rowcnt[c] = all;
        __syncthreads();   // before the next row's counters and sums
    }
}

struct CountVal {
    const int32_t *cnt;
    __device__ int64_t operator()(int64_t c) const { return cnt[c]; }
};

// Hub rows, step 1: every entry of hub row c becomes (rank(c) << 32 | C[u],
// w) at its segment hoff[c] + i (one block per row).
template <bool EW>
__global__ void __launch_bounds__(kTB) k_hub_fill(DGraph g, const int32_t *cmap, const int32_t *mate, const int32_t *crep,
                                                  const int32_t *list, const int32_t *counts, const int64_t *hoff,
                                                  const int64_t *hrank, uint64_t *key, int32_t *val,
                                                  int32_t *hub_c) {
    const int32_t nrows = counts[1];
    for (int64_t w = blockIdx.x; w < nrows; w += gridDim.x) {
        const int32_t c = list[w];
        const int32_t r = crep[c], m = mate[r];
        const int64_t degr = ld_xadj(g.xadj, (int64_t)r + 1) - ld_xadj(g.xadj, r);
        const int64_t bound = degr + (m >= 0 ? ld_xadj(g.xadj, (int64_t)m + 1) - ld_xadj(g.xadj, m) : 0);
        if (bound <= kSortSmem) continue;
        const int64_t off = hoff[c];
        const uint64_t hi = (uint64_t)hrank[c] << 32;
        if (threadIdx.x == 0) hub_c[hrank[c]] = c;
        for (int64_t i = threadIdx.x; i < bound; i += blockDim.x) {
            const unsigned long long e = row_entry<EW>(g, cmap, r, m, degr, i);
            key[off + i] = hi | (e >> 32);
            val[off + i] = (int32_t)(uint32_t)(e & 0xFFFFFFFFull);
        }
    }
}

// Hub rows, step 2 (after the stable sort by rank, then coarse id): the
// sorted entries of hub row c are the segment starting at hoff[c], in coarse
// id order.  An entry heads its output entry when it starts a run of equal
// (rank, coarse id) and the id is not the row's own; an exclusive scan of the
// head flags over all hub entries places every head (hs[p] - hs[hoff[c]]),
// so every row, however long, is spread over the whole grid.
struct HubHead {
    const uint64_t *key;
    const int32_t *hub_c;
    __device__ int64_t operator()(int64_t p) const {
        const uint64_t kp = key[p];
        if (p > 0 && key[p - 1] == kp) return 0;
        return (uint32_t)kp != (uint32_t)hub_c[kp >> 32] ? 1 : 0;
    }
};

__global__ void __launch_bounds__(kTB) k_hub_emit(int64_t htotal, const uint64_t *key, const int32_t *val,
                                                  const int32_t *hub_c, const int64_t *hoff, const int64_t *hs,
                                                  const int64_t *boff, int32_t *tadj, int32_t *tw) {
    const HubHead head{key, hub_c};
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < htotal; p += (int64_t)gridDim.x * blockDim.x) {
        if (!head(p)) continue;
        const uint64_t kp = key[p];
        const int32_t c = hub_c[kp >> 32];
        long long sum = 0;
        for (int64_t t = p; t < htotal && key[t] == kp; ++t) sum += (long long)(uint32_t)val[t];
        const int64_t q = boff[c] + (hs[p] - hs[hoff[c]]);
        tadj[q] = (int32_t)(uint32_t)kp;
        tw[q] = (int32_t)sum;
    }
}

// Hub rows, step 3: entries written per hub row (rank order; the segment of
// rank r ends where the next one starts).
__global__ void k_hub_rowcnt(int64_t nhub, int64_t htotal, const int32_t *hub_c, const int64_t *hoff, const int64_t *hs,
                             const int64_t *hs_total, int32_t *rowcnt) {
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nhub; r += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = hub_c[r];
        const int64_t beg = hoff[c];
        const int64_t end = r + 1 < nhub ? hoff[hub_c[r + 1]] : htotal;
        const int64_t he = end < htotal ? hs[end] : *hs_total;
        rowcnt[c] = (int32_t)(he - hs[beg]);
    }
}

// Long coarse rows (more than kWarpSort bound entries) are compacted by one
// block each; k_copy_rows leaves them out.
__global__ void __launch_bounds__(kTB) k_copy_long(const int32_t *list, const int32_t *counts, const int64_t *boff,
                                                   const int64_t *xadj_c, const int32_t *tadj, const int32_t *tw,
                                                   int32_t *adj_c, int32_t *ew_c) {
    pdl_enter();
    const int32_t nrows = counts[1];
    for (int64_t w = blockIdx.x; w < nrows; w += gridDim.x) {
        const int32_t c = list[w];
        const int64_t src = boff[c], dst = xadj_c[c], len = xadj_c[c + 1] - dst;
        for (int64_t i = threadIdx.x; i < len; i += blockDim.x) {
            adj_c[dst + i] = tadj[src + i];
            ew_c[dst + i] = tw[src + i];
        }
    }
}

// Compaction of the coarse rows: kCopyLanes lanes per row (the rows are
// short; a warp per row left most lanes idle and serialised the rows'
// round trips).
constexpr int kCopyLanes = 8;
__global__ void k_copy_rows(int32_t nc, const int64_t *boff, const int64_t *xadj_c, const int32_t *crep, const int32_t *mate,
                            const int32_t *vw, int32_t *vw_c, const int32_t *tadj, const int32_t *tw, int32_t *adj_c,
                            int32_t *ew_c) {
    pdl_enter();
    const int64_t groups = (int64_t)gridDim.x * blockDim.x / kCopyLanes;
    const int gl = (int)(threadIdx.x % kCopyLanes);
    for (int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kCopyLanes; c < nc; c += groups) {
        if (gl == 0) {   // the coarse vertex weight
            const int32_t r = crep[c], m = mate[r];
            vw_c[c] = vw[r] + (m >= 0 ? vw[m] : 0);
        }
        const int64_t src = boff[c], dst = xadj_c[c], len = xadj_c[c + 1] - dst;
        if (boff[c + 1] - src > kWarpSort) continue;   // k_copy_long
        for (int64_t i = gl; i < len; i += kCopyLanes) {
            adj_c[dst + i] = tadj[src + i];
            ew_c[dst + i] = tw[src + i];
        }
    }
}

// One coarsening level: matching, map, contraction.  longest: the level's longest
// row (-1: not known), then a bound on the coarse level's.  Returns JET_OK and sets
// stalled=true (without building the level) when n_c > 0.95 n.  Small levels are
// bound by launches and host waits: the row classes are made before the host
// knows the number of coarse vertices, so that it waits twice per level, for the
// sizes of the work and of the result, and empty classes are not launched (564
// launches, four waits and 2.9 ms for the 12 levels of a 110,592-vertex mesh before).
static int coarsen_level(Ctx &c, const DGraph &g, int64_t &longest, uint64_t seed, int32_t level, jet_hier *h, bool &stalled) {
    cudaStream_t s = c.stream;
    stalled = false;
    const int64_t n = g.n;
    auto a256 = [](size_t x) { return (x + 255) & ~size_t(255); };
    DevBuf scratch, cmapb, work, vb, eb, hubb, hsortb, hsb;   // scratch is freed in stream order
    const size_t nn = (size_t)n;
    JET_TRY(dev_alloc(scratch, 256 + 2 * a256((nn + 1) * 8) + a256((size_t)(scan_tiles_for(n) + 1) * 8) + 6 * a256(nn * 4), s));
    char *p = scratch.as<char>();
    auto take = [&](size_t b) { char *r = p; p += a256(b); return r; };
    LevelCount *lc = reinterpret_cast<LevelCount *>(take(sizeof(LevelCount)));
    int64_t *boff = reinterpret_cast<int64_t *>(take((nn + 1) * 8));
    int64_t *cidx = reinterpret_cast<int64_t *>(take((nn + 1) * 8));
    int64_t *scan_scr = reinterpret_cast<int64_t *>(take((size_t)(scan_tiles_for(n) + 1) * 8));
    int32_t *mate = reinterpret_cast<int32_t *>(take(nn * 4)), *crep = reinterpret_cast<int32_t *>(take(nn * 4));
    int32_t *warp_list = reinterpret_cast<int32_t *>(take(nn * 4)), *large_list = reinterpret_cast<int32_t *>(take(nn * 4));
    int32_t *t16_list = reinterpret_cast<int32_t *>(take(nn * 4)), *t32_list = reinterpret_cast<int32_t *>(take(nn * 4));
    JET_TRY(dev_alloc(cmapb, nn * 4, s));   // owned by the hierarchy
    int32_t *cmap = cmapb.as<int32_t>();
    JET_CUDA_TRY(cudaMemsetAsync(lc, 0, sizeof(LevelCount), s));
    JET_TRY(hem(c, g, longest, seed, level, c.opt.hem_rounds, mate));
    if (c.opt.flags & JET_FLAG_TWO_HOP) {
        int64_t added[3];
        JET_TRY(two_hop(c, g, mate, added));
    }
    JET_TRY(device_exscan(RepFlag{mate}, n, cidx, &lc->nc, scan_scr, s));
    JET_CUDA_TRY(launch_pdl(k_cmap, grid_for(n, kTB, 8192), kTB, 0, s, true, g.n, (const int32_t *)mate, (const int64_t *)cidx,
                            cmap, crep));
    JET_TRY(device_exscan(RowBound{g.xadj, crep, mate, &lc->nc}, n, boff, &lc->btotal, scan_scr, s));
    JET_CUDA_TRY(launch_pdl(k_row_classes, grid_for(n, kTB, num_sms() * 8), kTB, 0, s, true, g.n, (const int64_t *)boff, lc,
                            warp_list, large_list, t16_list, t32_list));
    c.launches += 2 + 2 * scan_launches(n);
    JET_CUDA_TRY(cudaMemcpyAsync(c.pinned, lc, sizeof(LevelCount), cudaMemcpyDeviceToHost, s));
    JET_CUDA_TRY(cudaStreamSynchronize(s));
    LevelCount hc;
    memcpy(&hc, c.pinned, sizeof(hc));
    const int64_t nc = hc.nc;
    longest = hc.longest;
    if (100 * nc > 95 * n) { stalled = true; return JET_OK; }
    const size_t ncl = (size_t)std::max<int64_t>(nc, 1);
    // merged rows
    const size_t bt = a256((size_t)std::max<int64_t>(hc.btotal, 1) * 4);
    JET_TRY(dev_alloc(work, 2 * bt + a256(ncl * 4) + 256, s));
    int32_t *tadj = work.as<int32_t>(), *tw = reinterpret_cast<int32_t *>(work.as<char>() + bt);
    int32_t *cnt = reinterpret_cast<int32_t *>(work.as<char>() + 2 * bt);
    int64_t *hub_total = reinterpret_cast<int64_t *>(work.as<char>() + 2 * bt + a256(ncl * 4));
    const size_t xb = a256((ncl + 1) * 8);
    JET_TRY(dev_alloc(vb, xb + ncl * 4, s));
    int64_t *xc = vb.as<int64_t>();
    int32_t *vwc = reinterpret_cast<int32_t *>(vb.as<char>() + xb);
    const int gl = num_sms() * 8;
    const int gwarp = std::min(gl, grid_for(hc.rows[0], kTB / 32)), glarge = std::max(1, std::min(num_sms() * 4, hc.rows[1]));
    const int32_t *cm = cmap, *mt = mate, *cr = crep, *cts = lc->rows;
    const int64_t *bo = boff;
    auto contract = [&](auto kern, int slot, int grid, const int32_t *list) -> int {
        if (hc.rows[slot] == 0) return JET_OK;
        JET_CUDA_TRY(launch_pdl(kern, grid, kTB, 0, s, true, g, cm, mt, cr, list, cts, bo, tadj, tw, cnt));
        c.launches += 1;
        return JET_OK;
    };
    JET_TRY(contract(g.ew ? k_contract_thread<true, 16> : k_contract_thread<false, 16>, 2, std::min(gl, grid_for(hc.rows[2], kTB)), t16_list));
    JET_TRY(contract(g.ew ? k_contract_thread<true, 32> : k_contract_thread<false, 32>, 3, std::min(gl, grid_for(hc.rows[3], kTB)), t32_list));
    JET_TRY(contract(g.ew ? k_contract_warp<true> : k_contract_warp<false>, 0, gwarp, warp_list));
    if (hc.rows[1] > 0) {
        auto kern = g.ew ? k_contract_large<true> : k_contract_large<false>;
        JET_CUDA_TRY(launch_pdl(kern, glarge, kLargeThreads, 0, s, true, g, cm, mt, cr, (const int32_t *)large_list, cts, bo, tadj,
                                tw, cnt, std::max(1, bits_for(nc - 1))));
        c.launches += 1;
    }
    if (hc.nhub > 0) {
        // hub rows: all their entries in one stable radix sort by (rank, coarse id)
        const int64_t htotal = hc.htotal, nhub = hc.nhub;
        JET_TRY(dev_alloc(hubb, 2 * a256(ncl * 8) + (size_t)nhub * 4, s));
        int64_t *hoff = hubb.as<int64_t>(), *hrank = reinterpret_cast<int64_t *>(hubb.as<char>() + a256(ncl * 8));
        int32_t *hub_c = reinterpret_cast<int32_t *>(hubb.as<char>() + 2 * a256(ncl * 8));
        const HubBound hb{crep, mate, g.xadj};
        JET_TRY(device_exscan(hb, nc, hoff, nullptr, scan_scr, s));
        JET_TRY(device_exscan(HubFlag{hb}, nc, hrank, nullptr, scan_scr, s));
        JET_TRY(dev_alloc(hsortb, sort_scratch_bytes(htotal), s));
        SortScratch sc;
        sort_scratch_carve(hsortb.as<char>(), htotal, sc);
        JET_TRY(dev_alloc(hsb, (size_t)htotal * 8 + (size_t)(scan_tiles_for(htotal) + 1) * 8 + 64, s));
        int64_t *hs = hsb.as<int64_t>(), *hs_scr = hs + htotal;
        if (g.ew) k_hub_fill<true><<<glarge, kTB, 0, s>>>(g, cmap, mate, crep, large_list, cts, hoff, hrank, sc.key[0], sc.val[0], hub_c);
        else k_hub_fill<false><<<glarge, kTB, 0, s>>>(g, cmap, mate, crep, large_list, cts, hoff, hrank, sc.key[0], sc.val[0], hub_c);
        JET_CUDA_TRY(cudaGetLastError());
        int which = 0;
        JET_TRY(sort_pairs(c, sc, htotal, 32 + bits_for(nhub - 1), &which));
        JET_TRY(device_exscan(HubHead{sc.key[which], hub_c}, htotal, hs, hub_total, hs_scr, s));
        k_hub_emit<<<std::min(gl, grid_for(htotal, kTB)), kTB, 0, s>>>(htotal, sc.key[which], sc.val[which], hub_c, hoff, hs,
                                                                      boff, tadj, tw);
        k_hub_rowcnt<<<grid_for(nhub, kTB, 1024), kTB, 0, s>>>(nhub, htotal, hub_c, hoff, hs, hub_total, cnt);
        c.launches += 3 + 2 * scan_launches(nc) + scan_launches(htotal);
        JET_CUDA_TRY(cudaGetLastError());
    }
    // coarse xadj
    JET_TRY(device_exscan(CountVal{cnt}, nc, xc, xc + nc, scan_scr, s));
    c.launches += scan_launches(nc);
    JET_CUDA_TRY(cudaMemcpyAsync(c.pinned, xc + nc, 8, cudaMemcpyDeviceToHost, s));
    JET_CUDA_TRY(cudaStreamSynchronize(s));
    const int64_t nnzc = c.pinned[0];
    const size_t ab = a256((size_t)std::max<int64_t>(nnzc, 1) * 4);
    JET_TRY(dev_alloc(eb, 2 * ab, s));
    int32_t *adj_c = eb.as<int32_t>(), *ew_c = reinterpret_cast<int32_t *>(eb.as<char>() + ab);
    if (hc.rows[1] > 0) {
        JET_CUDA_TRY(launch_pdl(k_copy_long, std::min(gl, hc.rows[1]), kTB, 0, s, true, (const int32_t *)large_list, cts, bo, (const int64_t *)xc,
                                (const int32_t *)tadj, (const int32_t *)tw, adj_c, ew_c));
        c.launches += 1;
    }
    JET_CUDA_TRY(launch_pdl(k_copy_rows, std::min(gl, grid_for(nc, kTB / kCopyLanes)), kTB, 0, s, true, (int32_t)nc, bo,
                            (const int64_t *)xc, cr, mt, g.vw, vwc, (const int32_t *)tadj, (const int32_t *)tw, adj_c, ew_c));
    c.launches += 1;
    JET_CUDA_TRY(cudaGetLastError());
    int32_t i = h->levels;
    h->cmap[i - 1] = cmap;
    h->n[i] = (int32_t)nc;
    h->nnz[i] = nnzc;
    h->xadj[i] = xc;
    h->adj[i] = adj_c;
    h->vw[i] = vwc;
    h->ew[i] = ew_c;
    h->levels = i + 1;
    h->bufs.push_back(std::move(cmapb));
    h->bufs.push_back(std::move(vb));
    h->bufs.push_back(std::move(eb));
    return JET_OK;   // the next level's work follows in stream order
}

__global__ void k_ones(int32_t *p, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) p[i] = 1;
}

// MLCoarsen of Alg. 1 (see jet_coarsen in jet.h for the stop rules).
int coarsen(Ctx &c, const DGraph &g0, int32_t k, uint64_t seed, jet_hier *h) {
    cudaStream_t s = c.stream;
    h->levels = 1;
    h->k = k;
    h->n[0] = g0.n;
    h->nnz[0] = g0.nnz;
    h->xadj[0] = g0.xadj;
    h->adj[0] = g0.adj;
    h->ew[0] = g0.ew;
    if (g0.vw) {
        h->vw[0] = g0.vw;
    } else {
        DevBuf ones;
        JET_TRY(dev_alloc(ones, (size_t)std::max<int32_t>(g0.n, 1) * 4, s));
        if (g0.n > 0) k_ones<<<grid_for(g0.n, kTB, 8192), kTB, 0, s>>>(ones.as<int32_t>(), g0.n);
        if (g0.n > 0) c.launches += 1;
        JET_CUDA_TRY(cudaGetLastError());
        h->vw[0] = ones.as<int32_t>();
        h->bufs.push_back(std::move(ones));
    }
    int32_t T = c.opt.coarsen_target > 0 ? c.opt.coarsen_target : std::max(8 * k, 256);
    int32_t maxl = std::min<int32_t>(c.opt.max_levels, JET_MAX_LEVELS);
    int64_t longest = h->longest0;
    while (h->n[h->levels - 1] > T && h->levels < maxl) {
        int32_t i = h->levels - 1;
        DGraph gi;
        gi.n = h->n[i]; gi.nnz = h->nnz[i]; gi.xadj = h->xadj[i]; gi.adj = h->adj[i]; gi.vw = h->vw[i]; gi.ew = h->ew[i];
        bool stalled = false;
        JET_TRY(coarsen_level(c, gi, longest, seed, i, h, stalled));
        if (stalled) break;
    }
    return JET_OK;
}

// ---------------------------------------------------------------------------
// projection (Alg. 1 ProjectPartition)
// ---------------------------------------------------------------------------
__global__ void k_project(int32_t n, const int32_t *cmap, const int32_t *pc, int32_t *pf) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        pf[v] = pc[cmap[v]];
}

int project(Ctx &c, int32_t n_fine, const int32_t *cmap, const int32_t *coarse_part, int32_t *fine_part) {
    if (n_fine > 0) k_project<<<grid_for(n_fine, kTB, 8192), kTB, 0, c.stream>>>(n_fine, cmap, coarse_part, fine_part);
    if (n_fine > 0) c.launches += 1;
    JET_CUDA_TRY(cudaGetLastError());
    return JET_OK;
}

}  // namespace jet
