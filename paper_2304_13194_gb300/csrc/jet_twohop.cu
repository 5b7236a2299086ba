// Two-hop matching (Sec. 3.1), added to heavy-edge matching when more than
// 25% of the vertices are still unmatched: leaves (degree-1 vertices with
// the same neighbour), twins (vertices with the same neighbourhood) and
// relatives (vertices with the same matchmaker: their lowest-id neighbour
// that is already matched and has degree <= kMatchmakerMaxDeg).  The stages
// run in that order, each only while 4u > n.  Inside a group the vertices
// pair in ascending id: first with second, third with fourth, ...
//
// Per stage, device-wide: one key per vertex (a sentinel for non-candidates;
// one warp per vertex so that hubs do not stall a thread), a stable radix
// sort of (key, vertex) with the vertices entering in id order, and the pairs of
// even rank in their group with their successor.  A twin's key is a 64-bit hash
// that only has to bring equal keys together: it is sorted by enough low bits that
// two different keys seldom share them, and should some do, a kernel finds out
// before any pair is made and the stage is repeated over all 64 bits.
#include "jet_internal.cuh"

#include <algorithm>

namespace jet {

namespace {

constexpr uint64_t kTwinSalt = 0x2545F4914F6CDD1DULL;
constexpr uint64_t kTwinDeg = 0x9FB21C651E98DF25ULL;

__global__ void k_count_unmatched(int32_t n, const int32_t *mate, int64_t *out) {
    __shared__ long long red[40];
    long long c = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        c += mate[v] < 0;
    c = block_sum_i64(c, red);
    if (threadIdx.x == 0 && c) atomic_add_i64(out, c);
}

// Stage keys, one warp per vertex: the neighbour of a leaf; the order-free
// neighbourhood hash of a twin candidate (wrapping sum, so the lane order does
// not matter); the lowest eligible matchmaker of a relative.
__global__ void __launch_bounds__(kTB) k_two_hop_keys(DGraph g, int stage, const int32_t *mate, uint64_t sentinel,
                                                      uint64_t *key, int32_t *val) {
    const int warps = blockDim.x >> 5;
    const unsigned lane = lane_id();
    pdl_enter();
    for (int64_t v = (int64_t)blockIdx.x * warps + (threadIdx.x >> 5); v < g.n; v += (int64_t)gridDim.x * warps) {
        uint64_t k = sentinel;
        if (mate[v] < 0) {
            const int64_t beg = ld_xadj(g.xadj, v), end = ld_xadj(g.xadj, v + 1);
            if (stage == 0) {
                if (end - beg == 1) k = (uint64_t)(uint32_t)__ldg(g.adj + beg);
            } else if (stage == 1) {
                unsigned long long h = 0;
#pragma unroll 4
                for (int64_t j = beg + lane; j < end; j += 32)
                    h += splitmix64((uint64_t)(uint32_t)__ldg(g.adj + j) ^ kTwinSalt);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
                h += splitmix64((uint64_t)(end - beg) ^ kTwinDeg);
                k = h == ~0ULL ? ~0ULL - 1 : h;
            } else {
                int32_t best = INT32_MAX;
                for (int64_t j0 = beg + lane; j0 < end; j0 += 4 * 32) {   // four entries in flight per lane
                    int32_t u[4], m[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) u[q] = j0 + 32 * q < end ? __ldg(g.adj + j0 + 32 * q) : INT32_MAX;
#pragma unroll
                    for (int q = 0; q < 4; ++q) m[q] = u[q] < best ? mate[u[q]] : -1;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (m[q] >= 0 && u[q] < best &&
                            ld_xadj(g.xadj, (int64_t)u[q] + 1) - ld_xadj(g.xadj, u[q]) <= kMatchmakerMaxDeg)
                            best = u[q];
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    int32_t t = __shfl_xor_sync(0xffffffffu, best, o);
                    best = t < best ? t : best;
                }
                if (best != INT32_MAX) k = (uint64_t)(uint32_t)best;
            }
        }
        if (lane == 0) {
            key[v] = k;
            val[v] = (int32_t)v;
        }
    }
}

// *mixed = 1 where two different keys share the sorted bits.
__global__ void __launch_bounds__(kTB) k_find_mixed(int64_t n, const uint64_t *key, uint64_t bits, int64_t *mixed) {
    pdl_enter();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i + 1 < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t x = key[i] ^ key[i + 1];
        if (x && !(x & bits)) *mixed = 1;
    }
}

// Position i of a group pairs with i + 1 when its rank in the group is even
// and i + 1 is in the same group.  The group's start is found by doubling steps
// back and bisection (most groups are short), which takes the place of a scan of the
// group heads and a scatter of the starts.  Nothing happens when *mixed is set.
__global__ void __launch_bounds__(kTB) k_pair_groups(int64_t n, const uint64_t *key, const int32_t *val, uint64_t sentinel,
                                                     const int64_t *mixed, int32_t *mate, int64_t *pairs) {
    __shared__ long long red[40];
    pdl_enter();
    if (*mixed) return;
    long long c = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i + 1 < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = key[i];
        if (k == sentinel || key[i + 1] != k) continue;
        int64_t in = i, step = 1;                        // key[in] == k
        while (in - step >= 0 && key[in - step] == k) { in -= step; step *= 2; }
        int64_t out = in - step < -1 ? -1 : in - step;   // key[out] != k, or -1
        while (in - out > 1) {
            const int64_t mid = out + (in - out) / 2;
            if (key[mid] == k) in = mid;
            else out = mid;
        }
        if (((i - in) & 1) == 0) {
            const int32_t a = val[i], b = val[i + 1];
            mate[a] = b;
            mate[b] = a;
            ++c;
        }
    }
    c = block_sum_i64(c, red);
    if (threadIdx.x == 0 && c) atomic_add_i64(pairs, c);
}

}  // namespace

int two_hop(Ctx &c, const DGraph &g, int32_t *mate, int64_t added[3]) {
    cudaStream_t s = c.stream;
    added[0] = added[1] = added[2] = 0;
    const int64_t n = g.n;
    if (n == 0) return JET_OK;
    // counters {unmatched, then pairs and mixed of every stage} | sort scratch
    DevBuf buf;
    JET_TRY(dev_alloc(buf, 256 + sort_scratch_bytes(n), s));
    int64_t *cnt = buf.as<int64_t>();
    SortScratch sc;
    sort_scratch_carve(buf.as<char>() + 256, n, sc);
    const int gv = std::min(num_sms() * 8, grid_for(n, kTB));
    const int gw = std::min(num_sms() * 8, grid_for(n, kTB / 32));
    JET_CUDA_TRY(cudaMemsetAsync(cnt, 0, 256, s));
    k_count_unmatched<<<gv, kTB, 0, s>>>((int32_t)n, mate, cnt);
    c.launches += 1;
    JET_CUDA_TRY(cudaGetLastError());
    auto read = [&](const int64_t *src) -> int {
        JET_CUDA_TRY(cudaMemcpyAsync(c.pinned, src, 16, cudaMemcpyDeviceToHost, s));
        JET_CUDA_TRY(cudaStreamSynchronize(s));
        return JET_OK;
    };
    JET_TRY(read(cnt));
    int64_t un = c.pinned[0];
    // two different hashes share 2 bits_for(n) + 6 bits with probability below 2^-7
    const int twin_bits = std::min(64, (2 * bits_for(n) + 6 + 7) / 8 * 8);
    for (int stage = 0, attempt = 0; stage < 3;) {
        if (4 * un <= n) break;
        // keys below n for leaves and relatives (sentinel n), any 64-bit value for twins
        const uint64_t sentinel = stage == 1 ? ~0ULL : (uint64_t)n;
        const int kbits = stage != 1 ? bits_for(n) : attempt ? 64 : twin_bits;
        int64_t *pairs = cnt + 2 + 4 * stage + 2 * attempt, *mixed = pairs + 1;
        JET_CUDA_TRY(launch_pdl(k_two_hop_keys, gw, kTB, 0, s, true, g, stage, (const int32_t *)mate, sentinel, sc.key[0], sc.val[0]));
        int which = 0;
        JET_TRY(sort_pairs(c, sc, n, kbits, &which));
        const uint64_t *key = sc.key[which];
        if (stage == 1 && kbits < 64) {
            JET_CUDA_TRY(launch_pdl(k_find_mixed, gv, kTB, 0, s, true, n, key, (1ULL << kbits) - 1, mixed));
            c.launches += 1;
        }
        JET_CUDA_TRY(launch_pdl(k_pair_groups, gv, kTB, 0, s, true, n, key, (const int32_t *)sc.val[which], sentinel,
                                (const int64_t *)mixed, mate, pairs));
        c.launches += 2;
        JET_TRY(read(pairs));
        if (c.pinned[1]) {   // only a twin stage over twin_bits, once
            attempt = 1;
            continue;
        }
        added[stage] = 2 * c.pinned[0];
        un -= added[stage];
        ++stage;
        attempt = 0;
    }
    return JET_OK;
}

}  // namespace jet
