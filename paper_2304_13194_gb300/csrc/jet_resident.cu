// Small and medium levels of a refinement: one thread-block cluster keeps a
// whole level in its shared memory and runs every iteration of Alg. 3 on it,
// level after level of a chain (coarsest first), in a single launch.
//
// Why: an iteration of such a level moves a few hundred kilobytes at most, so
// what it costs is the number of dependent steps times the latency of each.
// Kernels or cluster phases that keep the level's state in global memory pay
// an L2 round trip per step (about 0.7 us on this GPU, 40-57 us per iteration
// whether a level has 200 or 100,000 vertices).  Here the steps between two
// cluster barriers only touch shared memory, and an iteration has three
// barriers (Jetlp, Jetrw) or four (Jetrs) instead of five to eight phases:
//  * the blocks own equal runs of vertices.  Per-vertex state (row offsets,
//    neighbour counts ext, gains, slots, the best partition) lives with the
//    owner; the current parts P and the parts after the pending moves N (one
//    byte each for k <= 256) are replicated in every block, so that the
//    gathers over a row, which dominate, are local;
//  * a pass leaves its moves in a list in the owner's shared memory; after the
//    barrier every block reads all lists (coalesced) and updates its own N;
//  * a neighbour's gain is fetched from its owner only where N says that the
//    neighbour wants to move; ext of a mover's neighbours is updated with
//    atomics on the owner's shared memory;
//  * eviction order (slot, then vertex id) needs no tile sums: each block's
//    slot buckets, read by all blocks, give both the boundary slot and the
//    weight that earlier blocks hold in it; inside a block the warps own
//    consecutive runs;
//  * every block computes the Alg. 3 controller from the same sums, so its
//    decisions need no broadcast.
// Measured (us per iteration, this loop / the loops before it): 64 x 64 mesh
// levels 9-11 / 39-48 (cluster phases in global memory); random geometric
// levels of 51k to 2k vertices 20-14 / 41-55; weighted 48^3 mesh levels of 60k
// to 1k vertices 32-14 / 38-57 (CUDA-graph loop above 4,096 vertices).  What is
// left is instruction latency: a few hundred instructions per phase on few
// warps, three to four cluster barriers of 610 cycles (1024 threads), remote
// reads of 205 cycles.
// The rows themselves are kept in shared memory as far as they fit and read
// from L2 beyond that.  All decisions are integer comparisons with the fixed
// tie-breaks; results are those of the per-kernel loop, bit for bit.
// No block waits except at the hardware cluster barrier, every block reads the
// same mode from the same sums and so meets every barrier.
#include "jet_phases.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

namespace jet {

namespace cg = cooperative_groups;

extern __shared__ __align__(16) unsigned char res_arena[];

namespace {

constexpr int kRT = 1024;                 // most threads per block (small chains run half of them)
constexpr int kRWarps = kRT / 32;
static_assert(kSlots == kRWarps + 1, "the tables' memory holds one bucket array");
constexpr int kThreadRow = 48;            // rows up to this length: one thread (or a few lanes) each
constexpr int kSeen = 4;                  // distinct parts a thread keeps of its row; rows with more go to a warp
constexpr uint32_t kMoveBit = 0x8000u;    // list entry: the vertex is in M
constexpr uint32_t kDestMask = 0x3FFu;    // list entry: destination part (k <= 1024); local vertex id in the high half
constexpr uint8_t kNoSlot = 0xFF, kTakenSlot = 0xFE;

struct ResLevel {
    DGraph g;
    const int32_t *cmap;     // this level -> the next coarser one (null: the level starts from the given partition)
    int32_t *out;            // receives the level's refined partition
    ResStat *stat;           // the level's outcome (pinned host memory)
    uint64_t seed;           // Jetrw seed of the level
    int32_t cq16;            // first-filter ratio c of the level
    int32_t pad;
};
// One graph's chain of levels, coarsest first (a kernel parameter).
struct ResJob {
    const int32_t *init;     // partition that the first level starts from (through its cmap, or directly)
    int32_t *wdeg;           // scratch: weighted degrees where they do not fit in shared memory
    TraceRec *trace;         // iteration records of the chain's last level (pinned host memory; may be null)
    int64_t Llim, opt, sigma, phi_ppm;
    int32_t k, nlv, max_no_improve, weak_limit, max_iters, hub_deg;
    uint32_t abl, arena_bytes;
    ResLevel lv[JET_MAX_LEVELS];
};

// One block's share of an iteration's sums; the other blocks read it.
struct ResPart {
    int32_t dcut;
    uint32_t degm, nM, nX, degx, nbnd, nexam, degexam, ncand, takenw;
};
enum { kfDcut, kfDegm, kfNM, kfNX, kfDegx, kfNbnd, kfNexam, kfDegexam, kfNcand, kfTakenw, kPartFields };

// The level as a block sees it (in shared memory, read by all its threads).
struct ResView {
    int32_t n, S, base, own, k, rank, cs;
    int32_t wps;                           // log2 of the warps per source block when every block's data are read
    uint32_t magic;                        // owner of u = umulhi(u, magic) = u / S
    uint32_t oP, oN, oD, oBest, oRow, oExt, oF, oList, oBig, oFlag, oKey;   // byte offsets into the arena
    uint32_t oAct, oPw, oDelta, oExcess, oNeed, oAidx, oBs, oInB, oSs, oCap, oBk, oTot, oTab;
    uint32_t oVw, oWdeg, oAdj, oEw, cached;   // optional copies; cached = entries of the own rows held in shared memory
    const int32_t *gadj, *gew, *gvw;          // global arrays, at the own rows' / vertices' start
    int32_t *gwdeg;
    int32_t hasbig, hub;
    uint32_t abl;
    int32_t cq16, max_no_improve, weak_limit, max_iters;
    uint64_t seed;
    int64_t Llim, opt, sigma, phi_ppm;
};
struct ResCtl {
    int32_t mode, it, noimp, weak, hit_cap, best_bal, copy, nA, nB;
    int32_t kcount[4];
    int64_t cut, best_cut, best_maxw;
};
// Block-wide state, at the start of the arena.
struct ResShared {
    ResView v;
    ResCtl ctl;
    ResPart part[2];                       // by iteration parity
    unsigned long long acc[3][kPartFields + 2];   // block 0: sums over the level's iterations, by kind (then |A|, P_best copies)
    uint32_t wsum[32];                     // Jetrs: evicted weight by warp; the trace's sums
    int32_t red[4];
    uint16_t hubs[kHugeCap];
    int cnt, nact, nstage, nhub, anybig;
};

constexpr uint32_t kNone = 0xFFFFFFFFu;

__host__ __device__ constexpr uint32_t up16(uint32_t x) { return (x + 15u) & ~15u; }

// Offsets of the fixed part of the arena for slices of S vertices; returns
// its size.  ptb = bytes of a part id.
__host__ __device__ inline uint32_t res_layout(ResView &v, int32_t n, int32_t S, int32_t k, uint32_t ptb) {
    uint32_t p = up16((uint32_t)sizeof(ResShared));
    auto take = [&](uint32_t bytes) { const uint32_t r = p; p += up16(bytes); return r; };
    v.oP = take((uint32_t)n * ptb);
    v.oN = take((uint32_t)n * ptb);
    v.oBest = take((uint32_t)S * ptb);
    v.oRow = take((uint32_t)(S + 1) * 4);
    v.oExt = take((uint32_t)S * 4);
    v.oF = take((uint32_t)S * 4);
    v.oList = take((uint32_t)S * 4);
    v.oBig = take((uint32_t)S * 2);
    v.oAct = take((uint32_t)S * 2);
    v.oFlag = take((uint32_t)S);
    v.oKey = take((uint32_t)S);
    v.oD = take((uint32_t)S * ptb);
    v.oPw = take((uint32_t)k * 4);
    v.oDelta = take((uint32_t)k * 8);
    v.oExcess = take((uint32_t)k * 4);
    v.oNeed = take((uint32_t)k * 4);
    v.oAidx = take((uint32_t)k * 2);
    v.oBs = take((uint32_t)k * 2);
    v.oInB = take((uint32_t)k);
    v.oSs = take((uint32_t)k);
    v.oCap = take((uint32_t)(k + 1) * 8);
    v.oBk = take((uint32_t)k * kSlots * 4);
    v.oTot = (uint32_t)S >= (uint32_t)k * kSlots ? v.oF : take((uint32_t)k * kSlots * 4);   // F is idle in rebalancing
    v.oTab = take((uint32_t)k * (kRWarps + 1) * 4);   // per-warp tables; in the eviction the prefix buckets, then sums by warp
    return p;
}

int32_t res_slice(int64_t n, int cs) { return (int32_t)((((n + cs - 1) / cs) + 31) & ~int64_t(31)); }
__device__ __forceinline__ int32_t res_slice_dev(int32_t n, int32_t cs) { return ((n + cs - 1) / cs + 31) & ~31; }

__device__ __forceinline__ ResShared &rs() { return *reinterpret_cast<ResShared *>(res_arena); }

template <class T>
__device__ __forceinline__ T *arena_at(uint32_t off) { return reinterpret_cast<T *>(res_arena + off); }

// The same shared variable in block c of the cluster: its address in the
// cluster's shared window, and 32-bit (or 8-bit) accesses there.  (Accesses
// through generic addresses were not overlapped: 16 loads took 16 latencies.)
__device__ __forceinline__ uint32_t peer_addr(const void *p, int c) {
    uint32_t d;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(c));
    return d;
}
__device__ __forceinline__ uint32_t ld_cluster(uint32_t addr) {
    uint32_t x;
    asm volatile("ld.shared::cluster.b32 %0, [%1];" : "=r"(x) : "r"(addr));
    return x;
}
__device__ __forceinline__ uint32_t peer_ld(const void *p, int c) { return ld_cluster(peer_addr(p, c)); }
__device__ __forceinline__ void peer_add(const void *p, int c, int32_t x) {
    asm volatile("red.relaxed.cluster.shared::cluster.add.s32 [%0], %1;" ::"r"(peer_addr(p, c)), "r"(x) : "memory");
}

// A row: generic pointers, so that the copy in shared memory and the global
// array are read by the same instructions.  The loop's code is kept small
// throughout: most phases run a few hundred instructions on a few warps, and
// fetching them again in every iteration is what such a phase costs (a warp
// alone took about 25 cycles per instruction of straight-line code).
struct ResRow {
    const int32_t *a, *w;   // w null: unit weights
    int32_t d;
};
__device__ __forceinline__ ResRow row_of(const ResView &v, int i) {
    const uint32_t *row = arena_at<uint32_t>(v.oRow);
    const uint32_t b = row[i], e = row[i + 1];
    ResRow r;
    r.d = (int32_t)(e - b);
    const bool in = e <= v.cached;
    r.a = (in ? arena_at<int32_t>(v.oAdj) : v.gadj) + b;
    r.w = v.gew ? (in ? arena_at<int32_t>(v.oEw) : v.gew) + b : nullptr;
    return r;
}
// Entries t0, t0 + step, ... (pad where the row has ended) and their weights
// (1 there, and everywhere without edge weights).
template <int U>
__device__ __forceinline__ void row_entries(const ResRow &r, int t0, int step, int32_t pad, int32_t (&u)[U], int32_t (&w)[U]) {
#pragma unroll
    for (int q = 0; q < U; ++q) {
        const int t = t0 + q * step;
        u[q] = t < r.d ? r.a[t] : pad;
        w[q] = t < r.d && r.w ? r.w[t] : 1;
    }
}
__device__ __forceinline__ int32_t own_vw(const ResView &v, int i) {
    return v.oVw != kNone ? arena_at<int32_t>(v.oVw)[i] : __ldg(v.gvw + i);
}

// Appends from any subset of a warp's lanes (all lanes call it).
template <class T>
__device__ __forceinline__ void append(int *cnt, T *list, bool pred, T x) {
    const unsigned m = __ballot_sync(0xffffffffu, pred);
    if (!m) return;
    int b = 0;
    if (lane_id() == 0) b = atomicAdd(cnt, __popc(m));
    b = __shfl_sync(0xffffffffu, b, 0);
    if (pred) list[b + __popc(m & ((1u << lane_id()) - 1u))] = x;
}

__device__ __forceinline__ void sum_to(uint32_t *dst, uint32_t x) {   // all lanes; one shared atomic per warp
    x = __reduce_add_sync(0xffffffffu, x);
    if (lane_id() == 0 && x) atomicAdd(dst, x);
}

__device__ __noinline__ int32_t random_dest(int32_t u, int32_t it, int32_t nB) {
    const ResView &v = rs().v;
    const uint64_t h = splitmix64(v.seed ^ (0x9E3779B97F4A7C15ULL * (uint64_t)(it + 1)) ^ (uint64_t)(uint32_t)u);
    return (int32_t)arena_at<uint16_t>(v.oBs)[h % (uint64_t)nB];
}

// ---------------------------------------------------------------------------
// Step 1 of every pass: connectivity of the rows that the pass must read
// ---------------------------------------------------------------------------
// What one row gives: conn to the own part, and over the allowed parts (Jetlp:
// every other part; rebalancing: the parts of B) the best one with its conn
// (lowest id on ties; cb 0: none), the sum and the number of distinct ones.
struct RowEval {
    int32_t conn_s, cb, pb, sum, cnt;
};

// One thread, after a row's evaluation.  Jetlp: gain and first filter; returns
// the list entry when the vertex is in X, else kNone.  Rebalancing:
// destination, loss, slot and bucket.
template <class PT>
__device__ __noinline__ uint32_t row_decision(int32_t mode, int i, RowEval ev) {
    ResShared &s = rs();
    const ResView &v = s.v;
    if (mode == MODE_LP) {
        if (ev.cb == 0) return kNone;
        const int32_t gain = ev.cb - ev.conn_s;
        if (!first_filter(gain, ev.conn_s, v.cq16, v.abl)) return kNone;
        arena_at<int32_t>(v.oF)[i] = gain;
        return ((uint32_t)i << 16) | (uint32_t)ev.pb;
    }
    const int32_t a = arena_at<int16_t>(v.oAidx)[arena_at<PT>(v.oP)[v.base + i]];
    int32_t loss;
    if (mode == MODE_RW) {
        const int32_t dest = ev.cb ? ev.pb : random_dest(v.base + i, s.ctl.it, s.ctl.nB);
        arena_at<PT>(v.oD)[i] = (PT)dest;
        loss = ev.conn_s - ev.cb;
    } else {
        loss = ev.conn_s - (ev.cnt > 0 ? ev.sum / ev.cnt : 0);
    }
    const int slot = slot_of(loss);
    arena_at<uint8_t>(v.oKey)[i] = (uint8_t)slot;
    atomicAdd(&arena_at<uint32_t>(v.oBk)[a * kSlots + slot], (uint32_t)own_vw(v, i));
    return kNone;
}

// conn of the entries first, first + step, ... of a long row added into tab
// (four entries in flight per thread).
template <class PT>
__device__ __noinline__ void row_into(const ResRow r, int first, int step, int32_t *tab) {
    const PT *P = arena_at<PT>(rs().v.oP);
    constexpr int U = 4;
#pragma unroll 1
    for (int t0 = first; t0 < r.d; t0 += U * step) {
        int32_t u[U], w[U];
        row_entries<U>(r, t0, step, -1, u, w);
#pragma unroll
        for (int q = 0; q < U; ++q)
            if (u[q] >= 0) atomicAdd(&tab[P[u[q]]], w[q]);
    }
}

// The best allowed part, and the sums, over the parts p = first, first + step,
// ... of a table (one of `ntab` tables when the block shares a row); entries
// are cleared.
__device__ __forceinline__ RowEval scan_table(const ResView &v, bool lp, int32_t ps, int32_t *tab, int first, int step,
                                              int ntab) {
    const uint8_t *inB = arena_at<uint8_t>(v.oInB);
    RowEval ev{0, 0, INT32_MAX, 0, 0};
#pragma unroll 1
    for (int p = first; p < v.k; p += step) {
        int32_t c = 0;
#pragma unroll 1
        for (int w = 0; w < ntab; ++w) {
            c += tab[w * v.k + p];
            tab[w * v.k + p] = 0;
        }
        if (c != 0) {
            if (p == ps) {
                ev.conn_s = c;
            } else if (lp || inB[p]) {
                if (c > ev.cb) { ev.cb = c; ev.pb = p; }   // ascending p: the lowest id stays on ties
                ev.sum += c;
                ev.cnt += 1;
            }
        }
    }
    // over the warp
    const int32_t cb = __reduce_max_sync(0xffffffffu, ev.cb);
    ev.pb = __reduce_min_sync(0xffffffffu, ev.cb == cb ? ev.pb : INT32_MAX);
    ev.cb = cb;
    ev.conn_s = __reduce_add_sync(0xffffffffu, ev.conn_s);
    ev.sum = __reduce_add_sync(0xffffffffu, ev.sum);
    ev.cnt = __reduce_add_sync(0xffffffffu, ev.cnt);
    return ev;
}

// Rows that a thread could not take: one warp each with a k-entry table, hub
// rows by the whole block (every warp into its own table, then warp 0 sums
// them).
template <class PT>
__device__ __noinline__ void eval_long_rows(int32_t mode, int nlong, ResPart &part) {
    ResShared &s = rs();
    const ResView &v = s.v;
    const PT *P = arena_at<PT>(v.oP);
    uint32_t *list = arena_at<uint32_t>(v.oList);
    const uint16_t *big = arena_at<uint16_t>(v.oBig);
    int32_t *tabs = arena_at<int32_t>(v.oTab), *tab = tabs + (threadIdx.x >> 5) * v.k;
    const bool lp = mode == MODE_LP;
    uint32_t degx = 0;
    auto decide = [&](int i, int32_t d, const RowEval &ev) {   // one thread
        const uint32_t e = row_decision<PT>(mode, i, ev);
        if (e != kNone) {
            list[atomicAdd(&s.cnt, 1)] = e;
            degx += (uint32_t)d;
        }
    };
#pragma unroll 1
    for (int q = threadIdx.x >> 5; q < nlong; q += (int)(blockDim.x >> 5)) {
        const int i = big[q];
        const ResRow r = row_of(v, i);
        if (r.d > v.hub) {
            int slot = 0;
            if (lane_id() == 0) slot = atomicAdd(&s.nhub, 1);
            slot = __shfl_sync(0xffffffffu, slot, 0);
            if (slot < kHugeCap) {
                if (lane_id() == 0) s.hubs[slot] = (uint16_t)i;
                continue;
            }
        }
        row_into<PT>(r, (int)lane_id(), 32, tab);
        __syncwarp();
        const RowEval ev = scan_table(v, lp, P[v.base + i], tab, (int)lane_id(), 32, 1);
        __syncwarp();
        if (lane_id() == 0) decide(i, r.d, ev);
    }
    __syncthreads();
    const int nh = min(s.nhub, kHugeCap);
#pragma unroll 1
    for (int q = 0; q < nh; ++q) {
        const int i = s.hubs[q];
        const ResRow r = row_of(v, i);
        row_into<PT>(r, (int)threadIdx.x, (int)blockDim.x, tab);
        __syncthreads();
        if (threadIdx.x < 32) {
            const RowEval ev = scan_table(v, lp, P[v.base + i], tabs, (int)lane_id(), 32, (int)(blockDim.x >> 5));
            if (lane_id() == 0) decide(i, r.d, ev);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) s.nstage = s.nhub = 0;
    if (lane_id() == 0 && degx) atomicAdd(&part.degx, degx);
}

// Step 1.  First the vertices whose rows must be read go to a compact list
// (Jetlp: boundary and unlocked vertices; rebalancing: candidates with a
// neighbour in another part — the other candidates are finished on the spot).
// Then one thread takes a row: it keeps the allowed parts it meets, up to kSeen
// of them, with their connectivities in registers, which needs neither a table
// nor a second look at the row; a boundary row rarely sees more.  The few others
// are left to the warps.  (Lanes shared by a row, with match and shuffles, took
// three times the instructions; lists by row length, so that a warp's rows end
// together, cost more to build than they saved.)
template <class PT>
__device__ __forceinline__ void eval_rows(int32_t mode, ResPart &part) {
    ResShared &s = rs();
    const ResView &v = s.v;
    const PT *P = arena_at<PT>(v.oP);
    const int32_t *ext = arena_at<int32_t>(v.oExt);
    const uint8_t *inB = arena_at<uint8_t>(v.oInB);
    uint16_t *act = arena_at<uint16_t>(v.oAct), *big = arena_at<uint16_t>(v.oBig);
    const bool lp = mode == MODE_LP;
    const int lane = (int)lane_id(), first = (int)(threadIdx.x & ~31u);
    {
        const int32_t nB = s.ctl.nB, it = s.ctl.it;
        const bool use_locks = !ablate_locks(v.abl);
        uint32_t n1 = 0;                 // boundary vertices (Jetlp) or candidates
        if (!lp) {                       // the plan's sums (in memory that F holds in a Jetlp pass)
            int32_t *tot = arena_at<int32_t>(v.oTot);
            for (int i = threadIdx.x; i < s.ctl.nA * kSlots; i += blockDim.x) tot[i] = 0;
        }
#pragma unroll 1
        for (int i0 = first; i0 < v.own; i0 += blockDim.x) {
            const int i = i0 + lane;
            bool read = false, one = false;
            if (i < v.own) {
                if (lp) {
                    uint8_t *flag = arena_at<uint8_t>(v.oFlag);
                    one = ext[i] > 0;
                    read = one && !(use_locks && flag[i]);
                    flag[i] = 0;         // M of this Jetlp sets the next locks
                } else {
                    const int32_t ps = P[v.base + i];
                    const int32_t a = nB > 0 ? arena_at<int16_t>(v.oAidx)[ps] : -1;
                    int slot = kNoSlot;
                    if (a >= 0 && 2LL * own_vw(v, i) <= 3LL * ((int64_t)arena_at<int32_t>(v.oPw)[ps] - v.opt)) {
                        one = true;
                        read = ext[i] != 0;
                        if (!read) {     // the whole row is in the own (oversized) part
                            slot = slot_of(v.oWdeg != kNone ? arena_at<int32_t>(v.oWdeg)[i] : v.gwdeg[i]);
                            if (mode == MODE_RW) arena_at<PT>(v.oD)[i] = (PT)random_dest(v.base + i, it, nB);
                            atomicAdd(&arena_at<uint32_t>(v.oBk)[a * kSlots + slot], (uint32_t)own_vw(v, i));
                        }
                    }
                    arena_at<uint8_t>(v.oKey)[i] = (uint8_t)slot;
                }
            }
            n1 += __popc(__ballot_sync(0xffffffffu, one));
            append(&s.nact, act, read, (uint16_t)i);
        }
        if (lane == 0 && n1) atomicAdd(lp ? &part.nbnd : &part.ncand, n1);
    }
    __syncthreads();
    const int m = s.nact;
    uint32_t degrows = 0, degx = 0;
#pragma unroll 1
    for (int j0 = first; j0 < m; j0 += blockDim.x) {
        const int j = j0 + lane;
        const int i = j < m ? act[j] : 0;
        bool stage = false;
        uint32_t entry = kNone;
        if (j < m) {
            const ResRow r = row_of(v, i);
            const int32_t ps = P[v.base + i];
            degrows += (uint32_t)r.d;
            stage = r.d > kThreadRow;
            RowEval ev{0, 0, INT32_MAX, 0, 0};
            int32_t sp[kSeen], sc[kSeen];
#pragma unroll
            for (int q = 0; q < kSeen; ++q) { sp[q] = -1; sc[q] = 0; }
            constexpr int U = 4;
            const int d = stage ? 0 : r.d;
#pragma unroll 1
            for (int t0 = 0; t0 < d; t0 += U) {
                int32_t p[U], w[U];
                row_entries<U>(r, t0, 1, -1, p, w);
#pragma unroll
                for (int q = 0; q < U; ++q) p[q] = p[q] >= 0 ? P[p[q]] : -1;
#pragma unroll
                for (int q = 0; q < U; ++q) {
                    if (p[q] == ps) {
                        ev.conn_s += w[q];
                    } else if (p[q] >= 0 && (lp || inB[p[q]])) {
                        ev.sum += w[q];
                        bool hit = false;
#pragma unroll
                        for (int z = 0; z < kSeen; ++z) {
                            const bool eq = sp[z] == p[q];
                            sc[z] += eq ? w[q] : 0;
                            hit |= eq;
                        }
                        if (!hit) {   // the first free place (parts fill them in order)
#pragma unroll
                            for (int z = 0; z < kSeen; ++z)
                                if (z == ev.cnt) { sp[z] = p[q]; sc[z] = w[q]; }
                            ev.cnt += 1;
                        }
                    }
                }
            }
            if (ev.cnt > kSeen) stage = true;
#pragma unroll
            for (int z = 0; z < kSeen; ++z)
                if (sc[z] > ev.cb || (sc[z] == ev.cb && z < ev.cnt && sp[z] < ev.pb)) { ev.cb = sc[z]; ev.pb = sp[z]; }
            if (!stage) entry = row_decision<PT>(mode, i, ev);
            if (entry != kNone) degx += (uint32_t)r.d;
        }
        append(&s.cnt, arena_at<uint32_t>(v.oList), entry != kNone, entry);
        append(&s.nstage, big, stage, (uint16_t)i);
    }
    if (first < m) {
        sum_to(&part.degexam, degrows);
        if (lp) sum_to(&part.degx, degx);
    }
    if (threadIdx.x == 0) *(lp ? &part.nexam : &part.nbnd) = (uint32_t)m;
    __syncthreads();
    const int ns = s.nstage;
    if (ns > 0) eval_long_rows<PT>(mode, ns, part);
}

// ---------------------------------------------------------------------------
// move lists
// ---------------------------------------------------------------------------
// Every block reads the lists of all blocks into its copy of N: the wanted
// parts of X (final_ false), or the moves of M with the other members of the
// lists back at their own part (final_ true).  A list's first entries are
// fetched together with its length.
template <class PT>
__device__ __noinline__ void pull_lists(bool final_) {
    ResShared &s = rs();
    const ResView &v = s.v;
    const PT *P = arena_at<PT>(v.oP);
    PT *N = arena_at<PT>(v.oN);
    const int warp = (int)(threadIdx.x >> 5);
    const int c = warp >> v.wps;                          // source block; 1 << wps warps each
    const int step = 32 << v.wps;
    const uint32_t list = peer_addr(arena_at<uint32_t>(v.oList), c);
    const int32_t base = c * v.S;
    const int m = (int)peer_ld(&s.cnt, c);
    constexpr int U = 4;
#pragma unroll 1
    for (int j0 = (warp & ((1 << v.wps) - 1)) * 32 + (int)lane_id(); j0 < v.S; j0 += U * step) {
        uint32_t e[U];
#pragma unroll
        for (int q = 0; q < U; ++q) e[q] = j0 + q * step < v.S ? ld_cluster(list + 4u * (uint32_t)(j0 + q * step)) : 0u;
        if (j0 >= m) break;
#pragma unroll
        for (int q = 0; q < U; ++q) {
            if (j0 + q * step >= m) continue;
            const int32_t u = base + (int32_t)(e[q] >> 16);
            N[u] = final_ && !(e[q] & kMoveBit) ? P[u] : (PT)(e[q] & kDestMask);
        }
    }
}

// ---------------------------------------------------------------------------
// Afterburner (Alg. 4 second loop) and apply, over the own list
// ---------------------------------------------------------------------------
// Both walk the rows of list members: eight lanes per row of up to kThreadRow
// entries while the list is short, one thread when it fills the block, a warp
// per longer row, the block per hub row; `share(r, e, first,
// step, x, y)` adds a thread's part into x and y, `done(j, e, r, x, y)` runs in
// one thread with the sums.  take(e): whether the member's row is read.
template <class Take, class Share, class Done>
__device__ __forceinline__ void walk_list(int m, Take &&take, Share &&share, Done &&done) {
    ResShared &s = rs();
    const ResView &v = s.v;
    const uint32_t *list = arena_at<uint32_t>(v.oList);
    uint16_t *big = arena_at<uint16_t>(v.oBig);
    const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5), warps = (int)(blockDim.x >> 5);
    const int lw = m <= 4 * warps ? 3 : (m <= 16 * warps ? 1 : 0);   // log2 of the lanes per short row
    // pass 0: groups over the whole list; 1: warps over the staged rows; 2: the block over the hub rows
#pragma unroll 1
    for (int pass = 0; pass < (v.hasbig ? 3 : 1); ++pass) {
        const int width = pass == 0 ? 1 << lw : (pass == 1 ? 32 : (int)blockDim.x);
        int count = m;
        if (pass > 0) {
            __syncthreads();
            count = pass == 1 ? s.nstage : min(s.nhub, kHugeCap);
        }
        const int ipw = pass == 0 ? 32 >> lw : 1;            // items per warp and step
        const int q0 = pass == 2 ? 0 : warp * ipw, qs = pass == 2 ? 1 : warps * ipw;
#pragma unroll 1
        for (int q = q0; q < count; q += qs) {
            const int item = q + (pass == 0 ? lane >> lw : 0);
            bool on = item < count;
            int j = 0;
            if (on) j = pass == 0 ? item : (pass == 1 ? (int)big[item] : (int)s.hubs[item]);
            const uint32_t e = list[j];
            const ResRow r = row_of(v, (int)(e >> 16));
            on = on && take(e);
            if (pass == 0 && v.hasbig) {
                append(&s.nstage, big, on && r.d > kThreadRow && (lane & (width - 1)) == 0, (uint16_t)j);
                on = on && r.d <= kThreadRow;
            } else if (pass == 1 && r.d > v.hub) {
                int slot = 0;
                if (lane == 0) slot = atomicAdd(&s.nhub, 1);
                slot = __shfl_sync(0xffffffffu, slot, 0);
                if (slot < kHugeCap) {
                    if (lane == 0) s.hubs[slot] = (uint16_t)j;
                    continue;
                }
            }
            int32_t x = 0, y = 0;
            const int first = pass == 2 ? (int)threadIdx.x : (lane & (width - 1));
            if (on) share(r, e, first, width, x, y);
            __syncwarp();
#pragma unroll 1
            for (int o = min(width, 32) >> 1; o > 0; o >>= 1) {
                x += __shfl_xor_sync(0xffffffffu, x, o);
                y += __shfl_xor_sync(0xffffffffu, y, o);
            }
            bool last = on && first == 0;
            if (pass == 2) {
                if (threadIdx.x < 2) s.red[threadIdx.x] = 0;
                __syncthreads();
                if (lane == 0) {
                    atomicAdd(&s.red[0], x);
                    atomicAdd(&s.red[1], y);
                }
                __syncthreads();
                x = s.red[0];
                y = s.red[1];
                __syncthreads();
                last = threadIdx.x == 0;
            }
            if (last) done(j, e, r, x, y);
        }
    }
    if (v.hasbig) {
        __syncthreads();
        if (threadIdx.x == 0) s.nstage = s.nhub = 0;
    }
}

// Afterburner and second filter over the own X: sets the move bit of M.
template <class PT>
__device__ __forceinline__ void lp_afterburn(ResPart &part) {
    ResShared &s = rs();
    const ResView &v = s.v;
    const PT *P = arena_at<PT>(v.oP), *N = arena_at<PT>(v.oN);
    int32_t *F = arena_at<int32_t>(v.oF);
    uint32_t *list = arena_at<uint32_t>(v.oList);
    const int m = s.cnt;
    uint32_t nm = 0;
    if (v.abl & (ABL_NO_AFTERBURN | ABL_BASELINE_LP)) {
        for (int j = threadIdx.x; j < m; j += blockDim.x) {
            list[j] |= kMoveBit;
            nm += 1;
        }
    } else {
        walk_list(
            m, [](uint32_t) { return true; },
            [&](const ResRow &r, uint32_t e, int first, int step, int32_t &f2, int32_t &) {
                const int i = (int)(e >> 16);
                const int32_t me = v.base + i, ps = P[me], pd = (int32_t)(e & kDestMask), Fv = F[i];
                constexpr int U = 4;
#pragma unroll 1
                for (int t0 = first; t0 < r.d; t0 += U * step) {
                    int32_t u[U], w[U], pu[U], nu[U];
                    row_entries<U>(r, t0, step, -1, u, w);
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        pu[q] = u[q] >= 0 ? P[u[q]] : -1;
                        nu[q] = u[q] >= 0 ? N[u[q]] : -1;
                    }
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        if (nu[q] != pu[q]) {   // a member of X: it counts at its destination if it precedes v in ord
                            const int c = (int)__umulhi((uint32_t)u[q], v.magic);
                            const int32_t fu = (int32_t)peer_ld(F + (u[q] - c * v.S), c);
                            if (fu > Fv || (fu == Fv && u[q] < me)) pu[q] = nu[q];
                        }
                        f2 += pu[q] == pd ? w[q] : (pu[q] == ps ? -w[q] : 0);
                    }
                }
            },
            [&](int j, uint32_t e, const ResRow &, int32_t f2, int32_t) {
                if (f2 >= 0) {
                    list[j] = e | kMoveBit;
                    nm += 1;
                }
            });
    }
    sum_to(&part.nM, nm);
}

// Apply M: exact cut change, part weights, ext of the movers and of their
// neighbours, locks.
template <class PT>
__device__ __forceinline__ void apply_moves(ResPart &part, int32_t *delta, bool lp) {
    ResShared &s = rs();
    const ResView &v = s.v;
    const PT *P = arena_at<PT>(v.oP), *N = arena_at<PT>(v.oN);
    int32_t *ext = arena_at<int32_t>(v.oExt);
    int32_t dcut = 0;
    uint32_t degm = 0;
    walk_list(
        s.cnt, [](uint32_t e) { return (e & kMoveBit) != 0; },
        [&](const ResRow &r, uint32_t e, int first, int step, int32_t &c, int32_t &ne) {
            const int32_t me = v.base + (int)(e >> 16), a = P[me], b = (int32_t)(e & kDestMask);
            constexpr int U = 4;
#pragma unroll 1
            for (int t0 = first; t0 < r.d; t0 += U * step) {
                int32_t u[U], w[U], pu[U], pn[U];
                row_entries<U>(r, t0, step, -1, u, w);
#pragma unroll
                for (int q = 0; q < U; ++q) {
                    pu[q] = u[q] >= 0 ? P[u[q]] : 0;
                    pn[q] = u[q] >= 0 ? N[u[q]] : 0;
                }
#pragma unroll
                for (int q = 0; q < U; ++q) {
                    if (u[q] < 0) continue;
                    const int32_t diff = (int)(pn[q] != b) - (int)(pu[q] != a);
                    ne += pn[q] != b;
                    const bool stays = pn[q] == pu[q];
                    if (stays && diff) {
                        const int o = (int)__umulhi((uint32_t)u[q], v.magic);
                        peer_add(ext + (u[q] - o * v.S), o, diff);
                    }
                    // an edge whose ends both move counts at the smaller id
                    if (stays || u[q] > me) c += w[q] * diff;
                }
            }
        },
        [&](int, uint32_t e, const ResRow &r, int32_t c, int32_t ne) {
            const int i = (int)(e >> 16);
            const int32_t wv = own_vw(v, i);
            atomicAdd(&delta[P[v.base + i]], -wv);
            atomicAdd(&delta[e & kDestMask], wv);
            dcut += c;
            degm += (uint32_t)r.d;
            ext[i] = ne;
            if (lp) arena_at<uint8_t>(v.oFlag)[i] = 1;
        });
    dcut = __reduce_add_sync(0xffffffffu, dcut);
    if (lane_id() == 0 && dcut) atomicAdd(&part.dcut, dcut);
    sum_to(&part.degm, degm);
}

// ---------------------------------------------------------------------------
// rebalancing: eviction
// ---------------------------------------------------------------------------
// Boundary slot of each oversized part from all blocks' buckets, and the
// weight this block's members of that slot may still take: `need` less what
// the blocks before this one hold there.  A warp per (part, block) first adds
// the buckets up (all blocks', and those of the blocks before this one), then
// a warp per part finds the slot.
__device__ __noinline__ void rb_plan(int32_t nA) {
    const ResView &v = rs().v;
    const uint32_t *bk = arena_at<uint32_t>(v.oBk);
    int32_t *tot = arena_at<int32_t>(v.oTot), *pre = arena_at<int32_t>(v.oTab);   // zero when the plan begins
    const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5);
    const int lcs = 31 - __clz(v.cs);
#pragma unroll 1
    for (int q = warp; q < nA << lcs; q += (int)(blockDim.x >> 5)) {
        const int a = (q >> lcs) * kSlots, c = (q + v.rank) & (v.cs - 1);
        const int32_t x = (int32_t)peer_ld(bk + a + lane, c), x32 = (int32_t)peer_ld(bk + a + 32, c);
        if (x) {
            atomicAdd(&tot[a + lane], x);
            if (c < v.rank) atomicAdd(&pre[a + lane], x);
        }
        if (lane == 0 && x32) {
            atomicAdd(&tot[a + 32], x32);
            if (c < v.rank) atomicAdd(&pre[a + 32], x32);
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int a = warp; a < nA; a += (int)(blockDim.x >> 5)) {
        const int32_t t = tot[a * kSlots + lane], t32 = tot[a * kSlots + 32], ex = arena_at<int32_t>(v.oExcess)[a];
        int32_t inc = t;
#pragma unroll 1
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        const unsigned m = __ballot_sync(0xffffffffu, inc >= ex);
        const int32_t tot31 = __shfl_sync(0xffffffffu, inc, 31);
        const int32_t before = m ? __shfl_sync(0xffffffffu, inc - t, __ffs(m) - 1) : tot31;
        const int slot = m ? __ffs(m) - 1 : ((int64_t)tot31 + t32 >= ex ? 32 : kSlots);
        if (lane == 0) {
            arena_at<uint8_t>(v.oSs)[a] = (uint8_t)slot;
            arena_at<int32_t>(v.oNeed)[a] = slot < kSlots ? ex - before - pre[a * kSlots + slot] : 0;
        }
    }
}

// The run of consecutive own vertices that a warp takes, in order.
__device__ __forceinline__ int warp_run(const ResView &v) { return ((v.S + (int)(blockDim.x >> 5) - 1) / (int)(blockDim.x >> 5) + 31) & ~31; }

// Eviction in (slot, vertex id) order: per warp and part the weight of its
// run's boundary-slot members, an exclusive scan over the warps, then each
// warp walks its run 32 vertices at a time, one part after another.  Jetrw
// puts the taken vertices on the list; Jetrs marks them and returns the
// warp's evicted weight.
template <class PT>
__device__ __noinline__ uint32_t rb_take(int32_t mode, ResPart &part) {
    ResShared &s = rs();
    const ResView &v = s.v;
    const PT *P = arena_at<PT>(v.oP), *D = arena_at<PT>(v.oD);
    uint8_t *key = arena_at<uint8_t>(v.oKey);
    const int16_t *aidx = arena_at<int16_t>(v.oAidx);
    const uint8_t *ss = arena_at<uint8_t>(v.oSs);
    const int32_t *need = arena_at<int32_t>(v.oNeed);
    const int32_t nA = s.ctl.nA;
    int32_t *hist = arena_at<int32_t>(v.oTab);
    const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5);
    int32_t *run = hist + warp * nA;
#pragma unroll 1
    for (int a = lane; a < nA; a += 32) run[a] = 0;
    __syncwarp();
    const int chunk = warp_run(v);
    const int lo = warp * chunk, hi = min(lo + chunk, v.own);
#pragma unroll 1
    for (int i = lo + lane; i < hi; i += 32) {
        const int sl = key[i];
        if (sl != kNoSlot) {
            const int a = aidx[P[v.base + i]];
            if (sl == ss[a]) atomicAdd(&run[a], own_vw(v, i));
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int a = warp; a < nA; a += (int)(blockDim.x >> 5)) {   // lanes = warps
        const int32_t x0 = lane < (int)(blockDim.x >> 5) ? hist[lane * nA + a] : 0;
        int32_t x = x0;
#pragma unroll 1
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane < (int)(blockDim.x >> 5)) hist[lane * nA + a] = x - x0;
    }
    __syncthreads();
    uint32_t tw = 0, nm = 0;
#pragma unroll 1
    for (int i0 = lo; i0 < hi; i0 += 32) {       // whole warp
        const int i = i0 + lane;
        const int sl = i < hi ? key[i] : kNoSlot;
        const bool cand = sl != kNoSlot;
        if (!__any_sync(0xffffffffu, cand)) continue;
        const int a = cand ? aidx[P[v.base + i]] : -1;
        const int sb = cand ? ss[a] : 0;
        const bool member = cand && sl == sb;
        const int32_t w = cand ? own_vw(v, i) : 0;
        bool taken = cand && sl < sb;
        unsigned todo = __ballot_sync(0xffffffffu, member);
#pragma unroll 1
        while (todo) {                           // the members of one part: an inclusive scan of their weights
            const int a1 = __shfl_sync(0xffffffffu, a, __ffs(todo) - 1);
            const bool in = member && a == a1;
            int32_t x = in ? w : 0;
#pragma unroll 1
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            const int32_t base = run[a1];
            if (in) taken = base + x - w < need[a1];
            __syncwarp();
            if (lane == 31) run[a1] = base + x;
            __syncwarp();
            todo &= ~__ballot_sync(0xffffffffu, in);
        }
        if (mode == MODE_RW) {
            append(&s.cnt, arena_at<uint32_t>(v.oList), taken,
                   ((uint32_t)i << 16) | kMoveBit | (taken ? (uint32_t)D[i] : 0u));
            nm += taken;
        } else {
            if (i < hi) key[i] = taken ? kTakenSlot : kNoSlot;
            tw += taken ? (uint32_t)w : 0u;
        }
    }
    sum_to(&part.nM, nm);
    return __reduce_add_sync(0xffffffffu, tw);
}

// Jetrs cookie cutter: before = evicted weight of the vertices before this
// warp's run.
__device__ __noinline__ void rb_cookie(ResPart &part, int64_t before) {
    ResShared &s = rs();
    const ResView &v = s.v;
    const uint8_t *key = arena_at<uint8_t>(v.oKey);
    const int64_t *cap = arena_at<int64_t>(v.oCap);
    const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5);
    const int chunk = warp_run(v);
    const int lo = warp * chunk, hi = min(lo + chunk, v.own);
    const int32_t nB = s.ctl.nB;
    const int64_t total2 = 2 * cap[nB];
    uint32_t nm = 0;
#pragma unroll 1
    for (int i0 = lo; i0 < hi; i0 += 32) {
        const int i = i0 + lane;
        const int32_t w = i < hi && key[i] == kTakenSlot ? own_vw(v, i) : 0;
        if (!__any_sync(0xffffffffu, w > 0)) continue;
        int32_t x = w;
#pragma unroll 1
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        int32_t dest = -1;
        if (w > 0) {
            const int64_t mid2 = 2 * (before + x - w) + w;
            if (mid2 < total2) {
                int b0 = 0, b1 = nB - 1;   // largest b with 2 C_b <= mid2
#pragma unroll 1
                while (b0 < b1) {
                    const int mid = (b0 + b1 + 1) >> 1;
                    if (2 * cap[mid] <= mid2) b0 = mid;
                    else b1 = mid - 1;
                }
                if (mid2 < 2 * cap[b0 + 1]) dest = arena_at<uint16_t>(v.oBs)[b0];
            }
        }
        before += __shfl_sync(0xffffffffu, x, 31);
        append(&s.cnt, arena_at<uint32_t>(v.oList), dest >= 0, ((uint32_t)i << 16) | kMoveBit | (uint32_t)dest);
        nm += dest >= 0;
    }
    sum_to(&part.nM, nm);
}

// ---------------------------------------------------------------------------
// controller (Alg. 3), the same in every block
// ---------------------------------------------------------------------------
// Rebalancing classes, prepared whatever the next mode is, by two warps: A numbered in ascending id with its excess (which = 0), B listed with
// the capacity prefix (which = 1).
__device__ __noinline__ void res_classes(int which) {
    ResShared &s = rs();
    const ResView &v = s.v;
    const int32_t *pw = arena_at<int32_t>(v.oPw);
    const int lane = (int)lane_id();
    const unsigned lt = (1u << lane) - 1u;
    int32_t cnt = 0;
    long long cc = 0;
#pragma unroll 1
    for (int p0 = 0; p0 < v.k; p0 += 32) {
        const int p = p0 + lane;
        const long long w = p < v.k ? pw[p] : 0;
        const bool in = p < v.k && (which == 0 ? w > v.Llim : w <= v.sigma);
        const unsigned m = __ballot_sync(0xffffffffu, in);
        const int idx = cnt + __popc(m & lt);
        cnt += __popc(m);
        if (which == 0) {
            if (p < v.k) arena_at<int16_t>(v.oAidx)[p] = in ? (int16_t)idx : (int16_t)-1;
            if (in) arena_at<int32_t>(v.oExcess)[idx] = (int32_t)(w - v.Llim);
        } else {
            const long long room = in ? v.sigma - w : 0;
            long long x = room;
#pragma unroll 1
            for (int o = 1; o < 32; o <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (p < v.k) arena_at<uint8_t>(v.oInB)[p] = in ? 1 : 0;
            if (in) {
                arena_at<uint16_t>(v.oBs)[idx] = (uint16_t)p;
                arena_at<int64_t>(v.oCap)[idx] = cc + x - room;
            }
            cc += __shfl_sync(0xffffffffu, x, 31);
        }
    }
    if (lane == 0) {
        if (which == 0) {
            s.ctl.nA = cnt;
        } else {
            s.ctl.nB = cnt;
            arena_at<int64_t>(v.oCap)[cnt] = cc;
        }
    }
}

// Mode of the next iteration (as next_mode_of of the per-kernel loop).
__device__ __forceinline__ int32_t res_next_mode(const ResView &v, bool balanced, int32_t noimp, int32_t it,
                                                 int32_t &weak, int32_t &hit_cap) {
    if (noimp >= v.max_no_improve) return MODE_DONE;
    if (it >= v.max_iters) { hit_cap = 1; return MODE_DONE; }
    if (balanced) { weak = 0; return MODE_LP; }
    if (weak < v.weak_limit) { weak += 1; return MODE_RW; }
    return MODE_RS;
}

// Sum of one field over the blocks (a whole warp; lane c reads block c).
__device__ __forceinline__ uint32_t part_sum(const ResView &v, ResPart &part, int f) {
    uint32_t *p = reinterpret_cast<uint32_t *>(&part) + f;
    const uint32_t x = (int)lane_id() < v.cs ? peer_ld(p, (int)lane_id()) : 0u;
    return __reduce_add_sync(0xffffffffu, x);
}

// Part weights += every block's delta (each warp takes one block's share; the
// caller synchronises).
__device__ __forceinline__ void add_deltas(const ResView &v, int32_t *delta) {
    int32_t *pw = arena_at<int32_t>(v.oPw);
    const int warp = (int)(threadIdx.x >> 5);
    const uint32_t d = peer_addr(delta, warp >> v.wps);
#pragma unroll 1
    for (int p = (warp & ((1 << v.wps) - 1)) * 32 + (int)lane_id(); p < v.k; p += 32 << v.wps) {
        const int32_t x = (int32_t)ld_cluster(d + 4u * (uint32_t)p);
        if (x) atomicAdd(&pw[p], x);
    }
}
__device__ __forceinline__ int32_t warp_max_pw(const ResView &v) {
    const int32_t *pw = arena_at<int32_t>(v.oPw);
    int32_t m = 0;
#pragma unroll 1
    for (int p = lane_id(); p < v.k; p += 32) m = max(m, pw[p]);
    return __reduce_max_sync(0xffffffffu, m);
}

// ---------------------------------------------------------------------------
// a level
// ---------------------------------------------------------------------------
// Level start: layout, parts, own rows, ext, weighted degrees, part weights,
// cut, and the first mode.
template <class PT>
__device__ __noinline__ void res_level_start(const ResJob &job, int32_t lvi) {
    cg::cluster_group cl = cg::this_cluster();
    ResShared &s = rs();
    const ResLevel &lv = job.lv[lvi];
    const int32_t *prev = lvi > 0 ? job.lv[lvi - 1].out : job.init;
    if (threadIdx.x == 0) {
        ResView v;
        v.n = lv.g.n;
        v.k = job.k;
        v.rank = (int32_t)cl.block_rank();
        v.cs = (int32_t)cl.num_blocks();
        v.S = res_slice_dev(v.n, v.cs);
        v.base = v.rank * v.S;
        v.own = max(0, min(v.S, v.n - v.base));
        if (v.own == 0) v.base = v.n;
        v.magic = (uint32_t)(0x100000000ull / (uint32_t)v.S) + 1u;
        v.wps = 0;
        while ((v.cs << (v.wps + 1)) <= (int)(blockDim.x >> 5)) ++v.wps;
        uint32_t p = res_layout(v, v.n, v.S, v.k, (uint32_t)sizeof(PT));
        const int64_t e0 = lv.g.xadj[v.base], e1 = lv.g.xadj[v.base + v.own];
        v.gadj = lv.g.adj + e0;
        v.gew = lv.g.ew ? lv.g.ew + e0 : nullptr;
        v.gvw = lv.g.vw + v.base;
        v.gwdeg = job.wdeg + v.base;
        // what is left of the arena: vertex weights, weighted degrees, then rows
        const uint32_t vb = up16((uint32_t)v.S * 4);
        v.oVw = v.oWdeg = kNone;
        if (p + vb <= job.arena_bytes) { v.oVw = p; p += vb; }
        if (p + vb <= job.arena_bytes) { v.oWdeg = p; p += vb; }
        const uint32_t per = v.gew ? 8u : 4u;
        const uint32_t room = job.arena_bytes > p + 32u ? (job.arena_bytes - p - 32u) / per : 0u;
        v.cached = (uint32_t)min((int64_t)room, e1 - e0);
        v.oAdj = p;
        v.oEw = v.gew ? p + up16(v.cached * 4) : p;
        v.hasbig = 0;
        v.hub = job.hub_deg;
        v.abl = job.abl;
        v.cq16 = lv.cq16;
        v.max_no_improve = job.max_no_improve;
        v.weak_limit = job.weak_limit;
        v.max_iters = job.max_iters;
        v.seed = lv.seed;
        v.Llim = job.Llim; v.opt = job.opt; v.sigma = job.sigma; v.phi_ppm = job.phi_ppm;
        s.v = v;
        memset(&s.ctl, 0, sizeof(s.ctl));
        memset(s.part, 0, sizeof(s.part));
        memset(s.acc, 0, sizeof(s.acc));
        s.cnt = s.nact = s.nstage = s.nhub = s.anybig = 0;
    }
    __syncthreads();
    const ResView &v = s.v;
    PT *P = arena_at<PT>(v.oP), *N = arena_at<PT>(v.oN);
    {
        constexpr int U = 4;
#pragma unroll 1
        for (int u0 = threadIdx.x; u0 < v.n; u0 += U * (int)blockDim.x) {
            int32_t x[U];
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const int u = u0 + q * (int)blockDim.x;
                x[q] = u < v.n ? (lv.cmap ? __ldg(lv.cmap + u) : prev[u]) : 0;
            }
            if (lv.cmap) {
#pragma unroll
                for (int q = 0; q < U; ++q)
                    if (u0 + q * (int)blockDim.x < v.n) x[q] = prev[x[q]];
            }
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const int u = u0 + q * (int)blockDim.x;
                if (u < v.n) {
                    P[u] = (PT)x[q];
                    N[u] = (PT)x[q];
                }
            }
        }
    }
    uint32_t *row = arena_at<uint32_t>(v.oRow);
    {
        const int64_t e0 = lv.g.xadj[v.base];
        bool anybig = false;
#pragma unroll 1
        for (int i = threadIdx.x; i <= v.own; i += blockDim.x) {
            const int64_t b = lv.g.xadj[v.base + i];
            row[i] = (uint32_t)(b - e0);
            if (i < v.own) anybig |= lv.g.xadj[v.base + i + 1] - b > kThreadRow;
        }
        if (anybig) s.anybig = 1;   // every writer stores the same
        int32_t *sadj = arena_at<int32_t>(v.oAdj), *sew = arena_at<int32_t>(v.oEw);
#pragma unroll 1
        for (uint32_t j = threadIdx.x; j < v.cached; j += blockDim.x) {
            sadj[j] = __ldg(v.gadj + j);
            if (v.gew) sew[j] = __ldg(v.gew + j);
        }
        uint8_t *flag = arena_at<uint8_t>(v.oFlag);
#pragma unroll 1
        for (int i = threadIdx.x; i < v.own; i += blockDim.x) {
            flag[i] = 0;
            if (v.oVw != kNone) arena_at<int32_t>(v.oVw)[i] = __ldg(v.gvw + i);
        }
        int32_t *pw = arena_at<int32_t>(v.oPw), *delta = arena_at<int32_t>(v.oDelta);
#pragma unroll 1
        for (int p = threadIdx.x; p < v.k; p += blockDim.x) pw[p] = delta[p] = delta[v.k + p] = 0;
#pragma unroll 1
        for (int i = threadIdx.x; i < v.k * kSlots; i += blockDim.x) {
            arena_at<uint32_t>(v.oBk)[i] = 0;
            arena_at<int32_t>(v.oTab)[i] = 0;
        }
        // every own vertex goes on the list for the walk below (no move: destination = its part)
        uint32_t *list = arena_at<uint32_t>(v.oList);
#pragma unroll 1
        for (int i = threadIdx.x; i < v.own; i += blockDim.x) list[i] = (uint32_t)i << 16;
    }
    __syncthreads();
    if (threadIdx.x == 0) s.v.hasbig = s.anybig;
    __syncthreads();
    // ext, cut and weights of the own rows; the sums go where "iteration -1"
    // would leave them (part[1], delta[k..2k)).  The weighted degree is a
    // second walk over the rows.
    {
        int32_t *ext = arena_at<int32_t>(v.oExt);
        int32_t *wdeg = v.oWdeg != kNone ? arena_at<int32_t>(v.oWdeg) : v.gwdeg;
        PT *best = arena_at<PT>(v.oBest);
        int32_t *delta = arena_at<int32_t>(v.oDelta) + v.k;
        int32_t cut = 0;
#pragma unroll 1
        for (int round = 0; round < 2; ++round) {
            walk_list(
                v.own, [](uint32_t) { return true; },
                [&](const ResRow &r, uint32_t e, int first, int step, int32_t &c, int32_t &ne) {
                    const int32_t ps = P[v.base + (int)(e >> 16)];
                    constexpr int U = 4;
#pragma unroll 1
                    for (int t0 = first; t0 < r.d; t0 += U * step) {
                        int32_t u[U], w[U];
                        row_entries<U>(r, t0, step, -1, u, w);
#pragma unroll
                        for (int q = 0; q < U; ++q) {
                            const bool other = u[q] >= 0 && (round == 1 || P[u[q]] != ps);
                            c += other ? w[q] : 0;
                            ne += other ? 1 : 0;
                        }
                    }
                },
                [&](int i, uint32_t, const ResRow &, int32_t c, int32_t ne) {
                    if (round == 1) {
                        wdeg[i] = c;
                    } else {
                        const int32_t ps = P[v.base + i];
                        best[i] = (PT)ps;
                        atomicAdd(&delta[ps], own_vw(v, i));
                        cut += c;
                        ext[i] = ne;
                    }
                });
            __syncthreads();
        }
        // twice the cut: below 2^31 (the sum of all entries' weights is)
        cut = __reduce_add_sync(0xffffffffu, cut);
        if (lane_id() == 0 && cut) atomicAdd(&s.part[1].dcut, cut);
    }
    cl.sync();
    add_deltas(v, arena_at<int32_t>(v.oDelta) + v.k);
    __syncthreads();
    if (threadIdx.x < 32) {
        const int32_t maxw = warp_max_pw(v);
        const int64_t cut = (int64_t)part_sum(v, s.part[1], kfDcut) / 2;
        if (threadIdx.x == 0) {
            ResCtl &c = s.ctl;
            c.cut = c.best_cut = cut;
            c.best_maxw = maxw;
            c.best_bal = maxw <= v.Llim;
            c.mode = res_next_mode(v, maxw <= v.Llim, 0, 0, c.weak, c.hit_cap);
        }
    } else if (threadIdx.x < 64) {
        res_classes(0);
    } else if (threadIdx.x < 96) {
        res_classes(1);
    }
    __syncthreads();
}

// The whole loop of Alg. 3 on one level.
template <class PT>
__device__ __forceinline__ void res_level_loop(TraceRec *trace) {
    cg::cluster_group cl = cg::this_cluster();
    ResShared &s = rs();
    const ResView &v = s.v;
#pragma unroll 1
    for (;;) {
        const int32_t mode = s.ctl.mode;
        if (mode == MODE_DONE) break;
        const int buf = s.ctl.it & 1;
        const int32_t na = s.ctl.nA;
        ResPart &part = s.part[buf];
        int32_t *delta = arena_at<int32_t>(v.oDelta) + buf * v.k;
        eval_rows<PT>(mode, part);
        cl.sync();
        if (mode == MODE_LP) {
            if (threadIdx.x == 0) part.nX = (uint32_t)s.cnt;
            pull_lists<PT>(false);
            __syncthreads();
            lp_afterburn<PT>(part);
        } else {
            rb_plan(na);
            __syncthreads();
            const uint32_t tw = rb_take<PT>(mode, part);
            if (mode == MODE_RS) {
                if (lane_id() == 0) {
                    s.wsum[threadIdx.x >> 5] = tw;
                    if (tw) atomicAdd(&part.takenw, tw);
                }
                cl.sync();
                // evicted weight of the blocks before this one and of this
                // block's earlier warps
                const int lane = (int)lane_id();
                uint32_t x = lane < v.rank ? peer_ld(&part.takenw, lane) : 0u;
                x += lane < (int)(threadIdx.x >> 5) ? s.wsum[lane] : 0u;
                rb_cookie(part, (int64_t)__reduce_add_sync(0xffffffffu, x));
            }
        }
        cl.sync();
        pull_lists<PT>(true);
        {   // the next iteration's sums, and the buckets every block has read by now
            int32_t *next = arena_at<int32_t>(v.oDelta) + (buf ^ 1) * v.k;
#pragma unroll 1
            for (int p = threadIdx.x; p < v.k; p += blockDim.x) next[p] = 0;
            if (threadIdx.x < kPartFields) reinterpret_cast<uint32_t *>(&s.part[buf ^ 1])[threadIdx.x] = 0;
            if (mode != MODE_LP) {
#pragma unroll 1
                for (int i = threadIdx.x; i < na * kSlots; i += blockDim.x) {   // kSlots = kRWarps + 1: covers the tables' part too
                    arena_at<uint32_t>(v.oBk)[i] = 0;
                    arena_at<int32_t>(v.oTab)[i] = 0;
                }
            }
        }
        __syncthreads();
        apply_moves<PT>(part, delta, mode == MODE_LP);
        cl.sync();
        // controller: every block from the same sums
        add_deltas(v, delta);
        {
            // P := N (16 bytes at a time; both arrays are 16-byte aligned and padded)
            const int n16 = (int)(((uint32_t)v.n * sizeof(PT) + 15u) / 16u);
            const int4 *src = arena_at<int4>(v.oN);
            int4 *dst = arena_at<int4>(v.oP);
#pragma unroll 1
            for (int i = threadIdx.x; i < n16; i += blockDim.x) dst[i] = src[i];
        }
        const int warp = (int)(threadIdx.x >> 5);
        const int32_t dcut = warp == 0 ? (int32_t)part_sum(v, part, kfDcut) : 0;
        __syncthreads();
        if (warp == 0) {
            // decide: every lane alike, lane 0 stores
            ResCtl c = s.ctl;
            const int32_t maxw = warp_max_pw(v);
            const int64_t cut = c.cut + dcut;
            const bool bal = maxw <= v.Llim;
            c.noimp += 1;
            c.copy = 0;
            if (bal) {
                if (!c.best_bal || cut < c.best_cut) {
                    if (!c.best_bal || 1000000LL * cut < v.phi_ppm * c.best_cut) c.noimp = 0;
                    c.best_cut = cut; c.best_maxw = maxw; c.best_bal = 1;
                    c.copy = 1;
                }
            } else if (!c.best_bal && maxw < c.best_maxw) {
                c.best_cut = cut; c.best_maxw = maxw; c.noimp = 0;
                c.copy = 1;
            }
            const int32_t m = res_next_mode(v, bal, c.noimp, c.it + 1, c.weak, c.hit_cap);
            __syncwarp();
            if (lane_id() == 0) {
                ResCtl &o = s.ctl;
                o.cut = cut; o.noimp = c.noimp; o.copy = c.copy; o.weak = c.weak; o.hit_cap = c.hit_cap;
                o.best_cut = c.best_cut; o.best_maxw = c.best_maxw; o.best_bal = c.best_bal;
                o.kcount[mode] += 1;
                o.it = c.it + 1;
                o.mode = m;
                s.cnt = s.nact = 0;
                if (trace && v.rank == 0 && c.it < kTrace) {
                    trace[c.it].kind = mode;
                    trace[c.it].cut = cut;
                    trace[c.it].maxw = maxw;
                    trace[c.it].flags = c.copy;
                }
            }
        } else if (warp == 1) {
            res_classes(0);
        } else if (warp == 2) {
            res_classes(1);
        } else if (warp == 3 && v.rank == 0) {   // statistics: the fields' sums over the blocks
            const int lane = (int)lane_id();
            uint32_t f[kPartFields];
#pragma unroll
            for (int q = 0; q < kPartFields; ++q)
                f[q] = peer_ld(reinterpret_cast<uint32_t *>(&part) + q, min(lane, v.cs - 1));
            uint32_t x = 0;
#pragma unroll
            for (int q = 0; q < kPartFields; ++q) {
                const uint32_t t = __reduce_add_sync(0xffffffffu, lane < v.cs ? f[q] : 0u);
                if (lane == q) x = t;
            }
            if (lane == kPartFields) x = mode == MODE_LP ? 0u : (uint32_t)na;
            if (lane <= kPartFields && lane != kfDcut) s.acc[mode][lane] += x;
            if (trace) s.wsum[lane] = x;   // read by the trace writer below
        }
        __syncthreads();
        if (s.ctl.copy) {
            PT *best = arena_at<PT>(v.oBest);
            const PT *P = arena_at<PT>(v.oP);
#pragma unroll 1
            for (int i = threadIdx.x; i < v.own; i += blockDim.x) best[i] = P[v.base + i];
            // counted where the per-kernel loop copies: in the next iteration
            if (threadIdx.x == 0 && s.ctl.mode != MODE_DONE) s.acc[s.ctl.mode][kPartFields + 1] += 1;
        }
        if (trace && v.rank == 0 && warp == 3 && lane_id() == 0 && s.ctl.it <= kTrace) {
            TraceRec &r = trace[s.ctl.it - 1];
            const uint32_t *q = s.wsum;
            const bool lp = mode == MODE_LP;
            r.na = (int32_t)q[kPartFields]; r.pad = 0;
            r.nx = lp ? (int64_t)q[kfNX] : (int64_t)q[kfNcand];
            r.nm = q[kfNM];
            r.degx = q[kfDegx]; r.degm = q[kfDegm]; r.nbnd = q[kfNbnd]; r.nexam = q[kfNexam]; r.degexam = q[kfDegexam];
        }
    }
}

__device__ __forceinline__ int64_t global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return (int64_t)t;
}

// The level's bytes by the kernel that does the same work in the other loops
// (the byte model is linear in the sums).  They are the algorithm's traffic: here
// most of it stays in shared memory.  Eviction has no tiles in this loop: nothing is
// counted for them.
__device__ __noinline__ void res_bytes(int64_t *kb) {
    const ResShared &s = rs();
    const ResView &v = s.v;
    for (int i = 0; i < JET_K_COUNT; ++i) kb[i] = 0;
#pragma unroll 1
    for (int kind = 0; kind < 3; ++kind) {
        const unsigned long long *q = s.acc[kind];
        const int64_t its = s.ctl.kcount[kind];
        const bool lp = kind == MODE_LP;
        IterCounts c{lp ? (int64_t)q[kfNX] : 0, (int64_t)q[kfNM], (int64_t)q[kfDegx], (int64_t)q[kfDegm],
                     (int64_t)q[kfNbnd], (int64_t)q[kfNexam], (int64_t)q[kfDegexam], (int64_t)q[kfNcand],
                     0, 8 * (int64_t)v.n * (int64_t)q[kPartFields + 1]};
        int64_t b[JET_K_COUNT];
        iter_bytes(v.n * its, v.gew ? 8 : 4, 0, v.k * its, v.abl, kind, c, b);
        b[JET_K_RB_TILEHIST] = 0;
        for (int i = 0; i < JET_K_COUNT; ++i) kb[i] += b[i];
    }
}

template <class PT>
__global__ void __launch_bounds__(kRT, 1) k_refine_resident(const __grid_constant__ ResJob job) {
    cg::cluster_group cl = cg::this_cluster();
    ResShared &s = rs();
    const ResView &v = s.v;
#pragma unroll 1
    for (int32_t i = 0; i < job.nlv; ++i) {
        const int64_t t0 = global_ns();
        res_level_start<PT>(job, i);
        res_level_loop<PT>(i + 1 == job.nlv ? job.trace : nullptr);
        __syncthreads();
        const PT *best = arena_at<PT>(v.oBest);
        int32_t *out = job.lv[i].out;
#pragma unroll 1
        for (int u = threadIdx.x; u < v.own; u += blockDim.x) out[v.base + u] = best[u];
        if (v.rank == 0 && threadIdx.x == 0) {
            const ResCtl &c = s.ctl;
            ResStat &st = *job.lv[i].stat;
            st.best_cut = c.best_cut;
            st.best_maxw = c.best_maxw;
            st.it = c.it;
            st.best_bal = c.best_bal;
            st.hit_cap = c.hit_cap;
            for (int q = 0; q < 4; ++q) st.kcount[q] = c.kcount[q];
            int64_t kb[JET_K_COUNT];
            res_bytes(kb);
            for (int q = 0; q < JET_K_COUNT; ++q) st.kbytes[q] = kb[q];
            st.ns = global_ns() - t0;
        }
        cl.sync();   // the level's result is visible, and no block still reads this one's shared memory
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
uint32_t part_bytes(int32_t k) { return k <= 256 ? 1u : 2u; }

// Per device and part type: largest arena, and the largest cluster that one
// launch can co-schedule with it (0: none).
struct ResDevice {
    bool done = false;
    uint32_t arena = 0;
    int cluster = 0;
};

template <class PT>
int probe_device(ResDevice &d) {
    cudaFuncAttributes at{};
    int dev = 0, optin = 0;
    JET_CUDA_TRY(cudaGetDevice(&dev));
    JET_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    JET_CUDA_TRY(cudaFuncGetAttributes(&at, k_refine_resident<PT>));
    const int64_t arena = ((int64_t)optin - (int64_t)at.sharedSizeBytes) & ~int64_t(255);
    if (arena < 32768) return JET_OK;
    JET_CUDA_TRY(cudaFuncSetAttribute(k_refine_resident<PT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    JET_CUDA_TRY(cudaFuncSetAttribute(k_refine_resident<PT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)arena));
    d.arena = (uint32_t)arena;
    for (int cs = 16; cs >= 2; cs /= 2) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(cs);
        cfg.blockDim = dim3(kRT);
        cfg.dynamicSmemBytes = (size_t)arena;
        cudaLaunchAttribute la{};
        la.id = cudaLaunchAttributeClusterDimension;
        la.val.clusterDim.x = cs; la.val.clusterDim.y = 1; la.val.clusterDim.z = 1;
        cfg.attrs = &la;
        cfg.numAttrs = 1;
        int nclusters = 0;
        if (cudaOccupancyMaxActiveClusters(&nclusters, k_refine_resident<PT>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        if (nclusters >= 1) {
            d.cluster = cs;
            break;
        }
    }
    return JET_OK;
}

int device_info(int device, int32_t k, ResDevice &out) {
    static std::mutex mu;
    static ResDevice cache[2][256];
    out = ResDevice{};
    if (device < 0 || device >= 256) return JET_OK;
    std::lock_guard<std::mutex> lock(mu);
    const int idx = part_bytes(k) == 1 ? 0 : 1;
    ResDevice &d = cache[idx][device];
    if (!d.done) {
        JET_TRY(idx == 0 ? probe_device<uint8_t>(d) : probe_device<uint16_t>(d));
        d.done = true;
    }
    out = d;
    return JET_OK;
}

// Entries up to which a level of n vertices and k parts is kept.  Sixteen SMs
// read a level's rows slower than the whole GPU does, and a row that meets more
// than kSeen parts is walked again by a warp that then scans k table entries;
// how many rows a pass reads is not known here, so the lines are those of
// graphs without locality, where nearly every row lies on a boundary (uniform
// random graphs, R-MAT).  Measured there (the loop such a level takes otherwise
// / this one): n = 60,000, k = 8: 479,000 entries 1.05, 900,000 0.56; k = 64:
// n = 48,000, 335,000 entries 1.06, 479,000 0.84; n = 60,000, 299,000 1.11,
// 659,000 0.60; k = 128: n = 48,000, 239,000 1.14, 335,000 0.88; k = 256:
// n = 24,000, 191,000 1.04, 287,000 0.85; R-MAT s15 (883,000), k = 256: 0.51.
// Meshes and geometric graphs gain further on.  Inside a hierarchy they are told
// apart by the next coarser level: where the neighbours of a matched pair are
// neighbours of each other, contraction merges their entries, and it keeps 0.4 to
// 0.8 of them (random graphs, R-MAT and levels that stall keep 0.85 to 1).  Such
// levels of up to 16 entries per vertex may have twice as many (graph loop / this
// one): weighted 48^3 mesh, n = 59,800, 504,000 entries, k = 64 1.28; 80^3, n =
// 46,000, 591,000, k = 31 1.28; 60^3, n = 63,300, 671,000, k = 8 1.39; geometric
// of degree 12, n = 60,000, 714,000, k = 31 1.71; of degree 16, n = 40,000, 632,000,
// k = 64 1.72.  So may denser ones (400,000 entries where there are more than 40 per
// vertex) of which 0.65 is left: R-MAT s17 with two-hop matches, n = 8,400, 397,000,
// k = 64 1.9; between 0.65 and 0.8 such levels lose at times (0.81 to 1.5).  Levels of up to 8,192 vertices of any hierarchy gain up to
// about 400,000 entries whatever k <= 256 is, since the partition they start from is
// a refined one: means over R-MAT and random graphs of 350,000 to 400,000 entries 1.1
// (k = 2) to 2.4 (k = 64) at n <= 4,096, 1.1 to 1.8 up to 8,192.
// Up to 8,192 vertices 512 threads a block walk the rows: n = 8,000, k = 8,
// 342,000 entries 1.11, 398,000 0.93; n = 6,000, k = 192: 149,000 1.01,
// 197,000 0.87; k = 256: 59,000 1.11, 149,000 0.94; k = 384: 29,000 1.05,
// 95,000 0.91.  Up to 4,096 the loop to beat is the cluster loop: k = 256:
// 147,000 1.02, 198,000 0.98; k = 384: 99,000 1.13, 147,000 0.94; k = 480:
// 59,000 1.03, 147,000 0.86; above 400,000 entries this loop does not gain on it,
// nor on longer rows with few blocks (n = 1,000, k = 64: 258,000 1.05, 322,000 0.97).
int64_t res_entry_limit(int64_t n, int64_t nnz, int64_t nnz_coarser, int32_t k) {
    const int64_t wide = 76800000 / (160 + k);       // 480,000 / (1 + k / 160)
    int64_t most;
    if (n > 8192) most = wide;
    else if (nnz_coarser >= 0 && k <= 256) most = std::min<int64_t>(400000, 280 * n);
    else if (n > 4096) most = std::min<int64_t>({350000, wide, 5000000000 / ((int64_t)k * k)});
    else most = std::min<int64_t>({400000, 280 * n, 40000000 / k});
    const bool local = nnz_coarser >= 0 && ((10 * nnz_coarser <= 8 * nnz && nnz <= 16 * n) ||
                                            (20 * nnz_coarser <= 13 * nnz && (nnz <= 400000 || nnz <= 40 * n)));
    return local ? 2 * most : most;
}

bool res_fits(int64_t n, int32_t k, int cs, uint32_t arena) {
    if (n <= 0 || n > 262144) return false;
    const int32_t S = res_slice(n, cs);
    if (S > 16383) return false;   // 16-bit local ids, and the owner division stays exact
    ResView v;
    return res_layout(v, (int32_t)n, S, k, part_bytes(k)) + 64u <= arena;
}

}  // namespace

int resident_cluster(Ctx &c, int64_t n, int64_t nnz, int64_t nnz_coarser, int32_t k, int *cs) {
    *cs = 0;
    const int want = c.opt.cluster_blocks;
    // fewer blocks by choice: fewer entries (a small level's few blocks are enough for its rows)
    if (n <= 0 || n > c.opt.cluster_max_n ||
        nnz > res_entry_limit(n, nnz, nnz_coarser, k) * (want > 0 ? want : 16) / 16)
        return JET_OK;
    ResDevice d;
    JET_TRY(device_info(c.device, k, d));
    if (want > 0) {
        if (want <= d.cluster && res_fits(n, k, want, d.arena)) *cs = want;
        return JET_OK;
    }
    for (int s = 2; s <= d.cluster; s *= 2) {
        if (!res_fits(n, k, s, d.arena)) continue;
        *cs = s;
        if (n <= (int64_t)s * 256) break;
    }
    return JET_OK;
}

int resident_enqueue(Ctx &c, const ResChainLevel *lv, int32_t nlv, int32_t k, double eps, int64_t W, int cs,
                     const int32_t *init, bool want_trace) {
    if (nlv < 1 || nlv > JET_MAX_LEVELS) return JET_EINVAL;
    cudaStream_t s = c.stream;
    ResDevice d;
    JET_TRY(device_info(c.device, k, d));
    int64_t nmax = 1;
    for (int32_t i = 0; i < nlv; ++i) nmax = std::max<int64_t>(nmax, lv[i].g.n);
    DevBuf wdeg;   // released in stream order, after the launch
    JET_TRY(dev_alloc(wdeg, (size_t)nmax * 4, s));
    char *pin = reinterpret_cast<char *>(c.pinned);
    ResJob jb;
    memset(&jb, 0, sizeof(jb));
    jb.init = init;
    jb.wdeg = wdeg.as<int32_t>();
    jb.trace = want_trace ? reinterpret_cast<TraceRec *>(pin + kPinnedTraceOff) : nullptr;
    jb.Llim = balance_limit(W, k, eps, &jb.opt);
    jb.sigma = jb.opt + (jb.Llim - jb.opt) / 2;
    jb.phi_ppm = llround(c.opt.phi * 1e6);
    jb.k = k;
    jb.nlv = nlv;
    jb.max_no_improve = c.opt.max_no_improve;
    jb.weak_limit = c.opt.weak_limit;
    jb.max_iters = c.opt.max_iters_per_level;
    jb.hub_deg = c.opt.hub_degree > 0 ? c.opt.hub_degree : kHugeDeg;
    jb.abl = c.opt.flags & ABL_ALL;
    jb.arena_bytes = d.arena;
    for (int32_t i = 0; i < nlv; ++i) {
        ResLevel &l = jb.lv[i];
        if (lv[i].slot < 0 || lv[i].slot >= JET_MAX_LEVELS) return JET_EINVAL;
        l.g = lv[i].g;
        l.cmap = lv[i].cmap;
        l.out = lv[i].out;
        l.stat = reinterpret_cast<ResStat *>(pin + kPinnedResOff) + lv[i].slot;
        l.seed = lv[i].seed;
        l.cq16 = (int32_t)llround((lv[i].is_finest ? c.opt.c_fine : c.opt.c_coarse) * 65536.0);
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)cs);
    // slices of up to 512 vertices: half the threads (cheaper barriers: 470 against 610 cycles)
    cfg.blockDim = dim3(res_slice(nmax, cs) <= 512 ? kRT / 2 : kRT);
    cfg.dynamicSmemBytes = d.arena;
    cfg.stream = s;
    cudaLaunchAttribute la{};
    la.id = cudaLaunchAttributeClusterDimension;
    la.val.clusterDim.x = cs; la.val.clusterDim.y = 1; la.val.clusterDim.z = 1;
    cfg.attrs = &la;
    cfg.numAttrs = 1;
    if (part_bytes(k) == 1) JET_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_refine_resident<uint8_t>, jb));
    else JET_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_refine_resident<uint16_t>, jb));
    c.launches += 1;
    return JET_OK;
}

}  // namespace jet
