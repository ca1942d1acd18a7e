// Time-dependent shortest paths of the assignment loop on the GPU.
//
// The assignment loop (method of successive averages around the simulator)
// needs, every iteration, the earliest-arrival path of every trip under the
// link times of that iteration: routing is the step upstream of the
// simulation ("after the routing", Sec. 3.1), and re-routing between
// simulations is the paper's stated next step (Sec. 5).  Trips with the same
// origin and 30-minute departure period share one tree rooted at the middle
// of the period; at the regional scale that is some 10^5 trees per iteration
// on a 224k-node graph, far more than the host's threads finish in seconds.
//
// Networks of up to some 55 thousand nodes are searched with a tree's labels in
// a block's shared memory (td_trees_shared, below).  Beyond that every tree is
// searched by one warp (td_trees), thousands of warps at a time (a
// tree's frontier is a wave of a few hundred nodes; many trees in flight
// hide the memory latency each relaxation pays: on the 2.82M-trip day, 16
// trees per SM took 2.7 s per pass, 32 took 1.85 s, 64 took 1.78 s; the
// out-edges of a round's near nodes spread over the lanes took 32 to 1.7 s,
// a node's label, round stamp and far mark in one 16-byte record to
// 1.33 s, and 40 trees per SM (48 registers, no spills) to 1.26 s):
//   * label-correcting search in rounds over time buckets (near-far): the
//     near set's nodes relax their out-edges with the arrival function of
//     the bin holding their arrival time (FIFO by construction, see TD); a
//     node whose label improved joins the next round's near set when its
//     arrival is below the bucket threshold (once per round: a round stamp)
//     and the far pile otherwise (once: a mark); when the near set empties,
//     every label below the threshold is final, the threshold moves on by
//     the bucket width and the far nodes below it become the near set --
//     close to Dijkstra's work, with a whole near set relaxed per round;
//   * a label is (arrival ms << 32 | entering edge id) in one 64-bit word,
//     so atomicMin keeps the earliest arrival and, among equal arrivals, the
//     lower edge id -- the fixed point is exactly the tree the host's
//     Dijkstra builds (lpsim_assign_shortest_paths), with integer millisecond
//     link times making every arrival an exact sum;
//   * the search ends once every destination of the group is below the
//     threshold (settled); until then the latest destination label bounds
//     it: a node reached later cannot lie on any of their paths (link times
//     are positive), so it is not expanded;
//   * each trip's path is read back along the entering edges, written to the
//     output in travel order and timed from the trip's own departure;
//   * the labels the tree set are reset from its list of reached nodes, so a
//     warp's workspace is reused without clearing the whole graph.
// Every loop is bounded (rounds and path walks by the node count); a bound
// that is hit sets an error bit the host reports.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/lpsim_assign.h"
#include "assign_internal.h"
#include "host_par.h"

int lpsim_fail(int code, const std::string &msg);

using namespace lpsim_assign_detail;

namespace {

int fail(int code, const std::string &m) { return lpsim_fail(code, m); }

#define CU(call)                                                                                      \
    do {                                                                                              \
        cudaError_t e_ = (call);                                                                      \
        if (e_ != cudaSuccess) return fail(LPSIM_E_CUDA, std::string(#call ": ") + cudaGetErrorString(e_)); \
    } while (0)

constexpr uint64_t kUnreached = ~0ull;
constexpr uint32_t kNoEdge = 0xFFFFFFFFu;
#ifndef LPSIM_ASSIGN_WARPS_PER_SM
#define LPSIM_ASSIGN_WARPS_PER_SM 40
#endif
#ifndef LPSIM_ASSIGN_WORKSPACE_GIB
#define LPSIM_ASSIGN_WORKSPACE_GIB 48
#endif
constexpr int kWarpsPerBlock = 4;
constexpr int kBlocksPerSm = LPSIM_ASSIGN_WARPS_PER_SM / kWarpsPerBlock;   // trees searched at once per SM / 4
constexpr uint64_t kWorkspaceBudget = (uint64_t)LPSIM_ASSIGN_WORKSPACE_GIB << 30;  // per-warp workspaces at most
#ifndef LPSIM_ASSIGN_DELTA_MS
#define LPSIM_ASSIGN_DELTA_MS 60000
#endif
constexpr uint64_t kDeltaMs = LPSIM_ASSIGN_DELTA_MS;  // bucket width of the search thresholds (ms)

// error bits
constexpr uint32_t kErrUnreachable = 1u;  // a destination not reached (or equal to its origin)
constexpr uint32_t kErrCapacity = 2u;     // the path buffer was too small (the host retries)
constexpr uint32_t kErrBound = 4u;        // a round or path-walk bound was hit

struct GroupRec {
    uint32_t src;    // origin node
    uint32_t t0;     // root time (ms)
    uint32_t first;  // first position in the trip order
    uint32_t count;  // trips
};

// a node's search state in one 16-byte record, so the atomics of one
// relaxation (the label's minimum, then the round stamp or the far mark)
// touch one 32-byte sector
struct __align__(16) NodeRec {
    unsigned long long lab;  // (arrival ms << 32) | entering edge, or all ones while unreached
    uint32_t inq;            // round stamp of the last push onto a near set
    uint32_t fmark;          // tree mark while the node is in the far pile
};

constexpr uint64_t kWorkspacePerNode = sizeof(NodeRec) + 4 * 4;  // td_trees: bytes per node and warp

struct TreeArgs {
    uint32_t n_nodes, n_edges, n_bins, bin_ms;
    const uint32_t *out_off;  // n_nodes + 1
    const uint2 *adj;         // per out-edge position: {edge, head node}
    const uint32_t *pos;      // per edge: its out-edge position (nullptr: the edge id is the position)
    const uint32_t *src;      // per edge: tail node
    const uint32_t *in_off;   // n_nodes + 1
    const uint2 *in_adj;      // per in-edge, ascending edge ids: {out-edge position, tail node}
    // n_bins x n_edges by out-edge position: {link time ms, earliest arrival entering a later bin ms}; a search
    // reads a node's out-edges and their times side by side
    const uint2 *cms;
    // td_trees_shared, networks of at most kWide out-edges per node: positions are wide * node + k, so a node's
    // row is known without out_off (0: positions as above); n_pos of them per bin
    uint32_t wide, n_pos;
    uint32_t n_groups;
    const GroupRec *groups;
    const uint32_t *order;    // trip per position, group by group
    const uint32_t *dest;     // per trip
    const uint32_t *dep_ms;   // per trip: planned departure (ms)
    // outputs per trip
    unsigned long long *path_off;
    uint32_t *path_len;
    float *tsp;
    uint32_t *edges;          // path edges, travel order
    unsigned long long cap;   // entries of edges
    unsigned long long *cursor;
    // td_trees_shared: positions along each thread's path, scratch_len per thread
    uint32_t *scratch;
    uint32_t scratch_len;     // kScratch at most, less on small networks
    // td_trees: per-warp workspaces
    NodeRec *node;            // n_warps x n_nodes: label, round stamp of the last push, far-pile mark
    uint32_t *touched;        // n_warps x n_nodes
    uint32_t *fa, *fb;        // n_warps x n_nodes: near sets (this round, next round)
    uint32_t *far;            // n_warps x n_nodes: far pile (labels at or above the threshold)
    uint32_t *stamp;          // per warp: last round stamp used
    uint64_t delta_ms;        // bucket width of the thresholds
    uint32_t *next_group;
    uint32_t *err;
};

__device__ __forceinline__ uint32_t bin_of(const TreeArgs &A, uint64_t t) {
    const uint64_t b = t / A.bin_ms;
    return b < A.n_bins ? (uint32_t)b : A.n_bins - 1u;
}

// arrival when entering edge e at time t (ms): min(t + c, M) of t's bin
__device__ __forceinline__ uint64_t arrive(const uint2 lt, uint64_t t) {
    const uint64_t a = t + lt.x;
    return a < (uint64_t)lt.y ? a : (uint64_t)lt.y;
}

__device__ __forceinline__ uint32_t pos_of(const TreeArgs &A, uint32_t e) { return A.pos ? A.pos[e] : e; }

// Latest current arrival over the group's destinations (its trips'), or
// kUnreached while any is unreached; every lane gets the result.
__device__ __forceinline__ uint64_t dest_bound(const TreeArgs &A, const GroupRec &G, const NodeRec *nd,
                                               uint32_t lane) {
    uint64_t m = 0;
    for (uint32_t q = lane; q < G.count; q += 32) {
        const uint64_t l = __ldcg(&nd[A.dest[A.order[G.first + q]]].lab);
        const uint64_t t = l == kUnreached ? kUnreached : (l >> 32);
        m = t > m ? t : m;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t y = __shfl_xor_sync(0xFFFFFFFFu, m, o);
        m = y > m ? y : m;
    }
    return m;
}

__global__ void __launch_bounds__(kWarpsPerBlock * 32, kBlocksPerSm) td_trees(TreeArgs A) {
    const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
    const size_t gw = (size_t)blockIdx.x * kWarpsPerBlock + wib;
    NodeRec *nd = A.node + gw * A.n_nodes;
    uint32_t *touched = A.touched + gw * A.n_nodes;
    uint32_t *fa = A.fa + gw * A.n_nodes, *fb = A.fb + gw * A.n_nodes;
    uint32_t *far = A.far + gw * A.n_nodes;
    __shared__ uint32_t s_next[kWarpsPerBlock], s_touched[kWarpsPerBlock], s_far[kWarpsPerBlock];
    uint32_t stamp = A.stamp[gw];
    // rounds of a search at most: every round settles or re-labels a node,
    // and a node's label improves a bounded number of times
    const uint64_t max_rounds = 8ull * A.n_nodes + (1ull << 20);
    for (;;) {
        uint32_t g = 0;
        if (lane == 0) g = atomicAdd(A.next_group, 1u);
        g = __shfl_sync(0xFFFFFFFFu, g, 0);
        if (g >= A.n_groups) break;
        const GroupRec G = A.groups[g];
        const uint32_t tmark = ++stamp;  // this tree's mark of the nodes in its far pile
        if (lane == 0) {
            __stcg(&nd[G.src].lab, (unsigned long long)(((uint64_t)G.t0 << 32) | kNoEdge));
            __stcg(touched, G.src);
            __stcg(fa, G.src);
        }
        uint32_t nn = 1, nt = 1, nfar = 0;
        uint64_t theta = (uint64_t)G.t0 + A.delta_ms;  // labels below theta are expanded now, the rest wait
        uint64_t ub = kUnreached;  // latest destination arrival so far (ms), once all are reached
        __threadfence_block();
        __syncwarp();
        bool bounded = true;
        for (uint64_t round = 0;; round++) {
            if (round > max_rounds) {
                bounded = false;
                break;
            }
            if (nn > 0) {
                // one round of the near set: relax the out-edges of its nodes
                stamp++;
                if (lane == 0) {
                    s_next[wib] = 0;
                    s_touched[wib] = nt;
                    s_far[wib] = nfar;
                }
                __syncwarp();
                // 32 near nodes at a time, their out-edges spread over the
                // lanes (a warp scan of the degrees; each lane finds the node
                // of its edge by a binary search over the scan), so a round
                // with a few nodes of a few edges each keeps most lanes busy
                for (uint32_t c0 = 0; c0 < nn; c0 += 32) {
                    const uint32_t i = c0 + lane;
                    uint32_t u = 0, j0 = 0, deg = 0, tu = 0;  // a queued node is reached: its arrival has 32 bits
                    if (i < nn) {
                        u = __ldcg(fa + i);
                        tu = (uint32_t)(__ldcg(&nd[u].lab) >> 32);
                        j0 = A.out_off[u];
                        deg = tu < ub ? A.out_off[u + 1] - j0 : 0u;
                    }
                    uint32_t incl = deg;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                        if (lane >= (uint32_t)o) incl += y;
                    }
                    const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);
                    const uint32_t first = j0 - (incl - deg);  // edge t of the warp's is out-edge first + t of its owner
                    for (uint32_t b0 = 0; b0 < total; b0 += 32) {
                        const uint32_t t = b0 + lane;
                        // the lane whose node owns edge t: the first with incl > t
                        uint32_t owner = 0;
#pragma unroll
                        for (uint32_t step = 16; step > 0; step >>= 1) {
                            const uint32_t y = __shfl_sync(0xFFFFFFFFu, incl, (int)(owner + step - 1));
                            if (y <= t) owner += step;
                        }
                        const uint32_t o_first = __shfl_sync(0xFFFFFFFFu, first, (int)owner);
                        const uint32_t o_tu = __shfl_sync(0xFFFFFFFFu, tu, (int)owner);
                        if (t >= total) continue;
                        const uint32_t j = o_first + t;
                        const uint2 ev = A.adj[j];
                        const uint64_t at = arrive(A.cms[(size_t)bin_of(A, o_tu) * A.n_edges + j], o_tu);
                        if (at > 0xFFFFFFFFull || at > ub) continue;
                        const unsigned long long cand = (at << 32) | ev.x;
                        const unsigned long long old = atomicMin(&nd[ev.y].lab, cand);
                        if (cand < old) {
                            if (old == kUnreached) __stcg(touched + atomicAdd(&s_touched[wib], 1u), ev.y);
                            if (at < theta) {
                                if (atomicExch(&nd[ev.y].inq, stamp) != stamp)
                                    __stcg(fb + atomicAdd(&s_next[wib], 1u), ev.y);
                            } else if (atomicExch(&nd[ev.y].fmark, tmark) != tmark) {
                                __stcg(far + atomicAdd(&s_far[wib], 1u), ev.y);
                            }
                        }
                    }
                }
                __threadfence_block();
                __syncwarp();
                nn = s_next[wib];
                nt = s_touched[wib];
                nfar = s_far[wib];
                uint32_t *t = fa;
                fa = fb;
                fb = t;
                __syncwarp();
                continue;
            }
            // the near set is empty: every label below theta is final
            ub = dest_bound(A, G, nd, lane);
            if (ub < theta || nfar == 0) break;  // every destination settled (or nothing left)
            // next threshold: move the far nodes below it to the near set, keep
            // the rest (the far list holds each node once: its mark)
            uint64_t next = theta + A.delta_ms;
            for (int pass = 0; pass < 2 && nn == 0 && nfar > 0; pass++) {
                uint32_t kept = 0;
                uint64_t tmin = kUnreached;
                for (uint32_t c0 = 0; c0 < nfar; c0 += 32) {
                    const uint32_t i = c0 + lane;
                    uint32_t v = 0;
                    uint64_t tv = kUnreached;
                    if (i < nfar) {
                        v = __ldcg(far + i);
                        tv = __ldcg(&nd[v].lab) >> 32;
                    }
                    const bool drop = i < nfar && tv < theta;            // settled in an earlier bucket
                    const bool move = i < nfar && tv >= theta && tv < next;
                    const bool keep = i < nfar && tv >= next;
                    const uint32_t mk = __ballot_sync(0xFFFFFFFFu, keep), mm = __ballot_sync(0xFFFFFFFFu, move);
                    const uint32_t below = (1u << lane) - 1u;
                    __syncwarp();  // every lane has read its entry before any is overwritten
                    if (drop || move) __stcg(&nd[v].fmark, 0u);
                    if (keep) __stcg(far + kept + __popc(mk & below), v);
                    if (move) __stcg(fa + nn + __popc(mm & below), v);
                    kept += __popc(mk);
                    nn += __popc(mm);
                    uint64_t tk = keep ? tv : kUnreached;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const uint64_t y = __shfl_xor_sync(0xFFFFFFFFu, tk, o);
                        tk = y < tk ? y : tk;
                    }
                    tmin = tk < tmin ? tk : tmin;
                }
                nfar = kept;
                theta = next;
                // nothing below the threshold: jump to the earliest far label
                if (nn == 0 && nfar > 0) next = tmin + A.delta_ms;
            }
            __threadfence_block();
            __syncwarp();
        }
        if (!bounded && lane == 0) atomicOr(A.err, kErrBound);
        // far marks of the nodes still in the far pile (the others were cleared)
        for (uint32_t i = lane; i < nfar; i += 32) __stcg(&nd[__ldcg(far + i)].fmark, 0u);
        // paths of the group's trips, in travel order, timed from each trip's departure
        for (uint32_t q = lane; q < G.count; q += 32) {
            const uint32_t j = A.order[G.first + q];
            const uint32_t d = A.dest[j];
            A.path_len[j] = 0;
            const uint64_t ld = __ldcg(&nd[d].lab);
            if (ld == kUnreached || d == G.src || !bounded) {
                atomicOr(A.err, kErrUnreachable);
                continue;
            }
            uint32_t L = 0;
            bool ok = true;
            for (uint32_t v = d; v != G.src;) {
                const uint32_t e = (uint32_t)__ldcg(&nd[v].lab);
                if (++L > A.n_nodes || e >= A.n_edges) {
                    ok = false;
                    break;
                }
                v = A.src[e];
            }
            if (!ok) {
                atomicOr(A.err, kErrBound);
                continue;
            }
            const unsigned long long off = atomicAdd(A.cursor, (unsigned long long)L);
            if (off + L > A.cap) {
                atomicOr(A.err, kErrCapacity);
                continue;
            }
            uint32_t pos = L;
            for (uint32_t v = d; v != G.src && pos > 0;) {
                const uint32_t e = (uint32_t)__ldcg(&nd[v].lab);
                A.edges[off + --pos] = e;  // e < n_edges: the counting walk checked this chain
                v = A.src[e];
            }
            const uint64_t tj = A.dep_ms[j];
            uint64_t t = tj;
            for (uint32_t p = 0; p < L; p++)
                t = arrive(A.cms[(size_t)bin_of(A, t) * A.n_edges + pos_of(A, A.edges[off + p])], t);
            A.path_off[j] = off;
            A.path_len[j] = L;
            A.tsp[j] = (float)((double)(t - tj) / 1000.0);
        }
        // clear the labels this tree set
        __syncwarp();
        for (uint32_t i = lane; i < nt; i += 32)
            __stcg(&nd[__ldcg(touched + i)].lab, (unsigned long long)kUnreached);
        __threadfence_block();
        __syncwarp();
    }
    if (lane == 0) A.stamp[gw] = stamp;
}

// The same search with a tree's labels in shared memory: one block per tree,
// for networks whose labels fit (n_nodes * 4 bytes and a bit per node in a
// block's 227 KB: some 55 thousand nodes).  The label-correcting search is a
// chain of label reads and atomics; in device memory each costs a round trip to
// L2 or DRAM (thousands of trees' labels do not fit in L2), here a few cycles,
// and a block's threads relax a whole near set at once, four lanes per node.
//   * a label is the arrival alone, in ms after the root time, so a node takes
//     four bytes; the tree's entering edge of a node is found again where a path
//     is walked back: the lowest edge id among those that give its arrival, which
//     is the edge the 64-bit label holds;
//   * a bit per node says that it waits to be relaxed (cleared before its label is
//     read, so a later improvement queues it again); the waiting nodes' ids are
//     in a ring besides, and a round whose ids did not fit reads the bits;
//   * a node's out-edges and their times are looked up by 4 (or 8) times the
//     node where no node has more, so they come in one round trip to L2 instead
//     of two;
//   * no far pile: the nodes with a label in the next bucket are found by
//     scanning the labels (a node at or above the threshold was never relaxed).
// One block barrier per round: the counters rotate over three rounds.  Bound by
// the round trips to L2 of one round after another (some 400 a tree).
constexpr uint32_t kWide = 8;       // most out-edges per node for the wide rows
constexpr uint64_t kSharedDeltaMs = 240000;
constexpr uint32_t kRing = 1024;    // ids of waiting nodes (a power of two)
constexpr uint32_t kScratch = 512;  // positions kept per thread at most while a path is walked back
constexpr uint32_t kNever = 0xFFFFFFFFu;

__host__ __device__ inline size_t shared_tree_bytes(uint32_t n_nodes) {
    return (size_t)((n_nodes + 3) & ~3u) * 4 + (size_t)((n_nodes + 31) / 32) * 4 + kRing * 2;
}

template <int T, int PER_SM>
__global__ void __launch_bounds__(T, PER_SM) td_trees_shared(TreeArgs A) {
    extern __shared__ __align__(16) uint32_t s_lab[];
    const uint32_t n4 = (A.n_nodes + 3) & ~3u, nw = (A.n_nodes + 31) / 32;
    uint32_t *bits = s_lab + n4;
    uint16_t *ring = reinterpret_cast<uint16_t *>(bits + nw);
    __shared__ uint32_t s_group, s_cnt[3], s_min[3], s_red[32];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    volatile uint32_t *vlab = s_lab;
    uint32_t *scratch = A.scratch + (size_t)blockIdx.x * T * A.scratch_len + tid;
    const uint64_t max_rounds = 8ull * A.n_nodes + (1ull << 20);
    for (;;) {
        if (tid == 0) s_group = atomicAdd(A.next_group, 1u);
        __syncthreads();  // also: the last tree's paths have been read
        const uint32_t g = s_group;
        if (g >= A.n_groups) break;
        const GroupRec G = A.groups[g];
        const uint64_t t0 = G.t0;
        for (uint32_t i = tid; i < n4 / 4; i += T) reinterpret_cast<uint4 *>(s_lab)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
        for (uint32_t i = tid; i < nw; i += T) bits[i] = 0u;
        if (tid < 3) {
            s_cnt[tid] = tid == 2 ? 1u : 0u;  // the round before the first left one node: the root
            s_min[tid] = kNever;
        }
        __syncthreads();
        if (tid == 0) {
            s_lab[G.src] = 0u;
            bits[G.src >> 5] = 1u << (G.src & 31u);
            ring[0] = (uint16_t)G.src;
        }
        uint64_t theta = A.delta_ms;  // labels below theta are final or waiting
        uint64_t next = theta + A.delta_ms;
        uint32_t ub = kNever;         // latest destination label, once all are reached
        uint32_t base = 0, room = kRing, cur = 0, prev = 2;  // cur: this round's counters
        bool bounded = true, advanced = false;
        __syncthreads();
        for (uint64_t round = 0;; round++) {
            if (round > max_rounds) {
                bounded = false;
                break;
            }
            const uint32_t cnt = s_cnt[prev], low = s_min[prev];
            const bool over = cnt > room;  // ids did not fit: the bits say which nodes wait
            const uint32_t c = over ? 0u : cnt;
            room = kRing - c;
            auto queue = [&](uint32_t v, uint64_t below, uint32_t label) {
                if (label >= below) return;
                const uint32_t bit = 1u << (v & 31u);
                if (atomicOr(&bits[v >> 5], bit) & bit) return;
                const uint32_t p = atomicAdd(&s_cnt[cur], 1u);
                if (p < room) ring[(base + c + p) & (kRing - 1u)] = (uint16_t)v;
            };
            auto relax = [&](uint32_t u, uint32_t first, uint32_t step) {
                const uint32_t tu = vlab[u];
                if (tu >= ub) return;
                const uint64_t t = t0 + tu;
                const uint32_t j0 = A.wide ? u * A.wide : A.out_off[u], j1 = A.wide ? j0 + A.wide : A.out_off[u + 1];
                const uint2 *row = A.cms + (size_t)bin_of(A, t) * A.n_pos;
                for (uint32_t j = j0 + first; j < j1; j += step) {
                    const uint32_t v = A.adj[j].y;
                    const uint64_t at = arrive(row[j], t);
                    if (v == kNever || at > 0xFFFFFFFFull) continue;
                    const uint32_t rel = (uint32_t)(at - t0);
                    if (rel > ub) continue;
                    if (rel < atomicMin(&s_lab[v], rel)) queue(v, theta, rel);
                }
            };
            if (tid == 0) {
                const uint32_t after = cur == 2 ? 0u : cur + 1;
                s_cnt[after] = 0u;
                s_min[after] = kNever;
            }
            if (over) {
                for (uint32_t w = tid; w < nw; w += T) {
                    uint32_t m = atomicExch(&bits[w], 0u);
                    while (m) {
                        const uint32_t b = (uint32_t)__ffs((int)m) - 1u;
                        m &= m - 1u;
                        relax(32 * w + b, 0u, 1u);
                    }
                }
            } else if (c > 0) {
                for (uint32_t i0 = warp * 8; i0 < c; i0 += T / 4) {
                    const uint32_t i = i0 + (lane >> 2);
                    const uint32_t u = i < c ? ring[(base + i) & (kRing - 1u)] : 0u;
                    if (i < c && (lane & 3u) == 0) atomicAnd(&bits[u >> 5], ~(1u << (u & 31u)));
                    __syncwarp();  // the bit is cleared before any of the four lanes reads the label
                    if (i < c) relax(u, lane & 3u, 4u);
                    __syncwarp();
                }
            } else {
                // nothing waits: every label below theta is final
                if (advanced) {
                    if (low == kNever) break;  // no label at or above theta either
                    next = (uint64_t)low + A.delta_ms;  // an empty bucket: on to the earliest label
                }
                uint32_t m = 0;
                for (uint32_t q = tid; q < G.count; q += T) m = max(m, vlab[A.dest[A.order[G.first + q]]]);
                m = __reduce_max_sync(0xFFFFFFFFu, m);
                if (lane == 0) s_red[warp] = m;
                __syncthreads();
                ub = 0;
                for (uint32_t w = 0; w < T / 32; w++) ub = max(ub, s_red[w]);
                if (ub < theta) break;  // every destination settled
                uint32_t far = kNever;
                for (uint32_t i = tid; i < n4 / 4; i += T) {
                    const uint4 l = reinterpret_cast<const uint4 *>(s_lab)[i];
                    const uint32_t ls[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        if (ls[k] == kNever || ls[k] < theta) continue;
                        if (ls[k] >= next) far = min(far, ls[k]);
                        else queue(4 * i + k, next, ls[k]);
                    }
                }
                far = __reduce_min_sync(0xFFFFFFFFu, far);
                if (lane == 0 && far != kNever) atomicMin(&s_min[cur], far);
                theta = next;
                next = theta + A.delta_ms;
            }
            advanced = !over && c == 0;
            base += c;
            prev = cur;
            cur = cur == 2 ? 0u : cur + 1;
            __syncthreads();
        }
        if (!bounded && tid == 0) atomicOr(A.err, kErrBound);
        // paths of the group's trips, in travel order, timed from each trip's departure
        for (uint32_t q = tid; q < G.count; q += T) {
            const uint32_t jt = A.order[G.first + q];
            const uint32_t d = A.dest[jt];
            A.path_len[jt] = 0;
            if (s_lab[d] == kNever || d == G.src || !bounded) {
                atomicOr(A.err, kErrUnreachable);
                continue;
            }
            // the tree's edge into v: {its out-edge position, its tail}; position kNoEdge: none (never on a
            // finished search)
            auto entering = [&](uint32_t v) {
                const uint32_t tv = s_lab[v], i1 = A.in_off[v + 1];
                for (uint32_t i = A.in_off[v]; i < i1; i++) {
                    const uint2 in = A.in_adj[i];
                    const uint32_t tu = s_lab[in.y];
                    // (a tail reached as late as v gives its arrival only at the last millisecond, where all later ones stop)
                    if (tu > tv) continue;
                    const uint64_t t = t0 + tu;
                    if (arrive(A.cms[(size_t)bin_of(A, t) * A.n_pos + in.x], t) == t0 + tv) return in;
                }
                return make_uint2(kNoEdge, 0u);
            };
            uint32_t L = 0;
            bool ok = true;
            for (uint32_t v = d; v != G.src; L++) {
                const uint2 in = entering(v);
                if (L >= A.n_nodes || in.x == kNoEdge) {
                    ok = false;
                    break;
                }
                if (L < A.scratch_len) scratch[(size_t)L * T] = in.x;
                v = in.y;
            }
            if (!ok) {
                atomicOr(A.err, kErrBound);
                continue;
            }
            const unsigned long long off = atomicAdd(A.cursor, (unsigned long long)L);
            if (off + L > A.cap) {
                atomicOr(A.err, kErrCapacity);
                continue;
            }
            if (L > A.scratch_len) {  // a path longer than the scratch: its positions go through the output
                uint32_t p = L;
                for (uint32_t v = d; v != G.src && p > 0;) {
                    const uint2 in = entering(v);
                    A.edges[off + --p] = in.x;
                    v = in.y;
                }
            }
            const uint64_t tj = A.dep_ms[jt];
            uint64_t t = tj;
            for (uint32_t p = 0; p < L; p++) {
                const uint32_t j = L > A.scratch_len ? A.edges[off + p] : scratch[(size_t)(L - 1 - p) * T];
                A.edges[off + p] = A.adj[j].x;
                t = arrive(A.cms[(size_t)bin_of(A, t) * A.n_pos + j], t);
            }
            A.path_off[jt] = off;
            A.path_len[jt] = L;
            A.tsp[jt] = (float)((double)(t - tj) / 1000.0);
        }
    }
}

// cost_ms on the device: s * 1000 rounded to the nearest whole number (halves
// up), at least 1 (NaN too), at most 2^31 - 1.  In integers: the product of a
// 24-bit mantissa and 1000 is exact, as it is in the host's double (FP64
// instructions made the table kernel three times as long).
__device__ __forceinline__ uint32_t cost_ms_dev(float s) {
    if (!(s > 0.0f)) return 1u;
    if (s >= 4194304.0f) return 0x7FFFFFFFu;
    const uint32_t u = __float_as_uint(s), sh = 150u - (u >> 23);  // s = mantissa * 2^-sh, sh >= 2
    if (sh > 40u) return 1u;
    const uint64_t v = (uint64_t)((u & 0x7FFFFFu) | 0x800000u) * 1000u;
    const uint64_t r = (v + (1ull << (sh - 1u))) >> sh;
    return (uint32_t)(r < 1u ? 1u : r > 0x7FFFFFFFu ? 0x7FFFFFFFu : r);
}

// The link-time table of tt (n_edges x n_bins seconds) in whole milliseconds,
// by bin and position (adj: the edge at each, kNoEdge for none), as fill_link_times gives it on the host: per
// (edge, bin) the time to the nearest ms (at least 1, at most 2^31 - 1) and the
// earliest arrival entering a later bin.  A block takes 32 positions: its threads
// read and convert tiles of 32 bins, last bins first, one warp carries the
// minimum over the later bins and writes whole rows.  Bound by the bytes it
// moves.
__global__ void __launch_bounds__(256)
    link_table(const float *tt, const uint2 *adj, uint32_t n_pos, uint32_t n_bins, uint64_t bin_ms, uint2 *out) {
    __shared__ uint32_t c[32][33];
    const uint32_t j0 = blockIdx.x * 32, lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint64_t m = 0xFFFFFFFFull;
    for (uint32_t b1 = n_bins; b1 > 0;) {
        const uint32_t b0 = b1 > 32 ? b1 - 32 : 0;
        for (uint32_t r = warp; r < 32; r += 8) {
            const uint32_t e = j0 + r < n_pos ? adj[j0 + r].x : kNoEdge;
            if (e == kNoEdge || b0 + lane >= b1) continue;
            c[r][lane] = cost_ms_dev(tt[(size_t)e * n_bins + b0 + lane]);
        }
        __syncthreads();
        if (warp == 0 && j0 + lane < n_pos)
            for (uint32_t b = b1; b-- > b0;) {
                const uint32_t v = c[lane][b - b0];
                out[(size_t)b * n_pos + j0 + lane] = make_uint2(v, (uint32_t)m);
                const uint64_t a = (uint64_t)b * bin_ms + v;
                m = a < m ? a : m;
            }
        __syncthreads();
        b1 = b0;
    }
}

// every node unreached, with no round stamp and no far mark
__global__ void init_nodes(NodeRec *nd, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        nd[i] = NodeRec{(unsigned long long)kUnreached, 0u, 0u};
}

// Inflow per (edge, bin) of the routes: each trip walks its route from its
// planned departure with the arrival rule of the table, counting one entry
// in the bin of every link entry time (the host's lpsim_assign_load, on the
// device: integer counts, so the order of the atomics does not matter).
__global__ void load_routes(const ulonglong2 *span, const uint32_t *redge, const uint32_t *dep_ms,
                            uint64_t n, const uint2 *cms, const uint32_t *pos, uint32_t n_edges, uint32_t n_bins,
                            uint32_t bin_ms, uint32_t *inflow) {
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < n; j += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t t = dep_ms[j];
        const ulonglong2 r = span[j];
        for (unsigned long long q = r.x; q < r.y; q++) {
            const uint32_t e = redge[q];
            const uint64_t b = t / bin_ms;
            if (b < n_bins) atomicAdd(&inflow[(size_t)e * n_bins + b], 1u);
            t = arrive(cms[(size_t)(b < n_bins ? b : n_bins - 1) * n_edges + (pos ? pos[e] : e)], t);
        }
    }
}

}  // namespace

// Device copy of the graph, the trip table and the search workspaces.
struct AssignGpu {
    int device = -1;
    int n_sm = 0;
    cudaStream_t stream = nullptr;
    std::vector<void *> blocks;
    uint32_t n_warps = 0;
    TreeArgs A{};
    uint32_t period_steps = 0;  // grouping held in A.groups / A.order
    std::vector<uint64_t> order, gstart;
    unsigned long long cap = 0;
    // routes and inflow of lpsim_assign_load_gpu
    ulonglong2 *span = nullptr;
    uint32_t *redge = nullptr;
    uint64_t redge_cap = 0;
    uint64_t redge_here = 0, layout = 0;  // entries of the engine's on the device, of which layout
    uint64_t routes_version = ~0ull;      // of the routes on the device
    float *tt = nullptr;              // link times as given
    size_t tt_cells = 0;
    // td_trees_shared: its grid at most (0: td_trees searches), its arguments where they are not A's
    void (*shared_kernel)(TreeArgs) = nullptr;
    uint32_t shared_blocks = 0, shared_threads = 0;
    uint64_t scratch_cap = 0;  // entries of A.scratch
    const uint2 *wide_adj = nullptr, *wide_in = nullptr;
    uint32_t wide = 0;
    uint2 *table[2] = {};  // link-time tables: by out-edge position, by wide position
    size_t table_cells[2] = {};
    uint32_t *inflow = nullptr;
    size_t inflow_cells = 0;

    void *alloc(size_t bytes) {
        void *p = nullptr;
        if (cudaMalloc(&p, std::max<size_t>(bytes, 16)) != cudaSuccess) return nullptr;
        blocks.push_back(p);
        return p;
    }
    void release(void *p) {
        auto it = std::find(blocks.begin(), blocks.end(), p);
        if (it != blocks.end()) {
            blocks.erase(it);
            cudaFree(p);
        }
    }
    // room for n entries in place of p's block (contents not kept).  A failure
    // leaves p null and cap 0, so that the next call allocates again instead of
    // running on what is not there.
    template <class T, class N>
    bool regrow(T *&p, N &cap, size_t n) {
        if (p) release(const_cast<std::remove_const_t<T> *>(p));
        p = nullptr;
        cap = 0;
        p = static_cast<T *>(alloc(n * sizeof(T)));
        if (p) cap = (N)n;
        return p != nullptr;
    }
    ~AssignGpu() {
        if (stream) cudaStreamSynchronize(stream);
        for (void *b : blocks) cudaFree(b);
        if (stream) cudaStreamDestroy(stream);
    }
};

void assign_gpu_free(AssignGpu *g) { delete g; }

namespace {

template <class T>
int dput(AssignGpu *g, T *&dst, const T *src, size_t count) {
    dst = static_cast<T *>(g->alloc(count * sizeof(T)));
    if (!dst) return fail(LPSIM_E_OOM, "device allocation of " + std::to_string(count * sizeof(T)) + " bytes failed");
    if (count) CU(cudaMemcpyAsync(dst, src, count * sizeof(T), cudaMemcpyHostToDevice, g->stream));
    return LPSIM_OK;
}

#define TRY(x)                           \
    do {                                 \
        int rc_ = (x);                   \
        if (rc_ != LPSIM_OK) return rc_; \
    } while (0)

// The block that searches a tree in shared memory: the one of which most fit an
// SM (a tree is a chain of round trips, so trees in flight count first), of
// those the one with most threads, of those the one with most registers.
// Measured, ms per search with all its host work (td_trees_shared<256, 8> / <256, 4> /
// <512, 2> / <1024, 1>; trees per SM in brackets; lattices of the nodes given, 5 and 15 trips a
// node, the latter after the comma): 2,500 nodes (8 / 4 / 2 / 1) and 1,840 trees 0.55 / 0.69 / 1.01;
// 6,084 (8 / 4 / 2) and 2,860 trees 1.72 / 2.04 / 2.81; 8,464 (6 / 4 / 2 / 1) 1.70 / 1.69 / 2.34 / 3.76, 3.30
// / 3.92 / 5.80 / 9.84; 10,201 (5 / 4 / 2 / 1) 2.16 / 2.28 / 3.07 / 4.90, 5.96 / 6.19 / 7.78 / 12.5; 12,100 (4 / 4 /
// 2 / 1) 3.01 / 2.89 / 3.77 / 6.08, 7.12 / 6.82 / 9.55 / 15.8; 17,956 (3 / 3 / 2 / 1) - / 6.16 / 6.36 / 9.86; 18,225
// (2 / 2 / 2 / 1) - / 7.33 / 6.22 / 9.86; 27,225 (the same) - / 13.1 / 10.9 / 17.0; 27,556 (1 / 1 / 1 / 1) - / 22.9
// / 18.4 / 17.0.  (7,225 nodes with 1,803 trees, a little more than the seven per SM take at once, are the
// exception found: 1.81 / 1.59; with 4,758 trees 3.15 / 3.34.)  At 32 registers <256, 8> spills 24 bytes.
// Bucket widths of 60 / 120 / 240 / 480 s: 27,225 nodes 15.0 / 13.6 / 12.3 / 12.9
// (before the wide rows, which took 12.3 to 10.9).
using TreeKernel = void (*)(TreeArgs);
constexpr struct {
    TreeKernel kernel;
    int threads;
} kTreeBlocks[] = {{td_trees_shared<256, 8>, 256},
                   {td_trees_shared<256, 4>, 256},
                   {td_trees_shared<512, 2>, 512},
                   {td_trees_shared<1024, 1>, 1024}};  // more threads, then more registers, to the end

int choose_tree_block(AssignGpu *g, uint32_t n_nodes) {
    if (n_nodes > 0xFFFFu) return LPSIM_OK;  // ids in the ring have 16 bits
    const size_t smem = shared_tree_bytes(n_nodes);
    int max_smem = 0, most = 0;
    CU(cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, g->device));
    for (const auto &b : kTreeBlocks) {
        cudaFuncAttributes fa{};
        CU(cudaFuncGetAttributes(&fa, b.kernel));
        if (smem + fa.sharedSizeBytes > (size_t)max_smem) continue;
        CU(cudaFuncSetAttribute(b.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                max_smem - (int)fa.sharedSizeBytes));
        int per_sm = 0;
        CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, b.kernel, b.threads, smem));
        if (per_sm == 0 || per_sm < most) continue;
        most = per_sm;
        g->shared_kernel = b.kernel;
        g->shared_threads = (uint32_t)b.threads;
        g->shared_blocks = (uint32_t)(g->n_sm * per_sm);
    }
    return LPSIM_OK;
}

// graph, trips and workspaces (first call)
int gpu_setup(lpsim_assign *a) {
    auto *g = new (std::nothrow) AssignGpu();
    if (!g) return fail(LPSIM_E_OOM, "host allocation failed");
    a->gpu = g;
    CU(cudaGetDevice(&g->device));
    CU(cudaDeviceGetAttribute(&g->n_sm, cudaDevAttrMultiProcessorCount, g->device));
    CU(cudaStreamCreateWithFlags(&g->stream, cudaStreamNonBlocking));
    if (a->n >= 0xFFFFFFFFull) return fail(LPSIM_E_INVALID_ARG, "too many trips for the GPU search");
    TreeArgs &A = g->A;
    A.n_nodes = a->n_nodes;
    A.n_edges = a->n_edges;
    std::vector<uint2> adj(a->n_edges);
    for (uint32_t j = 0; j < a->n_edges; j++) adj[j] = make_uint2(a->out_edge[j], a->dst[a->out_edge[j]]);
    std::vector<uint32_t> dep_ms(a->n);
    for (uint64_t j = 0; j < a->n; j++) {
        const uint64_t t = to_ms((double)a->dep[j] * a->dt);
        if (t > 0xFFFFFFFFull) return fail(LPSIM_E_INVALID_ARG, "departure beyond the 32-bit millisecond range");
        dep_ms[j] = (uint32_t)t;
    }
    // positions of the edges among the out-edges, and the in-edges of every node by ascending edge id
    std::vector<uint32_t> pos(a->n_edges), in_off(a->n_nodes + 1, 0);
    bool identity = true;
    for (uint32_t j = 0; j < a->n_edges; j++) {
        pos[a->out_edge[j]] = j;
        identity = identity && a->out_edge[j] == j;
        in_off[adj[j].y + 1]++;
    }
    for (uint32_t v = 0; v < a->n_nodes; v++) in_off[v + 1] += in_off[v];
    std::vector<uint2> in_adj(a->n_edges);
    {
        std::vector<uint32_t> at(in_off.begin(), in_off.end() - 1);
        for (uint32_t e = 0; e < a->n_edges; e++) in_adj[at[a->dst[e]]++] = make_uint2(pos[e], a->src[e]);
    }
    uint32_t *oo, *sr, *de, *dm, *po = nullptr, *io;
    uint2 *ad, *ia;
    if (!identity) TRY(dput(g, po, pos.data(), pos.size()));
    TRY(dput(g, io, in_off.data(), in_off.size()));
    TRY(dput(g, ia, in_adj.data(), in_adj.size()));
    A.pos = po;
    A.in_off = io;
    A.in_adj = ia;
    TRY(dput(g, oo, a->out_off.data(), a->out_off.size()));
    TRY(dput(g, ad, adj.data(), adj.size()));
    TRY(dput(g, sr, a->src.data(), a->src.size()));
    TRY(dput(g, de, a->dest.data(), a->dest.size()));
    TRY(dput(g, dm, dep_ms.data(), dep_ms.size()));
    A.out_off = oo;
    A.adj = ad;
    A.src = sr;
    A.dest = de;
    A.dep_ms = dm;
    A.path_off = static_cast<unsigned long long *>(g->alloc(a->n * 8));
    A.path_len = static_cast<uint32_t *>(g->alloc(a->n * 4));
    A.tsp = static_cast<float *>(g->alloc(a->n * 4));
    A.cursor = static_cast<unsigned long long *>(g->alloc(8));
    A.next_group = static_cast<uint32_t *>(g->alloc(4));
    A.err = static_cast<uint32_t *>(g->alloc(4));
    if (!A.path_off || !A.path_len || !A.tsp || !A.cursor || !A.next_group || !A.err)
        return fail(LPSIM_E_OOM, "device allocation failed");
    A.delta_ms = kDeltaMs;
    // labels in shared memory where they fit
    TRY(choose_tree_block(g, a->n_nodes));
    if (g->shared_blocks) {
        uint32_t most = 0;
        for (uint32_t u = 0; u < a->n_nodes; u++) most = std::max(most, a->out_off[u + 1] - a->out_off[u]);
        if (most <= kWide) {
            const uint32_t w = most <= 4 ? 4 : 8;
            std::vector<uint2> wadj((size_t)w * a->n_nodes, make_uint2(kNoEdge, kNever)), win(a->n_edges);
            std::vector<uint32_t> at(in_off.begin(), in_off.end() - 1);
            for (uint32_t u = 0; u < a->n_nodes; u++)
                for (uint32_t j = a->out_off[u]; j < a->out_off[u + 1]; j++)
                    wadj[(size_t)u * w + (j - a->out_off[u])] = adj[j];
            for (uint32_t e = 0; e < a->n_edges; e++) {
                const uint32_t u = a->src[e];
                win[at[a->dst[e]]++] = make_uint2(u * w + (pos[e] - a->out_off[u]), u);
            }
            uint2 *wa, *wi;
            TRY(dput(g, wa, wadj.data(), wadj.size()));
            TRY(dput(g, wi, win.data(), win.size()));
            CU(cudaStreamSynchronize(g->stream));
            g->wide_adj = wa;
            g->wide_in = wi;
            g->wide = w;
        }
        // all resident threads' positions take no more than the workspaces of td_trees' warps would
        // (a longer path is written to the output in two walks)
        const uint64_t room = (uint64_t)kBlocksPerSm * kWarpsPerBlock * g->n_sm * kWorkspacePerNode * a->n_nodes / 4;
        A.scratch_len = (uint32_t)std::min<uint64_t>(std::min(kScratch, a->n_nodes),
                                                     room / ((uint64_t)g->shared_blocks * g->shared_threads) + 1);
        CU(cudaStreamSynchronize(g->stream));  // the host arrays go away
        return LPSIM_OK;
    }
    // workspaces: as many warps as fit the budget, at most kBlocksPerSm * kWarpsPerBlock per SM
    const uint64_t per_warp = (uint64_t)a->n_nodes * kWorkspacePerNode;
    uint64_t warps = std::min<uint64_t>((uint64_t)g->n_sm * kBlocksPerSm * kWarpsPerBlock,
                                        std::max<uint64_t>(kWorkspaceBudget / std::max<uint64_t>(per_warp, 1), 1));
    warps = std::max<uint64_t>(kWarpsPerBlock, warps / kWarpsPerBlock * kWarpsPerBlock);
    g->n_warps = (uint32_t)warps;
    const size_t nn = (size_t)warps * a->n_nodes;
    A.node = static_cast<NodeRec *>(g->alloc(nn * sizeof(NodeRec)));
    A.touched = static_cast<uint32_t *>(g->alloc(nn * 4));
    A.fa = static_cast<uint32_t *>(g->alloc(nn * 4));
    A.fb = static_cast<uint32_t *>(g->alloc(nn * 4));
    A.far = static_cast<uint32_t *>(g->alloc(nn * 4));
    A.stamp = static_cast<uint32_t *>(g->alloc(warps * 4));
    if (!A.node || !A.touched || !A.fa || !A.fb || !A.far || !A.stamp)
        return fail(LPSIM_E_OOM, "device allocation of the search workspaces failed");
    init_nodes<<<g->n_sm * 4, 256, 0, g->stream>>>(A.node, nn);
    CU(cudaGetLastError());
    CU(cudaMemsetAsync(A.stamp, 0, warps * 4, g->stream));
    CU(cudaStreamSynchronize(g->stream));
    return LPSIM_OK;
}

// the device copy, made at the first call (a failed attempt leaves none)
int gpu_ready(lpsim_assign *a) {
    if (a->gpu) return LPSIM_OK;
    const int rc = gpu_setup(a);
    if (rc) {
        assign_gpu_free(a->gpu);
        a->gpu = nullptr;
    }
    return rc;
}

// trip groups of a departure period length (kept between calls)
int gpu_groups(lpsim_assign *a, uint32_t period_steps) {
    AssignGpu *g = a->gpu;
    if (g->period_steps == period_steps) return LPSIM_OK;
    group_trips(a, period_steps, g->order, g->gstart);
    const uint64_t ng = g->gstart.size() - 1;
    std::vector<GroupRec> recs(ng);
    std::vector<uint32_t> ord(a->n);
    for (uint64_t i = 0; i < a->n; i++) ord[i] = (uint32_t)g->order[i];
    for (uint64_t q = 0; q < ng; q++) {
        const uint64_t j0 = g->order[g->gstart[q]];
        const uint64_t t0 = period_root_ms(a, a->dep[j0] / period_steps, period_steps);
        if (t0 > 0xFFFFFFFFull) return fail(LPSIM_E_INVALID_ARG, "departure period beyond the millisecond range");
        recs[q] = GroupRec{a->orig[j0], (uint32_t)t0, (uint32_t)g->gstart[q],
                           (uint32_t)(g->gstart[q + 1] - g->gstart[q])};
    }
    // no grouping until the new one is there
    g->period_steps = 0;
    if (g->A.groups) g->release(const_cast<GroupRec *>(g->A.groups));
    if (g->A.order) g->release(const_cast<uint32_t *>(g->A.order));
    g->A.groups = nullptr;
    g->A.order = nullptr;
    GroupRec *dg;
    uint32_t *dord;
    TRY(dput(g, dg, recs.data(), recs.size()));
    g->A.groups = dg;
    TRY(dput(g, dord, ord.data(), ord.size()));
    g->A.order = dord;
    g->A.n_groups = (uint32_t)ng;
    g->period_steps = period_steps;
    return LPSIM_OK;
}

}  // namespace

namespace {

// the link-time table of tt in whole milliseconds on the device (as the host
// searches' table), by out-edge position (A.cms) or, for a search with wide
// rows, by those
int gpu_table(lpsim_assign *a, const float *tt, uint32_t n_bins, uint32_t bin_steps, bool wide) {
    AssignGpu *g = a->gpu;
    TreeArgs &A = g->A;
    const uint64_t bin_ms = table_bin_ms(a, bin_steps);
    if (bin_ms > 0xFFFFFFFFull) return fail(LPSIM_E_INVALID_ARG, "bin longer than the 32-bit millisecond range");
    const uint32_t n_pos = wide ? g->wide * a->n_nodes : a->n_edges;
    const size_t in_cells = (size_t)n_bins * a->n_edges, cells = (size_t)n_bins * n_pos;
    if (cells > g->table_cells[wide] && !g->regrow(g->table[wide], g->table_cells[wide], cells))
        return fail(LPSIM_E_OOM, "device allocation of the link-time table failed");
    if (in_cells > g->tt_cells && !g->regrow(g->tt, g->tt_cells, in_cells))
        return fail(LPSIM_E_OOM, "device allocation of the link times failed");
    CU(cudaMemcpyAsync(g->tt, tt, in_cells * 4, cudaMemcpyHostToDevice, g->stream));
    if (n_pos)
        link_table<<<(n_pos + 31) / 32, 256, 0, g->stream>>>(g->tt, wide ? g->wide_adj : A.adj, n_pos, n_bins, bin_ms,
                                                            g->table[wide]);
    CU(cudaGetLastError());
    A.cms = g->table[wide];
    A.n_bins = n_bins;
    A.bin_ms = (uint32_t)bin_ms;
    return LPSIM_OK;
}

}  // namespace

extern "C" int lpsim_assign_load_gpu(const lpsim_assign *ac, const float *tt, uint32_t n_bins, uint32_t bin_steps,
                                     uint32_t *inflow) {
    lpsim_assign *a = const_cast<lpsim_assign *>(ac);
    if (!a || !tt || !inflow || n_bins == 0 || bin_steps == 0) return fail(LPSIM_E_INVALID_ARG, "bad argument");
    if (a->n == 0) {
        std::memset(inflow, 0, (size_t)a->n_edges * n_bins * 4);
        return LPSIM_OK;
    }
    TRY(gpu_ready(a));
    AssignGpu *g = a->gpu;
    int dev = -1;
    CU(cudaGetDevice(&dev));
    if (dev != g->device) return fail(LPSIM_E_STATE, "the device current at the first GPU call must be current");
    TRY(gpu_table(a, tt, n_bins, bin_steps, false));
    // the engine's routes stay on the device; a re-routing brings what it wrote
    if (!g->span) {
        g->span = static_cast<ulonglong2 *>(g->alloc(a->n * sizeof(ulonglong2)));
        if (!g->span) return fail(LPSIM_E_OOM, "device allocation of the route offsets failed");
    }
    if (g->routes_version != a->routes_version) {
        g->routes_version = ~0ull;
        if (g->layout != a->layout) g->redge_here = 0;
        if (a->redge_used > g->redge_cap) {
            g->redge_here = 0;
            if (!g->regrow(g->redge, g->redge_cap, a->redge.cap))
                return fail(LPSIM_E_OOM, "device allocation of the routes failed");
        }
        static_assert(sizeof(RouteSpan) == sizeof(ulonglong2), "route spans");
        CU(cudaMemcpyAsync(g->span, a->span.data(), a->n * sizeof(ulonglong2), cudaMemcpyHostToDevice, g->stream));
        if (a->redge_used > g->redge_here)
            CU(cudaMemcpyAsync(g->redge + g->redge_here, a->redge.p.get() + g->redge_here,
                               (a->redge_used - g->redge_here) * 4, cudaMemcpyHostToDevice, g->stream));
        CU(cudaStreamSynchronize(g->stream));
        g->redge_here = a->redge_used;
        g->layout = a->layout;
        g->routes_version = a->routes_version;
    }
    const size_t cells = (size_t)a->n_edges * n_bins;
    if (cells > g->inflow_cells && !g->regrow(g->inflow, g->inflow_cells, cells))
        return fail(LPSIM_E_OOM, "device allocation of the inflow table failed");
    CU(cudaMemsetAsync(g->inflow, 0, cells * 4, g->stream));
    load_routes<<<(unsigned)std::min<uint64_t>((a->n + 255) / 256, 65535), 256, 0, g->stream>>>(
        g->span, g->redge, g->A.dep_ms, a->n, g->A.cms, g->A.pos, a->n_edges, n_bins, g->A.bin_ms, g->inflow);
    CU(cudaGetLastError());
    CU(cudaMemcpyAsync(inflow, g->inflow, cells * 4, cudaMemcpyDeviceToHost, g->stream));
    CU(cudaStreamSynchronize(g->stream));
    return LPSIM_OK;
}

extern "C" int lpsim_assign_shortest_paths_gpu(lpsim_assign *a, const float *tt, uint32_t n_bins, uint32_t bin_steps,
                                               uint32_t period_steps, float *t_sp) {
    if (!a || !tt || n_bins == 0 || bin_steps == 0 || period_steps == 0)
        return fail(LPSIM_E_INVALID_ARG, "bad argument");
    if (a->n == 0) return LPSIM_OK;
    TRY(gpu_ready(a));
    AssignGpu *g = a->gpu;
    int dev = -1;
    CU(cudaGetDevice(&dev));
    if (dev != g->device) return fail(LPSIM_E_STATE, "the device current at the first GPU search must be current");
    TRY(gpu_groups(a, period_steps));
    TreeArgs &A = g->A;
    TRY(gpu_table(a, tt, n_bins, bin_steps, g->wide != 0));
    // positions along the paths: for the blocks these trees need, grown when another grouping has more
    const uint32_t blocks = std::min(g->shared_blocks, std::max(A.n_groups, 1u));
    const uint64_t scratch = (uint64_t)blocks * g->shared_threads * A.scratch_len;
    if (scratch > g->scratch_cap && !g->regrow(A.scratch, g->scratch_cap, scratch))
        return fail(LPSIM_E_OOM, "device allocation of the search workspaces failed");
    // path buffer: room for the current routes' length and half as much again
    if (!g->cap) {
        const uint64_t total = a->route_total;
        if (!g->regrow(A.edges, g->cap, std::max<uint64_t>(total + total / 2, 1u << 20)))
            return fail(LPSIM_E_OOM, "device allocation of the path buffer failed");
    }
    unsigned long long used = 0;
    uint32_t err = 0;
    for (int attempt = 0; attempt < 3; attempt++) {
        A.cap = g->cap;
        CU(cudaMemsetAsync(A.cursor, 0, 8, g->stream));
        CU(cudaMemsetAsync(A.next_group, 0, 4, g->stream));
        CU(cudaMemsetAsync(A.err, 0, 4, g->stream));
        if (g->shared_blocks) {
            TreeArgs S = A;
            S.delta_ms = kSharedDeltaMs;
            S.wide = g->wide;
            S.n_pos = g->wide ? g->wide * a->n_nodes : a->n_edges;
            if (g->wide) {
                S.adj = g->wide_adj;
                S.in_adj = g->wide_in;
            }
            g->shared_kernel<<<blocks, g->shared_threads, shared_tree_bytes(a->n_nodes), g->stream>>>(S);
        } else
            td_trees<<<g->n_warps / kWarpsPerBlock, kWarpsPerBlock * 32, 0, g->stream>>>(A);
        CU(cudaGetLastError());
        CU(cudaMemcpyAsync(&used, A.cursor, 8, cudaMemcpyDeviceToHost, g->stream));
        CU(cudaMemcpyAsync(&err, A.err, 4, cudaMemcpyDeviceToHost, g->stream));
        CU(cudaStreamSynchronize(g->stream));
        if (!(err & kErrCapacity)) break;
        // the paths did not fit: a buffer of the length they asked for, and again
        if (!g->regrow(A.edges, g->cap, used + used / 4 + 1024))
            return fail(LPSIM_E_OOM, "device allocation of the path buffer failed");
    }
    if (err & kErrBound) return fail(LPSIM_E_INVARIANT, "GPU path search exceeded its round or path-length bound");
    if (err & kErrUnreachable) return fail(LPSIM_E_INVALID_ARG, "a destination is unreachable from its origin");
    if (err & kErrCapacity) return fail(LPSIM_E_OOM, "path buffer still too small after resizing");
    // the candidates as the search left them: offsets, lengths and one array of edges
    std::fill(a->clen.begin(), a->clen.end(), 0u);
    if (!a->cedge.reserve(used)) return fail(LPSIM_E_OOM, "host allocation of the paths failed");
    static_assert(sizeof(unsigned long long) == sizeof(uint64_t), "path offsets");
    if (used) CU(cudaMemcpyAsync(a->cedge.p.get(), A.edges, used * 4, cudaMemcpyDeviceToHost, g->stream));
    CU(cudaMemcpyAsync(a->coff.data(), A.path_off, a->n * 8, cudaMemcpyDeviceToHost, g->stream));
    CU(cudaMemcpyAsync(a->tsp.data(), A.tsp, a->n * 4, cudaMemcpyDeviceToHost, g->stream));
    CU(cudaMemcpyAsync(a->clen.data(), A.path_len, a->n * 4, cudaMemcpyDeviceToHost, g->stream));
    CU(cudaStreamSynchronize(g->stream));
    if (t_sp) std::memcpy(t_sp, a->tsp.data(), a->n * 4);
    return LPSIM_OK;
}
