// GB300 (sm_103a) dynamic max-flow: device kernels and the C ABI of mf.h.
//
// The whole solve / repair of one graph is ONE persistent cooperative kernel
// (k_solve): its CTAs, one full wave or fewer for a small graph, run the phases
// below in lock-step, separated by a bounded grid barrier, so the loops (BFS
// levels, the push/relabel rounds) never return to the host (the paper also
// decides termination on the device, Sec. 3):
//
//   validate batch -> apply capacity changes (Alg. 5, lines 1-3)
//   -> clamp negative residuals (Alg. 5, lines 4-11)
//   -> saturate source arcs (Alg. 4 lines 3-7 / Alg. 1 third loop)
//   -> loop { height init with deficient vertices as sinks (Alg. 4)
//             backward BFS global relabel + active worklist (Sec. 5.3)
//             stop when no vertex is active
//             PushRelabel x KERNELCYCLES (Alg. 2)
//             RemoveInvalidEdges (Alg. 3)
//             stop when that round left nothing pending (Alg. 4's own test) }
//   -> flow = e(t) + sum of deficits (Alg. 4, final sum).
//
// Dynamic Push-Pull (Alg. 6-8) runs in the same loop, in the instance
// k_solve<true>: saturate the arcs across the previous cut, then push on its
// sink side and pull on its source side (one search, both heights in h), then
// the plain loop on the leftover subgraph P.  A batch that only raises
// capacities off the exact cut skips the loop (the flow cannot change).
//
// Residual capacities are kept twice: r[a] and its mirror rr[a] = r[rev[a]],
// so that the backward BFS reads the residual of the arc INTO the frontier
// vertex from a contiguous array instead of gathering r[rev[a]].  Every write
// to r[x] has a matching write to rr[rev[x]].
//
// Mutable arrays are read with ld.global.cg (L2, coherent across SMs), or
// through L1 (ld.ca) in phases during which they do not change or an early read
// is exact; the barrier's acquire drops what L1 holds, so nothing is relied on
// across one.
//
// The phases avoid atomics that the whole grid aims at one address: the
// items of a phase are dealt to the CTAs by a fixed stride and taken by their
// warps from a counter in shared memory, and each warp stages the BFS frontier
// it discovers in shared memory and publishes it a stage at a time.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "mf.h"
#include "mf_internal.h"
#include "mf_mlp.cuh"

namespace mf {

constexpr int kBlock = 768;   // one CTA per SM: 152 arrivals per grid barrier
constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned long long kWaitNs = 20ull * 1000ull * 1000ull * 1000ull;  // 20 s per barrier wait

// status bits (Ctl::status)
constexpr int ST_EINVAL = 1;   // rejected batch (state unchanged)
constexpr int ST_ITERS = 2;    // max_iters reached
constexpr int ST_WAIT = 4;     // a grid-barrier wait reached its time limit
constexpr int ST_TIME = 8;     // the kernel ran past its wall-clock limit
constexpr int ST_CHECK = 16;   // a debug_checks consistency check failed
constexpr int ST_STICKY = ST_ITERS | ST_WAIT | ST_TIME | ST_CHECK;

// JOB_REFRESH recomputes exact BFS heights (and the exact cut S = {h >= n})
// for a state whose last solve stopped without a final BFS; it does nothing
// when the heights are exact already.
enum JobKind { JOB_SOLVE = 0, JOB_REPAIR = 1, JOB_RECOMPUTE = 2, JOB_AUTO = 3, JOB_REFRESH = 4 };

// How the last solve/repair ended (mf_stats.exit_kind)
enum ExitKind { EXIT_BFS = 0, EXIT_CLEAN = 1, EXIT_NO_CUT_CHANGE = 2, EXIT_PUSH_PULL = 3 };

// Most PushRelabel rounds of the topology-driven mode per loop iteration
// (more on deep graphs), and the fewest
// cooperative cycles the high-degree vertices get per iteration (see k_solve).
constexpr int kMaxRounds = 16;
// The activation queue gets as long as the last BFS took (see k_solve), and
// serves at least kMinGen generations.  Measured per batch with a share of 1/2,
// 3/4, 1, 11/8 of it and 8 generations: unit assignment graph of 2^18 + 2^18
// vertices 1.28, 1.20, 1.15, 1.17 ms; 1023 x 769 grid 1.05, 0.96, 0.98, 0.95 ms;
// 2048^2 grid (push-pull) 2.17, 2.07, 1.95, 1.95 ms; RMAT-20 static solve 2.22,
// 2.18, 2.18, 2.23 ms; 1000-vertex graph 113, 116, 119, 128 us (134 with 12
// generations; with 6, short chains no longer end inside one phase).  A bound
// of max(16, BFS levels) generations instead, measured before the search got
// faster, cost the assignment graph 27 % and the grids 11-17 %.
constexpr int kMinGen = 8;         // activation generations served whatever the time
constexpr int kMinHubCycles = 4;
// The push-pull instance gives its hubs more cycles per pass: there a hub
// left active costs another dual search of the whole graph (measured on
// RMAT-20 100k batches: 3.2 -> 2.0-3.2 loop iterations, 1.24 -> 1.14 ms).
constexpr int kMinHubCyclesPP = 8;
// PushRelabel passes per loop iteration (hub cycles, then activation rounds;
// a pass that turns hubs active again hands them to the next pass, when
// there are at most kPassHubs of them).  The push-pull instance takes more:
// there the re-activated hubs are few and another pass costs much less than
// another dual BFS (measured on RMAT-20: 1.66 -> 1.32 ms per repair).
constexpr int kMaxPasses = 2;
constexpr int kMaxPassesPP = 4;
// BFS levels whose frontier has at most this many arcs and vertices (fewer in
// some graphs: search_rules) run on CTA 0 alone, with the frontiers in shared
// memory
constexpr long long kSoloArcs = 8192;
constexpr int kSoloCap = 4096;
// Above this many hubs the cycles file no activations and one pass over all
// vertices finds the active ones (7-10 us on 2^20 vertices); filing made every
// pushing item wait for its atomics, a stamp, a fence and a queue reservation
// (measured on RMAT-20 100k batches with ~2,000 hubs: 38 -> 29 us per push
// phase).  A few hubs are better off filing.
constexpr int kDeferHubs = 128;
constexpr int kPassHubs = 32;   // most re-activated hubs a further pass takes
constexpr int kPassHubsPP = 64;

constexpr int S_COUNT_MAX = 24;

// Device control block.  Fields marked (z) are zero whenever no k_solve is
// running: they are zeroed at creation, by mf_solve, and by the last thread
// of every k_solve that ends normally.
struct Ctl {
    int status;           // ST_* bits                      } read together by
    int batch_err;        // (z) set by batch validation    } mf_flow_value
    long long flow;       // result of the last solve/repair }
    unsigned bar_word;    // grid barrier: generation (high 16 bits), arrivals (z, low 16 bits)
    unsigned bar_pad;
    int qcnt[3];          // (z) BFS frontier sizes, rotating by level
    int ccnt[3];          // (z) BFS chunk-item counts, rotating by level
    long long asum[3];    // (z) sum of the degrees of each BFS frontier, rotating
    int acnt[3];          // (z) activation-round list sizes, rotating by round
    int rlcnt;            // (z) relabel list size
    unsigned stamp_base;  // first activation stamp of the next launch (kept across launches)
    unsigned bseq;        // sequence number of the last batch (duplicate-id stamps)
    int wcnt;             // (z) active worklist size (vertices of degree <= kHubDeg)
    int hcnt;             // (z) active hub list size (degree > kHubDeg)
    int hub_live[2];      // (z) hubs and items of a hub cycle's list, by cycle parity
    int hub_items[2];     // (z)
    int hub_act[2];       // (z) hubs still active after a short list's pushes, by cycle parity
    int pad0;
    long long dacc[2];    // (z) sum of deficits at the last height init
    long long iters;
    unsigned long long t_start;  // globaltimer at kernel entry
    int pol_kind;         // policy decision for the next JOB_AUTO launch
    int pol_kc;
    int pol_mode;         // processing mode chosen for it (MF_MODE_*)
    int pol_fallback;     // 1 if the learned policy fell back to the plain rule
    float feat[12];       // features of the last batch the policy kernel saw
    long long pol_acc[3]; // (z) k_policy's batch sums: increments, entries at s or t, sum |delta|
    int pol_done;         // (z) k_policy CTAs that have added their sums
    int pad3;
    int abort_loop;       // (z) set by thread 0 when the wall-clock limit passed
    int trace_n;          // trace records written by the current launch
    int ri_moved[2];      // (z) RemoveInvalidEdges saturated an arc, by iteration parity
    int phc[2];           // (z) hub lists of the next PushRelabel pass, by pass parity
    int rhcnt;            // (z) RemoveInvalidEdges items of relabelled hubs
    int pad2;
    int inc_block;        // (z) the batch holds a decrement or an increment across the cut
    int heights_exact;    // h is the BFS fixed point of the current residual graph
    int pairs_ok;         // r(a) + r(rev a) = cap(a) + cap(rev a) on every pair, and rr mirrors r
    int cut_exact;        // {h >= n} is exactly the set that cannot reach a sink
    int exit_kind;        // ExitKind of the last solve/repair
    int solo_L;           // BFS level at which CTA 0 hands a small-frontier run back
    long long solo_seen;  // frontier arcs counted up to that level
    long long st[S_COUNT_MAX];  // statistics, see enum Stat
    long long st_aux[S_COUNT_MAX];  // where a JOB_REFRESH counts, keeping st intact
    // the activation queue of a PushRelabel phase (see k_solve), one set per
    // pass parity: consumer tickets, producer reservations and finished
    // entries, each on its own 128-byte line (every warp of the grid polls or
    // bumps them)
    struct Queue {
        alignas(128) int head;   // (z)
        alignas(128) int tail;   // (z)
        alignas(128) int done;   // (z)
        alignas(128) int over;   // (z) an active vertex was left out (time, full queue)
        int maxgen;              // (z) highest generation enqueued
        alignas(128) int fin;    // (z) every queued entry has been processed
        __device__ void clear() { head = tail = done = over = maxgen = fin = 0; }
    } q[2];
    long long chk_where;        // first failed debug check: kind << 40 | index (kept until mf_solve)
};

enum Stat {
    S_LEVELS, S_BFS_VERTS, S_BFS_ARCS, S_WL, S_PR_ARCS, S_PUSH, S_RELABEL, S_RI_ARCS, S_RI_MOVES,
    S_BATCH, S_CLAMPED, S_RESAT,
    // phase times (ns, globaltimer of CTA 0 between grid barriers) and counts
    S_T_BATCH, S_T_RESET, S_T_BFS, S_T_PRW, S_T_HUB, S_T_RI, S_HUB_CYCLES, S_BARRIERS,
    S_BU_LEVELS, S_ROUNDS,
    S_COUNT
};
static_assert(S_COUNT <= S_COUNT_MAX, "statistics array too small");

// One trace record per grid barrier of k_solve (see mf_trace_read in mf.h).
struct TraceRec {
    short phase, mode;
    int iter, step, count;
    long long ns;
};

struct DevGraph {
    int n, s, t, m;
    long long A;
    int cap_limit;
    const int *row, *head, *rev, *arc_of_edge;
    const unsigned char *edge_st;   // per edge: 1 if it leaves s or enters t (policy feature), or nullptr
    int *cap, *r, *rr, *h, *cap_edge;
    long long *e;
    unsigned *stamp;
    int *qb0, *qb1, *wl;
    int2 *cb;
    int *hl;                  // active hubs
    int *hl2;                 // hub list of odd PushRelabel passes
    int2 *hri;                // RemoveInvalidEdges items of relabelled hubs (vertex, first arc)
    int *hlist0, *hlist1;     // hubs of a cycle's list (indices into hl or hl2), by cycle parity
    int4 *hit0, *hit1;        // their work items (HubItem), by cycle parity
    int *hikey;               // lowest residual-neighbour height per item of the current cycle
    int *hkey;                // per hub, by cycle parity (two each)
    long long *hrem;          // per-hub excess left to push in the current cycle
    TraceRec *trace;          // per-barrier trace records, or null
    int trace_cap;
    unsigned *astamp;         // per-vertex stamp of the last activation list joined
    unsigned *rstamp;         // per-vertex stamp of the last relabel list joined
    int *rl;                  // vertices relabelled in the current loop iteration
    unsigned char *part;      // push-pull partition per vertex (kPartT / kPartS / kPartP), or null
    Ctl *ctl;
    int al16;                 // head, r and rr start on 16-byte boundaries (16-byte staging copies)
    unsigned long long *aq;   // activation queue slots (generation << 32 | vertex + 1; 0 = empty)
    int qc;                   // its capacity
    int bu_long;              // bottom-up levels mostly read whole rows (search_rules)
    int solo_arcs;            // most arcs of a frontier that CTA 0 searches alone (<= kSoloArcs)
    int alpha;                // the search goes bottom-up when alpha x its frontier's arcs pass the unvisited arcs
};

// Push-pull partitions (Alg. 8): T can reach a sink, S cannot (the previous
// cut); P holds what neither stage-1 BFS reached.
constexpr unsigned char kPartT = 0, kPartS = 1, kPartP = 2;

struct Job {
    int kind, k, flags, kc, mode;
    int debug;           // debug_checks: list-entry bounds and the end-of-kernel invariants
    int exact_exit;      // 1: stop only after a BFS finds no active vertex
    int pp;              // 1: a repair by Dynamic Push-Pull (Alg. 8) when the cut is exact
    int sink_sat;        // 1: a solve from zero flow also saturates the arcs into t
    long long *st;       // statistics array (Ctl::st, or Ctl::st_aux for JOB_REFRESH)
    TraceRec *trace;     // trace records, or nullptr
    const int *k_dev;    // if set, the batch size is read from device memory
    long long max_iters;
    unsigned long long time_limit_ns;
    const int *ids, *caps;
    int *newc, *dlt;
};

// ---------------------------------------------------------------- helpers --
__device__ __forceinline__ int lcg(const int *p) { return __ldcg(p); }
__device__ __forceinline__ long long lcg(const long long *p) { return __ldcg(p); }
__device__ __forceinline__ int2 lcg(const int2 *p) { return __ldcg(p); }

// The height of a vertex in a phase that does not depend on heights written
// during it (see the callers): a plain load, which L1 may serve.
__device__ __forceinline__ int lheight(const int *p) {
    return __ldca(p);
}

__device__ __forceinline__ void add_ll(long long *p, long long v) {
    atomicAdd(reinterpret_cast<unsigned long long *>(p), static_cast<unsigned long long>(v));
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ int ld_acquire_s32(const int *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed_u64(unsigned long long *p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void fence_acq_rel() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// A value every lane of the warp must agree on (it steers warp-wide control
// flow): read once by lane 0 and broadcast.  A word that other warps write
// concurrently could otherwise reach the lanes as different values.
__device__ __forceinline__ int bcast_ld(const int *p) {
    return __shfl_sync(0xffffffffu, (threadIdx.x & 31) == 0 ? __ldcg(p) : 0, 0);
}
__device__ __forceinline__ long long bcast_ld(const long long *p) {
    return __shfl_sync(0xffffffffu, (threadIdx.x & 31) == 0 ? __ldcg(p) : 0ll, 0);
}

__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ long long warp_incl_scan(long long x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Warp-aggregated append: one atomicAdd per warp (Sec. 5.3: ballot, then the
// warp leader reserves space).  Must be called by all 32 lanes.
__device__ __forceinline__ void warp_append(bool pred, int val, int *cnt, int *buf) {
    const unsigned mask = __ballot_sync(kFull, pred);
    if (!mask) return;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(mask) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(cnt, __popc(mask));
    base = __shfl_sync(kFull, base, leader);
    if (pred) buf[base + __popc(mask & ((1u << lane) - 1u))] = val;
}

// A control word that was last written before the grid barrier the thread has
// just passed (list sizes, flags): a plain load, which may be served by L1.
// The barrier's acquire makes those writes visible to every thread of the CTA
// and drops what L1 held before.  All 24 warps of an SM then share one L2
// request; with ld.cg each of the grid's 3,648 warps sent its own to the one
// L2 slice that holds the word.
template <class T>
__device__ __forceinline__ T lctl(const T *p) {
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "control words");
    T v;
    if constexpr (sizeof(T) == 4) asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    else asm volatile("ld.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Two counters in the CTA's shared memory that are zero at the start of every
// phase (the grid barrier resets them).
__device__ __forceinline__ int *cta_words() {
    static __shared__ int w[2];
    return w;
}

// The next of the CTA's work items, to one warp: 0, 1, ...  All 32 lanes call.
__device__ __forceinline__ int cta_ticket(int *word) {
    int k = 0;
    if ((threadIdx.x & 31) == 0) k = atomicAdd(word, 1);
    return __shfl_sync(kFull, k, 0);
}

// The next of a phase's `count` work items, to one warp: each warp starts with
// item gwarp (item w belongs to CTA w mod gridDim.x) and takes further ones of
// its CTA's share as it gets free.  A fixed stride over the warps left them
// waiting at the barrier 33-58 % of the time in the search and hub phases; the
// slowest of 24 warps sets the CTA's time.  (RMAT-20 100k and static solve -4 %,
// 2048^2 grid -4 %; a counter of the whole grid would be one hot word.)
// Returns >= count when there is none.  All 32 lanes call.
__device__ __forceinline__ int next_item(int *word, int count) {
    const int first = (int)gridDim.x * (int)(blockDim.x >> 5);
    return count <= first ? count : first + cta_ticket(word) * (int)gridDim.x + (int)blockIdx.x;
}

// Bounded grid barrier for a cooperative (co-resident) grid.  One word holds
// the generation (high 16 bits) and the arrivals: the arrival's atomic
// returns the generation to wait on, and the last CTA to arrive starts the
// next generation with zero arrivals.  The CTA's earlier writes are released
// by the arrival and the others' acquired by the poll, so no separate fence
// stands on the path.  Every wait gives up after kWaitNs and sets ST_WAIT;
// returns false when this CTA gave up or saw that another one did (the kernel
// must then return; a CTA that had already passed sees the flag at its next
// barrier, which can no longer complete).
__device__ __forceinline__ bool grid_sync(Ctl *C) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int good = 1;
        unsigned old;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(&C->bar_word) : "memory");
        if ((old & 0xffffu) == gridDim.x - 1) {
            asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(&C->bar_word), "r"(0x10000u - gridDim.x)
                         : "memory");
        } else {
            unsigned long long t0 = 0;
            for (unsigned spins = 1; ((ld_acquire(&C->bar_word) ^ old) & 0xffff0000u) == 0; ++spins) {
                if ((spins & 63u) == 0) {
                    if (t0 == 0) t0 = gtimer();
                    if (__ldcg(&C->status) & ST_WAIT) good = 0;
                    else if (gtimer() - t0 > kWaitNs) {
                        atomicOr(&C->status, ST_WAIT);
                        good = 0;
                    }
                    if (!good) break;
                }
            }
        }
        ok = good;
        cta_words()[0] = cta_words()[1] = 0;
    }
    __syncthreads();
    return ok;
}

// ---------------------------------------------------------- BFS visiting --
// Per-thread work counters (32-bit to spare registers; added to the 64-bit
// statistics at the end of the kernel, and every 256 loop iterations so that
// no thread's count can wrap).  Adding them once per warp after every
// iteration cost ≈ 10 us per iteration: 3,648 atomics on each of 9 words.
struct Counters {
    unsigned bfs_arcs = 0, bfs_verts = 0, pr_arcs = 0, push = 0, relabel = 0, ri_arcs = 0,
             ri_moves = 0, clamped = 0, resat = 0, visits = 0;
};

constexpr int kIlp = 4;    // arcs in flight per lane in PushRelabel and RemoveInvalidEdges
constexpr int kIlpB = 4;   // arcs in flight per lane in the BFS

struct ArcRoundBfs {
    int ra[kIlpB], w[kIlpB];
};

// Warp-aggregated append of the lanes' flagged values of N slots: one
// atomicAdd for the whole warp and all slots.  All 32 lanes call.
template <int N>
__device__ __forceinline__ void warp_append_n(const bool (&pred)[N], const int (&val)[N], int *cnt, int *buf) {
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    unsigned m[N];
    int tot = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        m[j] = __ballot_sync(kFull, pred[j]);
        tot += __popc(m[j]);
    }
    if (tot == 0) return;
    int base = 0;
    if (lane == 0) base = atomicAdd(cnt, tot);
    base = __shfl_sync(kFull, base, 0);
#pragma unroll
    for (int j = 0; j < N; ++j) {
        if (pred[j]) buf[base + __popc(m[j] & below)] = val[j];
        base += __popc(m[j]);
    }
}

constexpr int kWq = 320;   // staged frontier entries per warp (24 warps: 7680 ints)
constexpr int kFl = 4;     // staged entries per lane in flight when a stage is published

// The next BFS frontier as one warp writes it.  The entries are staged in the
// warp's kWq ints of shared memory and reach the global queue buf a whole stage
// at a time (one reservation on cnt); the bookkeeping of the staged vertices
// (their degrees for the frontier's arc total, their excess for the active
// lists) is done when the stage is published, for up to 32 kFl vertices at
// once, instead of inside the arc scan that discovered them: the scan's chain
// of dependent accesses ends at the height CAS.  front_flush must run before
// the level's grid barrier.
struct Front {
    int *cnt, *buf;
    long long *asum;
    int *stage;     // this warp's kWq shared ints
    int sn;         // staged entries (warp-uniform)
    long long ds;   // arc total not yet added (warp-uniform)
};

// Publish the staged entries and do their bookkeeping: each joins the global
// frontier, its degree counts towards the frontier's arc total, and a vertex
// with positive excess (in the first stage of a push-pull repair, a deficient
// vertex of the pull side) is active: worklist (degree <= kHubDeg) or hub
// list.  All 32 lanes call.
__device__ __forceinline__ void front_flush_entries(const DevGraph &G, Front &F, bool dual, Counters &K) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    // (the reservation is on its way while the vertices are looked up)
    int base = 0;
    if (lane == 0) base = atomicAdd(F.cnt, F.sn);
    long long ds = 0;
    for (int i0 = 0; i0 < F.sn; i0 += 32 * kFl) {
        int v[kFl], deg[kFl];
        long long ev[kFl];
        bool ok[kFl], small[kFl], hub[kFl];
#pragma unroll
        for (int j = 0; j < kFl; ++j) {
            const int i = i0 + 32 * j + lane;
            ok[j] = i < F.sn;
            v[j] = ok[j] ? F.stage[i] : 0;
        }
#pragma unroll
        for (int j = 0; j < kFl; ++j) {
            deg[j] = ok[j] ? __ldg(&G.row[v[j] + 1]) - __ldg(&G.row[v[j]]) : 0;
            ev[j] = ok[j] ? lcg(&G.e[v[j]]) : 0;
        }
        if (i0 == 0) base = __shfl_sync(kFull, base, 0);
#pragma unroll
        for (int j = 0; j < kFl; ++j)
            if (ok[j]) F.buf[base + i0 + 32 * j + lane] = v[j];
#pragma unroll
        for (int j = 0; j < kFl; ++j) {
            // a vertex of the pull side (forward search) is active when deficient
            const bool pull = ok[j] && dual && G.part[v[j]] == kPartS;
            const bool act = ok[j] && (pull ? ev[j] < 0 : ev[j] > 0);
            ds += deg[j];
            K.bfs_verts += ok[j];
            hub[j] = act && deg[j] > kHubDeg;
            small[j] = act && !hub[j];
        }
        warp_append_n(small, v, &G.ctl->wcnt, G.wl);
        warp_append_n(hub, v, &G.ctl->hcnt, G.hl);
    }
    F.ds += warp_sum(ds);
    __syncwarp();
    F.sn = 0;
}

// Publish what the warp has staged.  All 32 lanes call.
__device__ __forceinline__ void front_flush(const DevGraph &G, Front &F, bool dual, Counters &K) {
    if (F.sn) front_flush_entries(G, F, dual, K);
    if (F.ds && (threadIdx.x & 31) == 0) add_ll(F.asum, F.ds);
    F.ds = 0;
}

// Stage the lanes' flagged values of N slots (at most 32 N <= kWq entries).
// All 32 lanes call.
template <int N>
__device__ __forceinline__ void front_stage_n(const DevGraph &G, const bool (&pred)[N], const int (&val)[N],
                                              Front &F, bool dual, Counters &K) {
    const unsigned below = (1u << (threadIdx.x & 31)) - 1u;
    unsigned m[N];
    int tot = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        m[j] = __ballot_sync(kFull, pred[j]);
        tot += __popc(m[j]);
    }
    if (tot == 0) return;
    if (F.sn + tot > kWq) front_flush_entries(G, F, dual, K);
    int base = F.sn;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        if (pred[j]) F.stage[base + __popc(m[j] & below)] = val[j];
        base += __popc(m[j]);
    }
    F.sn = base;
}

// Backward BFS step over kIlpB arcs per lane (a[j] of frontier vertex u, head
// v; ok[j] marks a real arc): the arc v -> u is residual iff rr[a] > 0; an
// unvisited v (height n) gets height L + 1 (global relabel, Sec. 2.2).  Newly
// reached vertices with positive excess are active and join the worklist
// (degree <= kHubDeg) or the hub list.  Slots whose bit is set in fwd belong
// to the pull side of a push-pull repair and search forward instead: u -> v
// residual (r[a] > 0), and a deficient v is active.  Every load of a round is
// issued before any of them is used.  All 32 lanes call.
__device__ __forceinline__ void bfs_visit_n(const DevGraph &G, const int (&a)[kIlpB], const bool (&ok)[kIlpB],
                                            unsigned fwd, bool dual, int L, Front &F, Counters &K) {
    const int n = G.n;
    int v[kIlpB], rin[kIlpB], hv[kIlpB];
    bool disc[kIlpB];
#pragma unroll
    for (int j = 0; j < kIlpB; ++j) {
        v[j] = ok[j] ? __ldg(&G.head[a[j]]) : 0;
        rin[j] = ok[j] ? lcg(((fwd >> j) & 1u) ? &G.r[a[j]] : &G.rr[a[j]]) : 0;
        K.bfs_arcs += ok[j];
    }
#pragma unroll
    for (int j = 0; j < kIlpB; ++j) hv[j] = (rin[j] > 0 && v[j] != G.s) ? lheight(&G.h[v[j]]) : -1;
#pragma unroll
    for (int j = 0; j < kIlpB; ++j) disc[j] = hv[j] == n && atomicCAS(&G.h[v[j]], n, L + 1) == n;
    front_stage_n(G, disc, v, F, dual, K);
}

// Expand up to 32 frontier vertices (one per lane, degree deg starting at
// arc beg, fwd for the pull side of a push-pull repair) with the arcs
// balanced over the lanes: lane i handles arcs k0 + 32 j + i of the
// concatenated lists.
__device__ __forceinline__ void bfs_expand_warp(const DevGraph &G, int beg, int deg, bool fwd, bool dual, int L,
                                                Front &F, Counters &K) {
    const unsigned fwd_lanes = __ballot_sync(kFull, fwd);
    const int lane = threadIdx.x & 31;
    int incl = deg;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(kFull, incl, 31);
    const int excl = incl - deg;
    for (int k0 = 0; k0 < total; k0 += 32 * kIlpB) {
        int a[kIlpB];
        bool ok[kIlpB];
        unsigned fw = 0;
#pragma unroll
        for (int jj = 0; jj < kIlpB; ++jj) {
            const int k = k0 + 32 * jj + lane;
            int j = 0;  // owner lane: largest j with excl_j <= k
#pragma unroll
            for (int step = 16; step >= 1; step >>= 1) {
                const int cand = j + step;
                const int ex = __shfl_sync(kFull, excl, cand & 31);
                if (cand < 32 && ex <= k) j = cand;
            }
            const int ob = __shfl_sync(kFull, beg, j);
            const int oe = __shfl_sync(kFull, excl, j);
            ok[jj] = k < total;
            a[jj] = ob + (k - oe);
            fw |= ((fwd_lanes >> j) & 1u) << jj;
        }
        bfs_visit_n(G, a, ok, fw, dual, L, F, K);
    }
}

// Bottom-up step of the backward BFS (direction-optimising search): the
// unvisited vertices v of V groups of 32 consecutive ids look for a residual
// arc v -> w into the current frontier (h(w) == L); the first one found gives
// h(v) = L + 1.  A lane scans its own vertices, kArcs arcs of each at a time,
// until it has found one: in the levels that matter most vertices find a
// parent among their first arcs.  (The group's arcs balanced over the lanes
// read whole rows, 128 arcs a round, before any vertex could stop, and paid
// seven shuffles a slot for the owner of each arc.  Per level: RMAT-20 27 -> 15
// us, 2048^2 grid 84 -> 40 us, 1023 x 769 grid 28 -> 13 us.)  Vertices of
// degree > kBigDeg become kChunk-arc items of the chunk list instead.  In the first
// stage of a push-pull repair (dual) a vertex of the pull side looks for a
// residual arc w -> v from the frontier instead, and only frontier vertices of
// the vertex's own side count.  All 32 lanes call.
// The many-vertex shape (2 vertices, 2 arcs of each) is for levels with pieces
// for every warp and parents among the first arcs (1 x 4, 2 x 4, 1 x 8: 0-25 %
// slower on RMAT-20 and grids).  The long-row shape (1 vertex, 4 arcs) is for
// graphs too small to give every warp a 64-vertex piece, where the rounds of
// one lane are the level's time, and for rows that are mostly read whole
// (search_rules): per level, many-vertex / long-row, 16,384 x 2 assignment
// graph 21.0 / 14.6 us, 262,144 x 2 one 37.7 / 34.5 (its 9.4M random height
// reads take 38 at the rate measured for L2), RMAT-16 8.2 / 7.3, 1,000-vertex
// graph 6.7 / 5.4 (1 x 6, 1 x 8, 2 x 4: 2-60 % above 1 x 4).
constexpr int kBuV = 2, kBuArcs = 2;
constexpr int kBuVLong = 1, kBuArcsLong = 4;

// The heights of a lane's vertices, loaded one piece ahead.  During a
// bottom-up level only the owning lane writes an unvisited vertex's height, so
// the early read is exact.
template <int V>
struct BuPre {
    int hv[V];
};

template <int V>
__device__ __forceinline__ BuPre<V> bu_prefetch(const DevGraph &G, long long base) {
    BuPre<V> p;
#pragma unroll
    for (int q = 0; q < V; ++q) {
        const long long v = base + 32 * q + (threadIdx.x & 31);
        p.hv[q] = v < G.n ? lcg(&G.h[v]) : -1;
    }
    return p;
}

template <int V, int kArcs>
__device__ __forceinline__ void bfs_bottom_up_group(const DevGraph &G, int base, const BuPre<V> &pre, bool dual, int L,
                                                    Front &F, int *ccnt, Counters &K) {
    const int lane = threadIdx.x & 31;
    int v[V], beg[V], left[V];   // left: arcs not yet scanned (0: found, or nothing to do)
    bool un[V], pull[V], any = false;
#pragma unroll
    for (int q = 0; q < V; ++q) {
        v[q] = base + 32 * q + lane;
        un[q] = pre.hv[q] == G.n && v[q] != G.s;
        any |= un[q];
    }
    if (!__any_sync(kFull, any)) return;
#pragma unroll
    for (int q = 0; q < V; ++q) {
        beg[q] = un[q] ? __ldg(&G.row[v[q]]) : 0;
        left[q] = un[q] ? __ldg(&G.row[v[q] + 1]) : 0;
        pull[q] = dual && un[q] && G.part[v[q]] == kPartS;
    }
#pragma unroll
    for (int q = 0; q < V; ++q) {
        left[q] -= beg[q];
        if (left[q] > kBigDeg) {
            const int nc = (left[q] + kChunk - 1) / kChunk;
            const int pos = atomicAdd(ccnt, nc);
            for (int c = 0; c < nc; ++c) G.cb[pos + c] = make_int2(v[q], beg[q] + c * kChunk);
            left[q] = 0;
        }
    }
    bool disc[V];
#pragma unroll
    for (int q = 0; q < V; ++q) disc[q] = false;
    for (;;) {
        int ra[V][kArcs], w[V][kArcs];
        any = false;
#pragma unroll
        for (int q = 0; q < V; ++q) any |= left[q] > 0;
        if (!__any_sync(kFull, any)) break;
#pragma unroll
        for (int q = 0; q < V; ++q)
#pragma unroll
            for (int j = 0; j < kArcs; ++j) {
                const bool ok = j < left[q];
                const int a = beg[q] + j;
                // (residuals do not change during the search)
                ra[q][j] = ok ? __ldca(pull[q] ? &G.rr[a] : &G.r[a]) : 0;
                w[q][j] = ok ? __ldg(&G.head[a]) : 0;
                K.bfs_arcs += ok;
            }
        bool hit[V][kArcs];
#pragma unroll
        for (int q = 0; q < V; ++q)
#pragma unroll
            for (int j = 0; j < kArcs; ++j) {
                const int hw = ra[q][j] > 0 ? lheight(&G.h[w[q][j]]) : -1;
                hit[q][j] = hw == L;
                if (dual && hit[q][j]) hit[q][j] = (G.part[w[q][j]] == kPartS) == pull[q];
            }
#pragma unroll
        for (int q = 0; q < V; ++q) {
#pragma unroll
            for (int j = 0; j < kArcs; ++j) disc[q] |= hit[q][j];
            beg[q] += kArcs;
            left[q] = disc[q] ? 0 : left[q] - kArcs;
        }
    }
#pragma unroll
    for (int q = 0; q < V; ++q)
        if (disc[q]) G.h[v[q]] = L + 1;
    front_stage_n(G, disc, v, F, dual, K);
}

// Bottom-up scan of one kChunk-arc item of a high-degree unvisited vertex;
// several items of one vertex may find a parent, the height CAS elects one.
__device__ __forceinline__ void bfs_bottom_up_item(const DevGraph &G, int2 item, bool dual, int L, Front &F,
                                                   Counters &K) {
    const int lane = threadIdx.x & 31;
    const int v = item.x;
    const int side = dual ? G.part[v] : kPartT;
    bool disc = false;
    if (bcast_ld(&G.h[v]) == G.n) {
        const int a1 = min(item.y + kChunk, __ldg(&G.row[v + 1]));
        bool hit = false;
        for (int a0 = item.y; a0 < a1 && !hit; a0 += 32 * kIlpB) {
            if (a0 != item.y && bcast_ld(&G.h[v]) != G.n) break;
            ArcRoundBfs R;
#pragma unroll
            for (int j = 0; j < kIlpB; ++j) {
                const int a = a0 + 32 * j + lane;
                R.ra[j] = a < a1 ? lcg(side == kPartS ? &G.rr[a] : &G.r[a]) : 0;
                R.w[j] = a < a1 ? __ldg(&G.head[a]) : 0;
                K.bfs_arcs += a < a1;
            }
            bool mine = false;
#pragma unroll
            for (int j = 0; j < kIlpB; ++j)
                mine |= R.ra[j] > 0 && lheight(&G.h[R.w[j]]) == L && (!dual || G.part[R.w[j]] == side);
            hit = __any_sync(kFull, mine);
        }
        if (hit && lane == 0) disc = atomicCAS(&G.h[v], G.n, L + 1) == G.n;
    }
    disc = __shfl_sync(kFull, disc, 0);
    const bool one[1] = {disc && lane == 0};
    const int val[1] = {v};
    front_stage_n(G, one, val, F, dual, K);
}

// ------------------------------------------------------ push / relabel --
// One push of d units along arc a (u -> v) with reverse arc b: both residual
// copies of the arc pair (reductions: nothing waits on them) and the head's
// excess; the caller subtracts the total from e(u).  Returns e(v) before.
// A push into s or t (never active) is a reduction too: the pusher does not
// wait in the queue of same-address atomics that the many pushes into the
// sink form at its L2 slice.
__device__ __forceinline__ long long push_arc(const DevGraph &G, int a, int b, int v, int d) {
    atomicSub(&G.r[a], d);
    atomicSub(&G.rr[b], d);
    atomicAdd(&G.r[b], d);
    atomicAdd(&G.rr[a], d);
    if (v == G.t || v == G.s) {
        add_ll(&G.e[v], d);
        return 1;
    }
    return (long long)atomicAdd(reinterpret_cast<unsigned long long *>(&G.e[v]), (unsigned long long)d);
}

// One pull of d units into u along arc a (u -> v) of u's list, reverse arc
// b: the arc v -> u loses d of residual and v loses d of excess
// (PullRelabel, Alg. 6); the caller adds the total to e(u).  Returns e(v)
// before the pull.
__device__ __forceinline__ long long pull_arc(const DevGraph &G, int a, int b, int v, int d) {
    atomicSub(&G.r[b], d);
    atomicSub(&G.rr[a], d);
    atomicAdd(&G.r[a], d);
    atomicAdd(&G.rr[b], d);
    if (v == G.t || v == G.s) {
        add_ll(&G.e[v], -(long long)d);
        return -1;
    }
    return (long long)atomicAdd(reinterpret_cast<unsigned long long *>(&G.e[v]), (unsigned long long)(-(long long)d));
}

// debug_checks: record a failed check (the first one's kind and index) and
// make the state invalid until the next mf_solve; the caller skips the
// access.  Kinds: 1 list entry out of range, 2 excess != net inflow, 3
// residual pair or mirror inconsistent.
__device__ __forceinline__ void check_fail(Ctl *C, int kind, long long where) {
    if ((atomicOr(&C->status, ST_CHECK) & ST_CHECK) == 0)
        C->chk_where = ((long long)kind << 40) | (where & 0xffffffffffll);
}

// Where the vertices that a push makes active go.
//
// Worklist vertices (degree <= kHubDeg), in the data-driven and push-pull
// modes: the activation queue, with generation gen.  The sign of the excess
// says who holds a vertex: the one atomic that takes e(v) from <= 0 to > 0
// (its returned old value tells) makes v active and hands it to the thread
// that issued it, which queues v or goes on with it; every later push finds
// e(v) > 0 and files nothing; and the warp that serves v lowers e(v) once, as
// the last thing it does with v, after a fence.  So a vertex is queued or
// served at most once at a time, with no mark to take and give back (the mark
// cost two returning atomics and two fences per activation).  A pull mirrors
// the signs.  In the topology-driven mode they are only counted: every round
// finds the active vertices by itself.
//
// Hubs (degree > kHubDeg): the next pass's hub list, once, by its stamp.
struct ActList {
    int *hcnt, *hlist;          // the next pass's hub list, its size and its stamp
    unsigned hstamp;
    unsigned long long *aq;     // activation queue, or nullptr: count only
    int qc, gen;                // its capacity; generation of what is filed (a phase has time for
                                // some millions at most: they fit the slot's upper half)
    const volatile unsigned long long *deadline;   // shared: when the phase ends (globaltimer)
    Ctl::Queue *Q;
    int count;                  // filed without a queue (warp-uniform)
    bool defer;                 // hub cycles: file nothing, a scan finds the active vertices
};

// Enqueue the lanes' flagged vertices of N slots into the activation queue
// with generation AL.gen (one reservation per warp); entries past the queue's
// capacity are dropped, counted as finished and flagged (the iteration then
// ends on another global relabel).  The caller has fenced what the entries'
// servers must see.  All 32 lanes call.
template <int N>
__device__ __forceinline__ void aq_push_n(const ActList &AL, const bool (&pred)[N], const int (&val)[N]) {
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    unsigned m[N];
    int tot = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        m[j] = __ballot_sync(kFull, pred[j]);
        tot += __popc(m[j]);
    }
    if (tot == 0) return;
    int base = 0;
    if (lane == 0) base = atomicAdd(&AL.Q->tail, tot);
    base = __shfl_sync(kFull, base, 0);
    int over = 0;
    const unsigned long long tag = (unsigned long long)(unsigned)AL.gen << 32;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        if (pred[j]) {
            const int pos = base + __popc(m[j] & below);
            if (pos < AL.qc) st_relaxed_u64(&AL.aq[pos], tag | (unsigned)(val[j] + 1));
            else ++over;
        }
        base += __popc(m[j]);
    }
    if (base > AL.qc) {   // warp-uniform: base is now past the warp's last entry
        over = (int)warp_sum((long long)over);
        if (lane == 0) {
            atomicAdd(&AL.Q->done, over);
            atomicExch(&AL.Q->over, 1);
        }
    }
    if (lane == 0) atomicMax(&AL.Q->maxgen, AL.gen);
}

// Single-thread enqueue of v (as aq_push_n; the caller has fenced).
__device__ __forceinline__ void aq_push_one(const ActList &AL, int v) {
    const int pos = atomicAdd(&AL.Q->tail, 1);
    if (pos < AL.qc) {
        st_relaxed_u64(&AL.aq[pos], ((unsigned long long)(unsigned)AL.gen << 32) | (unsigned)(v + 1));
    } else {
        atomicAdd(&AL.Q->done, 1);
        atomicExch(&AL.Q->over, 1);
    }
    atomicMax(&AL.Q->maxgen, AL.gen);
}

// File hubs that moves turned active.  All 32 lanes call.
template <int N>
__device__ __forceinline__ void file_hubs(const DevGraph &G, bool (&add_hub)[N], const int (&v)[N],
                                          const ActList &AL) {
    bool any = false;
#pragma unroll
    for (int j = 0; j < N; ++j) any |= add_hub[j];
    if (!__any_sync(kFull, any)) return;
#pragma unroll
    for (int j = 0; j < N; ++j)
        if (add_hub[j]) add_hub[j] = atomicExch(&G.astamp[v[j]], AL.hstamp) != AL.hstamp;
    warp_append_n(add_hub, v, AL.hcnt, AL.hlist);
}

// File the vertices that moves turned active (add: worklist vertices; add_hub:
// hubs; neither s nor t).  All 32 lanes call.
template <int N>
__device__ __forceinline__ void file_activations(const DevGraph &G, bool (&add)[N], bool (&add_hub)[N],
                                                 const int (&v)[N], ActList &AL) {
    file_hubs(G, add_hub, v, AL);
    bool any = false;
#pragma unroll
    for (int j = 0; j < N; ++j) any |= add[j];
    if (!__any_sync(kFull, any)) return;
    if (!AL.aq) {
#pragma unroll
        for (int j = 0; j < N; ++j) AL.count += __popc(__ballot_sync(kFull, add[j]));
        return;
    }
    __syncwarp();
    fence_acq_rel();
    aq_push_n(AL, add, v);
}

// The vertices a warp has relabelled, staged one per lane: they join the loop
// iteration's relabel list 32 at a time, each once (rstamp).  Only relabelled
// vertices can own arcs that RemoveInvalidEdges must saturate (the others
// keep their BFS height, which no residual arc can make steep).
struct Relabelled {
    int u = 0, cnt = 0;   // lane k's vertex; staged vertices (warp-uniform)
    unsigned stamp = 0;
};

__device__ __forceinline__ void relabelled_flush(const DevGraph &G, Relabelled &R) {
    const int lane = threadIdx.x & 31;
    bool add = lane < R.cnt;
    if (add) add = atomicExch(&G.rstamp[R.u], R.stamp) != R.stamp;
    warp_append(add, R.u, &G.ctl->rlcnt, G.rl);
    R.cnt = 0;
}

__device__ __forceinline__ void note_relabel(const DevGraph &G, int u, Relabelled &R) {
    if ((threadIdx.x & 31) == R.cnt) R.u = u;
    if (++R.cnt == 32) relabelled_flush(G, R);
}

// One round of a warp's arc scan: lane i holds arcs a0 + 32 j + i (j < kIlp)
// with their residual (0 past `end`), head and the head's height.  All loads of
// one kind are issued before any is used.
struct ArcRound {
    int ra[kIlp], v[kIlp], hv[kIlp];
};

// The residual is that of the arc u -> head (push) or head -> u (pull, the
// mirror rr).  With a partition array pt, an arc to a vertex of another part
// counts as absent (push-pull: each side works on its own vertices only).
template <bool PULL>
__device__ __forceinline__ void load_round_t(const DevGraph &G, int a0, int end, ArcRound &R,
                                             const unsigned char *pt, unsigned char side) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < kIlp; ++j) {
        const int a = a0 + 32 * j + lane;
        const bool ok = a < end;
        R.ra[j] = ok ? lcg(PULL ? &G.rr[a] : &G.r[a]) : 0;
        R.v[j] = ok ? __ldg(&G.head[a]) : 0;
    }
    if (pt) {
#pragma unroll
        for (int j = 0; j < kIlp; ++j)
            if (R.ra[j] > 0 && pt[R.v[j]] != side) R.ra[j] = 0;
    }
#pragma unroll
    for (int j = 0; j < kIlp; ++j) R.hv[j] = R.ra[j] > 0 ? lheight(&G.h[R.v[j]]) : 0;
}

__device__ __forceinline__ int round_arcs(int a0, int end) {
    const int lane = threadIdx.x & 31;
    int c = 0;
#pragma unroll
    for (int j = 0; j < kIlp; ++j) c += (a0 + 32 * j + lane) < end;
    return c;
}

// The amount moved along arc a (u -> v, reverse b) in one step: a push or a
// pull.
template <bool PULL>
__device__ __forceinline__ long long move_arc(const DevGraph &G, int a, int b, int v, int d) {
    return PULL ? pull_arc(G, a, b, v, d) : push_arc(G, a, b, v, d);
}

// ------------------------------------------------ staged arc ranges --
// A warp that scans the arcs of one vertex of degree 129 .. kStg copies them
// to its own shared memory first: residuals and heads as 16-byte cp.async
// copies (L2 only, so residuals written by other SMs' atomics are seen; no
// register holds an arc in flight), then the heights of the residual arcs'
// heads, gathered kGat per lane at a time.  A range of up to kStg arcs then
// takes three dependent round trips to memory instead of two per 128-arc
// round.  The staged range starts at the 16-byte boundary at or below the
// first arc: index i of a stage is arc (a0 & ~3) + i.
constexpr int kStg = 512;              // arcs one warp stages at a time
constexpr int kStgInts = kStg + 8;     // + the alignment slack of the first copy
constexpr int kStgWarp = 3 * kStgInts; // ints per warp: heads, residuals, heights
constexpr int kGat = 8;                // height gathers in flight per lane
static_assert(kHubDeg <= kStg, "a worklist vertex fits one stage");
constexpr int kDynSmem = (kBlock / 32) * kStgWarp * 4;   // bytes of dynamic shared memory of k_solve

__device__ __forceinline__ void cp_async16(int *dst, const int *src) {
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}

// Copy arcs [a0, a1) of the int array src (A entries) to dst[i], i = a -
// (a0 & ~3): 16 bytes per copy, except where the array is not 16-byte aligned
// or the copy would pass its end (plain L2 loads there).  Pair with
// stage_wait.  All 32 lanes call.
__device__ __forceinline__ void stage_copy(const int *src, int *dst, int a0, int a1, long long A, bool al16) {
    const int base = a0 & ~3;
    const int nch = (a1 - base + 3) >> 2;
    for (int c = threadIdx.x & 31; c < nch; c += 32) {
        const long long a = base + 4LL * c;
        if (al16 && a + 4 <= A) {
            cp_async16(dst + 4 * c, src + a);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (a + q < A) dst[4 * c + q] = __ldcg(src + a + q);
        }
    }
}

// Wait for this lane's copies, then make every lane's visible to the warp.
__device__ __forceinline__ void stage_wait() {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
}

// Heights of the heads of the staged residual arcs in [a0, a1): sh[i] = h of
// the head, or INT_MAX for no residual arc (out of range, zero residual, or,
// with a partition array pt, a head in another part: its residual is zeroed
// in sr).  Returns this lane's lowest height.
__device__ __forceinline__ unsigned stage_heights(const DevGraph &G, const int *sv, int *sr, int *sh,
                                                            int a0, int a1, const unsigned char *pt,
                                                            unsigned char side) {
    const int lane = threadIdx.x & 31;
    const int base = a0 & ~3, cnt = a1 - base;
    unsigned best = INT_MAX;
    for (int i0 = lane; i0 < cnt; i0 += 32 * kGat) {
        int hv[kGat];
        bool res[kGat];
        unsigned char pv[kGat];
#pragma unroll
        for (int j = 0; j < kGat; ++j) {
            const int i = i0 + 32 * j;
            res[j] = i < cnt && base + i >= a0 && sr[i] > 0;
            const int v = res[j] ? sv[i] : 0;
            hv[j] = res[j] ? lcg(&G.h[v]) : 0;
            pv[j] = (pt && res[j]) ? pt[v] : side;
        }
#pragma unroll
        for (int j = 0; j < kGat; ++j) {
            const int i = i0 + 32 * j;
            if (res[j] && pv[j] != side) {
                res[j] = false;
                sr[i] = 0;
            }
            if (i < cnt) sh[i] = res[j] ? hv[j] : INT_MAX;
            if (res[j]) best = min(best, (unsigned)hv[j]);
        }
    }
    __syncwarp();
    return best;
}

// The moves of N slots per lane (d[j] > 0: d[j] units along arc a[j] of u,
// reverse b[j], head v[j]) and the filing of the vertices they turn active: a
// push that raised e(v) above 0 (a pull that lowered it below 0) makes v active.
// The heads' degrees load beside the move atomics.  Returns this lane's total
// moved.  All 32 lanes call.
constexpr int kMv = 4;   // moves in flight per lane
template <bool PULL, int N>
__device__ __forceinline__ long long move_batch(const DevGraph &G, const int (&a)[N], const int (&b)[N],
                                                const int (&v)[N], const int (&d)[N], ActList &AL,
                                                Counters &K) {
    long long old[N], sent = 0;
    int deg[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        old[j] = 0;
        deg[j] = 0;
        if (d[j] > 0) {
            old[j] = move_arc<PULL>(G, a[j], b[j], v[j], d[j]);
            deg[j] = __ldg(&G.row[v[j] + 1]) - __ldg(&G.row[v[j]]);
            sent += d[j];
            ++K.push;
        }
    }
    bool add[N], add_hub[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const bool turned = PULL ? (old[j] >= 0 && old[j] - d[j] < 0) : (old[j] <= 0 && old[j] + d[j] > 0);
        const bool cand = d[j] > 0 && turned && v[j] != G.s && v[j] != G.t;
        add[j] = cand && deg[j] <= kHubDeg;
        add_hub[j] = cand && deg[j] > kHubDeg;
    }
    file_activations(G, add, add_hub, v, AL);
    return sent;
}

// The moves a decision to push at height hh makes along staged arcs [a0,
// a1): the amounts in arc order (min(rem, c_f) each, 32 arcs a step, over
// the arcs at height hh), written over the heights in sh, then all moves at
// once, kGat per lane in flight.  Returns the warp's total moved (all lanes).
template <bool PULL>
__device__ __forceinline__ long long stage_moves(const DevGraph &G, const int *sv, const int *sr, int *sh, int a0,
                                                 int a1, int hh, long long rem, ActList &AL, Counters &K) {
    const int lane = threadIdx.x & 31;
    const int base = a0 & ~3, cnt = a1 - base;
    int iend = 0;
    for (int i0 = 0; i0 < cnt && rem > 0; i0 += 32) {
        const int i = i0 + lane;
        const int ra = (i < cnt && sh[i] == hh) ? sr[i] : 0;
        const long long incl = warp_incl_scan(ra);
        const long long dj = rem - (incl - ra);
        if (i < cnt) sh[i] = dj < 0 ? 0 : (dj > ra ? ra : (int)dj);
        rem -= min(__shfl_sync(kFull, incl, 31), rem);
        iend = i0 + 32;
    }
    __syncwarp();
    long long sent = 0;
    const int lim = min(iend, cnt);
    // warp-uniform trip count: move_batch holds warp-wide ballots
    for (int i0 = 0; i0 < lim; i0 += 32 * kMv) {
        int a[kMv], b[kMv], v[kMv], d[kMv];
        bool any = false;
#pragma unroll
        for (int j = 0; j < kMv; ++j) {
            const int i = i0 + 32 * j + lane;
            d[j] = i < lim ? sh[i] : 0;
            a[j] = base + i;
            v[j] = d[j] > 0 ? sv[i] : 0;
            b[j] = d[j] > 0 ? __ldg(&G.rev[a[j]]) : 0;
            any |= d[j] > 0;
        }
        if (!__any_sync(kFull, any)) continue;
        sent += move_batch<PULL, kMv>(G, a, b, v, d, AL, K);
    }
    return warp_sum(sent);
}

// Minimum over the warp of a height (INT_MAX: none).
__device__ __forceinline__ int warp_min_height(unsigned h) { return (int)__reduce_min_sync(kFull, h); }

// Algorithm 2 on a vertex u of degree > 32 kIlp (<= kHubDeg) by one warp, up
// to kc steps, the arcs staged in the warp's shared memory (heads once,
// residuals and heights before every push).  A step scans u's arcs for the
// lowest residual neighbour height h^; if h(u) > h^ it performs the pushes
// that consecutive Alg. 2 steps would make to the arcs at height h^ -- in arc
// order, min(e, c_f) each, until e(u) is used up -- else it relabels u to
// h^ + 1 (the next step pushes along the arcs just scanned).  A vertex
// without residual arcs gets height n.  Only u's warp lowers r(u, .) and e(u)
// and changes h(u) during the phase; other warps only raise r(u, .) and e(u),
// so every amount pushed is available.  e(u) is lowered once, at the end
// (ActList).  With PULL the same steps are Algorithm 6 (PullRelabel) on a
// deficient u: residual arcs into u, pulls of min(-e, c_f) from the lowest of
// them.  Returns whether u is still active (all lanes).
template <bool PULL>
__device__ __forceinline__ bool visit_staged_t(const DevGraph &G, int u, int beg, int end, int kc, ActList &AL,
                                               const unsigned char *pt, unsigned char side, int *stg, Relabelled &RL,
                                               Counters &K) {
    const int lane = threadIdx.x & 31;
    int *sv = stg, *sr = stg + kStgInts, *sh = stg + 2 * kStgInts;
    stage_copy(G.head, sv, beg, end, G.A, G.al16);
    const int hu = bcast_ld(&G.h[u]);
    int h = hu;
    const long long e0 = bcast_ld(&G.e[u]);
    const long long want = PULL ? -e0 : e0;
    long long sent = 0;
    for (int c = 0; c < kc && h < G.n && sent < want; ++c) {
        stage_copy(PULL ? G.rr : G.r, sr, beg, end, G.A, G.al16);
        stage_wait();
        K.pr_arcs += (end - beg + 31 - lane) / 32;
        const int hh = warp_min_height(stage_heights(G, sv, sr, sh, beg, end, pt, side));
        if (h <= hh) {
            h = hh == INT_MAX ? G.n : hh + 1;
            if (lane == 0) {
                G.h[u] = h;
                ++K.relabel;
            }
            if (hh == INT_MAX || ++c >= kc || h >= G.n) break;
        }
        sent += stage_moves<PULL>(G, sv, sr, sh, beg, end, hh, want - sent, AL, K);
        __syncwarp();
    }
    if (h != hu) note_relabel(G, u, RL);
    bool active = sent < want;
    if (sent) {
        __syncwarp();
        fence_acq_rel();   // the moves and h(u), before another warp may take u
        if (lane == 0) {
            const unsigned long long d = PULL ? (unsigned long long)sent : (unsigned long long)(-sent);
            const long long now = (long long)(atomicAdd(reinterpret_cast<unsigned long long *>(&G.e[u]), d) + d);
            active = PULL ? now < 0 : now > 0;
        }
        active = __shfl_sync(kFull, active, 0);
    }
    __syncwarp();
    return active && h < G.n;
}

// Serve the active vertex u of generation AL.gen - 1 by one warp (its arcs in
// registers, <= 32 kIlp; larger vertices: visit_staged_t): steps of Algorithm 2
// (as visit_staged_t), each on the residuals and heights as they are then, until
// one has moved something, kc at most.  So KERNELCYCLES bounds the relabels of a
// visit here, and the pushes that further steps would make are left to u's next
// visit.  Heights only rise and residuals out of u only grow meanwhile, so the
// moves stay within the residuals, and an arc that a stale height made steep is
// RemoveInvalidEdges' to saturate, as with Alg. 2's own unlocked reads.  All moves
// are issued together at the end.
//
// Then the warp goes on with one of the vertices its moves turned active,
// whose arc range has come back beside the move atomics, and only the others
// go to the queue: a lone excess travels along its path at four dependent
// round trips per vertex (arcs; heads' heights; move atomics; fence), without
// the queue's three (reservation, slot, poll) and the row lookup.  What the
// excess of u became is looked at after the next vertex's first loads are
// issued.  In the topology-driven mode (AL.aq null) activations are counted
// and nothing is followed.  Past the deadline (globaltimer) no generation
// from kMinGen on is served: what is still active stays so, and the phase is
// flagged.
template <bool PULL>
__device__ __forceinline__ void visit_chain_t(const DevGraph &G, int u, int kc, ActList &AL, const unsigned char *pt,
                                              unsigned char side, int *stg, Relabelled &RL, Counters &K) {
    const int lane = threadIdx.x & 31;
    int beg = __ldg(&G.row[u]), end = __ldg(&G.row[u + 1]);
    const int gen0 = AL.gen;
    int pu = -1;            // the vertex served before, if it may still be active:
    long long pleft = 0;    // its excess after the visit (lane 0)
    // u goes back to the queue.  A visit that only relabelled has passed no
    // fence yet, and the next server must read this h(u) and write its own
    // after it.
    auto requeue = [&]() {
        if (!AL.aq) {
            ++AL.count;
        } else if (lane == 0) {
            fence_acq_rel();
            aq_push_one(AL, u);
        }
    };
    for (;;) {
        if (lane == 0) ++K.visits;
        const int deg = end - beg;
        if (deg > 32 * kIlp) {
            if (pu >= 0 && lane == 0 && (PULL ? pleft < 0 : pleft > 0)) {
                --AL.gen;
                aq_push_one(AL, pu);
                ++AL.gen;
            }
            pu = -1;
            __syncwarp();
            if (visit_staged_t<PULL>(G, u, beg, end, kc, AL, pt, side, stg, RL, K)) requeue();
            break;
        }
        int ra[kIlp], v[kIlp], hv[kIlp], rb[kIlp], d[kIlp];
        long long eu = lane == 0 ? lcg(&G.e[u]) : 0;
        int hu = lane == 0 ? lcg(&G.h[u]) : 0;
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            const int a = beg + 32 * j + lane;
            ra[j] = a < end ? lcg(PULL ? &G.rr[a] : &G.r[a]) : 0;
            v[j] = a < end ? __ldg(&G.head[a]) : 0;
            d[j] = 0;
            K.pr_arcs += a < end;
        }
        if (pu >= 0 && lane == 0 && (PULL ? pleft < 0 : pleft > 0)) {
            --AL.gen;
            aq_push_one(AL, pu);
            ++AL.gen;
        }
        pu = -1;
        eu = __shfl_sync(kFull, eu, 0);
        hu = __shfl_sync(kFull, hu, 0);
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            const int a = beg + 32 * j + lane;
            // (INT_MAX: not an arc to move along.  Arcs that a neighbour's push
            // may make residual during the visit are kept where they cost no
            // further round of loads)
            const bool in = ra[j] > 0 || (deg <= 32 && a < end);
            hv[j] = in ? lcg(&G.h[v[j]]) : INT_MAX;
            rb[j] = in ? __ldg(&G.rev[a]) : 0;
            if (pt && in && pt[v[j]] != side) hv[j] = INT_MAX;   // another part's arc counts as absent
        }
        const long long want = PULL ? -eu : eu;
        long long rem = want;
        int h = hu;
        for (int c = 0; c < kc && rem > 0 && h < G.n; ++c) {
            if (c > 0) {
                // the heads' heights again, and the residuals beside them: two
                // neighbours that both act on heights read before the other's
                // relabel push the same excess back and forth (one read per
                // visit: 30 -> 500-4,000 invalid arcs and 2-20x the iterations
                // on grids)
#pragma unroll
                for (int j = 0; j < kIlp; ++j) {
                    if (hv[j] == INT_MAX) continue;
                    const int a = beg + 32 * j + lane;
                    ra[j] = lcg(PULL ? &G.rr[a] : &G.r[a]);
                    hv[j] = lcg(&G.h[v[j]]);
                }
            }
            unsigned lo = INT_MAX;
#pragma unroll
            for (int j = 0; j < kIlp; ++j)
                if (ra[j] > d[j]) lo = min(lo, (unsigned)hv[j]);
            const int hh = warp_min_height(lo);
            if (h <= hh) {
                h = hh == INT_MAX ? G.n : hh + 1;
                if (lane == 0) ++K.relabel;
                continue;
            }
            // the moves at height hh, in arc order (slot j, then lane), until
            // the excess is used up; sums saturate at 2^31 - 1, the most that
            // one step moves
            const unsigned most = rem > INT_MAX ? INT_MAX : (unsigned)rem;
            unsigned left = most;
#pragma unroll
            for (int j = 0; j < kIlp; ++j) {
                const unsigned x = (ra[j] > d[j] && hv[j] == hh) ? (unsigned)(ra[j] - d[j]) : 0u;
                if (32 * j >= deg || !__any_sync(kFull, x > 0)) continue;   // warp-uniform
                unsigned incl = x;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned y = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl = min(incl + y, (unsigned)INT_MAX);
                }
                unsigned excl = __shfl_up_sync(kFull, incl, 1);
                if (lane == 0) excl = 0;
                d[j] += excl >= left ? 0 : (int)min(x, left - excl);
                left -= min(__shfl_sync(kFull, incl, 31), left);
            }
            rem -= most - left;
            // a step that moves is the visit's last: moves decided at one height
            // and issued after more steps found the heads relabelled, and the
            // steep arcs and deficits that this left cost further iterations
            // (unit assignment graph 15,386 + 3,000: 3-70 iterations a repair,
            // 23 ms, now 1, 0.29 ms; 10,187 + 2,673 recompute 3.8 -> 0.33 ms;
            // 2048^2 grid push-pull +5 %, the rest even)
            if (left < most) break;
        }
        if (h != hu) {
            if (lane == 0) G.h[u] = h;
            note_relabel(G, u, RL);
        }
        if (rem == want) {   // nothing moved: u keeps its excess
            if (h < G.n && rem > 0) requeue();
            break;
        }
        long long old[kIlp];
        int vb[kIlp], ve[kIlp];
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            old[j] = 0;
            vb[j] = ve[j] = 0;
            if (d[j] > 0) {
                old[j] = move_arc<PULL>(G, beg + 32 * j + lane, rb[j], v[j], d[j]);
                vb[j] = __ldg(&G.row[v[j]]);
                ve[j] = __ldg(&G.row[v[j] + 1]);
                ++K.push;
            }
        }
        bool add[kIlp], add_hub[kIlp];
        int nu = -1, nb = 0, ne = 0;
        unsigned tot = 0;
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            const bool turned = PULL ? (old[j] >= 0 && old[j] - d[j] < 0) : (old[j] <= 0 && old[j] + d[j] > 0);
            const bool cand = d[j] > 0 && turned && v[j] != G.s && v[j] != G.t;
            add[j] = cand && ve[j] - vb[j] <= kHubDeg;
            add_hub[j] = cand && !add[j];
            tot |= __ballot_sync(kFull, add[j]);
        }
        file_hubs(G, add_hub, v, AL);
        __syncwarp();
        fence_acq_rel();   // the moves and h(u), before another warp may take u or a head
        if (lane == 0) {
            const long long sent = want - rem;
            const unsigned long long x = PULL ? (unsigned long long)sent : (unsigned long long)(-sent);
            pleft = (long long)(atomicAdd(reinterpret_cast<unsigned long long *>(&G.e[u]), x) + x);
        }
        const bool maybe = h < G.n;   // u may still be active
        if (!AL.aq) {
#pragma unroll
            for (int j = 0; j < kIlp; ++j) AL.count += __popc(__ballot_sync(kFull, add[j]));
            AL.count += __shfl_sync(kFull, maybe && (PULL ? pleft < 0 : pleft > 0), 0);
            break;
        }
        if (AL.gen >= kMinGen && __any_sync(kFull, gtimer() > *AL.deadline)) {
            const bool self = __shfl_sync(kFull, maybe && (PULL ? pleft < 0 : pleft > 0), 0);
            if ((tot || self) && lane == 0) atomicExch(&AL.Q->over, 1);
            break;
        }
        // the first of the activated heads is served next by this warp
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            const unsigned m = __ballot_sync(kFull, add[j]);
            if (nu < 0 && m) {
                const int src = __ffs(m) - 1;
                nu = __shfl_sync(kFull, v[j], src);
                nb = __shfl_sync(kFull, vb[j], src);
                ne = __shfl_sync(kFull, ve[j], src);
                if (lane == src) add[j] = false;
            }
        }
        if (nu >= 0) {
            aq_push_n(AL, add, v);
            if (maybe) pu = u;
        } else {
            // no head: u itself, if it is still active
            if (!__shfl_sync(kFull, maybe && (PULL ? pleft < 0 : pleft > 0), 0)) break;
            nu = u;
            nb = beg;
            ne = end;
        }
        u = nu;
        beg = nb;
        end = ne;
        ++AL.gen;
    }
    __syncwarp();
    if (AL.aq && lane == 0 && AL.gen > gen0) atomicMax(&AL.Q->maxgen, AL.gen - 1);
}

__device__ __forceinline__ void visit_chain(const DevGraph &G, int u, int kc, ActList &AL, int *stg, Relabelled &RL,
                                            Counters &K) {
    visit_chain_t<false>(G, u, kc, AL, nullptr, 0, stg, RL, K);
}

// Algorithm 3 over the arcs [a0, a1) of vertex u (height hu) by one warp:
// every residual arc u -> v with h(u) > h(v) + 1 is saturated, moving its
// residual as excess to v.  With PULL it is the h- form (Algorithm 7): every
// residual arc v -> u with h(u) > h(v) + 1 is saturated, moving the residual
// into u.  With a partition array pt only arcs within u's part count.
// Returns this lane's share of the excess moved out of u (PULL: into u).
template <bool PULL>
__device__ __forceinline__ long long remove_invalid_range_t(const DevGraph &G, int hu, int a0, int a1,
                                                            const unsigned char *pt, unsigned char side,
                                                            Counters &K) {
    const int lane = threadIdx.x & 31;
    long long moved = 0;
    for (int b0 = a0; b0 < a1; b0 += 32 * kIlp) {
        ArcRound R;
        load_round_t<PULL>(G, b0, a1, R, pt, side);
        K.ri_arcs += round_arcs(b0, a1);
#pragma unroll
        for (int j = 0; j < kIlp; ++j) {
            if (R.ra[j] > 0 && hu > R.hv[j] + 1) {
                const int a = b0 + 32 * j + lane;
                move_arc<PULL>(G, a, __ldg(&G.rev[a]), R.v[j], R.ra[j]);
                moved += R.ra[j];
                ++K.ri_moves;
            }
        }
    }
    return moved;
}

template <bool PULL>
__device__ __forceinline__ void remove_invalid_warp_t(const DevGraph &G, int u, int *moved_flag,
                                                      const unsigned char *pt, unsigned char side, Counters &K) {
    const int lane = threadIdx.x & 31;
    const int beg = __ldg(&G.row[u]), end = __ldg(&G.row[u + 1]);
    const int hu = __shfl_sync(kFull, lane == 0 ? lcg(&G.h[u]) : 0, 0);
    const long long moved = warp_sum(remove_invalid_range_t<PULL>(G, hu, beg, end, pt, side, K));
    if (lane == 0 && moved) {
        add_ll(&G.e[u], PULL ? moved : -moved);
        *moved_flag = 1;   // once per warp
    }
}

// ------------------------------------------------- cooperative hubs --
// Hubs run PushRelabel over the whole grid in kPrChunk-arc items, in cycles
// of three phases (hub_list, hub_lowest, hub_push) between grid barriers.  An item's
// heads and residuals are copied to the warp's shared memory by cp.async one
// item ahead, and what the item needs of its hub is loaded two and one items
// ahead, so that an item waits only for the heights of its heads (kHubArcs
// per lane in flight) and for its share of the hub's excess.  What is decided
// per hub is decided one hub per lane over the grid: with the last item's warp
// deciding (arrival counters), a few warps took several decisions of five round
// trips each while the rest of the grid waited (38 % of the warps' time busy).
// Bound by the random reads of the heights (~140-240 G/s from L2 measured on
// hub-heavy index sets; 9.5M arcs a scan).  RMAT-20 100k, per phase: scan 15.6
// -> 9.9 us, pushes 31.9 -> 22.7 us; the static solve's scan 23.6 -> 13.1,
// pushes 38.8 -> 27.5 us.
constexpr int kHubArcs = kPrChunk / 32;    // arcs per lane of an item
constexpr int kHubBuf = kPrChunk + 8;      // ints per array of a staged item
static_assert(4 * kHubBuf <= kStgWarp, "two staged hub items per warp");

// x: index in the hub list, y, z: arcs, w: the hub, sign bit: on the pull side
// of a push-pull repair
using HubItem = int4;
__device__ __forceinline__ int hub_of(const HubItem &m) { return m.w & 0x7fffffff; }
__device__ __forceinline__ bool hub_pull(const HubItem &m) { return m.w < 0; }
__device__ __forceinline__ HubItem hub_item(const HubItem *items, int w, int nitems) {
    return w < nitems ? __ldcg(&items[w]) : make_int4(0, 0, 0, 0);
}

__device__ __forceinline__ void hub_issue(const DevGraph &G, const HubItem &m, int *buf) {
    stage_copy(G.head, buf, m.y, m.z, G.A, G.al16);
    stage_copy(hub_pull(m) ? G.rr : G.r, buf + kHubBuf, m.y, m.z, G.A, G.al16);
}

// Heights of the heads of the staged item's residual arcs, lane i holding arcs
// y + 32 j + i (INT_MAX: no residual arc, or, with a partition array, a head
// in another part); returns the lane's lowest.
__device__ __forceinline__ unsigned hub_heights(const DevGraph &G, const HubItem &m, const int *buf,
                                                const unsigned char *pt, int (&hv)[kHubArcs]) {
    const int at = (m.y & 3) + (threadIdx.x & 31), cnt = m.z - m.y - (threadIdx.x & 31);
    const unsigned char side = hub_pull(m) ? kPartS : kPartT;
    unsigned lo = INT_MAX;
#pragma unroll
    for (int j = 0; j < kHubArcs; ++j) {
        const bool res = 32 * j < cnt && buf[kHubBuf + at + 32 * j] > 0;
        const int v = res ? buf[at + 32 * j] : 0;
        hv[j] = res ? lheight(&G.h[v]) : INT_MAX;
        if (pt && res && pt[v] != side) hv[j] = INT_MAX;
    }
#pragma unroll
    for (int j = 0; j < kHubArcs; ++j) lo = min(lo, (unsigned)hv[j]);
    return lo;
}

// The item list of a cycle of parity par: the items of the hubs of the last
// cycle's list (of HL, in the first cycle; cnt hubs) that are active now, kHubsPerWarp hubs per
// warp, one per lane.  Sets what the cycle needs of each: hrem (the amount to
// move) and hkey (by cycle parity: the lowest residual-neighbour height, to
// be found; when the heights are those of the BFS just run (fresh), u's
// lowest residual neighbour sits one level below it, and no scan is needed).
// The hubs themselves are listed in hlist, by cycle parity.
constexpr int kHubsPerWarp = 8;
template <bool PP>
__device__ __forceinline__ void hub_list(const DevGraph &G, const int *HL, int par, int cnt, bool first, bool fresh,
                                         const unsigned char *pt, int gwarp, int nwarps, bool check) {
    const int lane = threadIdx.x & 31;
    HubItem *items = par ? G.hit1 : G.hit0;
    const int *from = par ? G.hlist0 : G.hlist1;
    int *to = par ? G.hlist1 : G.hlist0;
    for (int k0 = gwarp * kHubsPerWarp; k0 < cnt; k0 += nwarps * kHubsPerWarp) {
        const int k = k0 + lane;
        int i = 0, u = 0, beg = 0, end = 0, tag = 0, h = G.n;
        long long e = 0;
        if (lane < kHubsPerWarp && k < cnt) {
            i = first ? k : lcg(&from[k]);
            u = lcg(&HL[i]);
            if (check && (u < 0 || u >= G.n)) {
                check_fail(G.ctl, 1, u);
            } else {
                beg = __ldg(&G.row[u]);
                end = __ldg(&G.row[u + 1]);
                h = lcg(&G.h[u]);
                e = lcg(&G.e[u]);
                tag = u;
                if (PP && pt && pt[u] == kPartS) {
                    tag |= (int)0x80000000u;
                    e = -e;
                }
            }
        }
        const bool live = h < G.n && e > 0;
        const unsigned m = __ballot_sync(kFull, live);
        if (!m) continue;
        const int nit = live ? (end - beg + kPrChunk - 1) / kPrChunk : 0;
        const int incl = (int)warp_incl_scan(nit);
        int pos = 0, base = 0;
        if (lane == 0) base = atomicAdd(&G.ctl->hub_live[par], __popc(m));
        if (lane == 31) pos = atomicAdd(&G.ctl->hub_items[par], incl);
        base = __shfl_sync(kFull, base, 0);
        pos = __shfl_sync(kFull, pos, 31) + incl - nit;
        if (live) {
            to[base + __popc(m & ((1u << lane) - 1u))] = i;
            G.hrem[i] = e;
            G.hkey[2 * i + par] = fresh ? h - 1 : INT_MAX;
            G.hkey[2 * i + (par ^ 1)] = nit;   // items still to push (hub_push)
        }
        for (unsigned r = m; r; r &= r - 1u) {   // the items, all lanes a hub
            const int src = __ffs(r) - 1;
            const int n1 = __shfl_sync(kFull, nit, src), p1 = __shfl_sync(kFull, pos, src);
            const int i1 = __shfl_sync(kFull, i, src), t1 = __shfl_sync(kFull, tag, src);
            const int b1 = __shfl_sync(kFull, beg, src), e1 = __shfl_sync(kFull, end, src);
            for (int q = lane; q < n1; q += 32)
                items[p1 + q] = make_int4(i1, b1 + q * kPrChunk, min(b1 + (q + 1) * kPrChunk, e1), t1);
        }
    }
}

// The lowest residual neighbour of every listed hub (hkey) and item (hikey).
// No push or relabel runs meanwhile.
__device__ __forceinline__ void hub_lowest(const DevGraph &G, int nitems, int par, int gwarp, int nwarps, int *stg,
                                           const unsigned char *pt, Counters &K) {
    const int lane = threadIdx.x & 31;
    const HubItem *items = par ? G.hit1 : G.hit0;
    int *const tick = cta_words();
    int w = gwarp, w1 = next_item(tick, nitems);
    HubItem cur = hub_item(items, w, nitems), nxt = hub_item(items, w1, nitems);
    if (w < nitems) hub_issue(G, cur, stg);
    asm volatile("cp.async.commit_group;" ::: "memory");
    int b = 0;
    while (w < nitems) {
        if (w1 < nitems) hub_issue(G, nxt, stg + (b ^ 1) * 2 * kHubBuf);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const int w2 = next_item(tick, nitems);
        const HubItem nn = hub_item(items, w2, nitems);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        int hv[kHubArcs];
        unsigned lo = hub_heights(G, cur, stg + b * 2 * kHubBuf, pt, hv);
        K.pr_arcs += (cur.z - cur.y + 31 - lane) >> 5;
        lo = __reduce_min_sync(kFull, lo);
        if (lane == 0) {
            G.hikey[w] = (int)lo;
            if (lo < INT_MAX) atomicMin(&G.hkey[2 * cur.x + par], (int)lo);
        }
        __syncwarp();   // every lane is done with the item's buffer
        cur = nxt;
        nxt = nn;
        w = w1;
        w1 = w2;
        b ^= 1;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// The decisions of the listed hubs after hub_lowest: a hub that is not above
// its lowest residual neighbour is relabelled to one above it (to n without
// one); its pushes follow in the same cycle (a rescan in the next cycle cost a
// cycle per relabel).  Its items join the iteration's RemoveInvalidEdges list
// once.  One hub per lane.
__device__ __forceinline__ void hub_relabel(const DevGraph &G, const int *HL, int par, int cnt, unsigned rstamp,
                                            int gwarp, int nwarps, Counters &K) {
    const int lane = threadIdx.x & 31;
    const int *list = par ? G.hlist1 : G.hlist0;
    for (int k0 = gwarp * kHubsPerWarp; k0 < cnt; k0 += nwarps * kHubsPerWarp) {
        const int k = k0 + lane;
        int u = 0, beg = 0, nit = 0;
        if (lane < kHubsPerWarp && k < cnt) {
            const int i = lcg(&list[k]);
            u = lcg(&HL[i]);
            const int hh = lcg(&G.hkey[2 * i + par]), hu = lcg(&G.h[u]);
            if (hu <= hh) {
                G.h[u] = hh == INT_MAX ? G.n : hh + 1;
                ++K.relabel;
                if (atomicExch(&G.rstamp[u], rstamp) != rstamp) {
                    beg = __ldg(&G.row[u]);
                    nit = (__ldg(&G.row[u + 1]) - beg + kPrChunk - 1) / kPrChunk;
                }
            }
        }
        const unsigned m = __ballot_sync(kFull, nit > 0);
        if (!m) continue;
        const int incl = (int)warp_incl_scan(nit);
        int pos = 0;
        if (lane == 31) pos = atomicAdd(&G.ctl->rhcnt, incl);
        pos = __shfl_sync(kFull, pos, 31) + incl - nit;
        for (unsigned r = m; r; r &= r - 1u) {
            const int src = __ffs(r) - 1;
            const int n1 = __shfl_sync(kFull, nit, src), p1 = __shfl_sync(kFull, pos, src);
            const int u1 = __shfl_sync(kFull, u, src), b1 = __shfl_sync(kFull, beg, src);
            for (int q = lane; q < n1; q += 32) G.hri[p1 + q] = make_int2(u1, b1 + q * kPrChunk);
        }
    }
}

// Moves along the lowest arcs of the listed hubs, each warp reserving its
// share of the hub's excess with one atomic.  With AL.defer the vertices made
// active are not filed: the moves are reductions that nothing waits for, and
// a scan finds the active vertices afterwards (k_solve).  Otherwise the list is
// short and the warp that finishes a hub's last item looks whether the hub is
// still active (hub_act): mostly none is, and the next cycle's list phase need
// not run.  (The count-down is relaxed: an excess read too early reads too
// high, which only costs that phase.)
__device__ __forceinline__ void hub_push(const DevGraph &G, int nitems, int par, bool fresh, int gwarp, int nwarps,
                                         int *stg, const unsigned char *pt, ActList &AL, Counters &K) {
    const int lane = threadIdx.x & 31;
    const HubItem *items = par ? G.hit1 : G.hit0;
    // the height that item m (number w) pushes at, or -1: its hub has no
    // neighbour below n - 1 or nothing left to move, or no arc at its height here
    auto push_height = [&](const HubItem &m, int w) {
        if (w >= nitems) return -1;
        const int hh = lcg(&G.hkey[2 * m.x + par]);
        const int key = fresh ? hh : lcg(&G.hikey[w]);
        const long long rem = lcg(&G.hrem[m.x]);
        return __shfl_sync(kFull, hh < G.n - 1 && key == hh && rem > 0 ? hh : -1, 0);
    };
    int *const tick = cta_words();
    int w = gwarp, w1 = next_item(tick, nitems);
    HubItem cur = hub_item(items, w, nitems), nxt = hub_item(items, w1, nitems);
    int hh = push_height(cur, w);
    if (hh >= 0) hub_issue(G, cur, stg);
    asm volatile("cp.async.commit_group;" ::: "memory");
    int hn = push_height(nxt, w1);
    int b = 0;
    while (w < nitems) {
        if (hn >= 0) hub_issue(G, nxt, stg + (b ^ 1) * 2 * kHubBuf);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const int w2 = next_item(tick, nitems);
        const HubItem nn = hub_item(items, w2, nitems);
        if (hh >= 0) {
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncwarp();
            const int *buf = stg + b * 2 * kHubBuf;
            const int at = (cur.y & 3) + lane;
            int hv[kHubArcs], d[kHubArcs], rb[kHubArcs];
            hub_heights(G, cur, buf, pt, hv);
            if (fresh) K.pr_arcs += (cur.z - cur.y + 31 - lane) >> 5;   // (else counted by the scan)
            // d: the exclusive prefix of the item's residual at height hh, in
            // arc order; sums saturate at 2^31 - 1, the most an item moves
            unsigned tot = 0;
#pragma unroll
            for (int j = 0; j < kHubArcs; ++j) {
                const unsigned x = hv[j] == hh ? (unsigned)buf[kHubBuf + at + 32 * j] : 0u;
                rb[j] = x ? __ldg(&G.rev[cur.y + 32 * j + lane]) : 0;
                d[j] = (int)tot;
                if (!__any_sync(kFull, x > 0)) continue;   // warp-uniform
                unsigned incl = x;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned y = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl = min(incl + y, (unsigned)INT_MAX);
                }
                unsigned excl = __shfl_up_sync(kFull, incl, 1);
                if (lane == 0) excl = 0;
                d[j] = (int)min(tot + excl, (unsigned)INT_MAX);
                tot = min(tot + __shfl_sync(kFull, incl, 31), (unsigned)INT_MAX);
            }
            long long got = 0;
            if (tot) {
                if (lane == 0)
                    got = (long long)atomicAdd(reinterpret_cast<unsigned long long *>(&G.hrem[cur.x]),
                                               (unsigned long long)(-(long long)tot));
                got = __shfl_sync(kFull, got, 0);
            }
            if (got > 0) {   // warp-uniform
                const unsigned most = got > (long long)tot ? tot : (unsigned)got;
                const bool pull = hub_pull(cur);
                long long sent = 0;
#pragma unroll
                for (int half = 0; half < kHubArcs; half += 4) {
                    bool add[4], add_hub[4];
                    int v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int j = half + q;
                        add[q] = add_hub[q] = false;
                        v[q] = 0;
                        const unsigned x = hv[j] == hh ? (unsigned)buf[kHubBuf + at + 32 * j] : 0u;
                        const unsigned m = (unsigned)d[j] >= most ? 0u : min(x, most - (unsigned)d[j]);
                        if (m == 0) continue;
                        const int a = cur.y + 32 * j + lane;
                        v[q] = buf[at + 32 * j];
                        ++K.push;
                        sent += m;
                        // a push moves along a, a pull along its reverse
                        const int x0 = pull ? rb[j] : a, x1 = pull ? a : rb[j];
                        atomicSub(&G.r[x0], (int)m);
                        atomicSub(&G.rr[x1], (int)m);
                        atomicAdd(&G.r[x1], (int)m);
                        atomicAdd(&G.rr[x0], (int)m);
                        if (AL.defer || v[q] == G.t || v[q] == G.s) {
                            add_ll(&G.e[v[q]], pull ? -(long long)m : (long long)m);
                        } else {
                            const unsigned long long s = pull ? (unsigned long long)(-(long long)m) : m;
                            const long long old =
                                (long long)atomicAdd(reinterpret_cast<unsigned long long *>(&G.e[v[q]]), s);
                            const bool turned =
                                pull ? old >= 0 && old < (long long)m : old <= 0 && -old < (long long)m;
                            const int deg = __ldg(&G.row[v[q] + 1]) - __ldg(&G.row[v[q]]);
                            add[q] = turned && deg <= kHubDeg;
                            add_hub[q] = turned && deg > kHubDeg;
                        }
                    }
                    if (!AL.defer) file_activations(G, add, add_hub, v, AL);
                }
                sent = warp_sum(sent);
                if (lane == 0) add_ll(&G.e[hub_of(cur)], pull ? sent : -sent);
            }
            __syncwarp();   // every lane is done with the item's buffer
        }
        if (!AL.defer && lane == 0 && atomicSub(&G.hkey[2 * cur.x + (par ^ 1)], 1) == 1) {
            const int u = hub_of(cur);
            const long long eu = lcg(&G.e[u]);
            if (lcg(&G.h[u]) < G.n && (hub_pull(cur) ? eu < 0 : eu > 0)) atomicAdd(&G.ctl->hub_act[par], 1);
        }
        __syncwarp();
        cur = nxt;
        nxt = nn;
        hh = hn;
        hn = push_height(nxt, w2);
        w = w1;
        w1 = w2;
        b ^= 1;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// Add the warp's counters to the statistics st and clear them.  All 32 lanes
// call.
__device__ __forceinline__ void flush_counters(Counters &K, long long *st) {
    const unsigned vals[10] = {K.bfs_verts, K.bfs_arcs, K.pr_arcs, K.push, K.relabel, K.ri_arcs, K.ri_moves,
                               K.clamped, K.resat, K.visits};
    const int idx[10] = {S_BFS_VERTS, S_BFS_ARCS, S_PR_ARCS, S_PUSH, S_RELABEL, S_RI_ARCS, S_RI_MOVES, S_CLAMPED,
                         S_RESAT, S_WL};
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        const long long v = warp_sum((long long)vals[i]);
        if ((threadIdx.x & 31) == 0 && v) add_ll(&st[idx[i]], v);
    }
    K = Counters{};
}

// The same at the end of the kernel, summed over the CTA in shared memory
// first: one global atomic per statistic and CTA instead of one per warp.
// Every thread of the CTA calls.
__device__ __forceinline__ void flush_counters_cta(Counters &K, long long *st) {
    __shared__ unsigned long long s_sum[10];
    if (threadIdx.x < 10) s_sum[threadIdx.x] = 0;
    __syncthreads();
    const unsigned vals[10] = {K.bfs_verts, K.bfs_arcs, K.pr_arcs, K.push, K.relabel, K.ri_arcs, K.ri_moves,
                               K.clamped, K.resat, K.visits};
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        const long long v = warp_sum((long long)vals[i]);
        if ((threadIdx.x & 31) == 0 && v) atomicAdd(&s_sum[i], (unsigned long long)v);
    }
    __syncthreads();
    if (threadIdx.x < 10 && s_sum[threadIdx.x]) {
        int slot;
        switch (threadIdx.x) {
            case 0: slot = S_BFS_VERTS; break;
            case 1: slot = S_BFS_ARCS; break;
            case 2: slot = S_PR_ARCS; break;
            case 3: slot = S_PUSH; break;
            case 4: slot = S_RELABEL; break;
            case 5: slot = S_RI_ARCS; break;
            case 6: slot = S_RI_MOVES; break;
            case 7: slot = S_CLAMPED; break;
            case 8: slot = S_RESAT; break;
            default: slot = S_WL; break;
        }
        add_ll(&st[slot], (long long)s_sum[threadIdx.x]);
    }
    K = Counters{};
}

// ------------------------------------------- staged BFS work items --
// The grid-wide top-down item phase of a BFS level stages each kChunk-arc
// item's heads and residuals (the residual of the arc into the frontier
// vertex, or out of it on the pull side of a push-pull search) in the warp's
// shared memory by cp.async, one item ahead: the copies of the next item are
// in flight while the warp scans the current one from shared memory, so an
// arc round waits only for the heights of its heads.  Residuals do not change
// during a BFS level, so the early copy is exact.
constexpr int kItemBuf = kChunk + 8;       // ints per array of one staged item
constexpr int kItemWarp = 4 * kItemBuf;    // two items (heads, residuals) per warp
constexpr int kItemOff = 2 * kSoloCap;     // after the frontier stages
static_assert(kItemOff + (kBlock / 32) * kItemWarp <= kDynSmem / 4, "staged items exceed the shared memory");

struct ItemMeta {
    int x, y, a1;   // vertex, first arc, end of the item's arcs
    bool fwd;       // pull side of a push-pull search: forward residuals
};

__device__ __forceinline__ ItemMeta item_meta(const DevGraph &G, int c, bool dual) {
    const int2 it = lcg(&G.cb[c]);
    ItemMeta m;
    m.x = it.x;
    m.y = it.y;
    m.a1 = min(it.y + kChunk, __ldg(&G.row[it.x + 1]));
    m.fwd = dual && G.part[it.x] == kPartS;
    return m;
}

__device__ __forceinline__ void item_issue(const DevGraph &G, const ItemMeta &m, int *buf) {
    stage_copy(G.head, buf, m.y, m.a1, G.A, G.al16);
    stage_copy(m.fwd ? G.r : G.rr, buf + kItemBuf, m.y, m.a1, G.A, G.al16);
}

// bfs_visit_n over arcs whose heads and residuals are staged (index a - base).
__device__ __forceinline__ void bfs_visit_staged(const DevGraph &G, const int *sv, const int *sr, int base,
                                                 const int (&a)[kIlpB], const bool (&ok)[kIlpB], unsigned fwd,
                                                 bool dual, int L, Front &F, Counters &K) {
    const int n = G.n;
    int v[kIlpB], rin[kIlpB], hv[kIlpB];
    bool disc[kIlpB];
#pragma unroll
    for (int j = 0; j < kIlpB; ++j) {
        v[j] = ok[j] ? sv[a[j] - base] : 0;
        rin[j] = ok[j] ? sr[a[j] - base] : 0;
        K.bfs_arcs += ok[j];
    }
#pragma unroll
    for (int j = 0; j < kIlpB; ++j) hv[j] = (rin[j] > 0 && v[j] != G.s) ? lheight(&G.h[v[j]]) : -1;
#pragma unroll
    for (int j = 0; j < kIlpB; ++j) disc[j] = hv[j] == n && atomicCAS(&G.h[v[j]], n, L + 1) == n;
    front_stage_n(G, disc, v, F, dual, K);
}

// --------------------------------------- BFS levels of a small frontier --
// CTA 0 runs the levels of a small frontier alone, in step by __syncthreads
// only, while the rest of the grid waits at one barrier: until the frontier
// passes kSoloCap vertices or kSoloArcs arcs, the search would turn bottom-up,
// or the frontier empties; it then hands the frontier back in the global
// queue.  What bounds a level is its chain of round trips, so the frontier is
// kept in shared memory as the list of its arcs (sign bit: searched forward,
// on the pull side of a push-pull repair), written when a vertex is found: a
// level takes three trips (heads and residuals; heights; the claiming CAS and,
// with it, the rows of what it claims), two where few arcs make the height
// reads not worth their trip, and one __syncthreads.  A level of at most one
// arc per thread runs code for one (the four slots' instructions were a third
// of its time).  Which of the found vertices are active is looked up
// afterwards, for the whole run.  (Measured on grids, per level: frontier of
// vertices, rows and excesses looked up and global lists reserved in every
// level 4.6-5.7 us; rows after the claims, two barriers, four slots always
// 3.0-3.9 us; now 2.5-3.2 us.)
constexpr int kSoloWl = 12288;      // found vertices kept at most
constexpr int kSoloBig = 128;       // frontier vertices of degree > kBigDeg: at most kSoloArcs / (kBigDeg + 1)
constexpr int kSoloCas = 1024;      // arcs up to which every residual arc tries the CAS at once
static_assert(kSoloArcs / (kBigDeg + 1) <= kSoloBig, "big vertices of a small frontier");
static_assert(2 * kSoloArcs + 2 * kSoloCap + kSoloWl + 4 * kSoloBig <= kDynSmem / 4, "shared lists of a small frontier");

// A level's frontier, the next one's and the one before, rotating: with three
// a level needs one __syncthreads.
struct alignas(16) SoloFront {
    int nv, nbig;      // vertices, big ones
    int na;            // arcs of the others
    unsigned arcs;     // all arcs (fewer than 2^31)
};

__device__ __forceinline__ void bfs_solo(const DevGraph &G, int L, int cur, long long arcs_seen, bool dual, int *smem,
                                         long long *s_stat, unsigned long long &tprev, long long it, TraceRec *trace,
                                         Counters &K) {
    __shared__ SoloFront W[3];
    Ctl *C = G.ctl;
    const int n = G.n, tid = threadIdx.x, lane = tid & 31;
    int *const sv[2] = {smem, smem + kSoloCap};
    int *const sa[2] = {smem + 2 * kSoloCap, smem + 2 * kSoloCap + (int)kSoloArcs};
    int *const swl = smem + 2 * kSoloCap + 2 * (int)kSoloArcs;
    int2 *const sbig[2] = {reinterpret_cast<int2 *>(swl + kSoloWl), reinterpret_cast<int2 *>(swl + kSoloWl) + kSoloBig};

    int nw = 0;   // vertices found before the current level, and kept (CTA-uniform)

    // The lanes' flagged vertices of J slots, rows [beg, end), join frontier w,
    // lists q (positions from kSoloCap on go to spill); a sets the sign of
    // their arcs.  One reservation per warp and counter.  All 32 lanes call.
    auto add = [&](const auto &ok, const auto &v, const auto &beg, const auto &end, const auto &a, SoloFront *w, int q,
                   int *spill, bool found) {
        constexpr int J = sizeof(v) / sizeof(int);
        unsigned mine = 0;   // this lane's vertices (high half) and listed arcs (low half)
        unsigned all = 0;
#pragma unroll
        for (int j = 0; j < J; ++j)
            if (ok[j]) {
                const int deg = end[j] - beg[j];
                all += (unsigned)deg;
                mine += 0x10000u + (deg <= kBigDeg ? (unsigned)deg : 0u);
            }
        all = __reduce_add_sync(kFull, all);
        unsigned incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        int pv = 0, pa = 0;
        if (lane == 31) {
            pv = atomicAdd(&w->nv, (int)(incl >> 16));
            pa = atomicAdd(&w->na, (int)(incl & 0xffffu));
            atomicAdd(&w->arcs, all);
        }
        pv = __shfl_sync(kFull, pv, 31) + (int)((incl - mine) >> 16);
        pa = __shfl_sync(kFull, pa, 31) + (int)((incl - mine) & 0xffffu);
#pragma unroll
        for (int j = 0; j < J; ++j) {
            if (!ok[j]) continue;
            const int deg = end[j] - beg[j], sign = a[j] & (int)0x80000000u;
            (pv < kSoloCap ? sv[q] : spill)[pv] = v[j];
            if (found) swl[nw + pv] = v[j] | sign;
            ++pv;
            if (deg > kBigDeg) {
                const int k = atomicAdd(&w->nbig, 1);
                if (k < kSoloBig) sbig[q][k] = make_int2(beg[j] | sign, end[j]);
            } else {
                // (a frontier of more than kSoloArcs arcs is handed back: its
                // list need not be whole)
                if (pa + deg <= (int)kSoloArcs)
                    for (int i = 0; i < deg; ++i) sa[q][pa + i] = (beg[j] + i) | sign;
                pa += deg;
            }
        }
    };
    // J arcs per lane (ok[j]: arc a[j], sign set: searched forward)
    auto visit = [&](const auto &a, const auto &ok, bool cas, int Ls, SoloFront *w, int q, int *spill) {
        constexpr int J = sizeof(a) / sizeof(int);
        int v[J], rin[J], beg[J], end[J];
        bool disc[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int x = a[j] & 0x7fffffff;
            v[j] = ok[j] ? __ldg(&G.head[x]) : 0;
            rin[j] = ok[j] ? lcg(a[j] < 0 ? &G.r[x] : &G.rr[x]) : 0;
            K.bfs_arcs += ok[j];
        }
#pragma unroll
        for (int j = 0; j < J; ++j) disc[j] = rin[j] > 0 && v[j] != G.s;
        if (!cas) {
            int hv[J];
#pragma unroll
            for (int j = 0; j < J; ++j) hv[j] = disc[j] ? lcg(&G.h[v[j]]) : 0;
#pragma unroll
            for (int j = 0; j < J; ++j) disc[j] = disc[j] && hv[j] == n;
        }
        // (the rows of all that are tried, on the same trip as the claims)
        int old[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            old[j] = disc[j] ? atomicCAS(&G.h[v[j]], n, Ls + 1) : 0;
            beg[j] = disc[j] ? __ldg(&G.row[v[j]]) : 0;
            end[j] = disc[j] ? __ldg(&G.row[v[j] + 1]) : 0;
        }
        bool any = false;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            disc[j] = disc[j] && old[j] == n;
            any |= disc[j];
            K.bfs_verts += disc[j];
        }
        if (__any_sync(kFull, any)) add(disc, v, beg, end, a, w, q, spill, true);
    };
    // the level's listed arcs, J per thread at once
    auto scan = [&](auto jc, int na, int q, bool cas, int Ls, SoloFront *w, int *spill) {
        constexpr int J = decltype(jc)::value;
        for (int k0 = tid & ~31; k0 < na; k0 += J * kBlock) {
            int a[J];
            bool ok[J];
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int k = k0 + j * kBlock + lane;
                ok[j] = k < na;
                a[j] = ok[j] ? sa[q][k] : 0;
            }
            visit(a, ok, cas, Ls, w, q ^ 1, spill);
        }
    };
    // the active ones of the vertices found so far join the global lists (a
    // vertex of the pull side is active when deficient); every thread calls,
    // between barriers
    auto flush = [&]() {
        for (int i0 = 0; i0 < nw; i0 += kBlock) {
            const int i = i0 + tid;
            const int x = i < nw ? swl[i] : 0, v = x & 0x7fffffff;
            const long long ev = i < nw ? lcg(&G.e[v]) : 0;
            const int deg = i < nw ? __ldg(&G.row[v + 1]) - __ldg(&G.row[v]) : 0;
            const bool act = i < nw && (x < 0 ? ev < 0 : ev > 0);
            warp_append(act && deg <= kHubDeg, v, &C->wcnt, G.wl);
            warp_append(act && deg > kHubDeg, v, &C->hcnt, G.hl);
        }
        __syncthreads();
        nw = 0;
    };

    if (tid < 3) W[tid] = SoloFront{0, 0, 0, 0};
    __syncthreads();
    const int *F0 = (L & 1) ? G.qb1 : G.qb0;
    for (int i0 = 0; i0 < cur; i0 += kBlock) {
        const int i = i0 + tid;
        bool ok[kIlpB];
        int v[kIlpB], beg[kIlpB], end[kIlpB], a[kIlpB];
#pragma unroll
        for (int j = 0; j < kIlpB; ++j) {
            v[j] = j == 0 && i < cur ? lcg(&F0[i]) : 0;
            ok[j] = j == 0 && i < cur && v[j] >= 0 && v[j] < n;
            beg[j] = ok[j] ? __ldg(&G.row[v[j]]) : 0;
            end[j] = ok[j] ? __ldg(&G.row[v[j] + 1]) : 0;
            a[j] = ok[j] && dual && G.part[v[j]] == kPartS ? (int)0x80000000u : 0;
        }
        add(ok, v, beg, end, a, &W[0], 0, nullptr, false);   // (at most kSoloCap vertices)
    }
    __syncthreads();
    int Ls = L, b = 0, c = 0, cs = cur;   // b: the level's lists, c: its counts
    long long seen = arcs_seen, mfs = 0;
    SoloFront f = W[0];
    for (;;) {
        int *spill = (Ls & 1) ? G.qb0 : G.qb1;   // positions >= kSoloCap of the next frontier
        SoloFront *const w = &W[c == 2 ? 0 : c + 1];
        if (tid == 0) W[c == 0 ? 2 : c - 1] = SoloFront{0, 0, 0, 0};   // (read a barrier ago)
        if (f.na <= kBlock)
            scan(std::integral_constant<int, 1>{}, f.na, b, f.na <= kSoloCas, Ls, w, spill);
        else
            scan(std::integral_constant<int, kIlpB>{}, f.na, b, f.na <= kSoloCas, Ls, w, spill);
        for (int q = tid >> 5; q < f.nbig; q += kBlock / 32) {
            const int2 r = sbig[b][q];
            const int a0 = r.x & 0x7fffffff;
            for (int ab = a0; ab < r.y; ab += 32 * kIlpB) {
                int a[kIlpB];
                bool ok[kIlpB];
#pragma unroll
                for (int j = 0; j < kIlpB; ++j) {
                    const int x = ab + 32 * j + lane;
                    ok[j] = x < r.y;
                    a[j] = x | (r.x & (int)0x80000000u);
                }
                visit(a, ok, false, Ls, w, b ^ 1, spill);
            }
        }
        __syncthreads();
        if (tid == 0 && trace) {
            const unsigned long long now = gtimer();
            s_stat[S_T_BFS] += (long long)(now - tprev);
            const int k = C->trace_n++;
            if (k < G.trace_cap) trace[k] = TraceRec{(short)S_T_BFS, 4, (int)it, Ls, cs, (long long)(now - tprev)};
            tprev = now;
        }
        ++Ls;
        b ^= 1;
        c = c == 2 ? 0 : c + 1;
        f = *w;
        cs = f.nv;
        mfs = (long long)f.arcs;
        const bool out = cs == 0 || cs > kSoloCap || mfs > G.solo_arcs || (mfs * G.alpha > G.A - (seen + mfs) && cs * 64LL > n);
        nw += cs;
        if (out || nw > kSoloWl - (int)kSoloArcs) flush();
        if (out) break;
        seen += mfs;
    }
    // hand the frontier of level Ls back in the global queue
    int *Fg = (Ls & 1) ? G.qb1 : G.qb0;
    for (int i = tid; i < min(cs, kSoloCap); i += kBlock) Fg[i] = sv[b][i];
    if (tid == 0) {
        C->qcnt[Ls % 3] = cs;
        C->asum[Ls % 3] = mfs;
        C->qcnt[(Ls + 1) % 3] = 0;
        C->asum[(Ls + 1) % 3] = 0;
        C->ccnt[Ls % 3] = 0;
        C->solo_L = Ls;
        C->solo_seen = seen;   // arcs of the levels run, without level Ls
    }
}

// A vertex id read from a list or queue, checked when debug_checks is on.
__device__ __forceinline__ bool vertex_ok(const Job &J, Ctl *C, int u, int n) {
    if (!J.debug || (u >= 0 && u < n)) return true;
    check_fail(C, 1, u);
    return false;
}

// ------------------------------------------------------------ the kernel --
// Grid barrier inside k_solve; CTA 0's thread 0 charges the time since the
// previous barrier to a phase bucket of the statistics and, when tracing is
// on, appends a record (phase, loop iteration, step, mode, count, time).
#define ST (J.st)
#define TR (J.trace)
#define MF_SYNC_T(bucket, step, mode, aux)                                    \
    do {                                                                      \
        if (!grid_sync(C)) return;                                            \
        if (gtid == 0) {                                                      \
            const unsigned long long now_ = gtimer();                         \
            const long long dt_ = (long long)(now_ - tprev);                  \
            s_stat[bucket] += dt_;                                            \
            s_stat[S_BARRIERS] += 1;                                          \
            if (TR) {                                                         \
                const int k_ = C->trace_n++;                                  \
                if (k_ < G.trace_cap)                                         \
                    TR[k_] = TraceRec{(short)(bucket), (short)(mode),    \
                                           (int)it, (int)(step), (int)(aux), dt_}; \
            }                                                                 \
            tprev = now_;                                                     \
        }                                                                     \
    } while (0)
#define MF_SYNC(bucket) MF_SYNC_T(bucket, -1, 0, -1)
// PP: the instance that can run Dynamic Push-Pull (Alg. 8); the plain
// instance compiles without its code paths.
template <bool PP>
__global__ void __launch_bounds__(kBlock, 1) k_solve(DevGraph G, Job J) {
    Ctl *C = G.ctl;
    const int lane = threadIdx.x & 31;
    const long long gtid = (long long)blockIdx.x * kBlock + threadIdx.x;
    const long long gthreads = (long long)gridDim.x * kBlock;
    // consecutive numbers on different SMs: neighbouring work items (the hubs'
    // rows of a renumbered graph, the items of one hub) cost alike
    const int gwarp = (int)((threadIdx.x >> 5) * gridDim.x + blockIdx.x);
    const int nwarps = (int)(gthreads >> 5);
    const int n = G.n, s = G.s, t = G.t;
    Counters K;
    // dynamic shared memory (kDynSmem bytes), used by one kind of phase at a
    // time (grid barriers keep them apart): the BFS frontiers (CTA 0's small
    // ones, or the warps' staged entries) at its start, the warps' arc stages of
    // PushRelabel
    extern __shared__ __align__(16) int s_dyn[];
    int *const s_bfs = s_dyn;
    int *const stg = s_dyn + (threadIdx.x >> 5) * kStgWarp;
    __shared__ volatile unsigned long long s_deadline;           // end of the queue phase (globaltimer)
    __shared__ unsigned long long s_bfs_begin, s_bfs_end;   // the last BFS, as thread 0 saw it
    __shared__ int s_fin;   // the queue phase has ended (see the activation queue)
    if (threadIdx.x == 0) s_fin = 0;
    static_assert(2 * kSoloCap * 4 <= kDynSmem, "the shared frontiers exceed the dynamic shared memory");
    static_assert(kWq * (kBlock / 32) <= 2 * kSoloCap, "frontier stages exceed the shared frontier");
    static_assert(kWq >= 32 * kIlpB, "a stage holds one round of arcs");
    unsigned long long tprev = gtimer();
    long long it = -1;   // loop iteration (-1 before the loop, for trace records)

    // A sticky error (iteration cap, barrier wait) invalidates the state
    // until the next mf_solve, which clears it before launching.
    if (lctl(&C->status) & ST_STICKY) return;
    const unsigned stamp_base = lctl(&C->stamp_base) + 1u;
    // JOB_AUTO: the policy kernel launched just before chose repair or
    // recompute and KERNELCYCLES
    int kind = J.kind, kc = J.kc, jmode = J.mode;
    bool pp_pick = true;   // a fixed job of a push-pull graph repairs by push-pull
    if (kind == JOB_AUTO) {
        kind = lctl(&C->pol_kind);
        kc = lctl(&C->pol_kc);
        jmode = lctl(&C->pol_mode);
        pp_pick = jmode == MF_MODE_PUSH_PULL;
        if (pp_pick) jmode = MF_MODE_DATA_DRIVEN;   // the plain loop of push-pull's stage 2
    }
    if (kind == JOB_REFRESH && lctl(&C->heights_exact)) return;
    const bool batch_job = kind == JOB_REPAIR || kind == JOB_RECOMPUTE;
    const int kb = J.k_dev ? lctl(J.k_dev) : J.k;          // batch entries
    const unsigned seq = lctl(&C->bseq) + 1u;           // this batch's stamp
    // CTA 0's thread 0 keeps its counts and phase times in shared memory: a
    // read-modify-write of the global words after every barrier kept CTA 0's
    // first warp, and with it the whole grid, waiting for two L2 round trips
    __shared__ long long s_stat[S_COUNT_MAX];
    if (gtid == 0) {
        for (int i = 0; i < S_COUNT; ++i) ST[i] = s_stat[i] = 0;
        s_stat[S_BATCH] = batch_job ? kb : 0;
        C->t_start = gtimer();
        if (TR) C->trace_n = 0;
    }

    // Dynamic Push-Pull (Alg. 8) needs the exact cut of the previous state:
    // T = {h < n} can reach a sink, S = {h >= n} cannot
    const bool pp = PP && J.pp && pp_pick && kind == JOB_REPAIR && G.part && lctl(&C->cut_exact);
    if (pp)
        for (long long v0 = gtid; v0 < n; v0 += 4 * gthreads) {   // four heights in flight per thread
            int hv[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) hv[j] = v0 + j * gthreads < n ? lcg(&G.h[v0 + j * gthreads]) : 0;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (v0 + j * gthreads < n) G.part[v0 + j * gthreads] = hv[j] < n ? kPartT : kPartS;
        }

    // What a thread of the batch phases moves onto s and t: in a graph with
    // many terminal arcs every entry meets one of the two, and atomics of all
    // warps on two words serialise (131,000 entries at the terminals of a 2048^2
    // grid: clamping 50 us, now 7; saturation 35 us, now 5), so the CTA adds
    // them up first.
    __shared__ unsigned long long s_term[2];   // s, t
    if (threadIdx.x < 2) s_term[threadIdx.x] = 0;
    long long es = 0, et = 0;
    auto give = [&](int v, long long x) {
        if (v == s) es += x;
        else if (v == t) et += x;
        else add_ll(&G.e[v], x);
    };
    auto settle_terminals = [&]() {   // every thread calls, past a barrier since the last call
        if (!__syncthreads_or(es != 0 || et != 0)) return;
        es = warp_sum(es);
        et = warp_sum(et);
        if (lane == 0 && es) atomicAdd(&s_term[0], (unsigned long long)es);
        if (lane == 0 && et) atomicAdd(&s_term[1], (unsigned long long)et);
        __syncthreads();
        if (threadIdx.x < 2) {
            const long long x = (long long)s_term[threadIdx.x];
            if (x) add_ll(&G.e[threadIdx.x ? t : s], x);
            s_term[threadIdx.x] = 0;
        }
        es = et = 0;
    };

    // ---- batch: validate, then apply (Algorithm 5) ----------------------
    bool fast = false;   // pure-increment batch that cannot change the cut
    if (batch_job) {
        for (long long i = gtid; i < kb; i += gthreads) {
            const int eid = J.ids[i];
            bool bad = eid < 0 || eid >= G.m;
            int nc = 0;
            if (!bad) {
                long long v = J.caps[i];
                if (J.flags & MF_DELTA) {
                    v += lcg(&G.cap_edge[eid]);
                    if (v < 0) v = 0;
                }
                if (v < 0 || v > G.cap_limit) bad = true;
                else nc = (int)v;
                if (atomicExch(&G.stamp[eid], seq) == seq) bad = true;  // duplicate id
            }
            J.newc[i] = nc;
            if (bad) atomicOr(&C->batch_err, 1);
        }
        MF_SYNC(S_T_BATCH);
        if (lctl(&C->batch_err)) {
            grid_sync(C);
            if (gtid == 0) {
                for (int i = 0; i < S_COUNT; ++i) ST[i] = s_stat[i];
                atomicOr(&C->status, ST_EINVAL);
                C->batch_err = 0;
                C->bseq = seq;
            }
            return;
        }
        // c_f(u,v) += c'(u,v) - c(u,v)  (Alg. 5, lines 1-3)
        bool blocks = false;   // this thread saw a decrement or an increment across the cut
        for (long long i = gtid; i < kb; i += gthreads) {
            const int eid = J.ids[i];
            const int nc = lcg(&J.newc[i]);
            const int d = nc - lcg(&G.cap_edge[eid]);
            G.cap_edge[eid] = nc;
            J.dlt[i] = d;
            const int a = __ldg(&G.arc_of_edge[eid]);
            if (a >= 0 && d != 0) {
                atomicAdd(&G.cap[a], d);
                const int b = __ldg(&G.rev[a]);
                atomicAdd(&G.r[a], d);   // (a recompute needs the pairs' new sums)
                atomicAdd(&G.rr[b], d);
                if (kind == JOB_REPAIR) {
                    // an increment can raise the flow only on an arc from
                    // the side that cannot reach a sink to the side that can
                    if (d < 0 || (lcg(&G.h[__ldg(&G.head[b])]) >= n && lcg(&G.h[__ldg(&G.head[a])]) < n))
                        blocks = true;
                }
            }
        }
        // one store per CTA: thousands of same-address stores from every SM
        // serialise at one L2 slice
        if (__syncthreads_or(blocks) && threadIdx.x == 0) C->inc_block = 1;
        MF_SYNC(S_T_BATCH);
        // With the exact cut S = {h >= n} of the previous state (no residual
        // arc from S to T), increments on arcs that do not go from S to T
        // leave that cut saturated and its capacity unchanged, so the flow
        // value stays the same and the state stays terminal (Sec. 4: only
        // changes on the cut's arcs can change the maximum).
        fast = kind == JOB_REPAIR && lctl(&C->cut_exact) && !lctl(&C->inc_block);
        if (kind == JOB_REPAIR && !fast) {
            // flow above the new capacity goes back: the tail keeps it as
            // excess, the head becomes deficient (Alg. 5, lines 4-11; the
            // excess update is the exact incremental form of Alg. 4 line 2).
            for (long long i = gtid; i < kb; i += gthreads) {
                if (lcg(&J.dlt[i]) >= 0) continue;
                const int a = __ldg(&G.arc_of_edge[J.ids[i]]);
                if (a < 0) continue;
                const int old = atomicMax(&G.r[a], 0);
                if (old < 0) {
                    const int o = -old;
                    const int b = __ldg(&G.rev[a]);
                    atomicAdd(&G.rr[b], o);
                    atomicSub(&G.r[b], o);
                    atomicSub(&G.rr[a], o);
                    give(__ldg(&G.head[b]), o);
                    give(__ldg(&G.head[a]), -(long long)o);
                    ++K.clamped;
                }
            }
            settle_terminals();
            MF_SYNC(S_T_BATCH);
            if (pp) {
                // Alg. 8: saturate every residual arc from S to T.  Before the
                // batch the cut had none, so only raised batch arcs can have one.
                for (long long i = gtid; i < kb; i += gthreads) {
                    if (lcg(&J.dlt[i]) <= 0) continue;
                    const int a = __ldg(&G.arc_of_edge[J.ids[i]]);
                    if (a < 0) continue;
                    const int b = __ldg(&G.rev[a]);
                    const int u = __ldg(&G.head[b]), v = __ldg(&G.head[a]);
                    if (G.part[u] != kPartS || G.part[v] != kPartT) continue;
                    const int ra = atomicExch(&G.r[a], 0);
                    if (ra > 0) {
                        atomicSub(&G.rr[b], ra);
                        atomicAdd(&G.r[b], ra);
                        atomicAdd(&G.rr[a], ra);
                        give(u, -(long long)ra);
                        give(v, ra);
                    }
                }
                settle_terminals();
                MF_SYNC(S_T_BATCH);
            }
        }
    }
    const bool pp_ran = pp && !fast;
    int stage = pp_ran ? 1 : 0;   // 0 plain loop; push-pull: 1 push on T and pull on S, 2 push on P

    // ---- zero flow (Algorithm 1, first two loops) ------------------------
    if (kind == JOB_SOLVE || kind == JOB_RECOMPUTE) {
        // rr(a) = cap(rev a).  Read through rev that is a random gather over the
        // capacities (RMAT-20: 31M gathers, 2 GB of DRAM traffic, 200-225 us).  A
        // recompute of a state whose arc pairs are known to add up (pairs_ok)
        // takes it from the pair's sum instead, r(a) + rr(a) = cap(a) +
        // cap(rev a), which is all streaming (96 us).
        constexpr int kInit = 6;   // arcs in flight per thread
        if (kind == JOB_RECOMPUTE && lctl(&C->pairs_ok)) {
            for (long long a0 = gtid; a0 < G.A; a0 += kInit * gthreads) {
                int c0[kInit], r0[kInit], r1[kInit];
#pragma unroll
                for (int j = 0; j < kInit; ++j) {
                    const long long a = min(a0 + j * gthreads, G.A - 1);
                    c0[j] = lcg(&G.cap[a]);
                    r0[j] = lcg(&G.r[a]);
                    r1[j] = lcg(&G.rr[a]);
                }
#pragma unroll
                for (int j = 0; j < kInit; ++j) {
                    const long long a = a0 + j * gthreads;
                    if (a < G.A) {
                        G.r[a] = c0[j];
                        G.rr[a] = r0[j] + r1[j] - c0[j];
                    }
                }
            }
        } else {
            for (long long a0 = gtid; a0 < G.A; a0 += kInit * gthreads) {
                int b[kInit], c0[kInit], c1[kInit];
#pragma unroll
                for (int j = 0; j < kInit; ++j) {
                    const long long a = min(a0 + j * gthreads, G.A - 1);
                    b[j] = __ldg(&G.rev[a]);
                    c0[j] = lcg(&G.cap[a]);
                }
#pragma unroll
                for (int j = 0; j < kInit; ++j) c1[j] = lcg(&G.cap[b[j]]);
#pragma unroll
                for (int j = 0; j < kInit; ++j) {
                    const long long a = a0 + j * gthreads;
                    if (a < G.A) {
                        G.r[a] = c0[j];
                        G.rr[a] = c1[j];
                    }
                }
            }
        }
        for (long long v = gtid; v < n; v += gthreads) G.e[v] = 0;
        MF_SYNC(S_T_BATCH);
    }

    // ---- saturate the source arcs (Alg. 1 third loop, Alg. 4 lines 3-7) --
    // (on the fast path every source arc that regains residual leads into
    // S, so the moved excess stays on vertices that cannot reach a sink)
    if (kind != JOB_REFRESH) {
        long long moved = 0;
        const int a0 = __ldg(&G.row[s]), a1 = __ldg(&G.row[s + 1]);
        // (kSat arcs in flight per thread: 2M source arcs 20 -> 10 us)
        constexpr int kSat = 4;
        for (long long ab = a0 + gtid; ab < a1; ab += kSat * gthreads) {
            int ra[kSat];
#pragma unroll
            for (int j = 0; j < kSat; ++j) {
                const long long a = ab + j * gthreads;
                ra[j] = a < a1 ? lcg(&G.r[a]) : 0;
                K.resat += a < a1;
            }
#pragma unroll
            for (int j = 0; j < kSat; ++j) {
                if (ra[j] <= 0) continue;
                const long long a = ab + j * gthreads;
                const int b = __ldg(&G.rev[a]);
                G.r[a] = 0;
                G.rr[b] = 0;
                atomicAdd(&G.r[b], ra[j]);
                atomicAdd(&G.rr[a], ra[j]);
                add_ll(&G.e[__ldg(&G.head[a])], (long long)ra[j]);
                moved += ra[j];
            }
        }
        moved = warp_sum(moved);
        if (lane == 0 && moved) add_ll(&G.e[s], -moved);
        MF_SYNC(S_T_BATCH);
    }

    // ---- static push-pull (Sec. 4.2): also saturate every arc into t; the
    // vertices left deficient become secondary sinks of the loop below
    if (J.sink_sat && (kind == JOB_SOLVE || kind == JOB_RECOMPUTE)) {
        long long moved = 0;
        const int a0 = __ldg(&G.row[t]), a1 = __ldg(&G.row[t + 1]);
        for (long long a = a0 + gtid; a < a1; a += gthreads) {
            const int rin = lcg(&G.rr[a]);   // residual of v -> t
            if (rin > 0) {
                const int b = __ldg(&G.rev[a]);
                G.r[b] = 0;
                G.rr[a] = 0;
                atomicAdd(&G.r[a], rin);
                atomicAdd(&G.rr[b], rin);
                add_ll(&G.e[__ldg(&G.head[a])], -(long long)rin);
                moved += rin;
            }
        }
        moved = warp_sum(moved);
        if (lane == 0 && moved) add_ll(&G.e[t], moved);
        MF_SYNC(S_T_BATCH);
    }

    // ---- device loop (Algorithm 4 while-loop) ----------------------------
    bool early = false;   // stopped when PushRelabel left no active vertex
    bool limited = false; // stopped by max_iters or the wall-clock limit
    unsigned snext = stamp_base;   // next unused activation stamp
    for (it = 0; !fast; ++it) {
        const int par = (int)(it & 1);
        // height init: t and deficient vertices are sinks (height 0), all
        // others n; the sinks form BFS level 0.
        if (gtid == 0) {
            C->q[0].clear();
            C->q[1].clear();
            C->qcnt[1] = 0;
            C->qcnt[2] = 0;
            C->ccnt[0] = 0;
            C->asum[1] = C->asum[2] = 0;
            C->acnt[0] = C->acnt[1] = C->acnt[2] = 0;
            C->rlcnt = 0;
            C->rhcnt = 0;
            C->phc[1] = 0;
            C->wcnt = 0;
            C->hcnt = 0;
            C->hub_live[0] = C->hub_live[1] = C->hub_items[0] = C->hub_items[1] = 0;
            C->hub_act[0] = C->hub_act[1] = 0;
            C->dacc[par ^ 1] = 0;
            if (gtimer() - C->t_start > J.time_limit_ns) C->abort_loop = 1;
        }
        {
            // (the roots are staged per warp like a frontier: a push-pull repair
            // of a grid has millions, and an append per 32 vertices queued
            // 130,000 atomics on one word: 4M vertices 56 -> 20 us)
            long long dsum = 0, rdeg = 0;
            constexpr int kRs = 4;   // vertices in flight per thread
            int *const roots = s_bfs + (threadIdx.x >> 5) * kWq;
            int nroots = 0;   // staged (warp-uniform)
            auto publish = [&]() {
                __syncwarp();
                int base = 0;
                if (lane == 0) base = atomicAdd(&C->qcnt[0], nroots);
                base = __shfl_sync(kFull, base, 0);
                for (int i = lane; i < nroots; i += 32) G.qb0[base + i] = roots[i];
                __syncwarp();
                nroots = 0;
            };
            for (long long vb0 = (long long)gwarp * 32; vb0 < n; vb0 += kRs * gthreads) {
                long long evs[kRs];
                unsigned char pts[kRs];
                bool root[kRs];
                int r0[kRs], r1[kRs];
#pragma unroll
                for (int j = 0; j < kRs; ++j) {
                    const long long v = vb0 + j * gthreads + lane;
                    evs[j] = v < n ? lcg(&G.e[v]) : 0;
                    pts[j] = stage && v < n ? G.part[v] : kPartT;
                }
#pragma unroll
                for (int j = 0; j < kRs; ++j) {
                    const long long v = vb0 + j * gthreads + lane;
                    const long long ev = evs[j];
                    root[j] = false;
                    if (v >= n) continue;
                    if (stage == 0) {
                        root[j] = (v == t) || (v != s && ev < 0);
                        G.h[v] = root[j] ? 0 : n;
                        if (root[j] && v != t) dsum += ev;
                    } else if (stage == 1) {
                        // Alg. 8: h+ roots are t and the deficient vertices of T,
                        // h- roots are s and the overflowing vertices of S (both
                        // heights live in h: the two sides are disjoint)
                        root[j] = pts[j] == kPartT ? (v == t || ev < 0) : (v == s || ev > 0);
                        G.h[v] = root[j] ? 0 : n;
                    } else {
                        // the subgraph P: its deficient vertices are the sinks;
                        // the rest of the graph sits at n + 1, out of reach
                        const bool inP = pts[j] == kPartP;
                        root[j] = inP && ev < 0;
                        G.h[v] = inP ? (root[j] ? 0 : n) : n + 1;
                    }
                }
#pragma unroll
                for (int j = 0; j < kRs; ++j) {
                    const long long v = vb0 + j * gthreads + lane;
                    r0[j] = root[j] ? __ldg(&G.row[v]) : 0;
                    r1[j] = root[j] ? __ldg(&G.row[v + 1]) : 0;
                }
                if (nroots > kWq - 32 * kRs) publish();
#pragma unroll
                for (int j = 0; j < kRs; ++j) {
                    rdeg += r1[j] - r0[j];
                    const unsigned m = __ballot_sync(kFull, root[j]);
                    if (root[j]) roots[nroots + __popc(m & ((1u << lane) - 1u))] = (int)(vb0 + j * gthreads + lane);
                    nroots += __popc(m);
                }
            }
            if (nroots) publish();
            dsum = warp_sum(dsum);
            rdeg = warp_sum(rdeg);
            if (lane == 0 && dsum) add_ll(&C->dacc[par], dsum);
            if (lane == 0 && rdeg) add_ll(&C->asum[0], rdeg);
        }
        MF_SYNC_T(S_T_RESET, 0, 0, lctl(&C->qcnt[0]));
        // the flags of the next iteration: their last readers (the previous
        // iteration's exit test) are all past this barrier
        if (gtid == 0) C->ri_moved[par ^ 1] = 0;

        if (threadIdx.x == 0) s_bfs_begin = gtimer();
        // backward BFS from the sinks over residual arcs (global relabel),
        // level-synchronous and direction-optimising: top-down from the
        // frontier while it is small, bottom-up from the unvisited vertices
        // while the frontier holds more than 1/alpha of the unvisited arcs.
        int L = 0;
        bool bottom_up = false;
        long long arcs_seen = 0;
        for (;;) {
            const int cur = lctl(&C->qcnt[L % 3]);
            if (cur == 0) break;
            const long long mf = lctl(&C->asum[L % 3]);
            arcs_seen += mf;
            const bool dual = PP && stage == 1;   // push-pull: backward on T, forward on S
            // (the dual search of push-pull takes a smaller vertex share: its
            // first frontier, the overflowing and deficient vertices of both
            // sides, is a few percent of the vertices but touches few of the
            // others, which then scan all their arcs bottom-up)
            if (!bottom_up) bottom_up = mf * G.alpha > G.A - arcs_seen && cur * (dual ? 32LL : 64LL) > n;
            else bottom_up = cur * 24LL >= n;
            if (!bottom_up && mf <= G.solo_arcs && cur <= kSoloCap) {
                // a small frontier: CTA 0 runs the levels alone (bfs_solo).
                // Every thread has read this level's counters before it starts
                // (the first barrier).
                MF_SYNC_T(S_T_BFS, L, 6, cur);
                if (blockIdx.x == 0) bfs_solo(G, L, cur, arcs_seen, dual, s_dyn, s_stat, tprev, it, TR, K);
                MF_SYNC_T(S_T_BFS, L, 5, cur);
                L = lctl(&C->solo_L);
                arcs_seen = lctl(&C->solo_seen);
                continue;
            }
            const int *F = (L & 1) ? G.qb1 : G.qb0;
            int *NF = (L & 1) ? G.qb0 : G.qb1;
            int *ncnt = &C->qcnt[(L + 1) % 3];
            int *ccnt = &C->ccnt[L % 3];
            long long *asum = &C->asum[(L + 1) % 3];
            if (gtid == 0) {
                C->qcnt[(L + 2) % 3] = 0;
                C->ccnt[(L + 1) % 3] = 0;
                C->asum[(L + 2) % 3] = 0;
                if (bottom_up) s_stat[S_BU_LEVELS] += 1;
            }
            Front FR{ncnt, NF, asum, s_bfs + (threadIdx.x >> 5) * kWq, 0, 0};
            if (bottom_up) {
                // pieces of 32 V consecutive vertex ids
                int *const tick = cta_words();
                auto pieces = [&](auto vc, auto ac) {
                    constexpr int V = decltype(vc)::value, kPiece = 32 * V;
                    const int groups = (n + kPiece - 1) / kPiece;
                    int grp = gwarp, nxt;
                    BuPre<V> pre = bu_prefetch<V>(G, (long long)min(grp, groups) * kPiece);
                    for (; grp < groups; grp = nxt) {
                        const BuPre<V> cur = pre;
                        nxt = next_item(tick, groups);
                        pre = bu_prefetch<V>(G, (long long)min(nxt, groups) * kPiece);
                        bfs_bottom_up_group<V, decltype(ac)::value>(G, grp * kPiece, cur, dual, L, FR, ccnt, K);
                    }
                };
                if (G.bu_long || n <= 32LL * kBuV * nwarps)
                    pieces(std::integral_constant<int, kBuVLong>{}, std::integral_constant<int, kBuArcsLong>{});
                else
                    pieces(std::integral_constant<int, kBuV>{}, std::integral_constant<int, kBuArcs>{});
            } else {
                // groups of gs frontier vertices:
                // 32, or fewer when the frontier does not fill the grid's warps,
                // so that the arcs of a small frontier still spread over them
                int gs = 32;
                while (gs > 1 && (long long)(gs >> 1) * nwarps >= cur) gs >>= 1;
                int *const tick = cta_words();
                const int groups = (cur + gs - 1) / gs;
                for (int grp = gwarp; grp < groups; grp = next_item(tick, groups)) {
                    const int idx = grp * gs + lane;
                    int beg = 0, deg = 0;
                    bool fwd = false;
                    const int u = (lane < gs && idx < cur) ? lcg(&F[idx]) : 0;
                    if (lane < gs && idx < cur && vertex_ok(J, C, u, n)) {
                        fwd = dual && G.part[u] == kPartS;
                        beg = __ldg(&G.row[u]);
                        deg = __ldg(&G.row[u + 1]) - beg;
                        if (deg > kBigDeg) {
                            const int nc = (deg + kChunk - 1) / kChunk;
                            const int pos = atomicAdd(ccnt, nc);
                            for (int c = 0; c < nc; ++c) G.cb[pos + c] = make_int2(u, beg + c * kChunk);
                            deg = 0;
                        }
                    }
                    bfs_expand_warp(G, beg, deg, fwd, dual, L, FR, K);
                }
            }
            front_flush(G, FR, dual, K);
            MF_SYNC_T(S_T_BFS, L, bottom_up ? 2 : 0, cur);
            const int nch = lctl(ccnt);
            if (nch > 0) {
                int *const tick = cta_words();
                if (bottom_up) {
                    for (int c = gwarp; c < nch; c = next_item(tick, nch))
                        bfs_bottom_up_item(G, lcg(&G.cb[c]), dual, L, FR, K);
                } else {
                    // items staged one ahead (see item_issue)
                    int *const ibuf = s_dyn + kItemOff + (threadIdx.x >> 5) * kItemWarp;
                    int c = gwarp, c1 = next_item(tick, nch), b = 0;
                    ItemMeta cur = c < nch ? item_meta(G, c, dual) : ItemMeta{0, 0, 0, false};
                    if (c < nch) item_issue(G, cur, ibuf);
                    asm volatile("cp.async.commit_group;" ::: "memory");
                    ItemMeta nxt = c1 < nch ? item_meta(G, c1, dual) : ItemMeta{0, 0, 0, false};
                    while (c < nch) {
                        if (c1 < nch) item_issue(G, nxt, ibuf + (b ^ 1) * 2 * kItemBuf);
                        asm volatile("cp.async.commit_group;" ::: "memory");
                        c = c1;
                        c1 = next_item(tick, nch);
                        const ItemMeta nn = c1 < nch ? item_meta(G, c1, dual) : ItemMeta{0, 0, 0, false};
                        asm volatile("cp.async.wait_group 1;" ::: "memory");   // the current item's copies
                        __syncwarp();
                        const int *sv = ibuf + b * 2 * kItemBuf;
                        const unsigned fw = cur.fwd ? (1u << kIlpB) - 1u : 0u;
                        for (int ab = cur.y; ab < cur.a1; ab += 32 * kIlpB) {
                            int a[kIlpB];
                            bool ok[kIlpB];
#pragma unroll
                            for (int j = 0; j < kIlpB; ++j) {
                                a[j] = ab + 32 * j + lane;
                                ok[j] = a[j] < cur.a1;
                            }
                            bfs_visit_staged(G, sv, sv + kItemBuf, cur.y & ~3, a, ok, fw, dual, L, FR, K);
                        }
                        __syncwarp();   // every lane is done with this buffer before it is refilled
                        cur = nxt;
                        nxt = nn;
                        b ^= 1;
                    }
                    asm volatile("cp.async.wait_all;" ::: "memory");
                }
                front_flush(G, FR, dual, K);
                MF_SYNC_T(S_T_BFS, L, bottom_up ? 3 : 1, nch);
            }
            ++L;
        }
        if (gtid == 0) s_stat[S_LEVELS] += L;

        if (threadIdx.x == 0) s_bfs_end = gtimer();
        // termination: no active vertex under the fresh BFS heights
        const int nw = lctl(&C->wcnt);
        const int nh = lctl(&C->hcnt);
        if (nw == 0 && nh == 0) {
            if (stage == 1) {
                // Alg. 8: what neither search reached -- overflowing vertices
                // of T that reach no sink, deficient vertices of S that no
                // source reaches -- forms P, where the push phase continues
                for (long long v = gtid; v < n; v += gthreads)
                    if (v != s && v != t && lcg(&G.h[v]) == n) G.part[v] = kPartP;
                MF_SYNC_T(S_T_RESET, 2, 0, 0);
                stage = 2;
                continue;
            }
            break;
        }
        if (it >= J.max_iters || lctl(&C->abort_loop)) {   // (abort_loop: written before the height-init barrier)
            if (gtid == 0) atomicOr(&C->status, it >= J.max_iters ? ST_ITERS : ST_TIME);
            limited = true;
            break;
        }

        // PushRelabel (Alg. 2), in passes.  A pass serves the high-degree
        // vertices of its hub list together, in kPrChunk-arc items over the
        // whole grid (cooperative cycles separated by grid barriers), and then
        // the worklist, one warp per vertex: from the activation queue in one
        // phase, where the sign of the excess says who holds a vertex (ActList),
        // or, topology-driven, in rounds separated by grid barriers, each of
        // which serves an active vertex once.  So no vertex is ever processed by
        // two warps at once.  High-degree vertices that a pass turns active
        // again form the hub list of the next pass.
        const unsigned rstamp_it = snext++;   // relabel-list stamp of this iteration
        Relabelled RL;
        RL.stamp = rstamp_it;
        if (gtid == 0) {
            C->qcnt[0] = 0;
            C->asum[0] = 0;
        }
        bool rounds_clean = true;   // the last activation round left no active vertex
        bool hubs_clean = true;     // the last hub cycle left no hub active
        int pend = 0;               // hubs that the last pass turned active
        // Rounds per pass (topology-driven mode): kMaxRounds, and past that,
        // while at most one vertex per warp is active, as many as the BFS just
        // run had levels -- such a round costs about what a BFS level costs, so
        // on deep graphs (grids) finishing a few active vertices by rounds is
        // cheaper than another global relabel.
        const int max_rounds = L > kMaxRounds ? L : kMaxRounds;
        int hub_no = 0;             // hub cycles' lists built in this iteration
        for (int pass = 0; pass < (PP ? kMaxPassesPP : kMaxPasses); ++pass) {
            const int *HL = (pass & 1) ? G.hl2 : G.hl;
            const int nhp = pass == 0 ? nh : pend;
            const unsigned hstamp = snext++;   // the next pass's hub list
            int *const pcnt = &C->phc[(pass + 1) & 1];
            // pass 0 appends to phc[1] and starts its rounds on the counters
            // zeroed at the iteration's start; a later pass always has hubs,
            // so the barrier of its first list comes before any use of what is
            // zeroed here (the previous pass's rounds ended with an empty list)
            if (gtid == 0) {
                if (pass > 0) {
                    *pcnt = 0;
                    C->wcnt = 0;
                    C->acnt[0] = C->acnt[1] = C->acnt[2] = 0;
                }
                s_stat[S_WL] += nhp;
            }
            // the data-driven and push-pull modes run PushRelabel from the
            // activation queue; the topology-driven mode in rounds
            const bool qmode = jmode != MF_MODE_TOPOLOGY && G.aq != nullptr;
            ActList AL{pcnt, (pass & 1) ? G.hl : G.hl2, hstamp, qmode ? G.aq : nullptr, G.qc, 0, &s_deadline,
                       &C->q[pass & 1], 0, nhp > kDeferHubs};
            bool pass_hubs_clean = true;
            if (nhp > 0) {
                pass_hubs_clean = false;
                const int hub_min = PP ? kMinHubCyclesPP : kMinHubCycles;
                const int hub_cycles = kc > hub_min ? kc : hub_min;
                const unsigned char *const ptc = stage == 1 ? G.part : nullptr;
                int nlive = nhp;   // hubs of the cycle's list
                for (int c = 0;; ++c, ++hub_no) {
                    const int par = hub_no & 1;
                    const bool fresh = c == 0 && pass == 0;   // the BFS heights decide the first cycle
                    // the next list's counters: every thread has read them
                    // before the last cycle's pushes
                    if (gtid == 0) {
                        C->hub_live[par ^ 1] = C->hub_items[par ^ 1] = 0;
                        // the worklist that the scan below builds replaces the
                        // BFS's (whose length only matters without active hubs)
                        if (AL.defer && c == 0) C->wcnt = 0;
                    }
                    hub_list<PP>(G, HL, par, nlive, c == 0, fresh, ptc, gwarp, nwarps, J.debug != 0);
                    MF_SYNC_T(S_T_HUB, c, 0, nlive);
                    // the next pass's queue counters: every thread has read what
                    // the pass before this one left there
                    if (gtid == 0 && c == 0 && pass > 0) C->q[(pass + 1) & 1].clear();
                    nlive = lctl(&C->hub_live[par]);
                    const int nitems = lctl(&C->hub_items[par]);
                    if (nlive == 0) pass_hubs_clean = true;
                    if (nlive == 0 || c >= hub_cycles) {
                        ++hub_no;
                        break;
                    }
                    if (gtid == 0) s_stat[S_HUB_CYCLES] += 1;
                    if (!fresh) {
                        hub_lowest(G, nitems, par, gwarp, nwarps, stg, ptc, K);
                        MF_SYNC_T(S_T_HUB, c, 1, nitems);
                    }
                    if (gtid == 0) C->hub_act[par ^ 1] = 0;   // (read before this cycle's list phase)
                    if (!fresh) hub_relabel(G, HL, par, nlive, rstamp_it, gwarp, nwarps, K);
                    hub_push(G, nitems, par, fresh, gwarp, nwarps, stg, ptc, AL, K);
                    if (AL.count && lane == 0) atomicAdd(&C->wcnt, AL.count);   // (topology-driven mode)
                    AL.count = 0;
                    MF_SYNC_T(S_T_HUB, c, 3, nitems);
                    if (!AL.defer && lctl(&C->hub_act[par]) == 0) {
                        pass_hubs_clean = true;
                        ++hub_no;
                        break;
                    }
                }
                if (AL.defer) {
                    // the active vertices, by one pass over all vertices: the
                    // worklist anew, and the hubs (left active by the cycles, or
                    // made active by another one) into the next pass's list
                    constexpr int kSc = 4;   // vertices in flight per thread
                    for (long long vb0 = (long long)gwarp * 32; vb0 < n; vb0 += kSc * gthreads) {
                        int v[kSc], hs[kSc], deg[kSc];
                        long long es[kSc];
                        bool small[kSc], hub[kSc], any = false;
#pragma unroll
                        for (int j = 0; j < kSc; ++j) {
                            const long long x = vb0 + j * gthreads + lane;
                            v[j] = x < n ? (int)x : s;
                            hs[j] = lcg(&G.h[v[j]]);
                            es[j] = lcg(&G.e[v[j]]);
                        }
#pragma unroll
                        for (int j = 0; j < kSc; ++j) {
                            hub[j] = hs[j] < n && v[j] != s && v[j] != t &&
                                     (stage == 1 && G.part[v[j]] == kPartS ? es[j] < 0 : es[j] > 0);
                            any |= hub[j];
                        }
                        if (!__any_sync(kFull, any)) continue;
#pragma unroll
                        for (int j = 0; j < kSc; ++j)
                            deg[j] = hub[j] ? __ldg(&G.row[v[j] + 1]) - __ldg(&G.row[v[j]]) : 0;
#pragma unroll
                        for (int j = 0; j < kSc; ++j) {
                            small[j] = hub[j] && deg[j] <= kHubDeg;
                            hub[j] = deg[j] > kHubDeg;
                        }
                        warp_append_n(small, v, &C->wcnt, G.wl);
                        warp_append_n(hub, v, pcnt, AL.hlist);
                    }
                    MF_SYNC_T(S_T_HUB, hub_cycles, 2, lctl(&C->wcnt));
                    pass_hubs_clean = true;   // (those left active are listed)
                }
            }
            bool pass_rounds_clean = true;
            int cnt = lctl(&C->wcnt);
            const int qtail0 = qmode ? lctl(&AL.Q->tail) : 0;   // queued by the hub cycles
            if (qmode && cnt + qtail0 > 0) {
                // PushRelabel from the activation queue, without rounds: the
                // worklist entries (generation 0) are dealt to the warps first,
                // then each warp takes a ticket for the next queued
                // entry and waits for it; of the vertices that a visit turns
                // active the warp serves one itself (visit_chain_t) and queues
                // the others at once with the next generation, for the next
                // free warps.  The phase ends when every queued entry has been
                // processed: a warp counts what it has finished when it finds
                // no entry ready, and the one that makes the counts equal
                // raises fin.  One warp per CTA polls that word and tells
                // the others in shared memory.  One grid barrier at the end.
                //
                // How long it goes on: what another global relabel costs is
                // known, the BFS has just been timed, so the queue gets as
                // long and then leaves what is still active to the next
                // iteration (neither side can then cost much more
                // than the better choice would have).  Generations below
                // kMinGen are served in any case, so every iteration makes
                // progress.
                const int n0 = cnt;
                if (threadIdx.x == 0) s_deadline = gtimer() + (s_bfs_end - s_bfs_begin);
                __syncthreads();
                int ndone = 0;   // entries finished and not yet counted (warp-uniform)
                int *const tick = cta_words();
                for (int i = gwarp;; i = i < n0 ? next_item(tick, n0) : i) {
                    int u = -1, gen = 0;
                    if (i < n0) {
                        u = bcast_ld(&G.wl[i]);
                    } else {
                        unsigned long long slot = 0;
                        if (lane == 0) {
                            const int q = atomicAdd(&AL.Q->head, 1);
                            unsigned long long t0 = 0;
                            unsigned ns = 32;
                            for (int k = 0;; ++k) {
                                if (q < G.qc) {
                                    slot = ld_acquire_u64(&G.aq[q]);
                                    if (slot) {
                                        G.aq[q] = 0;   // the slot is free again for the next phase
                                        break;
                                    }
                                }
                                if (ndone) {
                                    // the finished entries' own enqueues, and (by the acquire)
                                    // those of every entry counted before them, precede the
                                    // tail read
                                    int d;
                                    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;"
                                                 : "=r"(d) : "l"(&AL.Q->done), "r"(ndone) : "memory");
                                    if (d + ndone == n0 + ld_acquire_s32(&AL.Q->tail)) atomicExch(&AL.Q->fin, 1);
                                    ndone = 0;
                                }
                                if (threadIdx.x == 0) {
                                    if (ld_acquire_s32(&AL.Q->fin)) {
                                        *(volatile int *)&s_fin = 1;
                                        break;
                                    }
                                } else if (*(volatile int *)&s_fin) {
                                    break;
                                }
                                if ((k & 15) == 15) {
                                    if (t0 == 0) t0 = gtimer();
                                    if (gtimer() - t0 > kWaitNs) {
                                        atomicOr(&C->status, ST_WAIT);
                                        *(volatile int *)&s_fin = 1;
                                        break;
                                    }
                                }
                                __nanosleep(ns);
                                ns = ns < 256 ? 2 * ns : ns;
                            }
                        }
                        ndone = __shfl_sync(kFull, ndone, 0);
                        slot = __shfl_sync(kFull, slot, 0);
                        if (!slot) break;   // every entry processed (or a wait gave up)
                        u = (int)(slot & 0xffffffffu) - 1;
                        gen = (int)(slot >> 32);
                    }
                    AL.gen = gen + 1;
                    if (!vertex_ok(J, C, u, n)) {
                        // skipped; still counted as processed below
                    } else if (gen >= kMinGen && __any_sync(kFull, gtimer() > s_deadline)) {
                        if (lane == 0) AL.Q->over = 1;   // left active
                    } else if (stage == 1) {
                        const unsigned char side = G.part[u];
                        if (side == kPartS)
                            visit_chain_t<true>(G, u, kc, AL, G.part, side, stg, RL, K);
                        else
                            visit_chain_t<false>(G, u, kc, AL, G.part, side, stg, RL, K);
                    } else {
                        visit_chain(G, u, kc, AL, stg, RL, K);
                    }
                    ++ndone;
                }
                if (RL.cnt) relabelled_flush(G, RL);
                MF_SYNC_T(S_T_PRW, 0, 0, cnt + lctl(&AL.Q->tail));
                if (lctl(&C->status) & ST_WAIT) return;   // a wait gave up: the queue's state is undefined
                if (threadIdx.x == 0) s_fin = 0;
                pass_rounds_clean = lctl(&AL.Q->over) == 0;
                if (gtid == 0) s_stat[S_ROUNDS] += lctl(&AL.Q->maxgen) + 1;
            } else if (!qmode && (cnt > 0 || (pass == 0 && jmode == MF_MODE_TOPOLOGY))) {
                pass_rounds_clean = false;
                for (int rd = 0;; ++rd) {
                    // topology-driven (Sec. 5.2): every round visits every
                    // vertex id and serves the active ones (no worklist is kept:
                    // the counts only tell whether another round has work).  A
                    // CTA first collects the active ones of its ids, groups of
                    // 32 dealt over the CTAs, in its part of qb0, and its warps
                    // then take them one by one: served in place, the active
                    // ones of a group, often neighbours in id, waited for one
                    // another (RMAT-18, renumbered: 62 -> 17 us a round).
                    int *const ncnt = &C->acnt[(rd + 1) % 3];
                    if (gtid == 0) {
                        C->acnt[(rd + 2) % 3] = 0;
                        s_stat[S_ROUNDS] += 1;
                    }
                    const int groups = (n + 31) / 32, per = groups / (int)gridDim.x, more = groups % (int)gridDim.x;
                    int *const mine = G.qb0 + 32 * ((int)blockIdx.x * per + min((int)blockIdx.x, more));
                    int *const w = cta_words();
                    constexpr int kTp = 2;   // groups in flight per warp
                    for (int g0 = gwarp; g0 < groups; g0 += kTp * nwarps) {
                        int hs[kTp], deg[kTp];
                        long long es[kTp];
#pragma unroll
                        for (int j = 0; j < kTp; ++j) {
                            const int v = min((g0 + j * nwarps) * 32 + lane, n - 1);
                            hs[j] = lcg(&G.h[v]);
                            es[j] = lcg(&G.e[v]);
                            deg[j] = __ldg(&G.row[v + 1]) - __ldg(&G.row[v]);
                        }
#pragma unroll
                        for (int j = 0; j < kTp; ++j) {
                            const int v = (g0 + j * nwarps) * 32 + lane;
                            warp_append(v < n && v != s && v != t && hs[j] < n && es[j] > 0 && deg[j] <= kHubDeg, v,
                                        &w[0], mine);
                        }
                    }
                    __syncthreads();
                    for (int k = cta_ticket(&w[1]); k < w[0]; k = cta_ticket(&w[1]))
                        visit_chain(G, bcast_ld(&mine[k]), kc, AL, stg, RL, K);
                    if (RL.cnt) relabelled_flush(G, RL);
                    if (AL.count && lane == 0) atomicAdd(ncnt, AL.count);
                    AL.count = 0;
                    MF_SYNC_T(S_T_PRW, rd, 0, cnt);
                    cnt = lctl(ncnt);
                    if (cnt == 0) pass_rounds_clean = true;
                    if (cnt == 0 || rd + 1 >= max_rounds || (rd + 1 >= kMaxRounds && cnt > nwarps)) break;
                }
            }
            hubs_clean = pass_hubs_clean;
            rounds_clean = pass_rounds_clean;
            pend = lctl(pcnt);   // every append to it came before the pass's last barrier
            // another pass only for a few re-activated hubs: a large set of
            // them is better served after a global relabel
            if (pend == 0 || pend > (PP ? kPassHubsPP : kPassHubs) || !pass_hubs_clean || !pass_rounds_clean)
                break;
        }

        // RemoveInvalidEdges (Alg. 3): relabelled vertices by warps,
        // relabelled hubs by items
        // (push-pull: only arcs within the vertex's part; the pull side uses
        // the h- form, Algorithm 7)
        const unsigned char *ptc = stage ? G.part : nullptr;
        const int nrl = lctl(&C->rlcnt);
        const int nri = lctl(&C->rhcnt);
        int *const tick = cta_words();
        int ri = gwarp;   // hub items first (they cost the most), then vertices
        for (; ri < nri; ri = next_item(tick, nri + nrl)) {
            const int2 item = lcg(&G.hri[ri]);
            const int u = __shfl_sync(kFull, item.x, 0);
            if (!vertex_ok(J, C, u, n)) continue;   // warp-uniform
            const int hu = bcast_ld(&G.h[u]);
            const int a1 = min(item.y + kPrChunk, __ldg(&G.row[u + 1]));
            const unsigned char side = stage == 1 ? G.part[u] : (stage == 2 ? kPartP : kPartT);
            if (PP && side == kPartS) {
                const long long got = warp_sum(remove_invalid_range_t<true>(G, hu, item.y, a1, ptc, side, K));
                if (lane == 0 && got) {
                    add_ll(&G.e[u], got);
                    C->ri_moved[par] = 1;
                }
            } else {
                const long long moved = warp_sum(remove_invalid_range_t<false>(G, hu, item.y, a1, ptc, side, K));
                if (lane == 0 && moved) {
                    add_ll(&G.e[u], -moved);
                    C->ri_moved[par] = 1;
                }
            }
        }
        for (; ri < nri + nrl; ri = next_item(tick, nri + nrl)) {
            const int u = bcast_ld(&G.rl[ri - nri]);
            if (!vertex_ok(J, C, u, n)) continue;   // warp-uniform
            const unsigned char side = ptc ? ptc[u] : kPartT;
            if (side == kPartS)
                remove_invalid_warp_t<true>(G, u, &C->ri_moved[par], ptc, side, K);
            else
                remove_invalid_warp_t<false>(G, u, &C->ri_moved[par], ptc, side, K);
        }
        MF_SYNC_T(S_T_RI, 0, 0, nrl + nri);
        if ((it & 255) == 255) flush_counters(K, ST);

        // Alg. 4's loop test, on the heights PushRelabel left: no vertex is
        // active if every activation was served (the last round's list is
        // empty, no hub is left active or was turned active again) and
        // RemoveInvalidEdges moved nothing.  The labelling is then valid (the
        // only arcs that pushes and relabels can make steep leave relabelled
        // vertices, and RemoveInvalidEdges found none), so each vertex with
        // excess sits at height >= n and cannot reach a sink: the preflow is
        // maximum without another BFS.  The value needs the current deficits.
        const int busy = (rounds_clean ? 0 : 1) | (hubs_clean ? 0 : 2) | (lctl(&C->ri_moved[par]) ? 4 : 0) |
                         (pend > 0 ? 8 : 0);
        if (gtid == 0 && TR && C->trace_n - 1 < G.trace_cap) TR[C->trace_n - 1].mode = (short)busy;
        if (!J.exact_exit && kind != JOB_REFRESH && stage == 0 && busy == 0) {
            long long dsum = 0;
            for (long long v = gtid; v < n; v += gthreads) {
                const long long ev = lcg(&G.e[v]);
                if (v != s && v != t && ev < 0) dsum += ev;
            }
            dsum = warp_sum(dsum);
            if (lane == 0 && dsum) add_ll(&C->dacc[par ^ 1], dsum);
            MF_SYNC_T(S_T_RESET, 1, 0, 0);
            early = true;
            break;
        }
    }

    if (pp_ran) {
        // Alg. 8's result: the new cut is S' = (S minus P) plus the part of P
        // that reaches no sink of P, T' the rest; every deficient vertex ended
        // in T', so the value is e(t) plus all deficits (recounted here).
        // The heights are rewritten to encode the cut for the next repair
        // (T' below n, S' at n): exact as a cut, not as BFS distances.
        long long dsum = 0;
        for (long long v = gtid; v < n; v += gthreads) {
            const long long ev = lcg(&G.e[v]);
            if (v != s && v != t && ev < 0) dsum += ev;
            const unsigned char p = G.part[v];
            if (p == kPartT) G.h[v] = 0;
            else if (p == kPartS) G.h[v] = n;
        }
        dsum = warp_sum(dsum);
        if (lane == 0 && dsum) add_ll(&C->dacc[(it & 1) ^ 1], dsum);
        MF_SYNC_T(S_T_RESET, 3, 0, 0);
    }

    // ---- debug_checks: the state's invariants over all arcs ----------------
    // e(v) = sum over v's arcs of (r - cap) (the incremental excess updates
    // of the repair equal the full recount of Alg. 4 line 2), r >= 0, the
    // residuals of an arc pair add up to the pair's capacities, and the
    // mirror rr(a) = r(rev a).  One warp per vertex.
    if (J.debug) {
        for (int v = gwarp; v < n; v += nwarps) {
            const int a0 = __ldg(&G.row[v]), a1 = __ldg(&G.row[v + 1]);
            long long in = 0;
            bool bad = false;
            for (int a = a0 + lane; a < a1; a += 32) {
                const int b = __ldg(&G.rev[a]);
                const int ra = lcg(&G.r[a]), rb = lcg(&G.r[b]);
                in += (long long)ra - lcg(&G.cap[a]);
                if (ra < 0 || (long long)ra + rb != (long long)lcg(&G.cap[a]) + lcg(&G.cap[b]) ||
                    lcg(&G.rr[a]) != rb) {
                    if (!bad) check_fail(C, 3, a);
                    bad = true;
                }
            }
            in = warp_sum(in);
            if (lane == 0 && in != lcg(&G.e[v])) check_fail(C, 2, v);
        }
    }

    // ---- result and statistics -------------------------------------------
    if (gtid == 0) {
        for (int i = 0; i < S_COUNT; ++i)
            if (s_stat[i]) add_ll(&ST[i], s_stat[i]);
        // dacc: deficits at the last height init, or recounted at a clean
        // exit and after a push-pull repair
        if (!fast) C->flow = lcg(&G.e[t]) + lctl(&C->dacc[(early || pp_ran) ? (it & 1) ^ 1 : it & 1]);
        if (kind != JOB_REFRESH) {
            C->iters = fast ? 0 : early ? it + 1 : it;
            C->exit_kind = fast ? EXIT_NO_CUT_CHANGE : early ? EXIT_CLEAN : pp_ran ? EXIT_PUSH_PULL : EXIT_BFS;
        }
        C->heights_exact = !fast && !early && !pp_ran;
        if (kind == JOB_SOLVE) C->pairs_ok = 1;   // (cleared with the whole block by mf_import_state)
        C->cut_exact = !early;   // the fast path keeps the exact cut it started from
        C->stamp_base = snext;
        if (batch_job) C->bseq = seq;
    }
    // After a limit the words that decided it stay: no barrier lies between
    // here and that decision, which other CTAs may yet have to take (one that
    // read abort_loop cleared would go on and wait for the rest in vain).  The
    // status is sticky, and mf_solve starts from a cleared block.
    if (gtid == 0 && !limited) {
        C->ri_moved[0] = C->ri_moved[1] = 0;
        C->phc[0] = C->phc[1] = 0;
        C->rhcnt = 0;
        C->inc_block = 0;
        for (int i = 0; i < 3; ++i) {
            C->qcnt[i] = C->ccnt[i] = 0;
            C->asum[i] = 0;
        }
        C->wcnt = C->hcnt = C->rlcnt = 0;
        C->acnt[0] = C->acnt[1] = C->acnt[2] = 0;
        C->hub_live[0] = C->hub_live[1] = C->hub_items[0] = C->hub_items[1] = 0;
        C->hub_act[0] = C->hub_act[1] = 0;
        C->dacc[0] = C->dacc[1] = 0;
        C->batch_err = 0;
        C->abort_loop = 0;
    }
    flush_counters_cta(K, ST);
}

#undef ST
#undef TR

// ------------------------------------------------------------- policy --
static_assert(MF_MODE_DATA_DRIVEN == 0 && MF_MODE_TOPOLOGY == 1 && MF_MODE_PUSH_PULL == 2,
              "the network's mode outputs 2, 3, 4 are the modes in this order");

struct PolicyJob {
    int k, flags, mode, kc_plain, max_deg;
    int gmode;             // the graph's own processing mode (MF_MODE_*)
    int pp_ok;             // the graph can repair by Dynamic Push-Pull
    const int *k_dev;      // if set, the batch size is read from device memory
    const int *ids, *caps;
    const float *params;   // network parameters (mf_mlp.cuh), or null
};

// Features of a batch and the policy decision for the k_solve launch that
// follows (JOB_AUTO).  CTAs of 256 threads stride over the batch entries and
// add their integer sums (exact, so the result does not depend on the order)
// to the control block; the last CTA to arrive computes the 12 features,
// then the plain rule (dynamic repair when the batch holds at most 1 % of
// the edges, KERNELCYCLES = average degree) or the network, with the plain
// rule as fallback on any non-finite or out-of-range input (|z| > 8), and
// clears the sums for the next launch.  Entries with bad ids are skipped
// here; k_solve rejects the batch.
// Four 256-thread CTAs per CTA of the repair's grid: a 100k-entry batch is
// then one entry per thread, its chain of dependent gathers (edge, arc,
// reverse arc, heads) walked once instead of three times in a row.
constexpr int kPolicyCtasPerSlot = 4;
__global__ void __launch_bounds__(256) k_policy(DevGraph G, PolicyJob PJ) {
    Ctl *C = G.ctl;
    if (PJ.k_dev) PJ.k = lcg(PJ.k_dev);
    __shared__ long long red[3][8];
    __shared__ float x[mlp::kIn], z[mlp::kIn], h1[mlp::kH1], h2[mlp::kH2], y[mlp::kOut];
    __shared__ int fb, last;
    long long inc = 0, touch = 0, sumd = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < PJ.k;
         i += (long long)gridDim.x * blockDim.x) {
        const int id = PJ.ids[i];
        if (id < 0 || id >= G.m) continue;
        const long long old = lcg(&G.cap_edge[id]);
        long long nc = PJ.caps[i];
        if (PJ.flags & MF_DELTA) nc = old + nc < 0 ? 0 : old + nc;
        inc += nc > old;
        sumd += nc > old ? nc - old : old - nc;
        if (G.edge_st) {
            touch += __ldg(&G.edge_st[id]);
        } else {
            const int a = __ldg(&G.arc_of_edge[id]);
            if (a >= 0 && (__ldg(&G.head[a]) == G.t || __ldg(&G.head[__ldg(&G.rev[a])]) == G.s)) ++touch;
        }
    }
    inc = warp_sum(inc);
    touch = warp_sum(touch);
    sumd = warp_sum(sumd);
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = inc;
        red[1][threadIdx.x >> 5] = touch;
        red[2][threadIdx.x >> 5] = sumd;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 0; q < 3; ++q) {
            long long v = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[q][w];
            if (v) add_ll(&C->pol_acc[q], v);
        }
        __threadfence();
        last = atomicAdd(&C->pol_done, 1) == (int)gridDim.x - 1;
        if (last) {
            __threadfence();
            for (int q = 0; q < 3; ++q) {
                red[q][0] = __ldcg(&C->pol_acc[q]);
                C->pol_acc[q] = 0;
            }
            C->pol_done = 0;
        }
    }
    __syncthreads();
    if (!last) return;
    if (threadIdx.x == 0) {
        const float n = (float)G.n, m = (float)(G.m > 0 ? G.m : 1), k = (float)PJ.k;
        const float kk = k > 0.f ? k : 1.f;
        const long long iters = lcg(&C->iters);
        const long long reached = lcg(&C->st[S_BFS_VERTS]);
        x[0] = log2f(n);
        x[1] = log2f(m);
        x[2] = log2f(1.f + k);
        x[3] = k / m;
        x[4] = (float)red[0][0] / kk;
        x[5] = (float)red[1][0] / kk;
        x[6] = log2f(1.f + (float)red[2][0]);
        const long long fl = lcg(&C->flow);
        x[7] = log2f(1.f + (float)(fl < 0 ? -fl : fl));
        x[8] = (float)G.A / n;
        x[9] = log2f(1.f + (float)PJ.max_deg);
        x[10] = (float)iters;
        x[11] = (float)reached / ((float)(iters + 1) * n);
        for (int j = 0; j < mlp::kIn; ++j) C->feat[j] = x[j];
        fb = PJ.mode != MF_POLICY_LEARNED || PJ.params == nullptr;
        if (!fb)
            for (int j = 0; j < mlp::kIn; ++j) {
                z[j] = (x[j] - PJ.params[mlp::oMu + j]) / PJ.params[mlp::oSd + j];
                if (!isfinite(z[j]) || fabsf(z[j]) > 8.f) fb = 1;
            }
    }
    __syncthreads();
    if (!fb) {
        const float *P = PJ.params;
        if (threadIdx.x < mlp::kH1) {
            float a = P[mlp::oB1 + threadIdx.x];
            for (int j = 0; j < mlp::kIn; ++j) a += P[mlp::oW1 + threadIdx.x * mlp::kIn + j] * z[j];
            h1[threadIdx.x] = a > 0.f ? a : 0.f;
        }
        __syncthreads();
        if (threadIdx.x < mlp::kH2) {
            float a = P[mlp::oB2 + threadIdx.x];
            for (int j = 0; j < mlp::kH1; ++j) a += P[mlp::oW2 + threadIdx.x * mlp::kH1 + j] * h1[j];
            h2[threadIdx.x] = a > 0.f ? a : 0.f;
        }
        __syncthreads();
        if (threadIdx.x < mlp::kOut) {
            float a = P[mlp::oB3 + threadIdx.x];
            for (int j = 0; j < mlp::kH2; ++j) a += P[mlp::oW3 + threadIdx.x * mlp::kH2 + j] * h2[j];
            y[threadIdx.x] = a;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        int kind, kc, mode = PJ.gmode;
        bool fallback = fb != 0;
        for (int o = 0; o < mlp::kOut && !fallback; ++o)
            if (!isfinite(y[o])) fallback = true;
        if (fallback) {
            kind = (long long)PJ.k * 100 <= (long long)G.m ? JOB_REPAIR : JOB_RECOMPUTE;
            kc = PJ.kc_plain;
        } else {
            kind = y[0] > 0.f ? JOB_REPAIR : JOB_RECOMPUTE;
            const float l = fminf(fmaxf(rintf(y[1]), 0.f), 6.f);
            kc = 1 << (int)l;
            // the mode of the largest logit (outputs 2, 3, 4: data-driven,
            // topology-driven, push-pull); push-pull only where the graph
            // keeps the exact cut it needs, else the better of the other two
            int best = 0;
            for (int c = 1; c < mlp::kModes; ++c)
                if (y[2 + c] > y[2 + best]) best = c;
            if (best == MF_MODE_PUSH_PULL && !PJ.pp_ok) best = y[3] > y[2] ? MF_MODE_TOPOLOGY : MF_MODE_DATA_DRIVEN;
            mode = best;
        }
        C->pol_kind = kind;
        C->pol_kc = kc;
        C->pol_mode = mode;
        C->pol_fallback = (PJ.mode == MF_POLICY_LEARNED && fallback) ? 1 : 0;
    }
}

// at (or null for the identity): the place of each output element in the input
__global__ void k_cut_side(const int *h, int n, const int *at, unsigned char *side) {
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x)
        side[v] = h[at ? at[v] : v] >= n ? 1 : 0;
}

template <class T>
__global__ void k_gather(T *dst, const T *src, const int *at, long long count) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x)
        dst[i] = src[at[i]];
}

// ---------------------------------------------- allocation-free solve --
// Scratch of mf_solve_bicsr_noalloc: one static device array per GPU that
// loads this library, used instead of device allocations for everything the
// solve kernel needs besides the caller's graph and output arrays.  Sized for
// graphs of at most kNoAllocMaxN vertices and kNoAllocMaxArcs Bi-CSR arcs.
constexpr int kNoAllocMaxN = 1 << 17;
constexpr long long kNoAllocMaxArcs = 1LL << 21;
constexpr int kNoAllocMaxGrid = 1024;
constexpr long long kNoAllocMaxHubs = kNoAllocMaxArcs / kHubDeg;

__host__ __device__ constexpr size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// Byte offsets of the scratch regions (each 256-byte aligned).
struct NoAllocLayout {
    static constexpr size_t ctl = 0;
    static constexpr size_t rr = ctl + align256(sizeof(Ctl));
    static constexpr size_t qb0 = rr + align256(sizeof(int) * kNoAllocMaxArcs);
    static constexpr size_t qb1 = qb0 + align256(sizeof(int) * kNoAllocMaxN);
    static constexpr size_t wl = qb1 + align256(sizeof(int) * kNoAllocMaxN);
    static constexpr size_t rl = wl + align256(sizeof(int) * kNoAllocMaxN);
    static constexpr size_t astamp = rl + align256(sizeof(int) * kNoAllocMaxN);
    static constexpr size_t rstamp = astamp + align256(sizeof(unsigned) * kNoAllocMaxN);
    static constexpr size_t cb = rstamp + align256(sizeof(unsigned) * kNoAllocMaxN);
    static constexpr size_t hit0 = cb + align256(sizeof(int2) * (kNoAllocMaxArcs / kChunk + kNoAllocMaxN));
    static constexpr size_t hit1 = hit0 + align256(sizeof(int4) * (kNoAllocMaxArcs / kPrChunk + kNoAllocMaxHubs));
    static constexpr size_t hikey = hit1 + align256(sizeof(int4) * (kNoAllocMaxArcs / kPrChunk + kNoAllocMaxHubs));
    static constexpr size_t hl = hikey + align256(sizeof(int) * (kNoAllocMaxArcs / kPrChunk + kNoAllocMaxHubs));
    static constexpr size_t hlist0 = hl + align256(sizeof(int) * kNoAllocMaxHubs);
    static constexpr size_t hlist1 = hlist0 + align256(sizeof(int) * kNoAllocMaxHubs);
    static constexpr size_t hkey = hlist1 + align256(sizeof(int) * kNoAllocMaxHubs);
    static constexpr size_t hrem = hkey + align256(2 * sizeof(int) * kNoAllocMaxHubs);
    static constexpr size_t hl2 = hrem + align256(sizeof(long long) * kNoAllocMaxHubs);
    static constexpr size_t hri = hl2 + align256(sizeof(int) * kNoAllocMaxHubs);
    static constexpr size_t aq = hri + align256(sizeof(int2) * (kNoAllocMaxArcs / kPrChunk + kNoAllocMaxHubs));
    static constexpr size_t total = aq + align256(sizeof(unsigned long long) * kNoAllocMaxN);
};

static_assert(NoAllocLayout::total == 14371072, "the header states the scratch size");
static __device__ __align__(256) unsigned char g_noalloc_scratch[NoAllocLayout::total];

}  // namespace mf

// =============================================================== C ABI ====
using namespace mf;

struct mf_graph {
    int dev = 0;
    int32_t n = 0, s = 0, t = 0;
    int64_t m = 0, A = 0;
    int32_t cap_limit = 0;
    int kc = 1;
    long long max_iters = 0;
    unsigned long long time_limit_ns = 0;
    int grid = 0, sms = 0;
    int max_grid = 0;   // one full wave of co-resident CTAs
    mf_options opt{};
    DevGraph dg{};
    std::vector<void *> owned;
    std::vector<size_t> owned_bytes;
    int *b_ids = nullptr, *b_caps = nullptr, *b_newc = nullptr, *b_dlt = nullptr;
    int64_t b_cap = 0;
    unsigned char *side_buf = nullptr;
    bool solved = false;
    int policy = MF_POLICY_FIXED;
    float *params = nullptr;   // policy network parameters on the device
    int max_deg = 0;
    cudaStream_t last = nullptr;
    // a renumbered graph (mf_build.cpp): the resident arrays are in the
    // library's own vertex ids, everything that crosses the C ABI in the
    // input's (s, t above too)
    std::vector<int32_t> ord, inv;   // input id of each vertex, and the inverse (empty: not renumbered)
    int *d_inv = nullptr;            // inv on the device
    HostArray<int32_t> ext_row, arc_at;   // the arcs in the input's order, made when first asked for
    int *d_arc_at = nullptr;                // and on the device, for exports to device buffers, where it fits
};

namespace {

thread_local std::string g_last_error;

// Per-device set-up of the allocation-free solve.
constexpr int kNoAllocMaxDevices = 64;
struct NoAllocDevice {
    unsigned char *base = nullptr;   // device address of g_noalloc_scratch
    int grid = 0;
    cudaError_t err = cudaSuccess;
};
NoAllocDevice g_noalloc_dev[kNoAllocMaxDevices];
std::once_flag g_noalloc_once[kNoAllocMaxDevices];

int set_err(int code, const std::string &msg) {
    g_last_error = msg;
    return code;
}

// k_solve takes kDynSmem bytes of dynamic shared memory (above the default
// 48 KB limit): both instances get the attribute once per device, before
// their first occupancy query or launch on it.
std::once_flag g_smem_once[kNoAllocMaxDevices];
cudaError_t g_smem_err[kNoAllocMaxDevices];

cudaError_t solve_kernels_prepare(int dev) {
    if (dev < 0 || dev >= kNoAllocMaxDevices) return cudaErrorInvalidDevice;
    std::call_once(g_smem_once[dev], [dev]() {
        cudaError_t e = cudaFuncSetAttribute(k_solve<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_solve<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmem);
        g_smem_err[dev] = e;
    });
    return g_smem_err[dev];
}

#define MF_CUDA(call)                                                                       \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess)                                                              \
            return set_err(MF_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_));   \
    } while (0)

void *dalloc(mf_graph *g, size_t bytes) {
    if (bytes == 0) bytes = 16;
    void *p = nullptr;
    if (g->opt.alloc) {
        p = g->opt.alloc(bytes, g->opt.alloc_ctx);
    } else if (cudaMalloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        p = nullptr;
    }
    return p;
}

void dfree(mf_graph *g, void *p) {
    if (!p) return;
    if (g->opt.free) g->opt.free(p, g->opt.alloc_ctx);
    else cudaFree(p);
}

template <class T>
T *dnew(mf_graph *g, size_t count) {
    T *p = static_cast<T *>(dalloc(g, count * sizeof(T)));
    if (p) {
        g->owned.push_back(p);
        g->owned_bytes.push_back(count * sizeof(T));
    }
    return p;
}

// Hub items are read 16 bytes at a time; an allocator callback may return
// blocks of any alignment.
HubItem *dnew_hub_items(mf_graph *g, size_t count) {
    const uintptr_t p = reinterpret_cast<uintptr_t>(dnew<HubItem>(g, count + 1));   // 0: failed, stays 0
    return reinterpret_cast<HubItem *>((p + 15) & ~uintptr_t(15));
}

void dforget(mf_graph *g, void *p) {
    for (size_t i = 0; i < g->owned.size(); ++i)
        if (g->owned[i] == p) {
            g->owned.erase(g->owned.begin() + long(i));
            g->owned_bytes.erase(g->owned_bytes.begin() + long(i));
            return;
        }
}

bool is_device_ptr(const void *p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice;
}

template <class T>
int host_copy(const T *src, size_t count, std::vector<T> &dst, const T **out) {
    if (is_device_ptr(src)) {
        dst.resize(count);
        if (count) MF_CUDA(cudaMemcpy(dst.data(), src, count * sizeof(T), cudaMemcpyDeviceToHost));
        *out = dst.data();
    } else {
        *out = src;
    }
    return MF_OK;
}

int read_ctl(mf_graph *g, Ctl *out, size_t bytes = sizeof(Ctl)) {
    MF_CUDA(cudaSetDevice(g->dev));
    MF_CUDA(cudaMemcpyAsync(out, g->dg.ctl, bytes, cudaMemcpyDeviceToHost, g->last));
    MF_CUDA(cudaStreamSynchronize(g->last));
    return MF_OK;
}

// Where the search changes hands (see k_solve).
//  alpha      bottom-up pays early where a vertex finds a parent soon: in a
//             renumbered graph, whose rows begin with the likely parents, and
//             where rows are short (1023 x 769 grid, degree 8, its searches 256
//             us with 14, 297 with 4).  Long rows of alike heads are mostly read
//             whole, and anything below 14 does (unit assignment graph of degree
//             18, alpha 14 / 8 / 4 / 3 / 2: 1.33 / 1.10 / 1.21 / 1.14 / 1.17 ms a
//             batch, runs of one value 5 % apart).  On grids of longer rows it
//             does not matter: 6-connected 128^3 (10 arcs a vertex, push-pull)
//             2.45 / 2.30 / 2.53 / 2.40 / 2.35, 8-connected 512^2 (12) 2.92 / 3.04 /
//             3.11 / 2.94 / 2.95, 26-connected 64^3 (30, push-pull) 2.45 / 2.32 /
//             2.45 / 2.68 / 2.49.
//  solo_arcs  one CTA keeps up with a thin wave of short rows (2048^2 grid: 4
//             us a level against 7.5 on the whole grid), less so with long
//             rows: the tails of a power-law search mostly lead back (RMAT-20
//             static solve with 8192 / 4096 / 2048: 2.33 / 2.28 / 2.23 ms), and
//             an assignment graph's levels are written out arc by arc (8192 /
//             2048: 4,777 + 3,483 vertices 267 / 197 us, 6,551 + 2,539 263 /
//             215, 2^18 + 2^18 1.14 / 1.13 ms).
void search_rules(DevGraph &D, bool renumbered) {
    const bool soon = renumbered || D.A <= 8LL * D.n;   // a parent is found soon
    D.alpha = soon ? 14 : 3;
    D.bu_long = !soon;
    D.solo_arcs = !renumbered && D.A <= 8LL * D.n ? int(kSoloArcs) : 2048;
}

// CTAs of a graph whose options leave the choice: one per 1,536 arcs or per
// 4,096 vertices, whichever are more, at least four, at most one full wave.  A
// small graph does not fill the chip's warps, and every barrier waits for all
// CTAs.  (A server's grids for small batches are shares of this, down to one.)
// For the arcs, a solve or a recompute, in which every vertex may be active, sets
// the line.  Measured per batch with one CTA per 6,144 / 1,536 arcs / full wave:
// recompute of a 1,507-vertex graph 217 / 210 / 227 us, RMAT-13 push-pull 608 /
// 477 / 562, unit assignment 6,869 + 4,497 737 / 305 / 332, solve of a 113 x 160
// grid 932 / 646 / 632; repairs of the same kinds 79 / 81 / 81, 549 / 393 / 396,
// 314 / 296 / 319.  The vertices count where arcs are few: the sweeps over all
// vertices (heights, cut sides, final sums) then set the time.  Per batch, data-driven / push-pull, of 2^20 vertices and 5,000 edges with 5,
// 38, 76, 152 CTAs: 182 / 469, 105 / 167, 95 / 146, 91 / 137 us; of 200,000 and
// 20,000 with 4, 25, 38, 152: 93 / 172, 88 / 115, 83 / 109, 80 / 105; of 50,000
// and 10,000 the same from 10 on.
int auto_grid(int full, int64_t arcs, int32_t n) {
    const int64_t want = std::max(arcs / 1536, int64_t(n) / 4096);
    return int(std::max<int64_t>(std::min(full, 4), std::min<int64_t>(full, want)));
}

int launch(mf_graph *g, const Job &job, cudaStream_t st) {
    DevGraph dg = g->dg;
    Job jb = job;
    jb.st = job.kind == JOB_REFRESH ? g->dg.ctl->st_aux : g->dg.ctl->st;
    jb.debug = g->opt.debug_checks != 0;
    jb.trace = job.kind == JOB_REFRESH ? nullptr : g->dg.trace;
    void *args[] = {&dg, &jb};
    // a push-pull graph keeps its cut exact (every job ends on a BFS) and
    // solves from zero flow by static push-pull
    if (g->opt.mode == MF_MODE_PUSH_PULL) {
        jb.exact_exit = 1;
        jb.sink_sat = 1;
    }
    const void *fn = job.pp ? (const void *)k_solve<true> : (const void *)k_solve<false>;
    cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(g->grid), dim3(kBlock), args, kDynSmem, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_err(MF_ECUDA, std::string("cooperative launch: ") + cudaGetErrorString(e));
    }
    g->last = st;
    return MF_OK;
}

int launch_policy(mf_graph *g, int64_t k, const int *ids, const int *caps, int flags, cudaStream_t st) {
    PolicyJob pj{};
    pj.k = int(k);
    pj.flags = flags;
    pj.mode = g->policy;
    pj.kc_plain = g->kc;
    pj.max_deg = g->max_deg;
    pj.ids = ids;
    pj.caps = caps;
    pj.params = g->params;
    pj.gmode = g->opt.mode;
    pj.pp_ok = g->opt.mode == MF_MODE_PUSH_PULL;
    cudaGetLastError();   // an earlier, unrelated failure of this thread is not this launch's
    k_policy<<<kPolicyCtasPerSlot * g->grid, 256, 0, st>>>(g->dg, pj);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_err(MF_ECUDA, std::string("policy launch: ") + cudaGetErrorString(e));
    return MF_OK;
}

int ensure_batch_capacity(mf_graph *g, int64_t k, cudaStream_t st) {
    if (k <= g->b_cap) return MF_OK;
    int64_t want = std::max<int64_t>(k, std::max<int64_t>(1024, g->b_cap * 2));
    MF_CUDA(cudaStreamSynchronize(st));
    if (g->last && g->last != st) MF_CUDA(cudaStreamSynchronize(g->last));
    int *ptrs[4] = {g->b_ids, g->b_caps, g->b_newc, g->b_dlt};
    for (int *p : ptrs) {
        if (!p) continue;
        dfree(g, p);
        dforget(g, p);
    }
    g->b_ids = dnew<int>(g, size_t(want));
    g->b_caps = dnew<int>(g, size_t(want));
    g->b_newc = dnew<int>(g, size_t(want));
    g->b_dlt = dnew<int>(g, size_t(want));
    if (!g->b_ids || !g->b_caps || !g->b_newc || !g->b_dlt) {
        g->b_cap = 0;
        return set_err(MF_ENOMEM, "batch staging allocation failed");
    }
    g->b_cap = want;
    return MF_OK;
}

int gather_blocks(const mf_graph *g, long long count) {
    return int(std::max<long long>(1, std::min<long long>(g->sms * 8, (count + 255) / 256)));
}

// Copy host memory to the device before anything that follows on the graph's
// stream.  (A plain cudaMemcpy runs on the legacy stream and may return with
// the transfer from pageable memory still under way; a non-blocking stream
// does not wait for it.)
int upload(mf_graph *g, void *dst, const void *src, size_t bytes) {
    MF_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, g->last));
    MF_CUDA(cudaStreamSynchronize(g->last));
    return MF_OK;
}

// Fill ext_row / arc_at of a renumbered graph.
int need_external_arcs(mf_graph *g) {
    if (g->ord.empty() || !g->ext_row.empty()) return MF_OK;
    try {
        HostArray<int32_t> row(size_t(g->n) + 1), head(size_t(g->A)), ext_row(size_t(g->n) + 1), at(size_t(g->A));
        MF_CUDA(cudaMemcpy(row.data(), g->dg.row, row.size() * 4, cudaMemcpyDeviceToHost));
        if (g->A) MF_CUDA(cudaMemcpy(head.data(), g->dg.head, head.size() * 4, cudaMemcpyDeviceToHost));
        external_arcs(g->n, row.data(), head.data(), g->ord.data(), g->inv.data(), ext_row.data(), at.data());
        g->ext_row = std::move(ext_row);
        g->arc_at = std::move(at);
    } catch (const std::bad_alloc &) {
        return set_err(MF_ENOMEM, "host allocation");
    }
    return MF_OK;
}

// arc_at on the device too, where it fits (a caller that finds d_arc_at null
// permutes on the host).
int need_arc_index(mf_graph *g) {
    if (g->d_arc_at || g->A == 0) return MF_OK;
    int *at = dnew<int>(g, size_t(g->A));
    if (!at) return MF_OK;
    const int rc = upload(g, at, g->arc_at.data(), size_t(g->A) * 4);
    if (rc == MF_OK) {
        g->d_arc_at = at;   // (never an index that is not there)
    } else {
        dforget(g, at);
        dfree(g, at);
    }
    return rc;
}

// Make h the exact BFS heights of the current state (a no-op on the device
// when they are exact already), on the graph's last stream.
int refresh_heights(mf_graph *g) {
    Job j{};
    j.kind = JOB_REFRESH;
    j.exact_exit = 1;
    j.kc = g->kc;
    j.mode = g->opt.mode;
    j.max_iters = g->max_iters;
    j.time_limit_ns = g->time_limit_ns;
    return launch(g, j, g->last);
}

int status_to_code(mf_graph *g, const Ctl &c) {
    if (c.status & ST_CHECK) {
        g->solved = false;
        static const char *kinds[] = {"?", "list entry out of range", "excess differs from the net inflow",
                                      "residual pair or mirror inconsistent"};
        const long long kind = c.chk_where >> 40;
        long long where = c.chk_where & 0xffffffffffll;
        // a renumbered graph's vertex or arc by the caller's numbers
        if (!g->ord.empty() && kind == 3 && where < g->A && need_external_arcs(g) == MF_OK)
            where = std::find(g->arc_at.begin(), g->arc_at.end(), int32_t(where)) - g->arc_at.begin();
        else if (!g->ord.empty() && (kind == 1 || kind == 2) && where < g->n)
            where = g->ord[size_t(where)];
        return set_err(MF_ECHECK, std::string("debug check failed: ") + kinds[kind >= 1 && kind <= 3 ? kind : 0] +
                                      " (index " + std::to_string(where) + ")");
    }
    if (c.status & ST_STICKY) {
        g->solved = false;
        return set_err(MF_ETIMEOUT, (c.status & ST_WAIT)   ? "device wait reached its time limit"
                                    : (c.status & ST_TIME) ? "device loop reached its wall-clock limit"
                                                           : "device loop reached max_iters");
    }
    if (c.status & ST_EINVAL) {
        int zero = c.status & ~ST_EINVAL;
        MF_CUDA(cudaMemcpyAsync(&g->dg.ctl->status, &zero, sizeof(int), cudaMemcpyHostToDevice, g->last));
        MF_CUDA(cudaStreamSynchronize(g->last));
        return set_err(MF_EINVAL, "batch rejected on the device (edge id out of range, duplicate id or capacity out of range)");
    }
    return MF_OK;
}

}  // namespace

extern "C" {

const char *mf_version(void) { return "0.1.0"; }

const char *mf_strerror(int code) {
    switch (code) {
        case MF_OK: return "ok";
        case MF_EINVAL: return "invalid argument";
        case MF_ENOMEM: return "out of memory";
        case MF_ECUDA: return "CUDA error";
        case MF_ENOTSOLVED: return "graph not solved";
        case MF_ETIMEOUT: return "device loop timeout";
        case MF_ECHECK: return "device consistency check failed";
        default: return "unknown error";
    }
}

const char *mf_last_error(void) { return g_last_error.c_str(); }

int mf_options_default(mf_options *opt) {
    if (!opt) return MF_EINVAL;
    std::memset(opt, 0, sizeof(*opt));
    opt->mode = MF_MODE_DATA_DRIVEN;
    return MF_OK;
}

int mf_bicsr_host(int32_t n, int64_t m, const int64_t *row_ptr, const int32_t *col, const int32_t *cap,
                  int32_t s, int32_t t, int64_t *arcs, int64_t *arc_row, int32_t *head, int32_t *rev,
                  int32_t *arc_cap, int32_t *arc_of_edge, int32_t *cap_limit) {
    if (!row_ptr || (m > 0 && (!col || !cap)) || !arcs) return set_err(MF_EINVAL, "null argument");
    HostBiCSR G;
    int rc = build_bicsr(n, m, row_ptr, col, cap, s, t, false, &G);
    if (rc) return set_err(rc == 2 ? MF_ENOMEM : MF_EINVAL, "graph rejected by the Bi-CSR builder");
    *arcs = G.arcs;
    if (arc_row) for (int32_t u = 0; u <= n; ++u) arc_row[u] = G.row[size_t(u)];
    if (head) std::copy(G.head.begin(), G.head.end(), head);
    if (rev) std::copy(G.rev.begin(), G.rev.end(), rev);
    if (arc_cap) std::copy(G.cap.begin(), G.cap.end(), arc_cap);
    if (arc_of_edge) std::copy(G.arc_of_edge.begin(), G.arc_of_edge.end(), arc_of_edge);
    if (cap_limit) *cap_limit = G.cap_limit;
    return MF_OK;
}

int mf_create(int32_t n, int64_t m, const int64_t *row_ptr, const int32_t *col, const int32_t *cap,
              int32_t s, int32_t t, const mf_options *opt, void *stream, mf_graph **out) {
    if (!out || !row_ptr || (m > 0 && (!col || !cap))) return set_err(MF_EINVAL, "null argument");
    *out = nullptr;
    if (n < 2 || m < 0 || m >= INT32_MAX || s < 0 || t < 0 || s >= n || t >= n || s == t)
        return set_err(MF_EINVAL, "bad sizes or terminals");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    std::vector<int64_t> hrow;
    std::vector<int32_t> hcol, hcap;
    const int64_t *prow;
    const int32_t *pcol = col, *pcap = cap;
    int rc = host_copy(row_ptr, size_t(n) + 1, hrow, &prow);
    if (rc) return rc;
    if (m > 0) {
        if ((rc = host_copy(col, size_t(m), hcol, &pcol))) return rc;
        if ((rc = host_copy(cap, size_t(m), hcap, &pcap))) return rc;
    }
    HostBiCSR H;
    rc = build_bicsr(n, m, prow, pcol, pcap, s, t, true, &H);
    if (rc) return set_err(rc == 2 ? MF_ENOMEM : MF_EINVAL, "graph rejected by the Bi-CSR builder");

    mf_graph *g = new (std::nothrow) mf_graph();
    if (!g) return set_err(MF_ENOMEM, "host allocation");
    if (opt) g->opt = *opt;
    else mf_options_default(&g->opt);
    auto fail = [&](int code, const std::string &msg) {
        mf_destroy(g);
        return set_err(code, msg);
    };
    if ((g->opt.alloc == nullptr) != (g->opt.free == nullptr)) return fail(MF_EINVAL, "alloc and free must both be set");
    if (g->opt.mode != MF_MODE_DATA_DRIVEN && g->opt.mode != MF_MODE_TOPOLOGY && g->opt.mode != MF_MODE_PUSH_PULL)
        return fail(MF_EINVAL, "unknown mode");
    if (cudaGetDevice(&g->dev) != cudaSuccess) return fail(MF_ECUDA, "no CUDA device");
    int coop = 0;
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, g->dev);
    cudaDeviceGetAttribute(&g->sms, cudaDevAttrMultiProcessorCount, g->dev);
    if (!coop) return fail(MF_ECUDA, "device does not support cooperative launch");
    int per_sm = 0;
    int per_sm_pp = 0;
    if (solve_kernels_prepare(g->dev) != cudaSuccess) return fail(MF_ECUDA, "shared-memory attribute of k_solve");
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_solve<false>, kBlock, kDynSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_pp, k_solve<true>, kBlock, kDynSmem) != cudaSuccess)
        return fail(MF_ECUDA, "occupancy query failed");
    per_sm = std::min(per_sm, per_sm_pp);
    if (per_sm < 1)
        return fail(MF_ECUDA, "occupancy query failed");
    g->max_grid = per_sm * g->sms;
    g->grid = g->opt.grid_blocks > 0 ? std::min(g->max_grid, int(g->opt.grid_blocks)) : auto_grid(g->max_grid, H.arcs, n);

    g->n = n; g->m = m; g->A = H.arcs; g->s = s; g->t = t;
    g->cap_limit = H.cap_limit;
    g->max_deg = H.max_deg;
    int64_t avg = (m + n / 2) / n;
    g->kc = g->opt.kernel_cycles > 0 ? g->opt.kernel_cycles : int(std::max<int64_t>(1, avg));
    g->max_iters = g->opt.max_iters > 0 ? g->opt.max_iters : 4LL * n + 1000;
    g->time_limit_ns = 1000000ull * (unsigned long long)(g->opt.time_limit_ms > 0 ? g->opt.time_limit_ms : 60000);

    const size_t A = size_t(std::max<int64_t>(H.arcs, 1)), N = size_t(n), M = size_t(std::max<int64_t>(m, 1));
    DevGraph &D = g->dg;
    D.n = n; D.s = s; D.t = t; D.m = int(m); D.A = H.arcs; D.cap_limit = H.cap_limit;
    if (!H.inv.empty()) {
        D.s = H.inv[size_t(s)];
        D.t = H.inv[size_t(t)];
        try {
            g->ord.assign(H.ord.begin(), H.ord.end());
            g->inv.assign(H.inv.begin(), H.inv.end());
        } catch (const std::bad_alloc &) {
            return fail(MF_ENOMEM, "host allocation");
        }
        if (!(g->d_inv = dnew<int>(g, N))) return fail(MF_ENOMEM, "device allocation failed");
    }
    int *row = dnew<int>(g, N + 1), *head = dnew<int>(g, A), *rev = dnew<int>(g, A), *aoe = dnew<int>(g, M);
    D.row = row; D.head = head; D.rev = rev; D.arc_of_edge = aoe;
    unsigned char *est = dnew<unsigned char>(g, M);
    D.edge_st = est;
    D.cap = dnew<int>(g, A); D.r = dnew<int>(g, A); D.rr = dnew<int>(g, A);
    D.h = dnew<int>(g, N); D.e = dnew<long long>(g, N);
    D.cap_edge = dnew<int>(g, M); D.stamp = dnew<unsigned>(g, M);
    D.qb0 = dnew<int>(g, N + 32); D.qb1 = dnew<int>(g, N); D.wl = dnew<int>(g, N);
    D.cb = dnew<int2>(g, size_t(std::max<int64_t>(H.chunk_items, 1)));
    const size_t NH = size_t(std::max<int64_t>(H.hubs, 1));
    D.hl = dnew<int>(g, NH);
    D.hl2 = dnew<int>(g, NH);
    D.hkey = dnew<int>(g, 2 * NH);
    D.hrem = dnew<long long>(g, NH);
    D.hlist0 = dnew<int>(g, NH);
    D.hlist1 = dnew<int>(g, NH);
    D.hit0 = dnew_hub_items(g, size_t(std::max<int64_t>(H.hub_chunk_items, 1)));
    D.hit1 = dnew_hub_items(g, size_t(std::max<int64_t>(H.hub_chunk_items, 1)));
    D.hikey = dnew<int>(g, size_t(std::max<int64_t>(H.hub_chunk_items, 1)));
    D.hri = dnew<int2>(g, size_t(std::max<int64_t>(H.hub_chunk_items, 1)));
    D.astamp = dnew<unsigned>(g, N);
    D.rstamp = dnew<unsigned>(g, N);
    D.rl = dnew<int>(g, N);
    D.part = g->opt.mode == MF_MODE_PUSH_PULL ? dnew<unsigned char>(g, N) : nullptr;
    D.qc = int(std::max<size_t>(N, 1024));
    D.aq = dnew<unsigned long long>(g, size_t(D.qc));
    D.ctl = dnew<Ctl>(g, 1);
    g->side_buf = dnew<unsigned char>(g, N);
    // an allocator callback may hand out blocks without 16-byte alignment:
    // the staging copies then fall back to plain loads
    auto al16 = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
    search_rules(D, !g->ord.empty());
    D.al16 = al16(D.head) && al16(D.r) && al16(D.rr);
    if (!row || !head || !rev || !aoe || !est || !D.cap || !D.r || !D.rr || !D.h || !D.e || !D.cap_edge || !D.stamp ||
        !D.qb0 || !D.qb1 || !D.wl || !D.cb || !D.ctl || !g->side_buf || !D.hl || !D.hkey ||
        !D.hrem || !D.hlist0 || !D.hlist1 || !D.hit0 || !D.hit1 || !D.hikey || !D.hl2 || !D.hri || !D.astamp ||
        !D.rstamp || !D.rl || !D.aq)
        return fail(MF_ENOMEM, "device allocation failed");
    auto up = [&](void *dst, const void *src, size_t bytes) {
        return bytes ? cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st) : cudaSuccess;
    };
    if (up(row, H.row.data(), (N + 1) * 4) || up(head, H.head.data(), size_t(H.arcs) * 4) ||
        up(rev, H.rev.data(), size_t(H.arcs) * 4) || up(aoe, H.arc_of_edge.data(), size_t(m) * 4) ||
        up(est, H.edge_st.data(), size_t(m)) || (g->d_inv && up(g->d_inv, H.inv.data(), N * 4)) ||
        up(D.cap, H.cap.data(), size_t(H.arcs) * 4) || up(D.cap_edge, pcap, size_t(m) * 4) ||
        cudaMemsetAsync(D.stamp, 0, M * 4, st) || cudaMemsetAsync(D.ctl, 0, sizeof(Ctl), st) ||
        cudaMemsetAsync(D.aq, 0, size_t(D.qc) * 8, st) ||
        cudaMemsetAsync(D.e, 0, N * 8, st) || cudaMemsetAsync(D.h, 0, N * 4, st) ||
        cudaMemsetAsync(D.astamp, 0, N * 4, st) || cudaMemsetAsync(D.rstamp, 0, N * 4, st) ||
        cudaMemsetAsync(D.r, 0, A * 4, st) || cudaMemsetAsync(D.rr, 0, A * 4, st) ||
        cudaStreamSynchronize(st)) {
        cudaGetLastError();
        return fail(MF_ECUDA, "upload failed");
    }
    g->last = st;
    *out = g;
    return MF_OK;
}

int mf_cap_limit(const mf_graph *g, int32_t *out) {
    if (!g || !out) return MF_EINVAL;
    *out = g->cap_limit;
    return MF_OK;
}

int mf_sizes(const mf_graph *g, int32_t *n, int64_t *m, int64_t *arcs) {
    if (!g) return MF_EINVAL;
    if (n) *n = g->n;
    if (m) *m = g->m;
    if (arcs) *arcs = g->A;
    return MF_OK;
}

int mf_solve(mf_graph *g, void *stream) {
    if (!g) return MF_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    MF_CUDA(cudaSetDevice(g->dev));
    MF_CUDA(cudaMemsetAsync(g->dg.ctl, 0, sizeof(Ctl), st));
    MF_CUDA(cudaMemsetAsync(g->dg.stamp, 0, size_t(std::max<int64_t>(g->m, 1)) * 4, st));
    MF_CUDA(cudaMemsetAsync(g->dg.astamp, 0, size_t(g->n) * 4, st));
    MF_CUDA(cudaMemsetAsync(g->dg.rstamp, 0, size_t(g->n) * 4, st));
    // a launch that gave up inside a PushRelabel phase may have left queue entries
    MF_CUDA(cudaMemsetAsync(g->dg.aq, 0, size_t(g->dg.qc) * 8, st));
    Job j{};
    j.kind = JOB_SOLVE;
    j.kc = g->kc;
    j.mode = g->opt.mode;
    j.max_iters = g->max_iters;
    j.time_limit_ns = g->time_limit_ns;
    int rc = launch(g, j, st);
    if (rc == MF_OK) g->solved = true;
    return rc;
}

int mf_apply_updates(mf_graph *g, int64_t k, const int32_t *edge_id, const int32_t *new_cap, int32_t flags,
                     void *stream) {
    if (!g) return MF_EINVAL;
    if (!g->solved) return set_err(MF_ENOTSOLVED, "call mf_solve first");
    if (k < 0 || k > g->m || (k > 0 && (!edge_id || !new_cap)))
        return set_err(MF_EINVAL, "bad batch size or null batch pointer");
    if (flags & ~(MF_DEVICE_PTRS | MF_DELTA | MF_RECOMPUTE)) return set_err(MF_EINVAL, "unknown flags");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    MF_CUDA(cudaSetDevice(g->dev));
    int rc = ensure_batch_capacity(g, std::max<int64_t>(k, 1), st);
    if (rc) return rc;
    const int *ids = edge_id, *caps = new_cap;
    if (!(flags & MF_DEVICE_PTRS) && k > 0) {
        MF_CUDA(cudaMemcpyAsync(g->b_ids, edge_id, size_t(k) * 4, cudaMemcpyHostToDevice, st));
        MF_CUDA(cudaMemcpyAsync(g->b_caps, new_cap, size_t(k) * 4, cudaMemcpyHostToDevice, st));
        ids = g->b_ids;
        caps = g->b_caps;
    }
    Job j{};
    j.kind = (flags & MF_RECOMPUTE) ? JOB_RECOMPUTE : JOB_REPAIR;
    if (!(flags & MF_RECOMPUTE) && g->policy != MF_POLICY_FIXED) {
        rc = launch_policy(g, k, ids, caps, flags, st);
        if (rc) return rc;
        j.kind = JOB_AUTO;
    }
    j.k = int(k);
    j.flags = flags;
    j.kc = g->kc;
    j.mode = g->opt.mode;
    j.pp = g->opt.mode == MF_MODE_PUSH_PULL;
    j.max_iters = g->max_iters;
    j.time_limit_ns = g->time_limit_ns;
    j.ids = ids;
    j.caps = caps;
    j.newc = g->b_newc;
    j.dlt = g->b_dlt;
    return launch(g, j, st);
}

int mf_apply_updates_dev(mf_graph *g, const int32_t *k_dev, int64_t k_max, const int32_t *edge_id,
                         const int32_t *new_cap, int32_t flags, void *stream) {
    if (!g || !k_dev || !edge_id || !new_cap) return set_err(MF_EINVAL, "null argument");
    if (!g->solved) return set_err(MF_ENOTSOLVED, "call mf_solve first");
    if (k_max < 0 || k_max > g->m) return set_err(MF_EINVAL, "bad k_max");
    if (flags & ~(MF_DELTA | MF_RECOMPUTE | MF_DEVICE_PTRS)) return set_err(MF_EINVAL, "unknown flags");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    MF_CUDA(cudaSetDevice(g->dev));
    if (g->b_cap < std::max<int64_t>(k_max, 1)) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        MF_CUDA(cudaStreamIsCapturing(st, &cs));
        if (cs != cudaStreamCaptureStatusNone)
            return set_err(MF_EINVAL, "batch staging must be sized (k_max) before stream capture");
        int rc = ensure_batch_capacity(g, std::max<int64_t>(k_max, 1), st);
        if (rc) return rc;
    }
    Job j{};
    j.kind = (flags & MF_RECOMPUTE) ? JOB_RECOMPUTE : JOB_REPAIR;
    if (!(flags & MF_RECOMPUTE) && g->policy != MF_POLICY_FIXED) {
        PolicyJob pj{};
        pj.k = 0;
        pj.k_dev = k_dev;
        pj.flags = flags & MF_DELTA;
        pj.mode = g->policy;
        pj.kc_plain = g->kc;
        pj.max_deg = g->max_deg;
        pj.ids = edge_id;
        pj.caps = new_cap;
        pj.params = g->params;
        pj.gmode = g->opt.mode;
        pj.pp_ok = g->opt.mode == MF_MODE_PUSH_PULL;
        cudaGetLastError();   // an earlier, unrelated failure of this thread is not this launch's
        k_policy<<<kPolicyCtasPerSlot * g->grid, 256, 0, st>>>(g->dg, pj);
        MF_CUDA(cudaGetLastError());
        j.kind = JOB_AUTO;
    }
    j.k = 0;
    j.k_dev = k_dev;
    j.flags = flags;
    j.kc = g->kc;
    j.mode = g->opt.mode;
    j.pp = g->opt.mode == MF_MODE_PUSH_PULL;
    j.max_iters = g->max_iters;
    j.time_limit_ns = g->time_limit_ns;
    j.ids = edge_id;
    j.caps = new_cap;
    j.newc = g->b_newc;
    j.dlt = g->b_dlt;
    return launch(g, j, st);
}

int mf_set_stream(mf_graph *g, void *stream) {
    if (!g) return MF_EINVAL;
    MF_CUDA(cudaSetDevice(g->dev));
    if (g->last) MF_CUDA(cudaStreamSynchronize(g->last));
    g->last = static_cast<cudaStream_t>(stream);
    return MF_OK;
}

int mf_flow_value_async(mf_graph *g, int64_t *result, void *stream) {
    if (!g || !result) return MF_EINVAL;
    MF_CUDA(cudaSetDevice(g->dev));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    MF_CUDA(cudaMemcpyAsync(result, g->dg.ctl, 16, cudaMemcpyDeviceToHost, st));
    return MF_OK;
}

int mf_device_bytes(const mf_graph *g, int64_t *bytes) {
    if (!g || !bytes) return MF_EINVAL;
    int64_t b = 0;
    for (size_t x : g->owned_bytes) b += int64_t(x);
    *bytes = b;
    return MF_OK;
}

int mf_grid_blocks(const mf_graph *g, int32_t *blocks) {
    if (!g || !blocks) return MF_EINVAL;
    *blocks = g->grid;
    return MF_OK;
}

int mf_set_grid_blocks(mf_graph *g, int32_t blocks) {
    if (!g || blocks < 1) return set_err(MF_EINVAL, "null graph or fewer than one CTA");
    g->grid = std::min(int(blocks), g->max_grid);
    return MF_OK;
}

int mf_sync(mf_graph *g) {
    if (!g) return MF_EINVAL;
    Ctl c;
    int rc = read_ctl(g, &c);
    if (rc) return rc;
    return status_to_code(g, c);
}

int mf_flow_value(mf_graph *g, int64_t *out) {
    if (!g || !out) return MF_EINVAL;
    Ctl c;
    int rc = read_ctl(g, &c, 16);   // status, batch_err, flow
    if (rc) return rc;
    if (c.status & ST_CHECK) {      // where the check failed, for the message
        rc = read_ctl(g, &c);
        if (rc) return rc;
    }
    rc = status_to_code(g, c);
    if (rc == MF_ETIMEOUT || rc == MF_ECHECK) return rc;
    if (!g->solved) return set_err(MF_ENOTSOLVED, "call mf_solve first");
    *out = c.flow;
    return rc;
}

int mf_min_cut(mf_graph *g, uint8_t *side, int32_t flags) {
    if (!g || !side) return MF_EINVAL;
    if (!g->solved) return set_err(MF_ENOTSOLVED, "call mf_solve first");
    MF_CUDA(cudaSetDevice(g->dev));
    int rc = refresh_heights(g);
    if (rc) return rc;
    unsigned char *dst = (flags & MF_DEVICE_PTRS) ? side : g->side_buf;
    int blocks = std::max(1, std::min(g->sms * 4, (g->n + 255) / 256));
    cudaGetLastError();   // an earlier, unrelated failure of this thread is not this launch's
    k_cut_side<<<blocks, 256, 0, g->last>>>(g->dg.h, g->n, g->d_inv, dst);
    MF_CUDA(cudaGetLastError());
    if (!(flags & MF_DEVICE_PTRS))
        MF_CUDA(cudaMemcpyAsync(side, g->side_buf, size_t(g->n), cudaMemcpyDeviceToHost, g->last));
    return mf_sync(g);
}

int mf_stats_get(mf_graph *g, mf_stats *out) {
    if (!g || !out) return MF_EINVAL;
    Ctl c;
    int rc = read_ctl(g, &c);
    if (rc) return rc;
    std::memset(out, 0, sizeof(*out));
    out->flow = c.flow;
    out->iterations = c.iters;
    out->bfs_levels = c.st[S_LEVELS];
    out->bfs_vertices = c.st[S_BFS_VERTS];
    out->bfs_arcs = c.st[S_BFS_ARCS];
    out->worklist = c.st[S_WL];
    out->pr_arcs = c.st[S_PR_ARCS];
    out->pushes = c.st[S_PUSH];
    out->relabels = c.st[S_RELABEL];
    out->ri_arcs = c.st[S_RI_ARCS];
    out->ri_moves = c.st[S_RI_MOVES];
    out->batch = c.st[S_BATCH];
    out->clamped = c.st[S_CLAMPED];
    out->resat_arcs = c.st[S_RESAT];
    out->n = g->n;
    out->m = g->m;
    out->arcs = g->A;
    out->t_batch_ns = c.st[S_T_BATCH];
    out->t_reset_ns = c.st[S_T_RESET];
    out->t_bfs_ns = c.st[S_T_BFS];
    out->t_pr_ns = c.st[S_T_PRW];
    out->t_hub_ns = c.st[S_T_HUB];
    out->t_ri_ns = c.st[S_T_RI];
    out->hub_cycles = c.st[S_HUB_CYCLES];
    out->barriers = c.st[S_BARRIERS];
    out->bfs_bottom_up_levels = c.st[S_BU_LEVELS];
    out->pr_rounds = c.st[S_ROUNDS];
    out->policy_kind = c.pol_kind == JOB_RECOMPUTE ? 1 : 0;
    out->policy_kernel_cycles = c.pol_kc;
    out->policy_fallback = c.pol_fallback;
    out->policy_mode = g->policy == MF_POLICY_LEARNED ? c.pol_mode : g->opt.mode;
    out->exit_kind = c.exit_kind;
    out->status = c.status;
    out->kernel_cycles = g->kc;
    out->grid_blocks = g->grid;
    out->block_threads = kBlock;
    return MF_OK;
}

int mf_export_graph(mf_graph *g, int64_t *arc_row, int32_t *head, int32_t *rev, int32_t *cap) {
    if (!g) return MF_EINVAL;
    MF_CUDA(cudaSetDevice(g->dev));
    MF_CUDA(cudaStreamSynchronize(g->last));
    if (!g->ord.empty()) {
        int rc = need_external_arcs(g);
        if (rc) return rc;
        if (arc_row) for (size_t i = 0; i < g->ext_row.size(); ++i) arc_row[i] = g->ext_row[i];
        try {
            HostArray<int32_t> tmp(static_cast<size_t>(g->A));
            if (cap && g->A) {
                MF_CUDA(cudaMemcpy(tmp.data(), g->dg.cap, tmp.size() * 4, cudaMemcpyDeviceToHost));
                gather_i32(tmp.data(), g->arc_at.data(), g->A, false, cap);
            }
            if (head && g->A) {
                MF_CUDA(cudaMemcpy(tmp.data(), g->dg.head, tmp.size() * 4, cudaMemcpyDeviceToHost));
                gather_i32(tmp.data(), g->arc_at.data(), g->A, false, head);
                gather_i32(g->ord.data(), head, g->A, false, head);
            }
            if (rev && g->A) {
                // the reverse arc's place in the input's order
                HostArray<int32_t> place(static_cast<size_t>(g->A));
                gather_i32(nullptr, g->arc_at.data(), g->A, true, place.data());
                MF_CUDA(cudaMemcpy(tmp.data(), g->dg.rev, tmp.size() * 4, cudaMemcpyDeviceToHost));
                gather_i32(tmp.data(), g->arc_at.data(), g->A, false, rev);
                gather_i32(place.data(), rev, g->A, false, rev);
            }
        } catch (const std::bad_alloc &) {
            return set_err(MF_ENOMEM, "host allocation");
        }
        return MF_OK;
    }
    if (arc_row) {
        std::vector<int32_t> row(size_t(g->n) + 1);
        MF_CUDA(cudaMemcpy(row.data(), g->dg.row, row.size() * 4, cudaMemcpyDeviceToHost));
        for (size_t i = 0; i < row.size(); ++i) arc_row[i] = row[i];
    }
    if (head && g->A) MF_CUDA(cudaMemcpy(head, g->dg.head, size_t(g->A) * 4, cudaMemcpyDeviceToHost));
    if (rev && g->A) MF_CUDA(cudaMemcpy(rev, g->dg.rev, size_t(g->A) * 4, cudaMemcpyDeviceToHost));
    if (cap && g->A) MF_CUDA(cudaMemcpy(cap, g->dg.cap, size_t(g->A) * 4, cudaMemcpyDeviceToHost));
    return MF_OK;
}

int mf_export_state(mf_graph *g, int32_t *r, int64_t *excess, int32_t *height, int32_t flags) {
    if (!g) return MF_EINVAL;
    MF_CUDA(cudaSetDevice(g->dev));
    if (height && g->solved) {
        int rc = refresh_heights(g);
        if (rc) return rc;
    }
    cudaMemcpyKind kind = (flags & MF_DEVICE_PTRS) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    if (!g->ord.empty()) {
        // in the input's order: gathered on the device into the caller's device
        // buffers, else (host buffers, or no room for arc_at) on the host
        if (r) {
            int rc = need_external_arcs(g);
            if (rc == MF_OK && (flags & MF_DEVICE_PTRS)) rc = need_arc_index(g);
            if (rc) return rc;
        }
        try {
            HostArray<int32_t> a, b;
            auto out32 = [&](int32_t *dst, const int *src, const auto &at, const int *d_at) -> int {
                const long long count = (long long)at.size();
                if (!dst || count == 0) return MF_OK;
                if ((flags & MF_DEVICE_PTRS) && d_at) {
                    k_gather<<<gather_blocks(g, count), 256, 0, g->last>>>(dst, src, d_at, count);
                    MF_CUDA(cudaGetLastError());
                    return MF_OK;
                }
                a.resize(at.size());
                MF_CUDA(cudaMemcpyAsync(a.data(), src, at.size() * 4, cudaMemcpyDeviceToHost, g->last));
                MF_CUDA(cudaStreamSynchronize(g->last));
                if (!(flags & MF_DEVICE_PTRS)) {
                    gather_i32(a.data(), at.data(), count, false, dst);
                    return MF_OK;
                }
                b.resize(at.size());
                gather_i32(a.data(), at.data(), count, false, b.data());
                return upload(g, dst, b.data(), at.size() * 4);
            };
            cudaGetLastError();   // an earlier, unrelated failure of this thread is not these launches'
            int rc = out32(r, g->dg.r, g->arc_at, g->d_arc_at);
            if (rc == MF_OK) rc = out32(height, g->dg.h, g->inv, g->d_inv);
            if (rc) return rc;
            if (excess && (flags & MF_DEVICE_PTRS)) {
                k_gather<<<gather_blocks(g, g->n), 256, 0, g->last>>>(reinterpret_cast<long long *>(excess), g->dg.e,
                                                                      g->d_inv, (long long)g->n);
                MF_CUDA(cudaGetLastError());
            } else if (excess) {
                HostArray<int64_t> e(static_cast<size_t>(g->n));
                MF_CUDA(cudaMemcpyAsync(e.data(), g->dg.e, e.size() * 8, cudaMemcpyDeviceToHost, g->last));
                MF_CUDA(cudaStreamSynchronize(g->last));
                for (int32_t v = 0; v < g->n; ++v) excess[v] = e[size_t(g->inv[size_t(v)])];
            }
        } catch (const std::bad_alloc &) {
            return set_err(MF_ENOMEM, "host allocation");
        }
        MF_CUDA(cudaStreamSynchronize(g->last));
        return MF_OK;
    }
    if (r && g->A) MF_CUDA(cudaMemcpyAsync(r, g->dg.r, size_t(g->A) * 4, kind, g->last));
    if (excess) MF_CUDA(cudaMemcpyAsync(excess, g->dg.e, size_t(g->n) * 8, kind, g->last));
    if (height) MF_CUDA(cudaMemcpyAsync(height, g->dg.h, size_t(g->n) * 4, kind, g->last));
    MF_CUDA(cudaStreamSynchronize(g->last));
    return MF_OK;
}

int mf_import_state(mf_graph *g, const int32_t *r, const int64_t *excess, const int32_t *height, int32_t flags) {
    if (!g || !r || !excess || !height) return MF_EINVAL;
    MF_CUDA(cudaSetDevice(g->dev));
    cudaMemcpyKind kind = (flags & MF_DEVICE_PTRS) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    MF_CUDA(cudaStreamSynchronize(g->last));
    if (!g->ord.empty()) {
        // given in the input's order: permuted on the host
        int rc = need_external_arcs(g);
        if (rc) return rc;
        const cudaMemcpyKind in = (flags & MF_DEVICE_PTRS) ? cudaMemcpyDeviceToHost : cudaMemcpyHostToHost;
        try {
            HostArray<int32_t> a(size_t(std::max<int64_t>(g->A, g->n))), b(a.size());
            HostArray<int64_t> x(static_cast<size_t>(g->n)), y(static_cast<size_t>(g->n));
            if (g->A) {
                MF_CUDA(cudaMemcpy(a.data(), r, size_t(g->A) * 4, in));
                gather_i32(a.data(), g->arc_at.data(), g->A, true, b.data());
                MF_CUDA(cudaMemcpy(g->dg.r, b.data(), size_t(g->A) * 4, cudaMemcpyHostToDevice));
            }
            MF_CUDA(cudaMemcpy(a.data(), height, size_t(g->n) * 4, in));
            gather_i32(a.data(), g->inv.data(), g->n, true, b.data());
            MF_CUDA(cudaMemcpy(g->dg.h, b.data(), size_t(g->n) * 4, cudaMemcpyHostToDevice));
            MF_CUDA(cudaMemcpy(x.data(), excess, size_t(g->n) * 8, in));
            for (int32_t v = 0; v < g->n; ++v) y[size_t(g->inv[size_t(v)])] = x[size_t(v)];
            MF_CUDA(cudaMemcpy(g->dg.e, y.data(), size_t(g->n) * 8, cudaMemcpyHostToDevice));
        } catch (const std::bad_alloc &) {
            return set_err(MF_ENOMEM, "host allocation");
        }
    } else {
        if (g->A) MF_CUDA(cudaMemcpy(g->dg.r, r, size_t(g->A) * 4, kind));
        MF_CUDA(cudaMemcpy(g->dg.e, excess, size_t(g->n) * 8, kind));
        MF_CUDA(cudaMemcpy(g->dg.h, height, size_t(g->n) * 4, kind));
    }
    long long flow = 0;
    try {
        // rebuild the mirror rr[a] = r[rev[a]] on the host side of the copy
        if (g->A) {
            HostArray<int32_t> hr(static_cast<size_t>(g->A)), hrev(hr.size()), hrr(hr.size());
            MF_CUDA(cudaMemcpy(hr.data(), g->dg.r, hr.size() * 4, cudaMemcpyDeviceToHost));
            MF_CUDA(cudaMemcpy(hrev.data(), g->dg.rev, hrev.size() * 4, cudaMemcpyDeviceToHost));
            gather_i32(hr.data(), hrev.data(), g->A, false, hrr.data());
            MF_CUDA(cudaMemcpy(g->dg.rr, hrr.data(), hrr.size() * 4, cudaMemcpyHostToDevice));
        }
        // value of the imported state: e(t) plus the deficits (Alg. 4, final sum)
        HostArray<int64_t> he(static_cast<size_t>(g->n));
        MF_CUDA(cudaMemcpy(he.data(), g->dg.e, he.size() * 8, cudaMemcpyDeviceToHost));
        const int32_t ds = g->dg.s, dt = g->dg.t;
        flow = he[size_t(dt)];
        for (int32_t v = 0; v < g->n; ++v)
            if (v != ds && v != dt && he[size_t(v)] < 0) flow += he[size_t(v)];
    } catch (const std::bad_alloc &) {
        return set_err(MF_ENOMEM, "host allocation");
    }
    MF_CUDA(cudaMemset(g->dg.ctl, 0, sizeof(Ctl)));
    MF_CUDA(cudaMemset(g->dg.stamp, 0, size_t(std::max<int64_t>(g->m, 1)) * 4));
    MF_CUDA(cudaMemset(g->dg.astamp, 0, size_t(g->n) * 4));
    MF_CUDA(cudaMemset(g->dg.rstamp, 0, size_t(g->n) * 4));
    MF_CUDA(cudaMemset(g->dg.aq, 0, size_t(g->dg.qc) * 8));
    MF_CUDA(cudaMemcpy(&g->dg.ctl->flow, &flow, sizeof(flow), cudaMemcpyHostToDevice));
    MF_CUDA(cudaDeviceSynchronize());
    g->solved = true;
    return MF_OK;
}

int mf_set_time_limit(mf_graph *g, int32_t time_limit_ms) {
    if (!g || time_limit_ms < 0) return set_err(MF_EINVAL, "null graph or negative time limit");
    g->opt.time_limit_ms = time_limit_ms;
    g->time_limit_ns = 1000000ull * (unsigned long long)(time_limit_ms > 0 ? time_limit_ms : 60000);
    return MF_OK;
}

void mf_destroy(mf_graph *g) {
    if (!g) return;
    cudaSetDevice(g->dev);
    if (g->last) cudaStreamSynchronize(g->last);
    cudaDeviceSynchronize();
    for (void *p : g->owned) dfree(g, p);
    delete g;
}

int mf_set_policy(mf_graph *g, int32_t mode, const float *params) {
    if (!g || mode < MF_POLICY_FIXED || mode > MF_POLICY_LEARNED) return MF_EINVAL;
    if (mode == MF_POLICY_LEARNED && !params && !g->params)
        return set_err(MF_EINVAL, "the learned policy needs network parameters");
    MF_CUDA(cudaSetDevice(g->dev));
    if (params) {
        if (!g->params) g->params = dnew<float>(g, mlp::kTotal);
        if (!g->params) return set_err(MF_ENOMEM, "policy parameter allocation failed");
        const int rc = upload(g, g->params, params, sizeof(float) * mlp::kTotal);
        if (rc) return rc;
    }
    g->policy = mode;
    return MF_OK;
}

int mf_policy_features(mf_graph *g, int64_t k, const int32_t *edge_id, const int32_t *new_cap, int32_t flags,
                       float *features) {
    if (!g || !features || k < 0 || k > g->m || (k > 0 && (!edge_id || !new_cap))) return MF_EINVAL;
    MF_CUDA(cudaSetDevice(g->dev));
    cudaStream_t st = g->last;
    int rc = ensure_batch_capacity(g, std::max<int64_t>(k, 1), st);
    if (rc) return rc;
    const int *ids = edge_id, *caps = new_cap;
    if (!(flags & MF_DEVICE_PTRS) && k > 0) {
        MF_CUDA(cudaMemcpyAsync(g->b_ids, edge_id, size_t(k) * 4, cudaMemcpyHostToDevice, st));
        MF_CUDA(cudaMemcpyAsync(g->b_caps, new_cap, size_t(k) * 4, cudaMemcpyHostToDevice, st));
        ids = g->b_ids;
        caps = g->b_caps;
    }
    rc = launch_policy(g, k, ids, caps, flags & MF_DELTA, st);
    if (rc) return rc;
    Ctl c;
    rc = read_ctl(g, &c);
    if (rc) return rc;
    for (int j = 0; j < mlp::kIn; ++j) features[j] = c.feat[j];
    return MF_OK;
}

int mf_trace_enable(mf_graph *g, int32_t capacity) {
    if (!g || capacity < 0) return MF_EINVAL;
    MF_CUDA(cudaSetDevice(g->dev));
    MF_CUDA(cudaStreamSynchronize(g->last));
    if (g->dg.trace) {
        dfree(g, g->dg.trace);
        dforget(g, g->dg.trace);
        g->dg.trace = nullptr;
        g->dg.trace_cap = 0;
    }
    if (capacity == 0) return MF_OK;
    g->dg.trace = dnew<TraceRec>(g, size_t(capacity));
    if (!g->dg.trace) return set_err(MF_ENOMEM, "trace buffer allocation failed");
    g->dg.trace_cap = capacity;
    return MF_OK;
}

int mf_trace_read(mf_graph *g, mf_trace_rec *out, int32_t max_records, int32_t *count) {
    if (!g || !count || max_records < 0 || (max_records > 0 && !out)) return MF_EINVAL;
    Ctl c;
    int rc = read_ctl(g, &c);
    if (rc) return rc;
    const int avail = std::min(c.trace_n, g->dg.trace_cap);
    *count = c.trace_n;
    const int k = std::min(avail, int(max_records));
    if (k <= 0 || !g->dg.trace) return MF_OK;
    std::vector<TraceRec> tmp(static_cast<size_t>(k));
    MF_CUDA(cudaMemcpy(tmp.data(), g->dg.trace, size_t(k) * sizeof(TraceRec), cudaMemcpyDeviceToHost));
    for (int i = 0; i < k; ++i) {
        int ph = MF_PHASE_BATCH;
        switch (tmp[size_t(i)].phase) {
            case S_T_RESET: ph = MF_PHASE_HEIGHT_INIT; break;
            case S_T_BFS: ph = MF_PHASE_BFS; break;
            case S_T_PRW: ph = MF_PHASE_PUSH_RELABEL; break;
            case S_T_HUB: ph = MF_PHASE_HUB; break;
            case S_T_RI: ph = MF_PHASE_REMOVE_INVALID; break;
            default: ph = MF_PHASE_BATCH; break;
        }
        out[i].phase = int16_t(ph);
        out[i].mode = tmp[size_t(i)].mode;
        out[i].iter = tmp[size_t(i)].iter;
        out[i].step = tmp[size_t(i)].step;
        out[i].count = tmp[size_t(i)].count;
        out[i].ns = tmp[size_t(i)].ns;
    }
    return MF_OK;
}

// Allocation-free static solve on a caller-provided Bi-CSR (see mf.h).
int mf_solve_bicsr_noalloc(int32_t n, int64_t arcs, const int32_t *row, const int32_t *head, const int32_t *rev,
                           const int32_t *cap, int32_t s, int32_t t, int32_t kernel_cycles, int32_t *r,
                           int64_t *excess, int32_t *height, int64_t *flow, void *stream) {
    if (n < 2 || s < 0 || t < 0 || s >= n || t >= n || s == t || arcs < 0)
        return set_err(MF_EINVAL, "bad sizes or terminals");
    if (n > kNoAllocMaxN || arcs > kNoAllocMaxArcs)
        return set_err(MF_EINVAL, "graph larger than the static scratch: at most " + std::to_string(kNoAllocMaxN) +
                                      " vertices and " + std::to_string(kNoAllocMaxArcs) + " arcs");
    if (!row || !head || !rev || !cap || !r || !excess || !height || !flow)
        return set_err(MF_EINVAL, "null argument");
    int dev = 0;
    MF_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kNoAllocMaxDevices) return set_err(MF_EINVAL, "device index out of range");
    // once per device: the device address of the static scratch array (host
    // code only sees a host-side stand-in for it) and the co-resident grid
    std::call_once(g_noalloc_once[dev], [dev]() {
        NoAllocDevice &D = g_noalloc_dev[dev];
        D.err = cudaGetSymbolAddress(reinterpret_cast<void **>(&D.base), g_noalloc_scratch);
        int per_sm = 0, sms = 0;
        if (D.err == cudaSuccess) D.err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (D.err == cudaSuccess) D.err = solve_kernels_prepare(dev);
        if (D.err == cudaSuccess)
            D.err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_solve<false>, kBlock, kDynSmem);
        D.grid = std::min(per_sm * sms, kNoAllocMaxGrid);
        if (D.err == cudaSuccess && D.grid < 1) D.err = cudaErrorInvalidConfiguration;
    });
    const NoAllocDevice &ND = g_noalloc_dev[dev];
    if (ND.err != cudaSuccess)
        return set_err(MF_ECUDA, std::string("scratch set-up: ") + cudaGetErrorString(ND.err));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char *b = ND.base;
    using Lo = NoAllocLayout;
    DevGraph D{};
    D.n = n; D.s = s; D.t = t; D.m = 0; D.A = arcs; D.cap_limit = 0;
    D.row = row; D.head = head; D.rev = rev; D.arc_of_edge = nullptr; D.edge_st = nullptr;
    D.cap = const_cast<int *>(cap);      // read only by a solve from zero flow
    D.r = r; D.e = reinterpret_cast<long long *>(excess); D.h = height;
    D.cap_edge = nullptr; D.stamp = nullptr;
    D.al16 = ((reinterpret_cast<uintptr_t>(head) | reinterpret_cast<uintptr_t>(r)) & 15u) == 0;
    D.ctl = reinterpret_cast<Ctl *>(b + Lo::ctl);
    D.rr = reinterpret_cast<int *>(b + Lo::rr);
    D.qb0 = reinterpret_cast<int *>(b + Lo::qb0);
    D.qb1 = reinterpret_cast<int *>(b + Lo::qb1);
    D.wl = reinterpret_cast<int *>(b + Lo::wl);
    D.rl = reinterpret_cast<int *>(b + Lo::rl);
    D.astamp = reinterpret_cast<unsigned *>(b + Lo::astamp);
    D.rstamp = reinterpret_cast<unsigned *>(b + Lo::rstamp);
    D.cb = reinterpret_cast<int2 *>(b + Lo::cb);
    D.hit0 = reinterpret_cast<int4 *>(b + Lo::hit0);
    D.hit1 = reinterpret_cast<int4 *>(b + Lo::hit1);
    D.hikey = reinterpret_cast<int *>(b + Lo::hikey);
    D.hl = reinterpret_cast<int *>(b + Lo::hl);
    D.hlist0 = reinterpret_cast<int *>(b + Lo::hlist0);
    D.hlist1 = reinterpret_cast<int *>(b + Lo::hlist1);
    D.hkey = reinterpret_cast<int *>(b + Lo::hkey);
    D.hrem = reinterpret_cast<long long *>(b + Lo::hrem);
    D.hl2 = reinterpret_cast<int *>(b + Lo::hl2);
    D.hri = reinterpret_cast<int2 *>(b + Lo::hri);
    D.aq = reinterpret_cast<unsigned long long *>(b + Lo::aq);
    D.qc = std::min(std::max(n, 1024), kNoAllocMaxN);
    search_rules(D, false);
    // the previous call's contents stay in the array: clear what must start at 0
    MF_CUDA(cudaMemsetAsync(D.ctl, 0, sizeof(Ctl), st));
    MF_CUDA(cudaMemsetAsync(D.aq, 0, sizeof(unsigned long long) * size_t(D.qc), st));
    MF_CUDA(cudaMemsetAsync(D.astamp, 0, sizeof(unsigned) * size_t(n), st));
    MF_CUDA(cudaMemsetAsync(D.rstamp, 0, sizeof(unsigned) * size_t(n), st));
    Job j{};
    j.kind = JOB_SOLVE;
    j.exact_exit = 1;   // the caller reads the cut {height >= n} from the heights
    j.st = D.ctl->st;
    j.trace = nullptr;
    j.kc = kernel_cycles > 0 ? kernel_cycles : int(std::max<int64_t>(1, (arcs / 2 + n / 2) / n));
    j.max_iters = 4LL * n + 1000;
    j.time_limit_ns = 60ull * 1000ull * 1000ull * 1000ull;
    void *args[] = {&D, &j};
    cudaError_t e =
        cudaLaunchCooperativeKernel((const void *)k_solve<false>, dim3(auto_grid(ND.grid, arcs, n)), dim3(kBlock), args,
                                    kDynSmem, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_err(MF_ECUDA, std::string("cooperative launch: ") + cudaGetErrorString(e));
    }
    int32_t status = 0;
    MF_CUDA(cudaMemcpyAsync(&status, &D.ctl->status, sizeof(status), cudaMemcpyDeviceToHost, st));
    MF_CUDA(cudaMemcpyAsync(flow, &D.ctl->flow, sizeof(*flow), cudaMemcpyDeviceToHost, st));
    MF_CUDA(cudaStreamSynchronize(st));
    if (status & ST_STICKY) return set_err(MF_ETIMEOUT, "device loop did not finish");
    return MF_OK;
}

}  // extern "C"
