// la_solve_sparse: exact minimum-cost perfect matching of a sparse bipartite
// graph (arcs in CSR form) by the same cost scaling as la_solve.
//
// The paper's implementation takes arbitrary bipartite graphs (Sect. 1 and
// Sect. 6); Sect. 5 reduces assignment to min-cost flow with u(x,y) = 1 on
// the graph's arcs. Here a free row's warp scans only its own arcs
// (coalesced loads of columns and costs, prices gathered at L2) for the best
// and second-best part-reduced cost, and commits the Goldberg-Kennedy double
// push with the same packed 64-bit atomicMin on the column key as the dense
// refine (Algorithm 5.4 as a double push, Algorithm 5.2's initialisation,
// Algorithm 5.0's eps loop on costs scaled by n + 1).
//
// Readings for graphs that are not complete:
//  * A row with one arc (or whose arcs all lead to one column) has no second
//    best: any price drop >= eps keeps it eps-optimal, since eps-CS compares
//    only the row's own arcs. It bids as on a tie (drop = eps).
//  * Parallel arcs x -> y are allowed; a matching uses the cheaper one, and
//    a bid against the other copy keeps eps-CS (it only shrinks the drop).
//  * Feasibility. A graph may have no perfect matching. A first refine
//    phase runs with every arc cost taken as 0 and eps = 1 from zero prices:
//    if a perfect matching M' exists it is 0-optimal there, and the
//    price-drop bound of cost scaling (the path argument behind Lemma 5.6's
//    use of eps-optimality: a column relabelled while it holds excess lies on
//    an alternating path to a free column, of at most 2n - 1 arcs) keeps every
//    price within (eps + 0)(2n - 1) of its start while bids alone move the
//    prices. A bid beyond 4n + 4 in the refine, which runs from zero prices,
//    therefore proves that no perfect matching exists (LA_ERR_INFEASIBLE).
//    The updates that end the phase (k_sp_finish) also lift columns that reach
//    no free column, which that argument says nothing about, so there no price
//    decides: a free row that reaches no free column in the residual graph has
//    no augmenting path, and the matching cannot become perfect
//    (LA_ERR_INFEASIBLE too); while every free row reaches one the rounds go
//    on. Then prices are reset and the cost phases run on a graph known to be
//    feasible.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <vector>

#include "la.h"
#include "la_device.cuh"
#include "la_grid.cuh"

using namespace la;

namespace {

constexpr int kMaxDevices = 64;
constexpr int kBlock = 256;

// Control words of the end-of-phase kernel (k_sp_finish), beside Ctrl.
struct FinCtrl {
    GridBar bar;
    int free_rows;                  // rows not yet matched in this phase (the refine counts down)
    int count[2];                   // free rows listed in this round (double buffered)
    int changed[3];                 // a potential fell in this sweep (triple buffered)
    unsigned long long need[3];     // largest distance of a free row to a free column, per epoch
    unsigned long long qmax[2];     // largest q before the update
};

__device__ __forceinline__ void sp_set_status(Ctrl *ctrl, int s) { atomicCAS(&ctrl->status, 0, s); }

// Structure of the CSR arrays, min / max cost, rows and columns without arcs.
__global__ void k_sp_validate(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ cols,
                              const int32_t *__restrict__ costs, int n, int nnz, int *__restrict__ colseen,
                              Ctrl *ctrl) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    bool bad = false, empty_row = false;
    for (int x = tid; x < n; x += stride) {
        const int b = row_ptr[x], e = row_ptr[x + 1];
        bad |= e < b || b < 0 || e > nnz;
        empty_row |= e == b;
    }
    if (tid == 0) bad |= row_ptr[0] != 0 || row_ptr[n] != nnz;
    int lo = INT_MAX, hi = INT_MIN;
    for (int k = tid; k < nnz; k += stride) {
        const int y = cols[k];
        if (y < 0 || y >= n) {
            bad = true;
            continue;
        }
        colseen[y] = 1;
        const int c = costs[k];
        lo = min(lo, c);
        hi = max(hi, c);
    }
    if (bad) sp_set_status(ctrl, LA_ERR_INVALID);
    if (empty_row) atomicExch(&ctrl->colseen_missing, 1);
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(&ctrl->cmin, lo);
        atomicMax(&ctrl->cmax, hi);
    }
}

__global__ void k_sp_colcheck(const int *__restrict__ colseen, int n, Ctrl *ctrl) {
    bool miss = false;
    for (int y = blockIdx.x * blockDim.x + threadIdx.x; y < n; y += gridDim.x * blockDim.x) miss |= colseen[y] == 0;
    if (miss) atomicExch(&ctrl->colseen_missing, 1);
}

__global__ void k_sp_qmin(const unsigned long long *__restrict__ key, int n, Ctrl *ctrl, int slot) {
    unsigned long long m = ~0ull;
    for (int y = blockIdx.x * blockDim.x + threadIdx.x; y < n; y += gridDim.x * blockDim.x)
        m = min(m, key_q(__ldcg(key + y)));
    m = warp_min(m);
    if ((threadIdx.x & 31) == 0) atomicMin(&ctrl->qmin[slot], m);
}

// Refine initialisation (Algorithm 5.2): every row free, prices kept and
// shifted so that min q = 0, the price mirror refreshed, the queue reset.
// zero = 1 restarts from zero prices (after the feasibility phase).
__global__ void k_sp_reset(unsigned long long *__restrict__ key, unsigned long long *__restrict__ qm, int n,
                           unsigned long long qlim, Ctrl *ctrl, FinCtrl *fin, int slot, int phase, int zero) {
    const unsigned long long qmin = zero ? 0ull : ctrl->qmin[slot];
    bool bad = false;
    for (int y = blockIdx.x * blockDim.x + threadIdx.x; y < n; y += gridDim.x * blockDim.x) {
        const unsigned long long q = zero ? 0ull : key_q(key[y]) - qmin;
        bad |= q > qlim;
        key[y] = pack_key(q, kNone);
        qm[y] = q;
    }
    if (bad) sp_set_status(ctrl, LA_ERR_OVERFLOW);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctrl->next_row = 0;
        ctrl->qmin[slot ^ 1] = ~0ull;
        ctrl->phase_start_scans[phase & 63] = ctrl->scans;
        fin->free_rows = n;
        for (int k = 0; k < 2; ++k) {
            fin->count[k] = 0;
            fin->qmax[k] = 0;
        }
        for (int k = 0; k < 3; ++k) {
            fin->changed[k] = 0;
            fin->need[k] = 0;
        }
    }
}

// One bid of row `row` (a warp): best and second best of
// v(x,y) = (C - cmin)(n+1) + q(y) over the row's arcs, then the double push
// as one atomicMin on the column key. Returns the row left without a column
// (the displaced one, `row` itself after a lost bid), or kMatched, or, with a
// status set, kFailed.
constexpr int kMatched = -1, kFailed = -2;
template <bool ZERO>
__device__ __forceinline__ int sp_bid(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ cols,
                                      const int32_t *__restrict__ costs, int n, int cmin, uint32_t np1,
                                      unsigned long long eps, unsigned long long qlim, unsigned long long qinf,
                                      unsigned long long *__restrict__ key, unsigned long long *__restrict__ qm,
                                      Ctrl *__restrict__ ctrl, int row, int lane, unsigned long long &wins,
                                      unsigned long long &displaced) {
    using V = unsigned long long;
    const V inf = ~0ull;
    const int b = __ldg(row_ptr + row), e = __ldg(row_ptr + row + 1);
    ScanResult<V> r{inf, inf, 0, INT_MAX};
    for (int k = b + lane; k < e; k += 32) {
        const int y = __ldg(cols + k);
        const V cs = ZERO ? 0ull : (V)(uint32_t)(__ldg(costs + k) - cmin) * np1;
        const V v = cs + __ldcg(qm + y);
        const bool better = v < r.b1 || (v == r.b1 && (unsigned)y < (unsigned)r.w);
        const V hi = better ? r.b1 : v;
        r.b2 = hi < r.b2 ? hi : r.b2;
        r.c1 = better ? cs : r.c1;
        r.w = better ? y : r.w;
        r.b1 = better ? v : r.b1;
    }
    warp_merge(r);
    if (r.b2 == inf) r.b2 = r.b1;     // a single arc: bid as on a tie
    const unsigned long long nq = (r.b1 - r.c1) + (r.b2 - r.b1) + eps;
    if (r.w >= n || nq > qlim || nq > qinf) {
        if (lane == 0)
            sp_set_status(ctrl, r.w >= n ? LA_ERR_INTERNAL : (nq > qinf ? LA_ERR_INFEASIBLE : LA_ERR_OVERFLOW));
        return kFailed;
    }
    const unsigned long long nk = pack_key(nq, (uint32_t)row);
    unsigned long long old = 0;
    if (lane == 0) {
        old = atomicMin(key + r.w, nk);
        atomicMax(qm + r.w, old > nk ? nq : key_q(old));
    }
    old = __shfl_sync(0xffffffffu, old, 0);
    if (old <= nk) return row;        // a lower price got there first: the row bids again
    ++wins;
    const uint32_t m = key_mate(old);
    if (m == kNone) return kMatched;
    ++displaced;
    return (int)m;
}

// One refine phase over the arcs: persistent grid, one warp per free row.
// ZERO: the feasibility phase (every arc cost taken as 0; a price drop past
// qinf proves that no perfect matching exists).
template <bool ZERO>
__global__ void __launch_bounds__(kBlock)
k_sp_refine(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ cols,
            const int32_t *__restrict__ costs, int n, int cmin, uint32_t np1, unsigned long long eps,
            unsigned long long qlim, unsigned long long qinf, unsigned long long *__restrict__ key,
            unsigned long long *__restrict__ qm, Ctrl *__restrict__ ctrl, unsigned long long budget,
            FinCtrl *__restrict__ fin, int hand_free) {
    constexpr unsigned kFlush = 8;
    const int lane = threadIdx.x & 31;
    if (*reinterpret_cast<volatile int *>(&ctrl->status) != 0) return;   // an earlier phase failed
    int row = -1;
    unsigned long long wins = 0, displaced = 0, total = 0;
    unsigned pending = 0;
    for (;;) {
        // few rows free: k_sp_finish ends the phase (the load overlaps the bid)
        const int fr = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile int *>(&fin->free_rows), 0);
        if (row < 0) {
            int r = 0;
            if (lane == 0) r = atomicAdd(&ctrl->next_row, 1);
            row = __shfl_sync(0xffffffffu, r, 0);
            if (row >= n) break;
        }
        if (pending == kFlush) {
            unsigned long long s = 0;
            int st = 0;
            if (lane == 0) {
                s = atomicAdd(&ctrl->scans, (unsigned long long)kFlush);
                st = *reinterpret_cast<volatile int *>(&ctrl->status);
            }
            s = __shfl_sync(0xffffffffu, s, 0);
            st = __shfl_sync(0xffffffffu, st, 0);
            pending = 0;
            if (st != 0) break;
            if (s + kFlush > budget) {
                if (lane == 0) sp_set_status(ctrl, LA_ERR_ITER_LIMIT);
                break;
            }
        }
        ++pending;
        ++total;
        row = sp_bid<ZERO>(row_ptr, cols, costs, n, cmin, np1, eps, qlim, qinf, key, qm, ctrl, row, lane, wins,
                           displaced);
        if (row == kFailed) break;
        if (row == kMatched && lane == 0) atomicSub(&fin->free_rows, 1);
        if (fr <= hand_free) break;
    }
    if (lane == 0 && total) {
        atomicAdd(&ctrl->scans, (unsigned long long)pending);
        atomicAdd(&ctrl->wins, wins);
        atomicAdd(&ctrl->displaced, displaced);
        atomicAdd(&ctrl->full_scans, total);
        atomicMax(&ctrl->max_chain, total);
    }
}

// The end of a phase: rounds of an exact global price update and of bids,
// until no row is free. With few rows free the refine is one or a few serial
// displacement chains of tens of thousands of bids (price wars: a column's
// price rises by eps per bid); the update moves all those prices at once.
//
// The update (Sect. 5.2, Algorithm 5.3) with distances in price units
// instead of buckets of eps: D(y) is the least length of a residual path
// from column y to a free column, where the arc M(x) = y -> x -> z has
// length l = v(x,z) - v(x,y) + eps >= 0 (eps-optimality). As a potential
// S(y) = q(y) + D(y) it is the largest solution of
//   S(y) = q(y) for a free column,
//   S(y) <= min over the arcs x -> z, z != y, of c~(x,z) + S(z), + eps - c~(x,y)
// found by Bellman-Ford sweeps that only ever lower S (values written by
// other CTAs in the same sweep may be used). With q <- min(S, q + K) every
// matched row stays eps-optimal: min(D(y), K) <= min(D(z), K) + l. K is the
// largest distance of a free row, so that every free row's best arc then
// starts a shortest path, and its bids walk along it (l = 0 up to ties)
// unless the paths of two rows cross; such rows go into the next round. A
// free row that reaches no free column has no augmenting path: no perfect
// matching exists (the only test for that here; no price bound).
//
// Two bounds keep the sweeps short. The free rows' distances at the
// potentials so far bound K from above: a column farther than that is not
// lowered, and after two short epochs the arcs longer than that are dropped
// (min(D, K) is the same). And the CTAs sweep on without waiting for each
// other; grid barriers come once an epoch. A CTA keeps the arcs of its
// columns' rows in shared memory for a round (8 bytes an arc, rows that find
// no room are read from global memory and leave the room to shorter ones),
// eight lanes per column (8..40 arcs a row in the graphs this serves); only
// the potentials are gathered from L2.
//
// A row of more than kFinLongRow arcs would keep its eight lanes through 16
// and more rounds of gathers while every other CTA waits at the barrier, and
// would fill the shared memory. Such rows are listed instead, and the CTA's 32
// warps read them in segments of kFinSeg arcs. Whole solves, ms, with bids
// alone, with eight lanes for every row, now: 9 arcs a row and 20 rows of 8,192
// at n = 8192 28, 39, 23; 16 rows of 2,048 at n = 2048 5.3-7.1, 9.9, 5.8-8.2; one
// of 16,384 at n = 16384 -, 64, 35; 4 rows of 20,000 at n = 65536 150-195
// and 49-58, 65 arcs a row there 223-263 and 60-66, 9 arcs a row at n = 10^6
// 2,560 and 1,610 (bids alone and now).
//
// The price field. An update lifts every column that lies far from a free
// column, or reaches none, by K, and K is hops times eps on graphs with long
// residual paths: prices then climb to many times C~ where bids alone climb to
// about C~. A lift cut short is no way out: bids alone climb a plateau that
// updates left in steps of eps. So an update that would lift a price above
// kFinTop, half of the field, gives the solve up (kGiveUp), and so does a bid
// that leaves the field; the host then solves again with bids alone, in the
// refine, as if there were no updates. Emulated bid by bid on the host, largest
// price / 2^44 with bids alone, with updates without a limit, and as it is
// now: row x to columns x .. x + 3 at n = 3000, costs to 3.6e8 0.54-0.79,
// overflow, 0.49; n = 6000, costs to 3e7 0.17-0.20, overflow, 0.18; n = 30000,
// costs to 2e5 0.02, 0.21, 0.21. What is lost is the first rounds, a few
// percent of the second attempt. With updates cut short at 2^40 and bids from
// there on the last graph took 22 million bids, with bids alone 7 million, with
// updates 0.6. Prices of the graphs timed below stay under 2^32.
//
// Measured on GB300, whole solves in turn with the code that had one refine
// launch per phase, ms: sparse-uniform n = 65536, 33 arcs a row, 261 -> 34;
// sparse-geometric n = 16384, 36 arcs a row, 360 -> 96. There the 50 updates
// take 58 ms (150 sweeps each, 4.5 us a sweep), the bids 18 ms. Bound by a
// sweep's latency: 59 % of the warp cycles are spent at the CTA barrier, 27 %
// on gathers, with L2 at 14 % of its rate (ncu). When this form was chosen (88 ms then): without the caching a sweep
// took 19 us; without the bound on K 60 % more sweeps. Chains of at most 64,
// 256 and 1024 bids a round: 107, 88 and 95 ms (and 36, 29, 31 on the uniform
// graph): short chains do not reach the end of their path, long ones are rows
// whose path was taken, in a price war that the next update ends sooner.
//
// Paths longer than 256 need longer chains, or each round moves every row 256
// columns on and pays a whole update for it: a chain may take as many bids as
// the update took sweeps (about the columns of its longest path, and a third
// of its time). And where paths lead through most of the graph bids alone are
// faster: kGiveUp if a phase's first update leaves a free row that has reached
// no free column after kFinReach sweeps (cycles of rows of two arcs: 150 to
// 2,000; random and search-window graphs of three arcs a row and more, n = 600
// to 65536: at most 28; row x to columns x .. x + 3: 76), or is not done after
// n / 2 (1,024 to 16,384; there at most n / 5). n = 30000, row x to columns x
// .. x + d - 1, ms, with bids alone, with 256 bids a chain (emulated), now:
// d = 2 230-960, 63,000, 310-440; d = 4 1,700-6,000, 3,000, 190-290; d = 8
// 2,300-5,300, 450 (n = 20000), 170-200.
constexpr int kFinBlock = 1024;
constexpr int kFinLanes = 8;                                // lanes per column in a sweep
constexpr int kFinPerWarp = 32 / kFinLanes;
constexpr int kFinFirst = 6;                                // sweeps of a round's first epoch
constexpr int kFinSweeps = 16;                              // sweeps of an epoch at most
constexpr int kFinQuiet = 3;                                // ... and sweeps without a change that end it
constexpr int kFinMinCols = 16;                             // columns per CTA at least
constexpr int kFinMetaCap = 4096;                           // columns per CTA with cached arcs
constexpr int kFinLongRow = 512;                            // rows of more arcs are read by whole warps
constexpr int kFinLongRows = 256;                           // ... so many of them per CTA
constexpr int kFinSeg = 512;                                // ... in segments of so many arcs
constexpr int kFinSmem = 200 * 1024;
constexpr unsigned long long kFar = 1ull << 62;             // no path found yet
constexpr int kFinBids = 256;                               // bids of a warp's chain in one round, at least
constexpr unsigned kFinReach = 128;                         // sweeps until every free row has reached a free column
constexpr unsigned long long kFinTop = kQMax / 2;           // no update lifts a price above it
constexpr int kGiveUp = -1;                                 // status: solve again with bids alone

__device__ __forceinline__ unsigned long long min_u64_group(unsigned long long v) {
#pragma unroll
    for (int o = kFinLanes / 2; o; o >>= 1) {
        const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, o);
        v = u < v ? u : v;
    }
    return v;
}

// *p read at L2 if `on`, else `other`; a predicated load, so that a lane's
// loads are issued together whatever their predicates.
__device__ __forceinline__ unsigned long long ld_if(const unsigned long long *p, bool on, unsigned long long other) {
    unsigned long long v = other;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p ld.global.cg.u64 %0, [%1];\n\t}"
                 : "+l"(v)
                 : "l"(p), "r"((int)on)
                 : "memory");
    return v;
}

template <bool ZERO>
__global__ void __launch_bounds__(kFinBlock)
k_sp_finish(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ cols,
            const int32_t *__restrict__ costs, int n, int cmin, uint32_t np1, unsigned long long eps,
            unsigned long long qlim, unsigned long long *__restrict__ key,
            unsigned long long *__restrict__ qm, unsigned long long *__restrict__ pot, int *__restrict__ rowcol,
            int *__restrict__ rows, Ctrl *__restrict__ ctrl, unsigned long long budget, FinCtrl *__restrict__ fin,
            int meta_cap, int arc_cap) {
    extern __shared__ unsigned long long fin_smem[];
    __shared__ int s_ok, s_used, s_nlong;
    // long rows of this CTA's columns: column, first arc, arcs, segments up to and with this row, cost of the
    // matched arc, price, S, and the best arc's value in a sweep
    __shared__ int l_y[kFinLongRows], l_b[kFinLongRows], l_deg[kFinLongRows], l_end[kFinLongRows];
    __shared__ unsigned l_cy[kFinLongRows];
    __shared__ unsigned long long l_q[kFinLongRows], l_cur[kFinLongRows], l_best[kFinLongRows];
    if (threadIdx.x == 0) s_ok = 1;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gtid = blockIdx.x * blockDim.x + tid, gthreads = gridDim.x * blockDim.x;
    const int sub = lane % kFinLanes;
    // this CTA's columns: chunks of kFinMinCols (one 128-byte line of potentials), CTAs in turn
    const int chunks = (n + kFinMinCols - 1) / kFinMinCols;
    const int mine = kFinMinCols * ((chunks - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x);
    auto column = [&](int j) {
        return ((j / kFinMinCols) * (int)gridDim.x + (int)blockIdx.x) * kFinMinCols + j % kFinMinCols;
    };
    unsigned long long *s_cur = fin_smem;                                          // [meta_cap] S of the CTA's columns
    unsigned long long *s_q = s_cur + meta_cap;                                    // [meta_cap] their prices
    int2 *s_at = reinterpret_cast<int2 *>(s_q + meta_cap);                         // [meta_cap] first arc, padded count
    unsigned *s_cy = reinterpret_cast<unsigned *>(s_at + meta_cap);                // [meta_cap] cost of the matched arc
    int2 *s_arc = reinterpret_cast<int2 *>(s_cy + ((meta_cap + 1) & ~1));          // [arc_cap] column, cost - cmin
    const unsigned max_first = min(16384u, max(1024u, (unsigned)n / 2));
    unsigned long long sweeps = 0;
    unsigned long long wins = 0, displaced = 0, total = 0, longest = 0, updates = 0;
    for (int round = 0;; ++round) {
        const int par = round & 1;
        // The status and the counters are read right after a barrier (or the
        // launch), and are written again only after a further one: every CTA
        // decides alike.
        if (*reinterpret_cast<volatile int *>(&ctrl->status) != 0 ||
            *reinterpret_cast<volatile int *>(&fin->free_rows) == 0)
            break;
        for (int x = gtid; x < n; x += gthreads) rowcol[x] = -1;
        if (!grid_barrier(&fin->bar, &ctrl->status, &s_ok)) return;
        unsigned long long qmx = 0;
        for (int y = gtid; y < n; y += gthreads) {
            const unsigned long long k = __ldcg(key + y);
            const uint32_t x = key_mate(k);
            qmx = max(qmx, key_q(k));
            if (x < (uint32_t)n) {
                rowcol[x] = y;
                pot[y] = kFar;
            } else {
                pot[y] = key_q(k);
            }
        }
        qmx = warp_max_u64(qmx);
        if (lane == 0) atomicMax(&fin->qmax[par], qmx);
        if (!grid_barrier(&fin->bar, &ctrl->status, &s_ok)) return;
        for (int x = gtid; x < n; x += gthreads)
            if (__ldcg(rowcol + x) < 0) rows[atomicAdd(&fin->count[par], 1)] = x;
        // the arcs of this CTA's columns' rows into shared memory, long rows into their list
        if (tid == 0) s_used = s_nlong = 0;
        __syncthreads();
        for (int j0 = warp * kFinPerWarp; j0 < mine; j0 += (kFinBlock / 32) * kFinPerWarp) {
            const int j = j0 + lane / kFinLanes;
            int deg = 0, b = 0;
            const int y = j < mine ? column(j) : n;
            if (y < n) {
                const uint32_t x = key_mate(__ldcg(key + y));
                if (x < (uint32_t)n) {
                    b = __ldg(row_ptr + x);
                    deg = __ldg(row_ptr + x + 1) - b;
                }
            }
            int at = -1;                           // place of the arcs; -2: in the list
            if (sub == 0 && deg > kFinLongRow) {
                const int k = atomicAdd(&s_nlong, 1);
                if (k < kFinLongRows) {
                    at = -2;
                    l_y[k] = y;
                    l_b[k] = b;
                    l_deg[k] = deg;
                    l_cy[k] = 0xffffffffu;
                    l_q[k] = key_q(__ldcg(key + y));
                    l_cur[k] = l_best[k] = kFar;
                }
            } else if (sub == 0 && deg && j < meta_cap) {
                const int pad = (deg + kFinLanes - 1) / kFinLanes * kFinLanes;
                if (*(volatile int *)&s_used + pad <= arc_cap) {
                    at = atomicAdd(&s_used, pad);
                    if (at + pad > arc_cap) {      // others took the room: leave it to shorter rows
                        atomicSub(&s_used, pad);
                        at = -1;
                    }
                }
            }
            at = __shfl_sync(0xffffffffu, at, lane & ~(kFinLanes - 1));
            const int pad = at == -2 ? 0 : (deg + kFinLanes - 1) / kFinLanes * kFinLanes;
            unsigned cy = 0xffffffffu;
            for (int k = sub; k < pad; k += kFinLanes) {
                int2 a = make_int2(-1, 0);     // no arc
                if (k < deg) {
                    a.x = __ldg(cols + b + k);
                    a.y = ZERO ? 0 : __ldg(costs + b + k) - cmin;
                    if (a.x == y) {    // the matched arc (the cheapest copy)
                        cy = min(cy, (unsigned)a.y);
                        a.x = -1;
                    }
                }
                if (at >= 0) s_arc[at + k] = a;
            }
#pragma unroll
            for (int o = kFinLanes / 2; o; o >>= 1) cy = min(cy, __shfl_xor_sync(0xffffffffu, cy, o));
            if (sub == 0 && y < n && j < meta_cap) {
                s_cur[j] = deg && at != -2 ? kFar : 0ull;      // 0: nothing to lower here
                s_q[j] = key_q(__ldcg(key + y));
                s_cy[j] = cy;
                s_at[j] = at >= 0 ? make_int2(at, pad) : make_int2(-1, 0);
            }
        }
        __syncthreads();
        const int nlong = min(s_nlong, kFinLongRows);
        // the list's rows in segments of kFinSeg arcs, the CTA's warps in turn: f(row of the list, first arc, arcs)
        auto segments = [&](auto &&f) {
            const int segs = l_end[nlong - 1];
            for (int k = 0, seg = warp; seg < segs; seg += kFinBlock / 32) {
                while (seg >= l_end[k]) ++k;
                const int off = (seg - (k ? l_end[k - 1] : 0)) * kFinSeg;
                f(k, l_b[k] + off, min(kFinSeg, l_deg[k] - off));
            }
        };
        if (nlong) {
            if (tid == 0)
                for (int k = 0, e = 0; k < nlong; ++k) l_end[k] = e += (l_deg[k] - 1) / kFinSeg + 1;
            __syncthreads();
            segments([&](int k, int b, int len) {
                unsigned cy = 0xffffffffu;
                for (int o = lane; o < len; o += 32)
                    if (__ldg(cols + b + o) == l_y[k]) cy = min(cy, ZERO ? 0u : (unsigned)(__ldg(costs + b + o) - cmin));
                cy = __reduce_min_sync(0xffffffffu, cy);
                if (lane == 0 && cy != 0xffffffffu) atomicMin(&l_cy[k], cy);
            });
            __syncthreads();
        }
        // Bellman-Ford sweeps until no potential falls. The CTAs sweep on
        // without waiting for each other (S only falls, so any mix of old and
        // new values is a valid relaxation) until kFinQuiet sweeps in a row
        // changed nothing here; an epoch in which no CTA changed anything
        // proves the fixed point.
        unsigned long long lim = kFar;     // no column farther than this matters
        unsigned used = 0;                 // sweeps of this update, at most (the same for every CTA)
        bool settled = false;
        for (int it = 0; it <= n + 1; ++it) {
            const int slot = it % 3;
            bool any = false;
            if ((it == 2 || it == 4) && lim < kFar) {
                // arcs longer than the limit cannot be on a path that matters:
                // the cached rows keep the others
                for (int j0 = warp * kFinPerWarp; j0 < mine; j0 += (kFinBlock / 32) * kFinPerWarp) {
                    const int j = j0 + lane / kFinLanes;
                    int2 at = make_int2(-1, 0);
                    unsigned long long vm = 0;
                    if (j < mine && column(j) < n && j < meta_cap && s_cur[j] != 0) {
                        at = s_at[j];
                        vm = (unsigned long long)s_cy[j] * np1 + s_q[j];
                    }
                    const int len = at.x >= 0 ? at.y : 0;
                    const int longest_row = __reduce_max_sync(0xffffffffu, len);
                    int w = 0;
                    for (int k = sub; k < longest_row; k += kFinLanes) {   // longest_row: a multiple of kFinLanes
                        int2 a = make_int2(-1, 0);
                        bool keep = false;
                        if (k < len) {
                            a = s_arc[at.x + k];
                            keep = a.x >= 0 &&
                                   (unsigned long long)(unsigned)a.y * np1 + __ldcg(qm + a.x) + eps <= vm + lim;
                        }
                        const unsigned votes = __ballot_sync(0xffffffffu, keep) >> (lane & ~(kFinLanes - 1));
                        if (keep) s_arc[at.x + w + __popc(votes & ((1u << sub) - 1))] = a;   // at or before its old place
                        w += __popc(votes & ((1u << kFinLanes) - 1));
                        __syncwarp();
                    }
                    const int pad = (w + kFinLanes - 1) / kFinLanes * kFinLanes;
                    if (len && w + sub < pad) s_arc[at.x + w + sub] = make_int2(-1, 0);
                    if (len && sub == 0) s_at[j].y = pad;
                }
                __syncthreads();
            }
            const int most = it < 2 ? kFinFirst : kFinSweeps;
            used += most;
            for (int sw = 0, quiet = 0; sw < most && quiet < kFinQuiet; ++sw) {
                bool fell = false;
                for (int j0 = warp * kFinPerWarp; j0 < mine; j0 += (kFinBlock / 32) * kFinPerWarp) {
                    const int j = j0 + lane / kFinLanes;
                    const int y = j < mine ? column(j) : n;
                    unsigned long long best = kFar, cur = 0, q = 0;
                    unsigned cy = 0;
                    if (y < n && j < meta_cap) {
                        cur = s_cur[j];
                        q = s_q[j];
                        cy = s_cy[j];
                        const int2 at = s_at[j];
                        if (cur != 0 && at.x >= 0) {
                            // four gathers in flight per lane
                            for (int k = sub; k < at.y; k += 4 * kFinLanes) {
                                unsigned long long v[4];
                                unsigned c[4];
#pragma unroll
                                for (int g = 0; g < 4; ++g) {
                                    int2 a = make_int2(-1, 0);
                                    if (k + g * kFinLanes < at.y) a = s_arc[at.x + k + g * kFinLanes];
                                    c[g] = (unsigned)a.y;
                                    v[g] = ld_if(pot + max(a.x, 0), a.x >= 0, kFar);
                                }
#pragma unroll
                                for (int g = 0; g < 4; ++g) best = min(best, (unsigned long long)c[g] * np1 + v[g]);
                            }
                        }
                    }
                    // a row that found no room: its arcs from global memory
                    if (y < n && (j >= meta_cap || (cur != 0 && s_at[j].x < 0))) {
                        const unsigned long long ky = __ldcg(key + y);
                        const uint32_t x = key_mate(ky);
                        int b = 0, deg = 0;
                        if (x < (uint32_t)n) {
                            b = __ldg(row_ptr + x);
                            deg = __ldg(row_ptr + x + 1) - b;
                        }
                        if (j >= meta_cap) {
                            q = key_q(ky);
                            cur = deg ? __ldcg(pot + y) : 0ull;
                            cy = 0xffffffffu;
                            if (deg > kFinLongRow)
                                for (int k = 0; k < nlong; ++k)
                                    if (l_y[k] == y) cur = 0;
                        }
                        for (int k = sub; cur != 0 && k < deg; k += 4 * kFinLanes) {
                            int z[4];
                            unsigned c[4];
#pragma unroll
                            for (int g = 0; g < 4; ++g) {
                                const bool on = k + g * kFinLanes < deg;
                                z[g] = on ? __ldg(cols + b + k + g * kFinLanes) : -1;
                                c[g] = on && !ZERO ? (unsigned)(__ldg(costs + b + k + g * kFinLanes) - cmin) : 0u;
                                if (z[g] == y) {
                                    cy = min(cy, c[g]);
                                    z[g] = -1;
                                }
                            }
#pragma unroll
                            for (int g = 0; g < 4; ++g)
                                best = min(best, (unsigned long long)c[g] * np1 + ld_if(pot + max(z[g], 0), z[g] >= 0, kFar));
                        }
                    }
                    if (mine > meta_cap)   // a column without a record: its matched arc was found by one of the lanes
#pragma unroll
                        for (int o = kFinLanes / 2; o; o >>= 1) cy = min(cy, __shfl_xor_sync(0xffffffffu, cy, o));
                    best = min_u64_group(best);
                    if (sub == 0 && best < kFar && best + eps < cur + (unsigned long long)cy * np1) {
                        const unsigned long long v = best + eps - (unsigned long long)cy * np1;
                        if (v <= q + lim) {
                            __stcg(pot + y, v);
                            if (j < meta_cap) s_cur[j] = v;
                            fell = true;
                        }
                    }
                }
                if (nlong) {
                    segments([&](int k, int b, int len) {
                        unsigned long long best = kFar;
                        for (int o = lane; o < len; o += 4 * 32) {
                            int z[4];
                            unsigned c[4];
#pragma unroll
                            for (int g = 0; g < 4; ++g) {
                                const bool on = o + 32 * g < len;
                                z[g] = on ? __ldg(cols + b + o + 32 * g) : -1;
                                c[g] = on && !ZERO ? (unsigned)(__ldg(costs + b + o + 32 * g) - cmin) : 0u;
                                if (z[g] == l_y[k]) z[g] = -1;
                            }
#pragma unroll
                            for (int g = 0; g < 4; ++g)
                                best = min(best, (unsigned long long)c[g] * np1 + ld_if(pot + max(z[g], 0), z[g] >= 0, kFar));
                        }
                        best = warp_min(best);
                        if (lane == 0 && best < kFar) atomicMin(&l_best[k], best);
                    });
                    __syncthreads();
                    if (tid < nlong) {
                        const unsigned long long best = l_best[tid], own = (unsigned long long)l_cy[tid] * np1;
                        l_best[tid] = kFar;
                        if (best < kFar && best + eps < l_cur[tid] + own) {
                            const unsigned long long v = best + eps - own;
                            if (v <= l_q[tid] + lim) {
                                __stcg(pot + l_y[tid], v);
                                l_cur[tid] = v;
                                fell = true;
                            }
                        }
                    }
                }
                ++sweeps;
                const bool f = __syncthreads_or(fell) != 0;
                any |= f;
                quiet = f ? 0 : quiet + 1;
            }
            if (any && tid == 0) fin->changed[slot] = 1;
            // The free rows' distances at the potentials so far bound the
            // level K from above. (The list of free rows is complete from the
            // second epoch on.)
            unsigned long long far = 0;
            if (it > 0) {
                const int count = __ldcg(&fin->count[par]);
                for (int i = warp * gridDim.x + blockIdx.x; i < count; i += gridDim.x * (blockDim.x >> 5)) {
                    const int x = __ldcg(rows + i);
                    const int b = __ldg(row_ptr + x), e = __ldg(row_ptr + x + 1);
                    unsigned long long m = ~0ull, t = ~0ull;
                    for (int k = b + lane; k < e; k += 32) {
                        const int z = __ldg(cols + k);
                        const unsigned long long c =
                            ZERO ? 0ull : (unsigned long long)(uint32_t)(__ldg(costs + k) - cmin) * np1;
                        m = min(m, c + __ldcg(qm + z));
                        t = min(t, c + __ldcg(pot + z));
                    }
                    m = warp_min(m);
                    t = warp_min(t);
                    far = max(far, t >= kFar ? kFar : t - m);
                }
            }
            if (lane == 0 && far) atomicMax(&fin->need[slot], far);
            // the next epoch's words were last read before the barrier every CTA has passed since
            if (gtid == 0) {
                fin->changed[(it + 1) % 3] = 0;
                fin->need[(it + 1) % 3] = 0;
            }
            if (!grid_barrier(&fin->bar, &ctrl->status, &s_ok)) return;
            if (it == 0) continue;
            lim = *reinterpret_cast<volatile unsigned long long *>(&fin->need[slot]);
            if (*reinterpret_cast<volatile int *>(&fin->changed[slot]) == 0) {
                settled = true;
                break;
            }
            if (updates == 0 && used > (lim >= kFar ? kFinReach : max_first)) break;   // paths too long for updates
        }
        ++updates;
        // lim is now the largest distance of a free row: the level K
        if (gtid == 0) {
            const unsigned long long qmax = *reinterpret_cast<volatile unsigned long long *>(&fin->qmax[par]);
            if (!settled) sp_set_status(ctrl, kGiveUp);
            else if (lim >= kFar) sp_set_status(ctrl, LA_ERR_INFEASIBLE);
            else if (qmax + lim > kFinTop) sp_set_status(ctrl, kGiveUp);
        }
        const int count = *reinterpret_cast<volatile int *>(&fin->count[par]);
        if (!grid_barrier(&fin->bar, &ctrl->status, &s_ok)) return;
        if (*reinterpret_cast<volatile int *>(&ctrl->status) != 0) break;
        const unsigned long long K = lim;
        for (int y = gtid; y < n && K > 0; y += gthreads) {
            const unsigned long long k = __ldcg(key + y);
            const unsigned long long q = key_q(k), s = __ldcg(pot + y), nq = s < q + K ? max(s, q) : q + K;
            if (nq == q) continue;
            key[y] = pack_key(nq, key_mate(k));
            qm[y] = nq;
        }
        if (gtid == 0) {   // the other parity's counters, for the next round
            fin->count[par ^ 1] = 0;
            fin->qmax[par ^ 1] = 0;
            for (int k = 0; k < 3; ++k) {   // every sweep's words have been read
                fin->changed[k] = 0;
                fin->need[k] = 0;
            }
        }
        if (!grid_barrier(&fin->bar, &ctrl->status, &s_ok)) return;
        // the free rows bid, one warp per row, spread over the SMs first; a chain may be as long as the paths
        const unsigned most_bids = max((unsigned)kFinBids, used);
        for (int i = warp * gridDim.x + blockIdx.x; i < count; i += gridDim.x * (blockDim.x >> 5)) {
            int row = __ldcg(rows + i);
            unsigned steps = 0;
            while (row >= 0 && steps < most_bids) {
                unsigned now = 0;      // the scans are counted every kFinBids bids
                while (row >= 0 && now < (unsigned)kFinBids) {
                    ++now;
                    row = sp_bid<ZERO>(row_ptr, cols, costs, n, cmin, np1, eps, qlim, ~0ull, key, qm, ctrl, row, lane,
                                       wins, displaced);
                }
                steps += now;
                if (lane == 0 && atomicAdd(&ctrl->scans, (unsigned long long)now) + now > budget)
                    sp_set_status(ctrl, LA_ERR_ITER_LIMIT);
            }
            if (row == kMatched && lane == 0) atomicSub(&fin->free_rows, 1);
            total += steps;
            longest = max(longest, (unsigned long long)steps);
            if (row == kFailed) break;
        }
        if (!grid_barrier(&fin->bar, &ctrl->status, &s_ok)) return;
    }
    if (lane == 0 && total) {
        atomicAdd(&ctrl->wins, wins);
        atomicAdd(&ctrl->displaced, displaced);
        atomicAdd(&ctrl->full_scans, total);
        atomicMax(&ctrl->max_chain, longest);
    }
    if (gtid == 0) {
        ctrl->pu_updates += updates;
        ctrl->pu_iters += sweeps;      // of the first CTA
    }
}

// The matching from the column keys; the exact cost sums the cheapest arc of
// every matched pair.
__global__ void k_sp_finalize(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ cols,
                              const int32_t *__restrict__ costs, int n, const unsigned long long *__restrict__ key,
                              int32_t *match, long long *cost, long long *prices, Ctrl *ctrl, int slot) {
    long long sum = 0;
    const unsigned long long qmin = prices ? ctrl->qmin[slot] : 0;
    for (int y = blockIdx.x * blockDim.x + threadIdx.x; y < n; y += gridDim.x * blockDim.x) {
        const unsigned long long k = key[y];
        const uint32_t m = key_mate(k);
        if (m >= (uint32_t)n) {
            sp_set_status(ctrl, LA_ERR_INTERNAL);
            continue;
        }
        if (match) match[m] = y;
        int best = INT_MAX;
        bool found = false;
        for (int a = row_ptr[m]; a < row_ptr[m + 1]; ++a)
            if (cols[a] == y) {
                best = min(best, costs[a]);
                found = true;
            }
        if (!found) sp_set_status(ctrl, LA_ERR_INTERNAL);
        sum += best;
        if (prices) prices[y] = -(long long)(key_q(k) - qmin);
    }
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0 && sum != 0)
        atomicAdd(reinterpret_cast<unsigned long long *>(cost), (unsigned long long)sum);
}

struct SparseWorkspace {
    int64_t cap = 0;
    unsigned long long *key = nullptr;
    unsigned long long *qm = nullptr;
    int *colseen = nullptr;
    unsigned long long *pot = nullptr;   // end-of-phase kernel: potentials, row -> column, free rows
    int *rowcol = nullptr;
    int *rows = nullptr;
    FinCtrl *fin = nullptr;
    Ctrl *ctrl = nullptr;
    Ctrl *h_ctrl = nullptr;
    int num_sms = 0;
    int occ = 0;
    int events = 0;                      // events made
    cudaEvent_t ev[2];
};

std::mutex g_smu;
SparseWorkspace g_sws[kMaxDevices];

la_status ensure_sws(SparseWorkspace &w, int64_t n) {
    // what a call that failed here has left out, the next one makes
    if (!w.num_sms) {
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return LA_ERR_CUDA;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return LA_ERR_CUDA;
        int o = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_sp_refine<false>, kBlock, 0);
        w.occ = std::max(1, o);
        w.num_sms = sms;
    }
    if (!w.ctrl && cudaMalloc(&w.ctrl, sizeof(Ctrl)) != cudaSuccess) return LA_ERR_NOMEM;
    if (!w.h_ctrl && cudaMallocHost(&w.h_ctrl, sizeof(Ctrl)) != cudaSuccess) return LA_ERR_NOMEM;
    if (!w.fin && cudaMalloc(&w.fin, sizeof(FinCtrl)) != cudaSuccess) return LA_ERR_NOMEM;
    for (; w.events < 2; ++w.events)
        if (cudaEventCreate(&w.ev[w.events]) != cudaSuccess) return LA_ERR_CUDA;
    if (w.cap < n) {
        cudaFree(w.key);
        cudaFree(w.qm);
        cudaFree(w.colseen);
        cudaFree(w.pot);
        cudaFree(w.rowcol);
        cudaFree(w.rows);
        w.pot = nullptr;
        w.rowcol = nullptr;
        w.rows = nullptr;
        w.key = nullptr;
        w.qm = nullptr;
        w.colseen = nullptr;
        w.cap = 0;
        const int64_t cap = std::max<int64_t>(n, 1024);
        if (cudaMalloc(&w.key, sizeof(unsigned long long) * cap) != cudaSuccess) return LA_ERR_NOMEM;
        if (cudaMalloc(&w.qm, sizeof(unsigned long long) * cap) != cudaSuccess) return LA_ERR_NOMEM;
        if (cudaMalloc(&w.colseen, sizeof(int) * cap) != cudaSuccess) return LA_ERR_NOMEM;
        if (cudaMalloc(&w.pot, sizeof(unsigned long long) * cap) != cudaSuccess) return LA_ERR_NOMEM;
        if (cudaMalloc(&w.rowcol, sizeof(int) * cap) != cudaSuccess) return LA_ERR_NOMEM;
        if (cudaMalloc(&w.rows, sizeof(int) * cap) != cudaSuccess) return LA_ERR_NOMEM;
        w.cap = cap;
    }
    return LA_OK;
}

// Free rows at which the refine hands a phase to the end-of-phase kernel.
// Measured (means of 12 solves, ms, +- 10 %) at n / 1000, n / 256, n / 64, n / 16:
// sparse-uniform n = 65536 34, 36, 36, 35; sparse-geometric n = 16384 182, 102,
// 92, 95, n = 65536 585, 413, 420, 418.
int sp_hand_free(int n) {
    return std::max(8, n / 64);
}

// Cost phases without the end-of-phase kernel: where a phase is shorter than
// its launch and a few grid barriers, and where rows have two arcs on average,
// so that residual paths are long and hardly branch. ms with the kernel in
// every phase, without: 9 arcs a row, n = 50 0.58, 0.37; n = 200 0.79, 0.54;
// n = 500 1.2, 1.2 (n = 1000: 2.0, 3.3 without); search windows, n = 256 0.63,
// 0.46. Two arcs a row, n = 600 1.4, 0.87; n = 65536 20-41, 14-22; cycles of
// two arcs a row, n = 2500 83, 18 (three arcs a row: 3.6, 6.4).
// The feasibility phase keeps the kernel, which finds in one update what takes
// bids alone a price war of 4n steps (12 rows on 11 columns among n = 600:
// 0.3 and 21.6 ms).
bool sp_bids_alone(int n, int nnz) { return n <= 512 || (int64_t)nnz * 2 <= (int64_t)n * 5; }

// The end-of-phase kernel on a co-resident grid: one CTA per SM, fewer when
// the graph has fewer columns than the grid has lane groups.
template <bool ZERO>
cudaError_t launch_finish(cudaStream_t s, SparseWorkspace &w, const int32_t *row_ptr, const int32_t *cols,
                          const int32_t *costs, int n, int cmin, uint32_t np1, unsigned long long eps,
                          unsigned long long qlim, unsigned long long budget) {
    const int grid = std::max(1, std::min(w.num_sms, (n + kFinMinCols - 1) / kFinMinCols));
    // shared memory: what this graph needs, up to kFinSmem
    const int chunks = (n + kFinMinCols - 1) / kFinMinCols;
    int meta_cap = std::min(kFinMetaCap, kFinMinCols * ((chunks + grid - 1) / grid));
    const int meta = 24 * meta_cap + 4 * ((meta_cap + 1) & ~1);
    int arc_cap = (kFinSmem - meta) / 8;
    const cudaError_t e =
        cudaFuncSetAttribute(k_sp_finish<ZERO>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFinSmem);
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)&row_ptr, (void *)&cols, (void *)&costs, (void *)&n, (void *)&cmin, (void *)&np1,
                    (void *)&eps, (void *)&qlim, (void *)&w.key, (void *)&w.qm, (void *)&w.pot,
                    (void *)&w.rowcol, (void *)&w.rows, (void *)&w.ctrl, (void *)&budget, (void *)&w.fin,
                    (void *)&meta_cap, (void *)&arc_cap};
    return cudaLaunchCooperativeKernel((const void *)k_sp_finish<ZERO>, dim3(grid), dim3(kFinBlock), args, kFinSmem, s);
}

}  // namespace

#define LA_SCK(call)                                   \
    do {                                               \
        if ((call) != cudaSuccess) return LA_ERR_CUDA; \
    } while (0)

static la_status sparse_locked(const int32_t *row_ptr, const int32_t *cols, const int32_t *costs, int32_t n,
                               int32_t nnz, const la_options *opt, cudaStream_t s, int32_t *match_out,
                               int64_t *cost_out, la_stats *st) {
    const int alpha = (opt && opt->alpha) ? opt->alpha : 10;
    const int64_t eps0 = opt ? opt->eps0 : 0;
    int64_t *prices_out = opt ? opt->prices_out : nullptr;
    const bool profile = opt && opt->profile;
    if (alpha < 2 || eps0 < 0 || (opt && opt->scan_budget < 0) || (opt && opt->init_prices)) return LA_ERR_INVALID;
    la_stats stats;
    std::memset(&stats, 0, sizeof(stats));
    stats.n = n;
    stats.wide = 1;
    if (n == 0) {
        LA_SCK(cudaMemsetAsync(cost_out, 0, sizeof(int64_t), s));
        LA_SCK(cudaStreamSynchronize(s));
        if (st) *st = stats;
        return LA_OK;
    }
    int dev = 0;
    LA_SCK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return LA_ERR_INVALID;
    SparseWorkspace &w = g_sws[dev];
    if (la_status e = ensure_sws(w, n)) return e;

    Ctrl init;
    std::memset(&init, 0, sizeof(init));
    init.cmin = INT_MAX;
    init.cmax = INT_MIN;
    init.qmin[0] = init.qmin[1] = ~0ull;
    *w.h_ctrl = init;
    LA_SCK(cudaMemcpyAsync(w.ctrl, w.h_ctrl, sizeof(Ctrl), cudaMemcpyHostToDevice, s));
    LA_SCK(cudaMemsetAsync(w.colseen, 0, sizeof(int) * n, s));
    LA_SCK(cudaMemsetAsync(w.fin, 0, sizeof(FinCtrl), s));
    int64_t launches = 0;
    const int vg = std::max(1, std::min((std::max(n, nnz) + kBlock - 1) / kBlock, 8 * w.num_sms));
    k_sp_validate<<<vg, kBlock, 0, s>>>(row_ptr, cols, costs, n, nnz, w.colseen, w.ctrl);
    const int sg = std::max(1, std::min((n + kBlock - 1) / kBlock, 4 * w.num_sms));
    k_sp_colcheck<<<sg, kBlock, 0, s>>>(w.colseen, n, w.ctrl);
    launches += 2;
    LA_SCK(cudaGetLastError());
    LA_SCK(cudaMemcpyAsync(w.h_ctrl, w.ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, s));
    LA_SCK(cudaStreamSynchronize(s));
    const Ctrl c0 = *w.h_ctrl;
    if (c0.status) return (la_status)c0.status;
    if (c0.colseen_missing) {   // a row or a column without arcs: Hall's condition fails
        if (st) *st = stats;
        return LA_ERR_INFEASIBLE;
    }
    const unsigned long long np1 = (unsigned long long)n + 1;
    const unsigned long long Ct = np1 * (unsigned long long)((long long)c0.cmax - (long long)c0.cmin);
    stats.scaled_range = (int64_t)Ct;
    if (Ct >= (1ull << 40)) return LA_ERR_OVERFLOW;
    std::vector<unsigned long long> sched;
    {
        unsigned long long e = eps0 > 0 ? (unsigned long long)eps0 : Ct;
        do {
            e = std::max<unsigned long long>(1, e / (unsigned long long)alpha);
            sched.push_back(e);
        } while (e > 1 && sched.size() < 64);
        if (sched.back() != 1) return LA_ERR_INVALID;
    }
    stats.eps_first = (int64_t)sched[0];
    const unsigned long long qlim = kQMax - 1;
    const unsigned long long budget = opt && opt->scan_budget ? (unsigned long long)opt->scan_budget
                                                              : 256ull * n * (sched.size() + 1) + (1ull << 22);
    const int grid = std::max(1, std::min(w.num_sms * w.occ, (n + kBlock / 32 - 1) / (kBlock / 32)));
    if (profile) LA_SCK(cudaEventRecord(w.ev[0], s));
    const unsigned long long qinf = 4ull * (unsigned long long)n + 4;
    // with end-of-phase updates; if those give up, again with bids alone
    Ctrl c1;
    int ph = 0;
    bool alone = false;
    const bool short_solve = sp_bids_alone(n, nnz);
    for (;; alone = true) {
        const int hand_free = alone ? -1 : sp_hand_free(n);          // of the feasibility phase
        const bool updates = !alone && !short_solve;                 // of the cost phases
        if (alone) {
            init.cmin = c0.cmin;
            init.cmax = c0.cmax;
            *w.h_ctrl = init;
            LA_SCK(cudaMemcpyAsync(w.ctrl, w.h_ctrl, sizeof(Ctrl), cudaMemcpyHostToDevice, s));
            LA_SCK(cudaMemsetAsync(w.fin, 0, sizeof(FinCtrl), s));
        }
        // feasibility phase: zero costs, eps = 1, prices from 0
        k_sp_reset<<<sg, kBlock, 0, s>>>(w.key, w.qm, n, qlim, w.ctrl, w.fin, 0, 0, 1);
        k_sp_refine<true><<<grid, kBlock, 0, s>>>(row_ptr, cols, costs, n, c0.cmin, (uint32_t)np1, 1ull, qlim,
                                                  qinf, w.key, w.qm, w.ctrl, budget, w.fin, hand_free);
        launches += 2;
        if (!alone) {
            LA_SCK(launch_finish<true>(s, w, row_ptr, cols, costs, n, c0.cmin, (uint32_t)np1, 1ull, qlim, budget));
            ++launches;
        }
        // cost phases (Algorithm 5.0), from zero prices again
        for (ph = 0; ph < (int)sched.size(); ++ph) {
            const int slot = ph & 1;
            if (ph > 0) {
                k_sp_qmin<<<sg, kBlock, 0, s>>>(w.key, n, w.ctrl, slot);
                ++launches;
            }
            k_sp_reset<<<sg, kBlock, 0, s>>>(w.key, w.qm, n, qlim, w.ctrl, w.fin, slot, ph + 1, ph == 0);
            k_sp_refine<false><<<grid, kBlock, 0, s>>>(row_ptr, cols, costs, n, c0.cmin, (uint32_t)np1, sched[ph],
                                                       qlim, ~0ull, w.key, w.qm, w.ctrl, budget, w.fin,
                                                       updates ? hand_free : -1);
            launches += 2;
            if (updates) {
                LA_SCK(launch_finish<false>(s, w, row_ptr, cols, costs, n, c0.cmin, (uint32_t)np1, sched[ph], qlim,
                                            budget));
                ++launches;
            }
        }
        if (profile) LA_SCK(cudaEventRecord(w.ev[1], s));
        const int fslot = ph & 1;
        if (prices_out) {
            k_sp_qmin<<<sg, kBlock, 0, s>>>(w.key, n, w.ctrl, fslot);
            ++launches;
        }
        LA_SCK(cudaMemsetAsync(cost_out, 0, sizeof(int64_t), s));
        k_sp_finalize<<<sg, kBlock, 0, s>>>(row_ptr, cols, costs, n, w.key, match_out,
                                            reinterpret_cast<long long *>(cost_out),
                                            reinterpret_cast<long long *>(prices_out), w.ctrl, fslot);
        ++launches;
        LA_SCK(cudaGetLastError());
        LA_SCK(cudaMemcpyAsync(w.h_ctrl, w.ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, s));
        LA_SCK(cudaStreamSynchronize(s));
        c1 = *w.h_ctrl;
        // LA_ERR_INTERNAL: a grid barrier's wait ran out, behind bids on rows so long that one warp
        // takes seconds (350,000 arcs, 256 bids); the refine has no barrier
        if (alone || (c1.status != kGiveUp && c1.status != LA_ERR_OVERFLOW && c1.status != LA_ERR_INTERNAL)) break;
    }
    stats.phases = (int64_t)sched.size();
    stats.scans = (int64_t)c1.scans;
    stats.wins = (int64_t)c1.wins;
    stats.displaced = (int64_t)c1.displaced;
    stats.launches = launches;
    stats.refine_launches = (alone || short_solve ? 1 : 2) * ((int64_t)sched.size() + 1) + (short_solve && !alone);
    stats.price_updates = (int64_t)c1.pu_updates;
    stats.price_update_sweeps = (int64_t)c1.pu_iters;
    stats.max_chain = (int64_t)c1.max_chain;
    stats.full_scans = (int64_t)c1.full_scans;
    for (int k = 0; k <= ph && k < LA_STATS_PHASES; ++k) {
        // phase 0 of the counters is the feasibility phase
        const unsigned long long end = (k < ph) ? c1.phase_start_scans[k + 1] : c1.scans;
        stats.phase_scans[k] = (int64_t)(end - c1.phase_start_scans[k]);
    }
    if (profile) {
        float t = 0;
        LA_SCK(cudaEventElapsedTime(&t, w.ev[0], w.ev[1]));
        stats.refine_ms = t;
    }
    if (st) *st = stats;
    return (la_status)c1.status;
}

extern "C" {

la_status la_solve_sparse_ex(const int32_t *row_ptr, const int32_t *cols, const int32_t *costs, int32_t n,
                             int32_t nnz, const la_options *opt, void *stream, int32_t *match_out,
                             int64_t *cost_out, la_stats *stats_out) {
    if (n < 0 || n > LA_MAX_N || nnz < 0 || !cost_out || (n > 0 && (!row_ptr || (nnz > 0 && (!cols || !costs)))))
        return LA_ERR_INVALID;
    std::lock_guard<std::mutex> lock(g_smu);
    return sparse_locked(row_ptr, cols, costs, n, nnz, opt, static_cast<cudaStream_t>(stream), match_out, cost_out,
                         stats_out);
}

la_status la_solve_sparse(const int32_t *row_ptr, const int32_t *cols, const int32_t *costs, int32_t n,
                          int32_t nnz, void *stream, int32_t *match_out, int64_t *cost_out) {
    return la_solve_sparse_ex(row_ptr, cols, costs, n, nnz, nullptr, stream, match_out, cost_out, nullptr);
}

}  // extern "C"
