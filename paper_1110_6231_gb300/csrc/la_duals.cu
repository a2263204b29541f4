// la_dual_certificate: exact integer LP duals (u, v) for an optimal
// assignment, in cost units.
//
// Given a perfect matching M (row x -> column M(x)), the duals of the
// assignment LP that are tight on M are the potentials v with
//   v(y) <= v(M(x)) + C[x][y] - C[x][M(x)]   for every row x and column y,
// u(x) = C[x][M(x)] - v(M(x)); they exist iff M is optimal (no negative
// cycle). This returns the largest such potential with v <= 0: the
// shortest-path distances from a virtual source joined to every column by a
// zero arc, computed by Bellman-Ford sweeps over the columns (k_dual_sweeps).
// Values only decrease, so sweeps may read values written during the same
// sweep. With them, u(x) + v(y) <= C[x][y]
// everywhere, with equality on M, and sum u + sum v = cost(M): a certificate
// of optimality that needs no solver to check.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <mutex>

#include "la.h"
#include "la_grid.cuh"

using namespace la;

namespace {

constexpr int kMaxDevices = 64;
constexpr int kDualBlock = 512;
constexpr int kDualRounds = 4;      // sweeps of a CTA between two grid barriers
constexpr int kDualBurst = 256;     // ... in the first epochs; one from there on

struct DualCtrl {
    GridBar bar;
    int bad;            // the matching is not a permutation
    int changed[3];     // a potential fell since the barrier before last (triple buffered)
    int status;
    int settled;
};

// v = 0, cm(x) = C[x][M(x)], last(x) = no base used yet; checks that M is a permutation.
__global__ void k_dual_init(const int32_t *__restrict__ C, int n, const int32_t *__restrict__ match,
                            long long *__restrict__ v, int *__restrict__ cm, long long *__restrict__ last,
                            int *__restrict__ seen, DualCtrl *ctrl) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n) return;
    v[x] = 0;
    last[x] = LLONG_MAX;
    const int y = match[x];
    if (y < 0 || y >= n) {
        atomicExch(&ctrl->bad, 1);
        return;
    }
    if (atomicAdd(seen + y, 1) != 0) atomicExch(&ctrl->bad, 1);
    cm[x] = C[(size_t)x * n + y];
}

// All Bellman-Ford sweeps in one cooperative launch:
//   v(y) <- min(v(y), C[x][y] + base(x)), base(x) = v(M(x)) - C[x][M(x)].
// A row whose base has not fallen since it was last applied has nothing new
// to offer, so a sweep reads only the rows that changed: on geometric costs
// at n = 2048 those are all rows in the first sweep, 41 % in the second and
// under 10 % from the tenth of fifty on. CTA b owns rows b, b + gridDim, ...
// (kept in its shared memory while it sweeps); W threads take four columns
// each of a row, and the CTA's kDualBlock / W groups take its changed rows in
// turn, so that narrow matrices still have every thread loading. Between two
// grid barriers a CTA sweeps up to kDualRounds times: v only falls, so any mix
// of old and new values is a valid relaxation, and the fixed point is the
// same. The launch ends when no CTA lowered anything between two barriers.
// After kDualBurst epochs the matching is most likely not optimal: rows fall in
// every sweep until n + 2 epochs prove it, and one sweep each is enough for that
// (two rows of an optimum swapped, n = 4096: 342 ms with four sweeps, 143 with
// one, 156 from one launch pair and host synchronisation per sweep).
// Bound by the latency of one row read and one barrier per epoch: 1.25 -> 0.27
// ms at n = 2048 (geometric), from one launch pair, a memset, a copy and a
// host synchronisation per sweep, whose 32 CTAs read the whole matrix.
template <bool VEC>
__global__ void __launch_bounds__(kDualBlock)
k_dual_sweeps(const int32_t *__restrict__ C, int n, const int32_t *__restrict__ match, const int *__restrict__ cm,
              long long *__restrict__ last, long long *__restrict__ v, int W, int max_epochs,
              DualCtrl *__restrict__ ctrl) {
    __shared__ int s_ok, s_cnt;
    __shared__ int s_row[kDualBlock];
    __shared__ long long s_base[kDualBlock];
    const int tid = threadIdx.x;
    if (*reinterpret_cast<volatile int *>(&ctrl->bad)) return;   // set by the launch before, the same for every CTA
    if (tid == 0) s_ok = 1;
    const int g = tid / W, G = kDualBlock / W, t = tid % W;
    for (int ep = 0; ep < max_epochs; ++ep) {
        const int slot = ep % 3;
        bool any = false;
        const int rounds = ep < kDualBurst ? kDualRounds : 1;
        for (int round = 0; round < rounds; ++round) {
            bool found = false;
            // the CTA's rows, kDualBlock at a time
            for (long long r0 = 0; blockIdx.x + r0 * gridDim.x < n; r0 += kDualBlock) {
                __syncthreads();
                if (tid == 0) s_cnt = 0;
                __syncthreads();
                const long long x = blockIdx.x + (r0 + tid) * gridDim.x;
                if (x < n) {
                    const long long base = __ldcg(v + __ldg(match + x)) - (long long)__ldg(cm + x);
                    if (base < last[x]) {
                        last[x] = base;
                        const int k = atomicAdd(&s_cnt, 1);
                        s_row[k] = (int)x;
                        s_base[k] = base;
                    }
                }
                __syncthreads();
                const int cnt = s_cnt;
                if (cnt == 0) continue;
                found = true;
                if (VEC) {
                    for (int y = 4 * t; y < n; y += 4 * W) {
                        long long b0 = LLONG_MAX, b1 = LLONG_MAX, b2 = LLONG_MAX, b3 = LLONG_MAX;
#pragma unroll 4
                        for (int k = g; k < cnt; k += G) {
                            const int4 c = __ldg(reinterpret_cast<const int4 *>(C + (size_t)s_row[k] * n + y));
                            const long long base = s_base[k];
                            b0 = min(b0, c.x + base);
                            b1 = min(b1, c.y + base);
                            b2 = min(b2, c.z + base);
                            b3 = min(b3, c.w + base);
                        }
                        if (g >= cnt) continue;
                        const longlong2 p = __ldcg(reinterpret_cast<const longlong2 *>(v + y));
                        const longlong2 q = __ldcg(reinterpret_cast<const longlong2 *>(v + y + 2));
                        if (b0 < p.x) atomicMin(v + y, b0), any = true;
                        if (b1 < p.y) atomicMin(v + y + 1, b1), any = true;
                        if (b2 < q.x) atomicMin(v + y + 2, b2), any = true;
                        if (b3 < q.y) atomicMin(v + y + 3, b3), any = true;
                    }
                } else {
                    for (int y = t; y < n; y += W) {
                        long long b = LLONG_MAX;
#pragma unroll 4
                        for (int k = g; k < cnt; k += G)
                            b = min(b, (long long)__ldg(C + (size_t)s_row[k] * n + y) + s_base[k]);
                        if (b < __ldcg(v + y)) atomicMin(v + y, b), any = true;
                    }
                }
            }
            if (!found) break;     // uniform: found follows s_cnt
            __threadfence();
        }
        if (any) ctrl->changed[slot] = 1;
        // the next epoch's flag was last read before the barrier every CTA has passed since
        if (blockIdx.x == 0 && tid == 0) ctrl->changed[(ep + 1) % 3] = 0;
        if (!grid_barrier(&ctrl->bar, &ctrl->status, &s_ok)) return;
        if (*reinterpret_cast<volatile int *>(&ctrl->changed[slot]) == 0) {
            if (blockIdx.x == 0 && tid == 0) ctrl->settled = 1;
            break;
        }
    }
}

__global__ void k_dual_u(const int32_t *__restrict__ C, int n, const int32_t *__restrict__ match,
                         const long long *__restrict__ v, long long *__restrict__ u, const DualCtrl *ctrl) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n || ctrl->bad || !ctrl->settled) return;
    const int y = match[x];
    u[x] = (long long)C[(size_t)x * n + y] - v[y];
}

struct DualWs {
    int cap = 0;
    int num_sms = 0;
    int *cm = nullptr;
    long long *last = nullptr;
    int *seen = nullptr;
    DualCtrl *ctrl = nullptr;
    DualCtrl *h_ctrl = nullptr;
};

std::mutex g_dmu;
DualWs g_dws[kMaxDevices];

}  // namespace

#define LA_DCK(call)                                   \
    do {                                               \
        if ((call) != cudaSuccess) return LA_ERR_CUDA; \
    } while (0)

extern "C" la_status la_dual_certificate(const int32_t *cost, int32_t n, const int32_t *match, void *stream,
                                         int64_t *u_out, int64_t *v_out) {
    if (n < 0 || n > LA_MAX_N || (n > 0 && (!cost || !match || !v_out))) return LA_ERR_INVALID;
    if (n == 0) return LA_OK;
    std::lock_guard<std::mutex> lock(g_dmu);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int dev = 0;
    LA_DCK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return LA_ERR_INVALID;
    DualWs &w = g_dws[dev];
    if (!w.h_ctrl) {
        LA_DCK(cudaDeviceGetAttribute(&w.num_sms, cudaDevAttrMultiProcessorCount, dev));
        if (!w.ctrl) LA_DCK(cudaMalloc(&w.ctrl, sizeof(DualCtrl)));
        LA_DCK(cudaMallocHost(&w.h_ctrl, sizeof(DualCtrl)));
    }
    if (w.cap < n) {
        cudaFree(w.cm);
        cudaFree(w.last);
        cudaFree(w.seen);
        w.cm = nullptr;
        w.last = nullptr;
        w.seen = nullptr;
        w.cap = 0;
        if (cudaMalloc(&w.cm, sizeof(int) * n) != cudaSuccess) return LA_ERR_NOMEM;
        if (cudaMalloc(&w.last, sizeof(long long) * n) != cudaSuccess) return LA_ERR_NOMEM;
        if (cudaMalloc(&w.seen, sizeof(int) * n) != cudaSuccess) return LA_ERR_NOMEM;
        w.cap = n;
    }
    long long *v = reinterpret_cast<long long *>(v_out);
    LA_DCK(cudaMemsetAsync(w.seen, 0, sizeof(int) * n, s));
    LA_DCK(cudaMemsetAsync(w.ctrl, 0, sizeof(DualCtrl), s));
    const int tb = 256, gb = (n + tb - 1) / tb;
    k_dual_init<<<gb, tb, 0, s>>>(cost, n, match, v, w.cm, w.last, w.seen, w.ctrl);
    LA_DCK(cudaGetLastError());
    // 16-byte loads of four columns, where every row and v start on a 16-byte boundary
    const bool vec = n % 4 == 0 && (reinterpret_cast<uintptr_t>(cost) & 15) == 0 &&
                     (reinterpret_cast<uintptr_t>(v) & 15) == 0;
    int W = 32;                                        // threads per row: a power of two, at most the block
    while (W < kDualBlock && W * (vec ? 4 : 1) < n) W *= 2;
    const int grid = std::max(1, std::min(w.num_sms, (n + 3) / 4));
    // shortest paths have at most n arcs, and every epoch sweeps at least once
    int max_epochs = n + 2;
    const int32_t *C = cost;
    int nn = n;
    void *args[] = {(void *)&C, (void *)&nn, (void *)&match, (void *)&w.cm, (void *)&w.last, (void *)&v,
                    (void *)&W, (void *)&max_epochs, (void *)&w.ctrl};
    LA_DCK(cudaLaunchCooperativeKernel(vec ? (const void *)k_dual_sweeps<true> : (const void *)k_dual_sweeps<false>,
                                       dim3(grid), dim3(kDualBlock), args, 0, s));
    if (u_out) {
        k_dual_u<<<gb, tb, 0, s>>>(cost, n, match, v, reinterpret_cast<long long *>(u_out), w.ctrl);
        LA_DCK(cudaGetLastError());
    }
    LA_DCK(cudaMemcpyAsync(w.h_ctrl, w.ctrl, sizeof(DualCtrl), cudaMemcpyDeviceToHost, s));
    LA_DCK(cudaStreamSynchronize(s));
    if (w.h_ctrl->bad) return LA_ERR_INVALID;         // not a permutation
    return w.h_ctrl->settled ? LA_OK : LA_ERR_INTERNAL;   // still falling after n + 2 epochs: M is not optimal
}
