// Breadth-first discovery order: the order in which a sequential breadth-first search from the hub would take the
// nodes off its queue, each node's unvisited neighbours in id order.  It batches sources that are close to
// each other (see order_prepare).
//
// One cooperative launch builds the queue level by level.  A level's nodes are queue[qb, qe); every unit
// (a warp, or a block while the level has fewer nodes than blocks, so that the hub's thousands of arcs
// do not wait on one warp) takes a contiguous piece of them:
//   1. par[v] = min over v's parents of their queue position (unplaced v only: the position of a parent of a
//      placed node lies below qb);
//   2. each node counts the heads it is the parent of; the units' totals go to global memory;
//   3. with the totals before it, each unit appends its nodes' children, in arc (= id) order.
// A level of few nodes and arcs is done by the first block alone, arc by arc and without grid barriers, and so are
// the levels after it while they stay small: long chains, and the first and last levels of any graph (whole calls on
// a path of 3,000 nodes 126 -> 77 ms, on a 400 x 400 grid 240 -> 232; n = 2,000, every node a target 0.81 -> 0.78).
// No sort, and nothing for the host to read between levels.  Replaces one kernel per level, each with a
// host check, and a radix sort of every level (17 launches each): whole calls 1.25 -> 0.75 ms (n = 2,000, every node
// a target), 8.0 -> 6.3 ms (Brandes++, n = 200,000, 200 targets).  Bound by its barriers (three per larger level).
#include <algorithm>

#include "gridbar.cuh"
#include "order.cuh"

namespace bcpp {
namespace {

constexpr int OR_THREADS = 256;
constexpr int OR_WARPS = OR_THREADS / 32;
constexpr int OR_BLOCKS_PER_SM = 4;
constexpr int OR_SOLO_NODES = OR_THREADS, OR_SOLO_ARCS = 2048;   // a level for one block
constexpr int CTL_QB = 3, CTL_QE = 4, CTL_LEVEL = 5, CTL_DONE = 6;

// totals of the units before this block, and of all (tot[gridDim.x * OR_WARPS])
__device__ __forceinline__ void unit_prefix(const int32_t* tot, int64_t& before, int64_t& all) {
    __shared__ int64_t s_b[OR_WARPS], s_a[OR_WARPS];
    const int nu = (int)gridDim.x * OR_WARPS, mine = (int)blockIdx.x * OR_WARPS;
    int64_t b = 0, a = 0;
    for (int i = threadIdx.x; i < nu; i += OR_THREADS) {
        const int64_t x = __ldcg(tot + i);
        a += x;
        if (i < mine) b += x;
    }
    b = warp_sum(b);
    a = warp_sum(a);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        s_b[threadIdx.x >> 5] = b;
        s_a[threadIdx.x >> 5] = a;
    }
    __syncthreads();
    before = all = 0;
    for (int w = 0; w < OR_WARPS; w++) {
        before += s_b[w];
        all += s_a[w];
    }
}

// Small levels from queue[qb, qe) on, by one block; leaves the next level to do in the control words.
__device__ __noinline__ void solo_levels(int64_t qb, int64_t qe, int L, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                            int32_t* par, int32_t* queue, uint32_t* ctl) {
    __shared__ int64_t s_a0[OR_SOLO_NODES];
    __shared__ int32_t s_end[OR_SOLO_NODES], s_sum[OR_WARPS];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned lt = (1u << lane) - 1u;
    bool done = false;
    while (qe - qb <= OR_SOLO_NODES && L < ORDER_MAX_LEVELS) {
        const int cnt = (int)(qe - qb);
        __syncthreads();
        int64_t a0 = 0, d = 0;
        if (t < cnt) {
            const int32_t u = __ldcg(queue + qb + t);
            a0 = __ldg(rp + u);
            d = __ldg(rp + u + 1) - a0;
        }
        // (a row of more arcs than a level may have counts as that many)
        const int incl = warp_incl_scan((int)min(d, (int64_t)OR_SOLO_ARCS + 1), lane);
        if (lane == 31) s_sum[warp] = incl;
        __syncthreads();
        int before = 0, T = 0;
        for (int w = 0; w < OR_WARPS; w++) {
            if (w < warp) before += s_sum[w];
            T += s_sum[w];
        }
        s_a0[t] = a0 - (before + incl - d);   // arc j of the level is a0 + j - (arcs before the node)
        s_end[t] = before + incl;
        __syncthreads();
        if (T > OR_SOLO_ARCS) break;
        // node (from 0) of arc j: the first whose arcs end after it
        auto node_of = [&](int j) {
            int lo = 0, hi = cnt - 1;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (s_end[mid] > j) hi = mid;
                else lo = mid + 1;
            }
            return lo;
        };
        for (int j = t; j < T; j += OR_THREADS) {
            const int k = node_of(j);
            const int32_t v = __ldg(col + s_a0[k] + j), i = (int32_t)qb + k;
            if (__ldcg(par + v) > i) atomicMin(par + v, i);
        }
        __syncthreads();
        int64_t out = qe;
        for (int j0 = 0; j0 < T; j0 += OR_THREADS) {
            int32_t v = -1;
            if (j0 + t < T) {
                const int k = node_of(j0 + t);
                v = __ldg(col + s_a0[k] + j0 + t);
                if (__ldcg(par + v) != (int32_t)qb + k) v = -1;
            }
            const unsigned m = __ballot_sync(FULL, v >= 0);
            if (lane == 0) s_sum[warp] = __popc(m);
            __syncthreads();
            int64_t o = out;
            for (int w = 0; w < OR_WARPS; w++) {
                if (w < warp) o += s_sum[w];
                out += s_sum[w];
            }
            if (v >= 0) queue[o + __popc(m & lt)] = v;
            __syncthreads();
        }
        if (out == qe) {
            done = true;
            break;
        }
        qb = qe;
        qe = out;
        L++;
    }
    if (t == 0) {
        __stcg(ctl + CTL_QB, (uint32_t)qb);
        __stcg(ctl + CTL_QE, (uint32_t)qe);
        __stcg(ctl + CTL_LEVEL, (uint32_t)L);
        __stcg(ctl + CTL_DONE, done ? 1u : 0u);
    }
}

__global__ void __launch_bounds__(OR_THREADS, OR_BLOCKS_PER_SM)
order_bfs_kernel(int32_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col, int32_t* par, int32_t* queue,
                 uint32_t* ctl, int32_t* depth, uint32_t* flags) {
    __shared__ int32_t s_cnt[OR_WARPS + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int wid = blockIdx.x * OR_WARPS + warp, nw = gridDim.x * OR_WARPS;
    const int64_t tid = (int64_t)blockIdx.x * OR_THREADS + threadIdx.x, nt = (int64_t)gridDim.x * OR_THREADS;
    unsigned long long* hub = reinterpret_cast<unsigned long long*>(ctl + CTL_WORDS);
    int32_t* tot = reinterpret_cast<int32_t*>(ctl + CTL_WORDS + 2);
    // the hub: max of (degree << 32 | ~id)
    unsigned long long best = 0;
    for (int64_t v = tid; v < n; v += nt) {
        par[v] = INT32_MAX;
        const unsigned long long key =
            ((unsigned long long)(__ldg(rp + v + 1) - __ldg(rp + v)) << 32) | (0xffffffffu - (uint32_t)v);
        best = key > best ? key : best;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(FULL, best, o);
        best = x > best ? x : best;
    }
    if (lane == 0 && best) atomicMax(hub, best);
    if (!grid_barrier(ctl, flags)) return;
    if (tid == 0) {
        const int32_t src = (int32_t)(0xffffffffu - (uint32_t)(__ldcg(hub) & 0xffffffffull));
        queue[0] = src;
        par[src] = -1;
    }
    int64_t qb = 0, qe = 1;
    int L = 0;
    for (; L < ORDER_MAX_LEVELS; L++) {
        if (qe - qb <= OR_SOLO_NODES) {
            if (blockIdx.x == 0) solo_levels(qb, qe, L, rp, col, par, queue, ctl);
            if (!grid_barrier(ctl, flags)) return;
            // (the words change again only after the barriers of the level below)
            qb = __ldcg(ctl + CTL_QB);
            qe = __ldcg(ctl + CTL_QE);
            L = (int)__ldcg(ctl + CTL_LEVEL);
            if (__ldcg(ctl + CTL_DONE) || L >= ORDER_MAX_LEVELS) break;
        }
        const int64_t cnt = qe - qb;
        const bool wide = cnt < (int64_t)gridDim.x;   // a block per node
        const int64_t units = wide ? gridDim.x : nw, unit = wide ? blockIdx.x : wid;
        const int64_t per = (cnt + units - 1) / units;
        const int64_t i0 = min(qe, qb + unit * per), i1 = min(qe, i0 + per);
        const int step = wide ? OR_THREADS : 32, at = wide ? (int)threadIdx.x : lane;
        for (int64_t i = i0; i < i1; i++) {
            const int32_t u = __ldcg(queue + i);
            const int64_t a1 = __ldg(rp + u + 1);
            for (int64_t a = __ldg(rp + u) + at; a < a1; a += step) {
                const int32_t v = __ldg(col + a);
                if (__ldcg(par + v) > (int32_t)i) atomicMin(par + v, (int32_t)i);
            }
        }
        if (!grid_barrier(ctl, flags)) return;
        int c = 0;
        for (int64_t i = i0; i < i1; i++) {
            const int32_t u = __ldcg(queue + i);
            const int64_t a1 = __ldg(rp + u + 1);
            for (int64_t a = __ldg(rp + u) + at; a < a1; a += step) c += __ldcg(par + __ldg(col + a)) == (int32_t)i;
        }
        c = warp_sum(c);
        if (lane == 0) __stcg(tot + wid, c);
        if (!grid_barrier(ctl, flags)) return;
        int64_t before, all;
        unit_prefix(tot, before, all);
        if (all == 0) break;
        int64_t out = qe + before;
        if (!wide) {
            __syncthreads();
            if (lane == 0) s_cnt[warp] = c;
            __syncthreads();
            for (int w = 0; w < warp; w++) out += s_cnt[w];
            for (int64_t i = i0; i < i1; i++) {
                const int32_t u = __ldcg(queue + i);
                const int64_t a0 = __ldg(rp + u), a1 = __ldg(rp + u + 1);
                for (int64_t b = a0; b < a1; b += 32) {
                    int32_t v = -1;
                    if (b + lane < a1) {
                        v = __ldg(col + b + lane);
                        if (__ldcg(par + v) != (int32_t)i) v = -1;
                    }
                    const unsigned m = __ballot_sync(FULL, v >= 0);
                    if (v >= 0) queue[out + __popc(m & lt)] = v;
                    out += __popc(m);
                }
            }
        } else {
            for (int64_t i = i0; i < i1; i++) {
                const int32_t u = __ldcg(queue + i);
                const int64_t a0 = __ldg(rp + u), a1 = __ldg(rp + u + 1);
                for (int64_t b = a0; b < a1; b += OR_THREADS) {
                    int32_t v = -1;
                    if (b + threadIdx.x < a1) {
                        v = __ldg(col + b + threadIdx.x);
                        if (__ldcg(par + v) != (int32_t)i) v = -1;
                    }
                    const unsigned m = __ballot_sync(FULL, v >= 0);
                    __syncthreads();
                    if (lane == 0) s_cnt[warp] = __popc(m);
                    __syncthreads();
                    int64_t o = out;
                    for (int w = 0; w < OR_WARPS; w++) {
                        if (w < warp) o += s_cnt[w];
                        out += s_cnt[w];
                    }
                    if (v >= 0) queue[o + __popc(m & lt)] = v;
                }
            }
        }
        qb = qe;
        qe += all;
        if (!grid_barrier(ctl, flags)) return;
    }
    if (tid == 0) {
        depth[0] = L;
        depth[1] = 0;
    }
    if (qe >= n) return;
    // the nodes not placed, by id
    const int64_t per = ((int64_t)n + nw - 1) / nw;
    const int64_t v0 = min((int64_t)n, wid * per), v1 = min((int64_t)n, v0 + per);
    int c = 0, c2 = 0;
    for (int64_t v = v0 + lane; v < v1; v += 32) {
        const bool on = __ldcg(par + v) == INT32_MAX;
        c += on;
        c2 += on && __ldg(rp + v + 1) - __ldg(rp + v) >= 2;
    }
    c = warp_sum(c);
    c2 = warp_sum(c2);
    // (every block has read the last level's totals: it passed unit_prefix before or after the barrier below)
    if (!grid_barrier(ctl, flags)) return;
    if (lane == 0) {
        __stcg(tot + wid, c);
        if (c2) atomicAdd(depth + 1, c2);
    }
    if (!grid_barrier(ctl, flags)) return;
    int64_t before, all;
    unit_prefix(tot, before, all);
    __syncthreads();
    if (lane == 0) s_cnt[warp] = c;
    __syncthreads();
    int64_t out = qe + before;
    for (int w = 0; w < warp; w++) out += s_cnt[w];
    for (int64_t b = v0; b < v1; b += 32) {
        const int64_t v = b + lane;
        const bool on = v < v1 && __ldcg(par + v) == INT32_MAX;
        const unsigned m = __ballot_sync(FULL, on);
        if (on) queue[out + __popc(m & lt)] = (int32_t)v;
        out += __popc(m);
    }
}

__global__ void order_mark_kernel(const int32_t* __restrict__ S, int64_t ns, uint8_t* mem) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ns; i += (int64_t)gridDim.x * blockDim.x)
        mem[S[i]] = 1;
}
__global__ void order_flag_kernel(const int32_t* __restrict__ queue, int32_t n, const uint8_t* __restrict__ mem, int32_t* f) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        f[i] = mem[queue[i]];
}
__global__ void order_compact_kernel(const int32_t* __restrict__ queue, const int32_t* __restrict__ f,
                                     const int64_t* __restrict__ pos, int32_t n, uint32_t* out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        if (f[i]) out[pos[i]] = (uint32_t)queue[i];
}

inline unsigned blocks_for(int64_t n) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 8192)); }

}  // namespace

int64_t order_ctl_words(int num_sms) { return CTL_WORDS + 2 + (int64_t)num_sms * OR_BLOCKS_PER_SM * OR_WARPS; }

cudaError_t order_bfs_launch(int32_t n, const int64_t* rp, const int32_t* col, int32_t* par, int32_t* queue, uint32_t* ctl,
                             int32_t* depth, uint32_t* flags, int num_sms, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(ctl, 0, (size_t)order_ctl_words(num_sms) * sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, order_bfs_kernel, OR_THREADS, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorLaunchOutOfResources;
    per_sm = std::min(per_sm, OR_BLOCKS_PER_SM);
    // small graphs: fewer blocks, cheaper barriers
    const int blocks = (int)std::min<int64_t>((int64_t)per_sm * num_sms, std::max<int64_t>(num_sms / 2, ((int64_t)n + 63) / 64));
    void* args[] = {&n, &rp, &col, &par, &queue, &ctl, &depth, &flags};
    return cudaLaunchCooperativeKernel((const void*)order_bfs_kernel, dim3(blocks), dim3(OR_THREADS), args, 0, st);
}

void order_member(const int32_t* S, int64_t ns, const int32_t* queue, int32_t n, uint8_t* mem, int32_t* f, cudaStream_t st) {
    if (n <= 0) return;
    if (ns > 0) order_mark_kernel<<<blocks_for(ns), 256, 0, st>>>(S, ns, mem);
    order_flag_kernel<<<blocks_for(n), 256, 0, st>>>(queue, n, mem, f);
}

void order_compact(const int32_t* queue, const int32_t* f, const int64_t* pos, int32_t n, uint32_t* out, cudaStream_t st) {
    if (n > 0) order_compact_kernel<<<blocks_for(n), 256, 0, st>>>(queue, f, pos, n, out);
}

}  // namespace bcpp
