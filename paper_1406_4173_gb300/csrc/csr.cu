// CSR build and validation for the input graph G(V, E, W) (Sec. 3): undirected graphs with
// non-negative weights, restricted here to integer weights >= 1.  Building expands every
// undirected edge into two arcs, orders them by (tail, head), and rejects self-loops, repeated edges
// and zero weights.  Arcs are counted per tail (the count's atomics also give every arc a place in
// its row), scattered to their rows, and each row is sorted where it lies: in a warp's registers up to 32
// arcs, in shared memory up to CSR_LONG_ROW.  Nothing but the arcs themselves and one 32-bit place per arc
// is moved, and both fit the 129 MB L2 at 16 M arcs: 1.97 -> 0.70 ms for 8 M edges on 1 M nodes.  The arcs of longer rows
// are sorted together by the library's radix sort of 64-bit (row index, head) keys (all arcs of the graph that way
// before: star of 8 M edges 2.27 -> 1.49 ms).
#include <algorithm>

#include "csr.cuh"

namespace bcpp {

namespace {

// One more arc of tail u for every lane (all of mask m): its place in the row.  Lanes of one tail share an atomic.
__device__ __forceinline__ uint32_t next_place(uint32_t* counts, int32_t u, unsigned m) {
    const unsigned same = __match_any_sync(m, u);
    const int first = __ffs(same) - 1, lane = threadIdx.x & 31;
    uint32_t base = 0;
    if (lane == first) base = atomicAdd(&counts[u], (uint32_t)__popc(same));
    return __shfl_sync(same, base, first) + (uint32_t)__popc(same & ((1u << lane) - 1u));
}

// counts[u] = arcs of tail u (zeroed before); place[a] = place of arc a in its row (undirected: arc 2i is
// u -> v, arc 2i + 1 is v -> u).  Atomics to one address go one after the other, so the lanes of a warp that have a tail
// in common share one: first ends are looked at always (edge lists are often grouped by them), second ends where
// neighbouring lanes have the same.  8 M edges: star 7.7 -> 1.5 ms, random 0.48 -> 0.46; 2,000 nodes of degree
// 2,000: 0.56 -> 0.27.
__global__ void csr_count_kernel(int32_t n, int64_t m, const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                                 const uint32_t* __restrict__ ew, int directed, uint32_t* counts,
                                 uint32_t* __restrict__ place, uint32_t* flags) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t u = eu[i], v = ev[i];
        if (u < 0 || u >= n || v < 0 || v >= n) { flag_invalid(flags, WHY_RANGE); continue; }
        if (u == v) flag_invalid(flags, WHY_SELF_LOOP);
        if (ew && ew[i] == 0) flag_invalid(flags, WHY_WEIGHT_ZERO);
        const unsigned m = __activemask();
        const uint32_t p = next_place(counts, u, m);
        if (directed) {
            place[i] = p;
        } else {
            const int32_t before = __shfl_up_sync(m, v, 1);
            const bool shared = __any_sync(m, (threadIdx.x & 31) > 0 && v == before);
            reinterpret_cast<uint2*>(place)[i] = make_uint2(p, shared ? next_place(counts, v, m) : atomicAdd(&counts[v], 1u));
        }
    }
}

// the longest row, and the rows above CSR_LONG_ROW: their list and lengths (in any order) and all their arcs
__global__ void csr_longest_kernel(const uint32_t* __restrict__ counts, int32_t n, CsrLong* L, int32_t* rows, int64_t* len) {
    uint32_t x = 0;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t c = counts[u];
        x = max(x, c);
        if (c > CSR_LONG_ROW) {
            const uint32_t k = atomicAdd(&L->rows, 1u);
            rows[k] = (int32_t)u;
            len[k] = c;
            atomicAdd(&L->arcs, (unsigned long long)c);
        }
    }
    x = __reduce_max_sync(FULL, x);
    if ((threadIdx.x & 31) == 0 && x) atomicMax(&L->longest, x);
}

// keys of the arcs of row rows[blockIdx.y + ...]: (its index, head)
__global__ void csr_gather_kernel(int32_t n, int32_t nrows, const int32_t* __restrict__ rows, const int64_t* __restrict__ off,
                                  const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                  const uint32_t* __restrict__ w, uint64_t* __restrict__ keys, uint32_t* __restrict__ vals) {
    for (int32_t r = blockIdx.y; r < nrows; r += gridDim.y) {
        const int64_t a0 = rp[rows[r]], o = off[r], d = off[r + 1] - o;
        for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < d; j += (int64_t)gridDim.x * blockDim.x) {
            keys[o + j] = (uint64_t)r * (uint64_t)n + (uint32_t)col[a0 + j];
            vals[o + j] = w ? w[a0 + j] : 1u;
        }
    }
}
// ... and back, sorted; flags repeated arcs
__global__ void csr_return_kernel(int32_t n, int64_t arcs, const int32_t* __restrict__ rows, const int64_t* __restrict__ off,
                                  const int64_t* __restrict__ rp, const uint64_t* __restrict__ keys,
                                  const uint32_t* __restrict__ vals, int32_t* col, uint32_t* w, uint32_t* flags) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < arcs; j += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = keys[j], r = k / (uint64_t)n;
        const int64_t p = rp[rows[r]] + (j - off[r]);
        col[p] = (int32_t)(k - r * (uint64_t)n);
        if (w) w[p] = vals[j];
        if (j > 0 && keys[j - 1] == k) flag_invalid(flags, WHY_DUPLICATE);
    }
}

__global__ void csr_scatter_kernel(int64_t m, const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                                   const uint32_t* __restrict__ ew, int directed, const int64_t* __restrict__ rp,
                                   const uint32_t* __restrict__ place, int32_t* col, uint32_t* w) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t u = eu[i], v = ev[i];
        if (directed) {
            const int64_t p = rp[u] + place[i];
            col[p] = v;
            if (w) w[p] = ew[i];
        } else {
            const uint2 q = reinterpret_cast<const uint2*>(place)[i];
            const int64_t p = rp[u] + q.x, r = rp[v] + q.y;
            col[p] = v;
            col[r] = u;
            if (w) w[p] = w[r] = ew[i];
        }
    }
}

// A row's sort key: the head, with its weight behind it when there are weights.
template <bool W>
struct RowKey {
    using T = uint32_t;
    static __device__ __forceinline__ T load(const int32_t* col, const uint32_t*, int64_t p) { return (uint32_t)col[p]; }
    static __device__ __forceinline__ void store(int32_t* col, uint32_t*, int64_t p, T k) { col[p] = (int32_t)k; }
    static __device__ __forceinline__ uint32_t head(T k) { return k; }
};
template <>
struct RowKey<true> {
    using T = uint64_t;
    static __device__ __forceinline__ T load(const int32_t* col, const uint32_t* w, int64_t p) {
        return ((uint64_t)(uint32_t)col[p] << 32) | w[p];
    }
    static __device__ __forceinline__ void store(int32_t* col, uint32_t* w, int64_t p, T k) {
        col[p] = (int32_t)(k >> 32);
        w[p] = (uint32_t)k;
    }
    static __device__ __forceinline__ uint32_t head(T k) { return (uint32_t)(k >> 32); }
};

constexpr int CSR_WARP_ROW = 512;   // longest row a warp sorts in its shared memory
constexpr int CSR_SORT_WARPS = 8;

// bitonic sort of x[0, size) (size a power of two) by the nt threads t of a group that `sync` joins
template <typename T, class S>
__device__ __forceinline__ void bitonic(T* x, int size, int t, int nt, S&& sync) {
    for (int k = 2; k <= size; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = t; i < size / 2; i += nt) {
                const int a = 2 * i - (i & (j - 1)), b = a + j;
                const T xa = x[a], xb = x[b];
                if ((xa > xb) == ((a & k) == 0)) {
                    x[a] = xb;
                    x[b] = xa;
                }
            }
            sync();
        }
}

// Sorts the keys of each group of G lanes (G a power of two; at least `most` of them used, the others ~0).
template <int G, typename T>
__device__ __forceinline__ T sort_lanes(T k, int lane, int most) {
    const int l = lane & (G - 1);
#pragma unroll
    for (int s = 2; s <= G; s <<= 1) {
        if (s >= 2 * most) break;
#pragma unroll
        for (int j = s >> 1; j > 0; j >>= 1) {
            const T y = __shfl_xor_sync(FULL, k, j);
            k = ((l & j) == 0) == ((l & s) == 0) ? min(k, y) : max(k, y);
        }
    }
    return k;
}

// One warp per two rows, side by side when both have up to 16 arcs (8 M edges on 1 M nodes: 706 -> 683 us against a
// row at a time; the longer rows in shared memory take most of what is left); rows above CSR_WARP_ROW go on the list.
template <bool W>
__global__ void __launch_bounds__(CSR_SORT_WARPS * 32)
csr_sort_rows_kernel(int32_t n, const int64_t* __restrict__ rp, int32_t* col, uint32_t* w, int32_t* longrows,
                     uint32_t* nlong, uint32_t* flags) {
    using K = RowKey<W>;
    using T = typename K::T;
    __shared__ T s_x[CSR_SORT_WARPS][CSR_WARP_ROW];
    const int lane = threadIdx.x & 31;
    T* x = s_x[threadIdx.x >> 5];
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u0 = 2 * (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); u0 < n; u0 += 2 * nw) {
        const int64_t own = u0 + (lane >> 4);
        const int64_t own0 = own < n ? rp[own] : 0;
        const int64_t ownd = own < n ? rp[own + 1] - own0 : 0;
        const unsigned most = __reduce_max_sync(FULL, (unsigned)min(ownd, (int64_t)17));
        if (most < 2) continue;
        if (most <= 16) {
            const int l = lane & 15;
            const T k = sort_lanes<16>(l < ownd ? K::load(col, w, own0 + l) : ~(T)0, lane, (int)most);
            const uint32_t before = __shfl_up_sync(FULL, K::head(k), 1);
            if (l < ownd) {
                K::store(col, w, own0 + l, k);
                if (l > 0 && before == K::head(k)) flag_invalid(flags, WHY_DUPLICATE);
            }
            continue;
        }
        for (int64_t u = u0; u < min((int64_t)n, u0 + 2); u++) {
        const int64_t a0 = rp[u];
        const int64_t deg = rp[u + 1] - a0;
        if (deg < 2) continue;
        if (deg <= 32) {
            const T k = sort_lanes<32>(lane < deg ? K::load(col, w, a0 + lane) : ~(T)0, lane, (int)deg);
            const uint32_t before = __shfl_up_sync(FULL, K::head(k), 1);
            if (lane < deg) {
                K::store(col, w, a0 + lane, k);
                if (lane > 0 && before == K::head(k)) flag_invalid(flags, WHY_DUPLICATE);
            }
        } else if (deg <= CSR_WARP_ROW) {
            int size = 64;
            while (size < deg) size <<= 1;
            for (int i = lane; i < size; i += 32) x[i] = i < deg ? K::load(col, w, a0 + i) : ~(T)0;
            __syncwarp();
            bitonic(x, size, lane, 32, [] { __syncwarp(); });
            for (int i = lane; i < deg; i += 32) {
                K::store(col, w, a0 + i, x[i]);
                if (i > 0 && K::head(x[i - 1]) == K::head(x[i])) flag_invalid(flags, WHY_DUPLICATE);
            }
            __syncwarp();
        } else if (lane == 0) {
            longrows[atomicAdd(nlong, 1u)] = (int32_t)u;
        }
        }
    }
}

// One block per listed row of up to CSR_LONG_ROW arcs (dynamic shared memory: the longest one's power of two).
template <bool W>
__global__ void csr_sort_long_kernel(const int64_t* __restrict__ rp, int32_t* col, uint32_t* w,
                                     const int32_t* __restrict__ longrows, const uint32_t* __restrict__ nlong,
                                     uint32_t* flags) {
    using K = RowKey<W>;
    using T = typename K::T;
    extern __shared__ __align__(16) unsigned char s_raw[];
    T* x = reinterpret_cast<T*>(s_raw);
    for (uint32_t r = blockIdx.x; r < *nlong; r += gridDim.x) {
        const int64_t a0 = rp[longrows[r]];
        const int deg = (int)(rp[longrows[r] + 1] - a0);
        if (deg > (int)CSR_LONG_ROW) continue;   // sorted apart
        int size = 2 * CSR_WARP_ROW;
        while (size < deg) size <<= 1;
        for (int i = threadIdx.x; i < size; i += blockDim.x) x[i] = i < deg ? K::load(col, w, a0 + i) : ~(T)0;
        __syncthreads();
        bitonic(x, size, (int)threadIdx.x, (int)blockDim.x, [] { __syncthreads(); });
        for (int i = threadIdx.x; i < deg; i += blockDim.x) {
            K::store(col, w, a0 + i, x[i]);
            if (i > 0 && K::head(x[i - 1]) == K::head(x[i])) flag_invalid(flags, WHY_DUPLICATE);
        }
        __syncthreads();
    }
}

// One warp per row: sorted strictly increasing heads in range, no self-loop, weights >= 1,
// and for undirected graphs the reverse arc with the same weight.
// With node_off (graph arenas) heads are graph-local ids of the row's graph.
__global__ void csr_check_kernel(int32_t n, int64_t na, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                 const uint32_t* __restrict__ w, int directed, uint32_t* flags,
                                 unsigned long long* wmax, const int64_t* __restrict__ node_off, int32_t ngraphs) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    if (warp == 0 && lane == 0) {
        if (rp[0] != 0 || rp[n] != na) flag_invalid(flags, WHY_ROWPTR);
    }
    uint32_t local_max = 0;
    for (int64_t u = warp; u < n; u += nwarps) {
        const int64_t a0 = rp[u], a1 = rp[u + 1];
        if (a0 > a1 || a0 < 0 || a1 > na) {
            if (lane == 0) flag_invalid(flags, WHY_ROWPTR);
            continue;
        }
        int64_t gb = 0, ge = n;   // node range of the row's graph
        if (node_off) {
            int32_t lo = 0, hi = ngraphs;   // last g with node_off[g] <= u
            while (hi - lo > 1) {
                int32_t mid = (lo + hi) >> 1;
                if (node_off[mid] <= u) lo = mid; else hi = mid;
            }
            gb = node_off[lo];
            ge = node_off[lo + 1];
        }
        for (int64_t p = a0 + lane; p < a1; p += 32) {
            const int64_t vl = col[p];
            if (vl < 0 || vl >= ge - gb) { flag_invalid(flags, WHY_RANGE); continue; }
            const int64_t v = gb + vl;
            if (v == u) flag_invalid(flags, WHY_SELF_LOOP);
            if (p > a0 && col[p - 1] >= vl) flag_invalid(flags, WHY_UNSORTED);
            const uint32_t wv = w ? w[p] : 1u;
            if (wv == 0) flag_invalid(flags, WHY_WEIGHT_ZERO);
            if (wv > local_max) local_max = wv;
            if (!directed) {
                int64_t lo = rp[v], hi = rp[v + 1];
                if (lo < 0 || hi > na || lo > hi) { flag_invalid(flags, WHY_ROWPTR); continue; }
                const int32_t ul = (int32_t)(u - gb);
                while (lo < hi) {
                    int64_t mid = (lo + hi) >> 1;
                    if (col[mid] < ul) lo = mid + 1; else hi = mid;
                }
                if (lo >= rp[v + 1] || col[lo] != ul || (w && w[lo] != wv)) flag_invalid(flags, WHY_ASYMMETRIC);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) local_max = max(local_max, __shfl_xor_sync(FULL, local_max, o));
    if (lane == 0 && local_max) atomicMax(wmax, (unsigned long long)local_max);
}

// stats[0] = most arcs of rows [32 i, 32 i + 32), stats[1] = of one row (both zeroed before; a malformed row_ptr gives
// any number).  In the check itself, whose warps take a row each, it cost 130 us at n = 1,000,000.
__global__ void csr_stats_kernel(int32_t n, const int64_t* __restrict__ rp, unsigned long long* stats) {
    __shared__ unsigned long long s_max[2];
    if (threadIdx.x < 2) s_max[threadIdx.x] = 0ull;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    int64_t tile = 0, row = 0;
    for (int64_t u0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; u0 < n; u0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = u0 + lane, a0 = rp[min(u, (int64_t)n)], a1 = rp[min(u + 1, (int64_t)n)];
        row = max(row, a1 - a0);
        tile = max(tile, __shfl_sync(FULL, a1, 31) - __shfl_sync(FULL, a0, 0));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) row = max(row, __shfl_xor_sync(FULL, row, o));
    if (lane == 0) {
        atomicMax(&s_max[0], (unsigned long long)tile);
        atomicMax(&s_max[1], (unsigned long long)row);
    }
    __syncthreads();
    if (threadIdx.x < 2) atomicMax(stats + threadIdx.x, s_max[threadIdx.x]);
}

// Targets: in range and distinct; sets in_s[v] = 1 for v in S.
__global__ void targets_kernel(const int32_t* __restrict__ S, int32_t nS, int32_t n, uint8_t* in_s,
                               uint32_t* cnt, uint32_t* flags) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nS; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t s = S[i];
        if (s < 0 || s >= n) { flag_invalid(flags, WHY_TARGET); continue; }
        if (atomicAdd(&cnt[s], 1u) != 0) flag_invalid(flags, WHY_TARGET);
        in_s[s] = 1;
    }
}

// CSR transpose: count in-degrees (pass 0) or scatter (pass 1, cursor = row starts).
__global__ void transpose_kernel(int32_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                 const uint32_t* __restrict__ w, int64_t* counts_or_cursor, int32_t* tcol,
                                 uint32_t* tw, int pass) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = warp; u < n; u += nwarps) {
        for (int64_t p = rp[u] + lane; p < rp[u + 1]; p += 32) {
            const int32_t v = col[p];
            if (pass == 0) {
                atomicAdd((unsigned long long*)&counts_or_cursor[v], 1ull);
            } else {
                const int64_t q = (int64_t)atomicAdd((unsigned long long*)&counts_or_cursor[v], 1ull);
                tcol[q] = (int32_t)u;
                if (tw) tw[q] = w[p];
            }
        }
    }
}

// Disjoint union of graphs: heads must stay inside the row's graph; lcol = head - graph start.
__global__ void localize_kernel(int32_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                const int64_t* __restrict__ node_off, int32_t ngraphs, int32_t* __restrict__ lcol,
                                uint32_t* flags) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = warp; u < n; u += nwarps) {
        int32_t lo = 0, hi = ngraphs;
        while (hi - lo > 1) {
            int32_t mid = (lo + hi) >> 1;
            if (node_off[mid] <= u) lo = mid; else hi = mid;
        }
        const int64_t gb = node_off[lo], ge = node_off[lo + 1];
        for (int64_t p = rp[u] + lane; p < rp[u + 1]; p += 32) {
            const int32_t v = col[p];
            if (v < gb || v >= ge) flag_invalid(flags, WHY_RANGE);
            lcol[p] = (int32_t)(v - gb);
        }
    }
}

inline unsigned grid_for(int64_t work, int threads, int max_blocks = 8192) {
    int64_t b = (work + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (unsigned)b;
}

}  // namespace

void csr_count(int32_t n, int64_t m, const int32_t* eu, const int32_t* ev, const uint32_t* ew, int directed,
               uint32_t* counts, uint32_t* place, CsrLong* L, int32_t* rows, int64_t* len, uint32_t* flags,
               cudaStream_t st) {
    if (m <= 0) return;
    csr_count_kernel<<<grid_for(m, 256), 256, 0, st>>>(n, m, eu, ev, ew, directed, counts, place, flags);
    csr_longest_kernel<<<grid_for(n, 256, 1024), 256, 0, st>>>(counts, n, L, rows, len);
}

void csr_gather_rows(int32_t n, int32_t nrows, const int32_t* rows, const int64_t* off, const int64_t* rp, const int32_t* col,
                     const uint32_t* w, uint64_t* keys, uint32_t* vals, cudaStream_t st) {
    const dim3 grid((unsigned)std::max(8, 152 * 8 / std::max(nrows, 1)), (unsigned)std::min(nrows, 65535));
    if (nrows > 0) csr_gather_kernel<<<grid, 256, 0, st>>>(n, nrows, rows, off, rp, col, w, keys, vals);
}

void csr_return_rows(int32_t n, int64_t arcs, const int32_t* rows, const int64_t* off, const int64_t* rp, const uint64_t* keys,
                     const uint32_t* vals, int32_t* col, uint32_t* w, uint32_t* flags, cudaStream_t st) {
    if (arcs > 0) csr_return_kernel<<<grid_for(arcs, 256), 256, 0, st>>>(n, arcs, rows, off, rp, keys, vals, col, w, flags);
}

void csr_scatter(int64_t m, const int32_t* eu, const int32_t* ev, const uint32_t* ew, int directed, const int64_t* rp,
                 const uint32_t* place, int32_t* col, uint32_t* w, cudaStream_t st) {
    if (m > 0) csr_scatter_kernel<<<grid_for(m, 256), 256, 0, st>>>(m, eu, ev, ew, directed, rp, place, col, w);
}

template <bool W>
static cudaError_t csr_sort_t(int32_t n, uint32_t longest, const int64_t* rp, int32_t* col, uint32_t* w, int32_t* longrows,
                              uint32_t* nlong, uint32_t* flags, cudaStream_t st) {
    csr_sort_rows_kernel<W><<<grid_for((int64_t)n * 16, CSR_SORT_WARPS * 32, 152 * 64), CSR_SORT_WARPS * 32, 0, st>>>(
        n, rp, col, w, longrows, nlong, flags);
    if (longest <= (uint32_t)CSR_WARP_ROW) return cudaSuccess;
    size_t size = 2 * CSR_WARP_ROW;
    while (size < std::min(longest, CSR_LONG_ROW)) size <<= 1;
    const size_t bytes = size * sizeof(typename RowKey<W>::T);
    const cudaError_t e =
        cudaFuncSetAttribute(csr_sort_long_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    csr_sort_long_kernel<W><<<152 * 8, 256, bytes, st>>>(rp, col, w, longrows, nlong, flags);
    return cudaSuccess;
}

cudaError_t csr_sort_rows(int32_t n, uint32_t longest, const int64_t* rp, int32_t* col, uint32_t* w, int32_t* longrows,
                          uint32_t* nlong, uint32_t* flags, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    return w ? csr_sort_t<true>(n, longest, rp, col, w, longrows, nlong, flags, st)
             : csr_sort_t<false>(n, longest, rp, col, w, longrows, nlong, flags, st);
}

void csr_check(int32_t n, int64_t na, const int64_t* rp, const int32_t* col, const uint32_t* w, int directed,
               uint32_t* flags, unsigned long long* wmax, cudaStream_t st, const int64_t* node_off, int32_t ngraphs) {
    csr_check_kernel<<<grid_for((int64_t)n * 32, 256), 256, 0, st>>>(n, na, rp, col, w, directed, flags, wmax,
                                                                      node_off, ngraphs);
}

void csr_stats(int32_t n, const int64_t* rp, unsigned long long* stats, cudaStream_t st) {
    if (n > 0) csr_stats_kernel<<<grid_for(n, 256, 152 * 4), 256, 0, st>>>(n, rp, stats);
}

void csr_localize(int32_t n, const int64_t* rp, const int32_t* col, const int64_t* node_off, int32_t ngraphs,
                  int32_t* lcol, uint32_t* flags, cudaStream_t st) {
    if (n > 0 && ngraphs > 0)
        localize_kernel<<<grid_for((int64_t)n * 32, 256), 256, 0, st>>>(n, rp, col, node_off, ngraphs, lcol, flags);
}

void targets_check(const int32_t* S, int32_t nS, int32_t n, uint8_t* in_s, uint32_t* cnt, uint32_t* flags,
                   cudaStream_t st) {
    if (nS > 0) targets_kernel<<<grid_for(nS, 256), 256, 0, st>>>(S, nS, n, in_s, cnt, flags);
}

void csr_transpose_count(int32_t n, const int64_t* rp, const int32_t* col, int64_t* counts, cudaStream_t st) {
    transpose_kernel<<<grid_for((int64_t)n * 32, 256), 256, 0, st>>>(n, rp, col, nullptr, counts, nullptr, nullptr, 0);
}

void csr_transpose_fill(int32_t n, const int64_t* rp, const int32_t* col, const uint32_t* w, int64_t* cursor,
                        int32_t* tcol, uint32_t* tw, cudaStream_t st) {
    transpose_kernel<<<grid_for((int64_t)n * 32, 256), 256, 0, st>>>(n, rp, col, w, cursor, tcol, tw, 1);
}

}  // namespace bcpp
