// The Centrality step (Eq. 13): distances, counts and dependencies of the non-frontier nodes from their
// part's frontiers.
//
// Eq. 13 ranges over all of a part's frontiers, but only those with sigma_i(f,v) > 0 matter: a shortest
// path from s to v enters v's part for the last time through some frontier f, and what follows it is a
// shortest f-v path inside the part without another frontier, so d(s,f) + d_i(f,v) = d(s,v) and
// sigma_i(f,v) > 0 (Dijkstra_SK counts exactly these paths, Eq. 10); every other frontier's sum is at least
// d(s,v) and its term of the count is zero.  The same holds for the exits.  So each node keeps a short list of (frontier,
// distance, count), compacted once from the tables (a few per cent of them: most paths between a node
// and a far frontier pass another frontier), and the per-batch work is a visit of these lists.
//
// A warp takes a (batch, node), lanes are the batch's 32 sources.  Entries: the minimum of d(s,f) +
// d_i(f,v); then the counts of those that attain it.  Exits: frontiers with d(s,f) = d(s,v) + d_i(v,f)
// add sigma_i(v,f) c(s,f).  Rows of one part's frontiers are read by its nodes one after the other, so they
// come from L1 and L2.
//
// Replaces a min-plus product over all of a part's frontiers (three sweeps over the tables per batch): Chung-Lu
// n = 1,000,000, 2,048 targets 273 -> 16.0 ms (about 750 frontiers per part, lists of a few); n = 100,000, 512
// targets 7.2 -> 0.45 ms; 200,000 nodes in 100 parts of about 60 frontiers (nearly all of them listed),
// 200 targets 3.2 -> 2.6 ms.  The last is bound by instruction issue (73% of the cycles) and FP64 (31%);
// adding every entry for all lanes, as soon as one source needs it, kept it at 4.3 ms with FP64 at 77%.
#include <algorithm>

#include "skeleton.cuh"

namespace bcpp {
namespace {

constexpr int CT_WARPS = 8;
constexpr int CT_STAGE = 128;    // list entries a warp keeps in shared memory (longer lists: a stage at a time)

template <typename DT>
struct CtSm {
    int2 ft[CT_STAGE];
    uint64_t mu[CT_STAGE];
    DT md[CT_STAGE];     // the count as the dependency type
};

// non-zero counts of each node's table row (unit.pad = index of the unit's first node)
__global__ void ct_count_kernel(const CentralityUnit* __restrict__ units, int nunits, SkTables T, bool exits,
                                int64_t* cnt) {
    const int lane = threadIdx.x & 31;
    const uint64_t* ts = exits ? T.tsr : T.ts;
    for (int b = blockIdx.x; b < nunits; b += gridDim.x) {
        const CentralityUnit U = units[b];
        const int32_t nf = T.nf[U.part];
        for (int32_t v = U.v0 + (threadIdx.x >> 5); v < U.v1; v += CT_WARPS) {
            const uint64_t* row = ts + T.toff[U.part] + (int64_t)v * nf;
            int c = 0;
            for (int32_t f = lane; f < nf; f += 32) c += __ldg(row + f) != 0ull;
            c = warp_sum(c);
            if (lane == 0) cnt[U.pad + v - U.v0] = c;
        }
    }
}

// the lists themselves, in frontier order: skeleton row of the frontier, distance, count
__global__ void ct_fill_kernel(const CentralityUnit* __restrict__ units, int nunits, SkTables T, bool exits,
                               const int32_t* __restrict__ skbase, const int64_t* __restrict__ rp, int2* ft,
                               uint64_t* mu) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const uint64_t* ts = exits ? T.tsr : T.ts;
    const int32_t* td = exits ? T.tdr : T.td;
    for (int b = blockIdx.x; b < nunits; b += gridDim.x) {
        const CentralityUnit U = units[b];
        const int32_t nf = T.nf[U.part];
        for (int32_t v = U.v0 + (threadIdx.x >> 5); v < U.v1; v += CT_WARPS) {
            const int64_t t0 = T.toff[U.part] + (int64_t)v * nf;
            int64_t out = rp[U.pad + v - U.v0];
            for (int32_t f0 = 0; f0 < nf; f0 += 32) {
                const int32_t f = f0 + lane;
                const uint64_t x = f < nf ? __ldg(ts + t0 + f) : 0ull;
                const unsigned m = __ballot_sync(FULL, x != 0ull);
                if (x) {
                    const int64_t q = out + __popc(m & lt);
                    ft[q] = make_int2(skbase[U.part] + f, __ldg(td + t0 + f));
                    mu[q] = x;
                }
                out += __popc(m);
            }
        }
    }
}

// LISTS: both lists are there; else those that are not are read from the tables (entries without paths add nothing: their
// distance is that of a path, their count zero).
template <typename DT, bool LISTS>
__global__ void __launch_bounds__(CT_WARPS * 32, 5)
centrality_kernel(const CentralityUnit* __restrict__ units, int nslots, SkTables T, const uint32_t* __restrict__ pnodes,
                  const int32_t* __restrict__ skbase, CentralityLists E, CentralityLists X,
                  const int32_t* __restrict__ d_all,
                  const uint64_t* __restrict__ sg_all, const DT* __restrict__ dl_all, int64_t cap_n, double* bc_sum,
                  double* bc_cmp, int64_t cap_bc, const uint32_t* __restrict__ skip, uint32_t* flags) {
    __shared__ CtSm<DT> s_warp[CT_WARPS];
    CtSm<DT>& sm = s_warp[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const CentralityUnit U = units[blockIdx.x];
    bool ovf = false;
    for (int slot = blockIdx.y; slot < nslots; slot += gridDim.y) {
        if (skip && __ldg(skip + slot)) continue;   // a batch without rows
        // rows of this slot, this lane's source
        const int32_t* dr = d_all + (int64_t)slot * cap_n * 32 + lane;
        const uint64_t* sr = sg_all + (int64_t)slot * cap_n * 32 + lane;
        const DT* cr = dl_all + (int64_t)slot * cap_n * 32 + lane;
        for (int32_t v = U.v0 + (threadIdx.x >> 5); v < U.v1; v += CT_WARPS) {
            const int32_t q = U.pad + v - U.v0;
            // f(entries staged) for every stage of a list; the stage of a short list stays for a second visit
            auto staged = [&](const CentralityLists& L, bool exits, bool again, auto&& f) {
                const bool list = LISTS || L.rp;
                const int64_t a0 = list ? __ldg(L.rp + q) : T.toff[U.part] + (int64_t)v * T.nf[U.part];
                const int cnt = list ? (int)(__ldg(L.rp + q + 1) - a0) : T.nf[U.part];
                for (int c0 = 0; c0 < cnt; c0 += CT_STAGE) {
                    const int m = min(CT_STAGE, cnt - c0);
                    if (!again || cnt > CT_STAGE) {
                        __syncwarp();
                        for (int k = lane; k < m; k += 32) {
                            const int64_t e = a0 + c0 + k;
                            sm.ft[k] = list ? __ldg(L.ft + e)
                                            : make_int2(skbase[U.part] + c0 + k, __ldg((exits ? T.tdr : T.td) + e));
                            const uint64_t mu = __ldg((list ? L.mu : exits ? T.tsr : T.ts) + e);
                            sm.mu[k] = mu;
                            sm.md[k] = (DT)mu;
                        }
                        __syncwarp();
                    }
                    f(m);
                }
            };
            // distances (two of them at most DINF = 2^31 - 1, so a sum never wraps; DINF and above: none)
            uint32_t best = (uint32_t)DINF;
            staged(E, false, false, [&](int m) {
                int k = 0;
                for (; k + 4 <= m; k += 4) {
                    uint32_t d[4];
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const int2 e = sm.ft[k + j];
                        d[j] = (uint32_t)dr[(int64_t)e.x * 32] + (uint32_t)e.y;
                    }
                    best = min(best, min(min(d[0], d[1]), min(d[2], d[3])));
                }
                for (; k < m; k++) {
                    const int2 e = sm.ft[k];
                    best = min(best, (uint32_t)dr[(int64_t)e.x * 32] + (uint32_t)e.y);
                }
            });
            if (!__any_sync(FULL, best < (uint32_t)DINF)) continue;
            // counts over the entries that attain it, dependencies over the exits on a shortest path
            uint64_t sv = 0;
            DT acc = (DT)0;
            // (each source first marks its own entries of 32, then adds them: a warp-wide FP64 operation
            // costs 16 SM cycles, and the sources' entries differ)
            auto sums = [&](int m, bool entries, bool exits) {
                for (int k0 = 0; k0 < m; k0 += 32) {
                    unsigned in = 0u, out = 0u;
                    if (best < (uint32_t)DINF) {
                        const int n = min(32, m - k0);
#pragma unroll 4
                        for (int k = 0; k < n; k++) {
                            const int2 e = sm.ft[k0 + k];
                            const uint32_t d = (uint32_t)dr[(int64_t)e.x * 32];
                            if (d + (uint32_t)e.y == best) in |= 1u << k;
                            if (best + (uint32_t)e.y == d && d != (uint32_t)DINF) out |= 1u << k;
                        }
                    }
                    if (!entries) in = 0u;
                    if (!exits) out = 0u;
                    while (in) {
                        const int k = k0 + __ffs(in) - 1;
                        in &= in - 1u;
                        const int k2 = in ? k0 + __ffs(in) - 1 : k;
                        const uint64_t x = sr[(int64_t)sm.ft[k].x * 32];
                        const uint64_t x2 = in ? sr[(int64_t)sm.ft[k2].x * 32] : 0ull;
                        in &= in - 1u;
                        sv = madd_ck(sv, x, sm.mu[k], ovf);
                        sv = madd_ck(sv, x2, sm.mu[k2], ovf);
                    }
                    while (out) {
                        const int k = k0 + __ffs(out) - 1;
                        out &= out - 1u;
                        const int k2 = out ? k0 + __ffs(out) - 1 : k;
                        const DT x = cr[(int64_t)sm.ft[k].x * 32];
                        const DT x2 = out ? cr[(int64_t)sm.ft[k2].x * 32] : (DT)0;
                        out &= out - 1u;
                        if (x != (DT)0) acc += sm.md[k] * x;      // with few targets most c are zero
                        if (x2 != (DT)0) acc += sm.md[k2] * x2;
                    }
                    __syncwarp();
                }
            };
            if (T.ts == T.tsr) {   // undirected: one list for both
                staged(E, false, true, [&](int m) { sums(m, true, true); });
            } else {
                staged(E, false, true, [&](int m) { sums(m, true, false); });
                staged(X, true, false, [&](int m) { sums(m, false, true); });
            }
            double delta = (double)((DT)sv * acc);
            if (!__any_sync(FULL, delta != 0.0)) continue;
            const double tot = warp_sum(delta);
            if (lane == 0 && tot != 0.0) {
                const int64_t ix = (int64_t)slot * cap_bc + pnodes[T.pstart[U.part] + v];
                double s0 = bc_sum[ix], c0 = bc_cmp[ix];
                neumaier_add(s0, c0, tot);
                bc_sum[ix] = s0;
                bc_cmp[ix] = c0;
            }
        }
    }
    if (__any_sync(FULL, ovf) && lane == 0) atomicOr(&flags[FLAG_SIGMA_OVF], 1u);
}

}  // namespace

void ct_count(const CentralityUnit* units, int nunits, SkTables T, bool exits, int64_t* cnt, cudaStream_t st) {
    if (nunits > 0)
        ct_count_kernel<<<std::min(nunits, 152 * 64), CT_WARPS * 32, 0, st>>>(units, nunits, T, exits, cnt);
}

void ct_fill(const CentralityUnit* units, int nunits, SkTables T, bool exits, const int32_t* skbase, const int64_t* rp,
             int2* ft, uint64_t* mu, cudaStream_t st) {
    if (nunits > 0)
        ct_fill_kernel<<<std::min(nunits, 152 * 64), CT_WARPS * 32, 0, st>>>(units, nunits, T, exits, skbase, rp, ft, mu);
}

void centrality_launch(bool fp32_delta, const CentralityUnit* units, int nunits, int nslots, SkTables T,
                       const uint32_t* pnodes, const int32_t* skbase, CentralityLists E, CentralityLists X, const int32_t* d,
                       const uint64_t* sg, const void* dl, int64_t cap_n, double* bc_sum, double* bc_cmp,
                       int64_t cap_bc, const uint32_t* skip, uint32_t* flags, cudaStream_t st) {
    if (nunits <= 0 || nslots <= 0) return;
    // neighbouring blocks take one batch's neighbouring nodes: their frontier rows are shared in L2
    const dim3 grid((unsigned)nunits, (unsigned)std::min(nslots, 65535));
    auto go = [&](auto kernel, auto* c) {
        kernel<<<grid, CT_WARPS * 32, 0, st>>>(units, nslots, T, pnodes, skbase, E, X, d, sg, c, cap_n, bc_sum, bc_cmp, cap_bc,
                                               skip, flags);
    };
    const bool lists = E.rp && X.rp;
    if (fp32_delta) {
        const float* c = static_cast<const float*>(dl);
        if (lists) go(centrality_kernel<float, true>, c);
        else go(centrality_kernel<float, false>, c);
    } else {
        const double* c = static_cast<const double*>(dl);
        if (lists) go(centrality_kernel<double, true>, c);
        else go(centrality_kernel<double, false>, c);
    }
}

}  // namespace bcpp
