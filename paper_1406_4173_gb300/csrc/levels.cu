// Level-mask passes of plain Brandes (Eq. 2 / Eq. 5-7) and Brandes_SK (Eq. 11 / Eq. 12) for many batches of 32 sources at once.
//
// Layout.  A row is one (batch, node) pair; its 32 positions are the batch's sources.  Instead of a
// distance per source, a row has one 32-bit mask per distance level: bit s of lev[D][row] says that
// source s reaches the node at distance D.  One 4-byte gather then answers for 32 sources what a
// distance row answers with 32 to 128 bytes.
//
// Forward, level D (pull): every row that some source has not reached gathers lev[D - w] of its
// in-neighbours; the sources found there and not seen before are the row's new mask, and their path
// counts are the sums over exactly the arcs whose gathered mask has the source's bit.  No tentative
// distances, no buckets, no settle lists, no atomics on global memory.
// Backward, level D from the deepest: a row with a mask at D gathers lev[D + w] of its
// out-neighbours; c(s,u) = (I + delta) / sigma is summed over the arcs whose mask has the bit.  A
// pair whose c is zero (no target behind it) is taken out of the mask, so nobody adds it.
//
// Work split.  The whole GPU takes one level of all batches of a wave at a time (a cooperative launch
// with a grid barrier per level); warps take tiles of 32 rows in order, so that the SMs sweep one or
// two batches at a time, whose count rows (n * 128 bytes) stay in L2.  In a tile, arcs are spread
// over lanes (a lane per arc: heads and masks), the few arcs with a bit in common are compacted
// in shared memory, and then (row, source) pairs are spread over lanes: a lane sums the counts (or
// dependencies) of its pair over the row's compacted arcs.  So neither low degrees nor rows with
// few active sources leave lanes idle, and the FP64 adds of the backward pass, which GB300 issues at
// 2 lanes per SM and cycle, are done for packed pairs only.
//
// Measured against the lockstep kernel (whole call, FP64): Chung-Lu n = 50,000, every node a target
// 251 -> 119 ms; n = 1,000,000, 4,096 targets 709 -> 135 ms; directed, n = 100,000, weights 1 to 16,
// 2,000 targets 141 -> 34 ms; 4,096 random graphs 427 -> 177 ms; n = 2,000, every node 1.76 -> 0.77 ms.
// Brandes_SK (Eq. 11 / Eq. 12: weights, multiplicities, 64-bit counts, and the distance rows that the
// Centrality step reads) 51 -> 4.1 ms at n = 100,000 and 512 targets, 695 -> 133 ms at n = 1,000,000 and
// 2,048 targets.
// Bound by the latency of its gathers (a profile at n = 10,000: instructions issued on 40% of the
// cycles, FP64 pipe busy 38%) and, in the backward pass, by FP64 adds (pipe busy 63% of it).
//
// Giving back.  A batch that reaches a level past those provided for, or a path count of 2^32 in 32-bit rows, is marked
// (LmArgs::back), left out of the backward pass and run by the lockstep kernel; the others finish.
#include <algorithm>
#include <type_traits>

#include "gridbar.cuh"
#include "levels.cuh"

namespace bcpp {
namespace {

constexpr int LM_THREADS = 256;
constexpr int LM_WARPS = LM_THREADS / 32;
// Resident blocks per SM: 5 (48 registers, 40 warps) with 32-bit counts, 4 with 64-bit counts.  The two large
// Chung-Lu and the batched workload below on 4 blocks: 126 / 151 / 184 ms, on 5: 119 / 136 / 174, on 6
// (spills): 128 / 152 / 183.
constexpr int lm_min_blocks(bool narrow) { return narrow ? 5 : 4; }
// Values in flight per pair (unit weights: 2 131 / 166 / 195 ms, 3 119 / 137 / 173, 4 121 / 140 / 174 on the
// three workloads above) and chunks of 32 arcs whose gathers overlap (1 127 / 154 / 181, 2 125 / 144 / 178;
// with weights, Brandes_SK at n = 1,000,000: 1 148 ms, 2 139, 3 135).
template <bool WEIGHTED>
constexpr int LM_PAIRS = WEIGHTED ? 4 : 3;
template <bool WEIGHTED>
constexpr int LM_GATHERS = WEIGHTED ? 3 : 2;
constexpr int LM_MAX_SUB = 3;      // units of 4 rows at least
constexpr int LM_CAP = 256;        // arcs of one round of a tile (rows of larger degree go one by one)
constexpr int CTL_WIDE = 3, CTL_BACK = 4;   // batches with a path count past 32 bits; batches given back
constexpr int CTL_MOST = 5;                 // batches given back that take the others with them, less one
constexpr int CTL_LVL = CTL_WORDS;
constexpr unsigned LVL_ANY = 1u, LVL_STOP = 2u;
constexpr int PROBE_WORDS = 6;
// Words between two batches' depths: a 128-byte line each, since every SM stores to them once per level (side by
// side, stores of 152 SMs to a few lines held up everyone's loads: n = 10,000, every node a target 7.4 -> 6.3 ms,
// Brandes++ at n = 100,000 8.6 -> 7.8 ms).
constexpr int DEPTH_STRIDE = 32;

// 1/x for small path counts, correctly rounded by the compiler
constexpr int RCP_N = 1024;
struct RcpTable {
    double v[RCP_N];
    constexpr RcpTable() : v() {
        for (int i = 1; i < RCP_N; i++) v[i] = 1.0 / i;
    }
};
__device__ const RcpTable c_rcp{};

__device__ __forceinline__ double recip_of(uint64_t s) {
    if (s < (uint64_t)RCP_N) return __ldg(&c_rcp.v[(int)s]);
    // single-precision seed and one Newton-Raphson step (relative error below 1.5e-14)
    const double x = (double)s;
    const double r = (double)__frcp_rn((float)x);
    return fma(r, fma(-x, r, 1.0), r);
}

template <typename DT>
__device__ __forceinline__ DT recip_as(uint64_t s) {
    if constexpr (sizeof(DT) == 4) return 1.0f / (float)s;
    else return recip_of(s);
}

// FP32 sums are taken in the lockstep kernel's order, so that both give the same bits: with a sources at the
// row's distance and K = 32 / (a rounded up to a power of two), arc j of the row goes to partial sum j mod K, in
// order, and the partial sums are added pairwise (neighbours first).  Terms come as (arc, value); eight
// partial sums are held at a time.
struct TreeSum {
    float (*p)[32];   // [8][lane], in shared memory: few terms, and a register array would cost eight selects each
    int lane;
    float a, b;
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int z = 0; z < 8; z++) p[z][lane] = 0.0f;
    }
    __device__ __forceinline__ void add(int arc, int K, int part, float t) {
        const int z = arc & (K - 1);
        if (t != 0.0f && (z >> 3) == part) p[z & 7][lane] += t;
    }
    // after the terms of partial sums 8 part .. 8 part + 7
    __device__ __forceinline__ void close(int part) {
        const float t = ((p[0][lane] + p[1][lane]) + (p[2][lane] + p[3][lane])) +
                        ((p[4][lane] + p[5][lane]) + (p[6][lane] + p[7][lane]));
        if (part == 0) a = t;
        else if (part == 1) a = a + t;
        else if (part == 2) b = t;
        else b = b + t;
    }
    __device__ __forceinline__ float total(int K) const { return K > 16 ? a + b : a; }
};
__device__ __forceinline__ int partial_sums(uint32_t at_distance) {
    const int a = __popc(at_distance);
    return 32 >> (a <= 1 ? 0 : 32 - __clz(a - 1));
}

template <bool MULT, bool TREE = false>
struct WarpSm {
    uint2 list[LM_CAP];        // arcs with a bit in common: head row, mask
    uint64_t mult[MULT ? LM_CAP : 1];   // their multiplicities (uint64 forward, double backward)
    int seg[33];               // first list entry of each candidate
    uint32_t nm[32];           // masks found, by candidate
    uint32_t rowm[32];         // masks found, by row of the tile
    double ds[32];             // dependencies, by row of the tile
    int idx[32];               // compaction scratch
    float part[TREE ? 8 : 1][32];   // TreeSum
};

// position of the n-th set bit (from 0) of x; n < popc(x)
__device__ __forceinline__ int nth_bit(uint32_t x, int n) {
    int pos = 0;
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) {
        const int c = __popc(x & ((1u << h) - 1u));
        const bool up = n >= c;
        n -= up ? c : 0;
        pos += up ? h : 0;
        x = up ? x >> h : x;
    }
    return pos;
}

// 32 x 32 bit transpose: bit s of lane j's x becomes bit j of lane s's result
__device__ __forceinline__ uint32_t transpose_bits(uint32_t x, int lane) {
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) {
        // bits whose index has the h bit clear
        const uint32_t lowm = h == 16 ? 0x0000ffffu : h == 8 ? 0x00ff00ffu : h == 4 ? 0x0f0f0f0fu
                                                  : h == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(FULL, x, h);
        x = lane & h ? (x & ~lowm) | ((y >> h) & lowm) : (x & lowm) | ((y << h) & ~lowm);
    }
    return x;
}

// Every (lane, bit) of the lanes' masks, in order, U chunks of 32 at a time: f(ok[], k[], s[], first[]) for
// source s of lane k's mask; `first` has a bit for every lane of the chunk that starts a new k.
template <int U, class F>
__device__ __forceinline__ void for_pairs(uint32_t mask, int lane, int* idx, F&& f) {
    const unsigned le = 0xffffffffu >> (31 - lane);
    const unsigned nb = __ballot_sync(FULL, mask != 0u);
    if (nb == 0u) return;
    if (mask) idx[__popc(nb & (le >> 1))] = lane;
    const int cnt = __popc(mask);
    const int incl = warp_incl_scan(cnt, lane);
    const int total = __shfl_sync(FULL, incl, 31);
    const int st = incl - cnt;
    __syncwarp();
    int kb = -1;
    for (int p0 = 0; p0 < total; p0 += 32 * U) {
        unsigned first[U];
        int k[U], s[U];
        bool ok[U];
#pragma unroll
        for (int g = 0; g < U; g++) {
            const unsigned at = (unsigned)(st - p0 - 32 * g);
            first[g] = __reduce_or_sync(FULL, mask != 0u && at < 32u ? 1u << at : 0u);
            k[g] = idx[kb + __popc(first[g] & le)];
            kb += __popc(first[g]);
            const uint32_t mk = __shfl_sync(FULL, mask, k[g]);
            const int n = p0 + 32 * g + lane - __shfl_sync(FULL, st, k[g]);
            ok[g] = p0 + 32 * g + lane < total;
            s[g] = ok[g] ? nth_bit(mk, n) : 0;
        }
        f(ok, k, s, first);
    }
    __syncwarp();
}

// The tile's sums over its candidates' arcs.  FWD: in-arcs, masks at D - w, counts; else out-arcs,
// masks at D + w, dependencies.  need / a0 / deg: this lane's row (need = 0: none).  Found masks go to
// sm.rowm by row (zeroed by the caller).
//   pair_done(ok, r, s, acc, first): the sum of source s of the tile's row r (packed pairs)
//   row_done(r, mask, acc): the same for all 32 sources of one row, lane = source
//   ovf: a 64-bit count wrapped
// TABLE (Dijkstra_SK): a frontier other than the source (nodes below nf, distance above 0) takes part in the
// distances but not in the counts, so its arcs add to the found masks only.
template <bool FWD, bool WEIGHTED, bool MULT, bool TABLE, typename V, typename ACC, class SM, class PD, class RD>
__device__ __forceinline__ void tile_sums(const LmArgs& A, SM& sm, int lane, uint32_t need, int64_t a0, int deg,
                                          int D, int bd, int64_t rb, const int32_t* __restrict__ col,
                                          const int32_t* __restrict__ wt, const V* vals, int32_t nf, bool& ovf,
                                          PD&& pair_done,
                                          RD&& row_done) {
    constexpr bool TREE = std::is_same<V, float>::value;
    constexpr int PU = LM_PAIRS<WEIGHTED>, GU = LM_GATHERS<WEIGHTED>;
    // A row of many arcs: with unit weights many of a chunk's arcs have a bit in common, and each source takes
    // its own of them; with weights few have, and the warp takes them one after the other.
    constexpr int BU = WEIGHTED ? 4 : 2, BG = 4;
    const unsigned le = 0xffffffffu >> (31 - lane), lt = le >> 1;
    const bool cand = need != 0u && deg > 0;
    const unsigned cm = __ballot_sync(FULL, cand);
    if (cm == 0u) return;
    // candidates to the front lanes; with unit weights (many pairs per visit) by degree, so that
    // neighbouring pairs have sums of similar length (n = 50,000: 125 -> 121 ms; with weights the sort
    // costs more than it gives)
    const int K = __popc(cm);
    int crow;
    if constexpr (WEIGHTED) {
        if (cand) sm.idx[__popc(cm & lt)] = lane;
        __syncwarp();
        crow = lane < K ? sm.idx[lane] : 0;
        __syncwarp();
    } else {
        uint32_t key = cand ? ((uint32_t)min(deg, 1 << 26) << 5) | (uint32_t)lane : 0xffffffffu;
#pragma unroll
        for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
            for (int j = k >> 1; j > 0; j >>= 1) {
                const uint32_t y = __shfl_xor_sync(FULL, key, j);
                key = ((lane & j) == 0) == ((lane & k) == 0) ? min(key, y) : max(key, y);
            }
        crow = lane < K ? (int)(key & 31u) : 0;
    }
    const uint32_t cneed = __shfl_sync(FULL, need, crow);
    const uint32_t ca0 = __shfl_sync(FULL, (uint32_t)a0, crow);   // fewer than 2^31 arcs
    const int cd = __shfl_sync(FULL, deg, crow);
    const int cdeg = lane < K ? cd : 0;
    const int pre = warp_incl_scan(cdeg, lane);
    const uint32_t* L1 = A.lev + (int64_t)(FWD ? D - 1 : D + 1) * A.rows + rb;   // unit weights
    auto gather = [&](int32_t v, int32_t w) -> uint32_t {
        if constexpr (!WEIGHTED) return L1[v];
        const int d2 = FWD ? D - w : D + w;
        return (FWD ? d2 >= 0 : d2 <= bd) ? A.lev[(int64_t)d2 * A.rows + rb + v] : 0u;
    };
    // multiplicity of arc a, as 64 bits
    auto mult_of = [&](uint32_t a) -> uint64_t {
        if constexpr (!MULT) return 0;
        else return FWD ? __ldg(A.imu + a) : (uint64_t)__double_as_longlong(__ldg(A.mud + a));
    };
    // acc += mult * t
    auto add = [&](ACC& acc, V t, uint64_t mu) {
        if constexpr (sizeof(V) == 4) acc += t;   // fewer than 2^31 counts below 2^32
        else if constexpr (!FWD) acc = MULT ? fma(__longlong_as_double((long long)mu), t, acc) : acc + t;
        else acc = MULT ? madd_ck(acc, t, mu, ovf) : add_ck(acc, t, ovf);
    };
    auto counts = [&](int32_t v, int32_t w) { return !TABLE || v >= nf || D == w; };
    int k0 = 0;
    while (k0 < K) {
        const int base = __shfl_sync(FULL, pre - cdeg, k0);
        const unsigned fit = __ballot_sync(FULL, lane >= k0 && lane < K && pre - base <= LM_CAP);
        if (fit == 0u) {
            // one row of many arcs: lane = source
            const uint32_t nd = __shfl_sync(FULL, cneed, k0);
            const uint32_t b0 = __shfl_sync(FULL, ca0, k0);
            const int dg = __shfl_sync(FULL, cdeg, k0);
            const int r = __shfl_sync(FULL, crow, k0);
            ACC acc = (ACC)0;
            uint32_t found = 0u;
            TreeSum tree{sm.part, lane, 0.0f, 0.0f};
            const int parts = TREE ? partial_sums(nd) : 1;
            for (int part = 0; part < (TREE ? (parts + 7) / 8 : 1); part++) {
            if (TREE && parts > 1) tree.clear();
            for (int c4 = 0; c4 < dg; c4 += 32 * BG) {
                // The masks of BG chunks at once, since at most levels none of them has a bit in common and a row of
                // thousands of arcs was a chain of round trips (50,000 nodes on 60 hubs, 1,000 sources: 34.4 ->
                // 17.2 ms; star of 200,000, 1,000 sources: 16.5 -> 10.7; directed, weights up to 16: 34.8 -> 33.6).
                // Kept in shared memory: registers spill.
                bool any = false;
                int32_t v4[BG], w4[BG];
#pragma unroll
                for (int q = 0; q < BG; q++) {
                    const int c = c4 + 32 * q + lane;
                    v4[q] = c < dg ? __ldg(col + b0 + c) : -1;
                    w4[q] = WEIGHTED && c < dg ? __ldg(wt + b0 + c) : 1;
                }
#pragma unroll
                for (int q = 0; q < BG; q++) {
                    uint32_t m = v4[q] >= 0 ? gather(v4[q], w4[q]) & nd : 0u;
                    found |= m;
                    if (!counts(v4[q], w4[q])) m = 0u;
                    any |= m != 0u;
                    sm.list[32 * q + lane] = make_uint2((uint32_t)v4[q], m);
                }
                if (!__any_sync(FULL, any)) continue;
#pragma unroll 1
                for (int q = 0; q < BG; q++) {
                const uint2 x = sm.list[32 * q + lane];
                const int32_t v = (int32_t)x.x;
                const uint32_t m = x.y;
                const uint64_t mu = MULT && m ? mult_of(b0 + c4 + 32 * q + lane) : 0;
                uint32_t own = WEIGHTED ? __ballot_sync(FULL, m != 0u) : transpose_bits(m, lane);
                while (__any_sync(FULL, own != 0u)) {
                    V t[BU];
                    uint64_t muq[BU];
                    int jq[BU];
#pragma unroll
                    for (int q = 0; q < BU; q++) {
                        const int j = own ? __ffs(own) - 1 : 0;
                        jq[q] = j;
                        const int32_t vq = __shfl_sync(FULL, v, j);
                        muq[q] = MULT ? shfl_u64(mu, j) : 0;
                        uint32_t mq = 0xffffffffu;
                        if constexpr (WEIGHTED) mq = __shfl_sync(FULL, m, j);
                        const bool on = own != 0u && (mq >> lane) & 1u;
                        t[q] = on ? vals[(rb + vq) * 32 + lane] : (V)0;
                        own &= own - 1u;
                    }
#pragma unroll
                    for (int q = 0; q < BU; q++)
                        if (TREE && parts > 1) tree.add(jq[q], parts, part, t[q]);
                        else if (q == 0 || FWD || __any_sync(FULL, t[q] != (V)0)) add(acc, t[q], muq[q]);
                }
                }
            }
            if (TREE && parts > 1) tree.close(part);
            }
            if (TREE && parts > 1) acc = tree.total(parts);
            found = __reduce_or_sync(FULL, found);
            if (found) {
                if (lane == 0) sm.rowm[r] = found;
                row_done(r, found, acc);
            }
            k0++;
            continue;
        }
        const int k1 = k0 + __popc(fit);
        const int T = __shfl_sync(FULL, pre, k1 - 1) - base;
        const bool inr = lane >= k0 && lane < k1;
        const int st = pre - cdeg - base;
        sm.nm[lane] = 0u;
        __syncwarp();
        int pos = 0, kb = k0 - 1;
        for (int i0 = 0; i0 < T; i0 += 32 * GU) {
            unsigned first[GU];
            int k[GU];
            uint32_t a[GU], m[GU];
            int32_t v[GU], w[GU], stk[GU];
#pragma unroll
            for (int g = 0; g < GU; g++) {
                const unsigned at = (unsigned)(st - i0 - 32 * g);
                first[g] = __reduce_or_sync(FULL, inr && at < 32u ? 1u << at : 0u);
                k[g] = kb + __popc(first[g] & le);
                kb += __popc(first[g]);
                a[g] = __shfl_sync(FULL, ca0 - (uint32_t)st, k[g]) + (uint32_t)(i0 + 32 * g + lane);
                m[g] = __shfl_sync(FULL, cneed, k[g]);
                stk[g] = TREE ? __shfl_sync(FULL, st, k[g]) : 0;
                v[g] = 0;
                w[g] = 1;
                if (i0 + 32 * g + lane < T) {
                    v[g] = __ldg(col + a[g]);
                    if (WEIGHTED) w[g] = __ldg(wt + a[g]);
                } else {
                    m[g] = 0u;
                }
            }
#pragma unroll
            for (int g = 0; g < GU; g++)
                if (m[g]) {
                    m[g] &= gather(v[g], w[g]);
                    if (TABLE && m[g] && !counts(v[g], w[g])) {
                        atomicOr(&sm.nm[k[g]], m[g]);
                        m[g] = 0u;
                    }
                }
#pragma unroll
            for (int g = 0; g < GU; g++) {
                const unsigned tb = __ballot_sync(FULL, m[g] != 0u);
                const int p = pos + __popc(tb & lt);
                if (m[g]) {
                    // (FP32: the arc's place in its row, mod 32, above the head's 25 bits)
                    const uint32_t at = TREE ? (uint32_t)(i0 + 32 * g + lane - stk[g]) << 27 : 0u;
                    sm.list[p] = make_uint2((uint32_t)v[g] | at, m[g]);
                    if constexpr (MULT) sm.mult[p] = mult_of(a[g]);
                    atomicOr(&sm.nm[k[g]], m[g]);
                }
                if ((first[g] >> lane) & 1u) sm.seg[k[g]] = p;
                pos += __popc(tb);
            }
        }
        if (lane == 0) sm.seg[k1] = pos;
        __syncwarp();
        const uint32_t nm = inr ? sm.nm[lane] : 0u;
        if (nm) sm.rowm[crow] = nm;
        for_pairs<1>(nm, lane, sm.idx, [&](const bool* ok, const int* k, const int* s, const unsigned* first) {
            // the row's listed arcs, in step for all its sources (their values share cache lines)
            const int e1 = ok[0] ? sm.seg[k[0] + 1] : 0;
            int e = ok[0] ? sm.seg[k[0]] : 0;
            const int r = __shfl_sync(FULL, crow, k[0]);
            const V* vs = vals + rb * 32 + s[0];
            ACC acc = (ACC)0;
            if constexpr (TREE) {
                const int parts = partial_sums(__shfl_sync(FULL, cneed, k[0]));
                TreeSum tree{sm.part, lane, 0.0f, 0.0f};
                for (int part = 0; parts > 1 && part < (parts + 7) / 8; part++) {
                    tree.clear();
                    for (int i = e; i < e1; i += PU) {
                        V t[PU];
                        uint2 x[PU];
#pragma unroll
                        for (int q = 0; q < PU; q++) {
                            t[q] = (V)0;
                            x[q] = i + q < e1 ? sm.list[i + q] : make_uint2(0u, 0u);
                            if ((x[q].y >> s[0]) & 1u) t[q] = vs[(int64_t)(x[q].x & 0x1ffffffu) * 32];
                        }
#pragma unroll
                        for (int q = 0; q < PU; q++) tree.add((int)(x[q].x >> 27), parts, part, t[q]);
                    }
                    tree.close(part);
                }
                if (parts > 1) acc = tree.total(parts);   // (one partial sum: in order, below)
                if (parts > 1) e = e1;
            }
            while (e < e1) {
                V t[PU];
#pragma unroll
                for (int q = 0; q < PU; q++) {
                    t[q] = (V)0;
                    if (e + q < e1) {
                        const uint2 x = sm.list[e + q];
                        if ((x.y >> s[0]) & 1u) t[q] = vs[(int64_t)(TREE ? x.x & 0x1ffffffu : x.x) * 32];
                    }
                }
#pragma unroll
                for (int q = 0; q < PU; q++)
                    add(acc, t[q], MULT ? sm.mult[min(e + q, e1 - 1)] : 0);
                e += PU;
            }
            pair_done(ok[0], r, s[0], acc, first[0]);
        });
        __syncwarp();
        k0 = k1;
    }
}

// Pairs reached by level D, by D / 2 and by 3 D / 4, and all pairs, of a sample of the unfinished batches' rows; rows of
// these batches, and all rows sampled.  (Its own function: inlined, it cost the kernel's loops registers, n = 10,000:
// 6.1 -> 6.9 ms.)
__device__ __noinline__ void probe_levels(const uint32_t* lev, int64_t rows, int D, int wmax, const uint32_t* bdepth,
                                          const LsItem* items, const int32_t* tile_item, int32_t item_base, int32_t tpb,
                                          uint32_t* probe) {
    const int64_t nt = (int64_t)gridDim.x * LM_THREADS, step = max((int64_t)1, rows / nt);
    uint32_t b1 = 0, b2 = 0, b3 = 0, pairs = 0, open = 0, total = 0;
    for (int64_t row = ((int64_t)blockIdx.x * LM_THREADS + threadIdx.x) * step; row < rows; row += nt * step) {
        const int32_t t = (int32_t)(row >> 5);
        const int it = tile_item ? __ldg(tile_item + t) - item_base : t / tpb;
        total++;
        if ((int)bdepth[it * DEPTH_STRIDE] + wmax < D) continue;   // (a batch that is done has no masks there)
        open++;
        pairs += __ldg(&items[it].nsrc);
        for (int l = 0; l <= D; l++) {
            const uint32_t c = __popc(__ldcg(lev + (int64_t)l * rows + row));
            b2 += c;
            if (l <= D / 2) b1 += c;
            if (l <= D - D / 4) b3 += c;
        }
    }
    b1 = __reduce_add_sync(FULL, b1);
    b2 = __reduce_add_sync(FULL, b2);
    b3 = __reduce_add_sync(FULL, b3);
    pairs = __reduce_add_sync(FULL, pairs);
    open = __reduce_add_sync(FULL, open);
    total = __reduce_add_sync(FULL, total);
    if ((threadIdx.x & 31) == 0 && total) {
        atomicAdd(probe, b1);
        atomicAdd(probe + 1, b2);
        atomicAdd(probe + 2, pairs);
        atomicAdd(probe + 3, open);
        atomicAdd(probe + 4, total);
        atomicAdd(probe + 5, b3);
    }
}
// D (pairs / b2)^(1 / dim) levels needed, with 2^dim = b2 / b1: more than 2^k D?  Not when fewer pairs are found in the
// last quarter than in the one before, by `keep`: the search runs out (directed graphs, where most pairs are never
// reached; 20,000 nodes without cycles, weights up to 9, 300 targets: 4.1 -> 3.2 ms).
__device__ __noinline__ bool looks_deep(const uint32_t* probe, int k, float keep) {
    const float b1 = (float)__ldcg(probe), b2 = (float)__ldcg(probe + 1), b3 = (float)__ldcg(probe + 5), g = b2 / b1;
    float x = (float)__ldcg(probe + 2) / b2;
    for (; k > 0; k--) x /= g;
    return b1 > 0.0f && g >= 1.5f && x > 1.0f && b2 - b3 >= keep * (b3 - b1);
}

// Marks the batches that are given back: those deeper than `most`, which could still grow past the level where the
// pass was cut, and those with a path count past 32 bits.  The backward pass takes them for empty.
__device__ __noinline__ void mark_back(uint32_t* bdepth, int nitems, int most, uint32_t* back, uint32_t* ctl,
                                       uint32_t* flags) {
    for (int it = blockIdx.x * LM_THREADS + threadIdx.x; it < nitems; it += gridDim.x * LM_THREADS) {
        uint32_t* b = bdepth + (int64_t)it * DEPTH_STRIDE;
        const uint32_t why = ((int)b[0] > most ? MASKS_DEEP : 0u) | (b[1] ? MASKS_COUNT : 0u);
        if (why) {
            b[0] = 0u;
            back[it] = 1u;
            atomicOr(&flags[FLAG_MASKS], why);
            atomicAdd(ctl + CTL_BACK, 1u);
        }
    }
}

// A batch has a path count past 32 bits; more than ctl[CTL_MOST] of them: the level is the last.  (Not inlined: n = 1,000,000,
// 4,096 targets 135.9 -> 135.3 ms.)
__device__ __noinline__ void note_wide(uint32_t* b, uint32_t* ctl, int D) {
    if (atomicExch(b + 1, 1u) == 0u && atomicAdd(ctl + CTL_WIDE, 1u) + 1u > __ldcg(ctl + CTL_MOST)) atomicOr(ctl + CTL_LVL + D, LVL_STOP);
}

template <typename SG, typename DT, bool WEIGHTED, bool MULT, bool TABLE>
__global__ void __launch_bounds__(LM_THREADS, lm_min_blocks(sizeof(SG) == 4))
lm_kernel(const LmArgs A, const int sub_log) {
    using Sm = WarpSm<MULT, std::is_same<DT, float>::value>;
    __shared__ Sm s_warp[LM_WARPS];
    __shared__ int s_last;   // last level of the forward pass
    const int lane = threadIdx.x & 31;
    Sm& sm = s_warp[threadIdx.x >> 5];
    const int wid = blockIdx.x * LM_WARPS + (threadIdx.x >> 5);
    const int nw = gridDim.x * LM_WARPS;
    SG* sg = static_cast<SG*>(A.sg);
    DT* cc = static_cast<DT*>(A.cc);
    uint32_t* lvl = A.ctl + CTL_LVL;
    uint32_t* bdepth = lvl + A.lcap + 1;
    const int wmax = WEIGHTED ? A.wmax : 1;
    unsigned long long t0 = 0, t1 = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0 && A.phase_ns) asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));

    struct Tile {
        LsItem I;
        int32_t n, u;
        int64_t base, rb;
        int it;
    };
    auto tile_of = [&](int t) {
        Tile x;
        int tile0;
        if (A.item_tile0) {
            x.it = __ldg(A.tile_item + t + A.tile_base) - A.item_base;
            tile0 = __ldg(A.item_tile0 + x.it) - A.tile_base;
        } else {
            x.it = t / A.tpb;
            tile0 = x.it * A.tpb;
        }
        const int4 q = __ldg(reinterpret_cast<const int4*>(A.items) + x.it);
        x.I.g = q.x; x.I.src_off = q.y; x.I.nsrc = q.z; x.I.aux = q.w;
        x.base = __ldg(A.node_off + x.I.g);
        x.n = (int32_t)(__ldg(A.node_off + x.I.g + 1) - x.base);
        x.u = (t - tile0) * 32 + lane;
        x.rb = (int64_t)tile0 * 32;
        return x;
    };

    // an earlier wave of the pass looked too deep (only set past a barrier of this launch, if by it)
    if (__ldcg(A.flags + FLAG_MASKS) & MASKS_ALL) {
        for (int it = blockIdx.x * LM_THREADS + threadIdx.x; it < A.nitems; it += gridDim.x * LM_THREADS) A.back[it] = 1u;
        return;
    }

    // With few tiles per warp a unit is a part of a tile (32 >> sub_log rows), so that a level's last and
    // fullest tiles do not leave the other warps waiting (see lm_go for the rule).
    // Units go out in order: the first of every warp by its index, the others from one counter per
    // pass and level, a few at a time (a fixed assignment of all of them left warps waiting for the
    // rows of high degree: 245 -> 164 ms on 1,000,000 nodes and 4,096 sources).
    uint32_t* work = bdepth + (int64_t)A.nitems * DEPTH_STRIDE;
    const int nunits = A.ntiles << sub_log;
    const int grab = max(1, min(8, nunits / (16 * nw)));
    auto for_units = [&](uint32_t* ctr, auto&& f) {
        const bool more = nunits > nw;
        int mine = 0;
        if (more && lane == 0) mine = nw + (int)atomicAdd(ctr, (uint32_t)grab);
        if (wid < nunits) f(wid);
        if (!more) return;
        for (;;) {
            const int t0 = __shfl_sync(FULL, mine, 0);
            if (t0 >= nunits) break;
            if (lane == 0) mine = nw + (int)atomicAdd(ctr, (uint32_t)grab);   // the next ones, while these run
            const int t1 = min(t0 + grab, nunits);
            for (int t = t0; t < t1; t++) f(t);
        }
    };

    if (blockIdx.x == 0 && threadIdx.x == 0) A.ctl[CTL_MOST] = (uint32_t)(A.nitems / (A.few ? 3 : 2));
    // level 0: each batch's sources
    for (int t = wid; t < A.ntiles; t += nw) {
        const Tile x = tile_of(t);
        const int64_t row = (int64_t)t * 32 + lane;
        const int32_t src = lane < x.I.nsrc ? __ldg(A.srcs + x.I.src_off + lane) : -1;
        const int local = src - (x.u - lane);
        sm.rowm[lane] = 0u;
        if (sizeof(SG) == 8 && A.drow) {
            int4* dr = reinterpret_cast<int4*>(A.drow + (int64_t)t * 1024);
            double2* cr = reinterpret_cast<double2*>(cc + (int64_t)t * 1024);   // (64-bit counts come with FP64 only)
#pragma unroll 4
            for (int i = lane; i < 256; i += 32) dr[i] = make_int4(DINF, DINF, DINF, DINF);
            if (cc)
#pragma unroll 4
                for (int i = lane; i < 512; i += 32) cr[i] = make_double2(0.0, 0.0);
        }
        __syncwarp();
        if (src >= 0 && local >= 0 && local < 32) {
            atomicOr(&sm.rowm[local], 1u << lane);
            sg[(x.rb + src) * 32 + lane] = (SG)1;
            if (sizeof(SG) == 8 && A.drow) A.drow[(x.rb + src) * 32 + lane] = 0;
            if constexpr (TABLE) {
                const int64_t o = __ldg(A.toff + x.I.g) + (int64_t)src * __ldg(A.nfront + x.I.g) + x.I.aux + lane;
                A.td[o] = 0;
                A.ts[o] = 1ull;
            }
        }
        __syncwarp();
        const uint32_t m = sm.rowm[lane];
        A.lev[row] = m;
        A.seen[row] = m;
        A.dsum[row] = 0.0;
        __syncwarp();
    }
    if (!grid_barrier(A.ctl, A.flags)) return;

    // ------------------------------------------------------------------ forward
    // A batch that may reach a later level when the pass is cut, and one with a path count past 32 bits (second word
    // beside its depth), is given back; the others go on.
    // (The last level is kept in shared memory: a register for it cost the weighted instances 1 to 3%.)
    int depth = 0;
    for (int D = 1; D < A.lcap; D++) {
        bool any = false, ovf = false;
        for_units(work + D, [&](int unit) {
            const int t = unit >> sub_log;
            const bool mine = lane >> (5 - sub_log) == (unit & ((1 << sub_log) - 1));
            const Tile x = tile_of(t);
            // finished batches: nothing new within the largest weight.  (A cached load: the values of
            // earlier levels decide, and this SM's own store below shows up in it.)
            const int bd = (int)bdepth[x.it * DEPTH_STRIDE];
            if (bd + wmax < D) return;
            const int64_t row = (int64_t)t * 32 + lane;
            const uint32_t full = x.I.nsrc >= 32 ? 0xffffffffu : (1u << x.I.nsrc) - 1u;
            uint32_t seen = 0u, need = 0u;
            int64_t a0 = 0;
            int deg = 0;
            if (mine && x.u < x.n) {
                seen = A.seen[row];
                need = full & ~seen;
                if (need) {
                    const int64_t* rp = A.irp + x.base + x.u;
                    a0 = __ldg(rp);
                    deg = (int)(__ldg(rp + 1) - a0);
                }
            }
            sm.rowm[lane] = 0u;
            __syncwarp();
            SG* srow = sg + (int64_t)t * 1024;
            int32_t* drow = sizeof(SG) == 8 && A.drow ? A.drow + (int64_t)t * 1024 : nullptr;
            const int32_t nf = TABLE ? __ldg(A.nfront + x.I.g) : 0;
            const int64_t tab = TABLE ? __ldg(A.toff + x.I.g) + (int64_t)(x.u - lane) * nf + x.I.aux : 0;
            auto settle = [&](bool ok, int r, int s, uint64_t acc) {
                if (ok) {
                    srow[r * 32 + s] = (SG)acc;
                    if constexpr (TABLE) {
                        A.td[tab + (int64_t)r * nf + s] = D;
                        A.ts[tab + (int64_t)r * nf + s] = acc;
                    }
                    if (drow) drow[r * 32 + s] = D;
                    if (sizeof(SG) == 4 && (acc >> 32) != 0) note_wide(bdepth + x.it * DEPTH_STRIDE, A.ctl, D);
                }
            };
            tile_sums<true, WEIGHTED, MULT, TABLE, SG, uint64_t>(
                A, sm, lane, need, a0, deg, D, 0, x.rb, A.icol, A.iw, sg, nf, ovf,
                [&](bool ok, int r, int s, uint64_t acc, unsigned) { settle(ok, r, s, acc); },
                [&](int r, uint32_t mask, uint64_t acc) { settle((mask >> lane) & 1u, r, lane, acc); });
            __syncwarp();
            const uint32_t got = sm.rowm[lane];
            if (mine) A.lev[(int64_t)D * A.rows + row] = got;
            if (got) A.seen[row] = seen | got;
            if (__any_sync(FULL, got != 0u)) {
                any = true;
                if (lane == 0 && bd != D) bdepth[x.it * DEPTH_STRIDE] = (uint32_t)D;
            }
            __syncwarp();
        });
        if (sizeof(SG) == 8 && __any_sync(FULL, ovf) && lane == 0) atomicOr(&A.flags[FLAG_SIGMA_OVF], 1u);
        if (any && lane == 0 && __ldcg(lvl + D) == 0u) atomicOr(lvl + D, LVL_ANY);
        if (threadIdx.x == 0) s_last = D;
        if (!grid_barrier(A.ctl, A.flags)) return;
        // every block reads the same word: nobody writes level D's status any more
        const uint32_t w = __ldcg(lvl + D);
        if (w & LVL_ANY) depth = D;
        if (D - depth >= wmax || (sizeof(SG) == 4 && (w & LVL_STOP))) break;
        // Too deep a graph shows early: an eighth and a quarter of the way the pairs reached by now and by half of that
        // give the dimension that the balls around the sources grow with, and with it the level at which
        // they hold every pair; past the levels provided for (at an eighth: past twice as many), the unfinished batches
        // are given back without going there first, and with them the later waves of a graph, when they are most of
        // the wave.  (Binary tree of 131,071 nodes, weights up to 30, 512 sources: 92.7 -> 90.1 ms, 88.2 without the attempt.)
        // Balls that hardly grow any more belong to stragglers, not to a deep graph.
        const int part = A.lcap / 8;
        const bool early = D <= part + 1;   // (small waves: the test costs about as much as it saves)
        if (A.probe && (D == part || D == part + 1 || D == 2 * part || D == 2 * part + 1) && (!early || A.ntiles >= nw)) {
            uint32_t* probe = work + 2 * A.lcap + (early ? 0 : PROBE_WORDS);
            if (D == part || D == 2 * part) {
                probe_levels(A.lev, A.rows, D, wmax, bdepth, A.items, A.item_tile0 ? A.tile_item + A.tile_base : nullptr,
                             A.item_base, A.tpb, probe);
            } else if (looks_deep(probe, early ? 4 : 2, TABLE ? 0.0f : 0.9f)) {
                if (blockIdx.x == 0 && threadIdx.x == 0 && !A.item_tile0 && 2 * __ldcg(probe + 3) > __ldcg(probe + 4))
                    atomicOr(&A.flags[FLAG_MASKS], MASKS_ALL);
                break;
            }
        }
    }
    // Cut: the batches could still grow.  (With a bound, weighted skeletons, only empty levels are missing.)
    const uint32_t nwide = sizeof(SG) == 4 ? __ldcg(A.ctl + CTL_WIDE) : 0u;
    const bool cut = s_last - depth < wmax && (sizeof(SG) == 4 || !A.bounded);
    if (cut || nwide) {
        const int some = A.nitems / (A.few ? 3 : 2);
        mark_back(bdepth, A.nitems, (int)nwide > some ? -1 : cut ? s_last - wmax : INT32_MAX, A.back, A.ctl, A.flags);
        if (!grid_barrier(A.ctl, A.flags)) return;
        const int back = (int)__ldcg(A.ctl + CTL_BACK);
        if (back == A.nitems) return;
        if (A.few && back > some) {
            for (int it = blockIdx.x * LM_THREADS + threadIdx.x; it < A.nitems; it += gridDim.x * LM_THREADS) A.back[it] = 1u;
            return;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && A.phase_ns) asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));

    if (TABLE || !cc) return;
    // ------------------------------------------------------------------ backward
    // (level 0 is the sources themselves: nothing is credited to them and nobody reads their c)
    for (int D = depth; D >= 1; D--) {
        for_units(work + A.lcap + D, [&](int unit) {
            const int t = unit >> sub_log;
            const bool mine = lane >> (5 - sub_log) == (unit & ((1 << sub_log) - 1));
            const int64_t row = (int64_t)t * 32 + lane;
            const Tile x = tile_of(t);
            const int bd = (int)bdepth[x.it * DEPTH_STRIDE];
            if (D > bd) return;
            uint32_t* lrow = A.lev + (int64_t)D * A.rows + row;
            const uint32_t need = mine ? *lrow : 0u;
            if (!__any_sync(FULL, need != 0u)) return;
            int64_t a0 = 0;
            int deg = 0;
            bool tgt = false;
            if (need) {
                if (D < bd) {
                    const int64_t* rp = A.rp + x.base + x.u;
                    a0 = __ldg(rp);
                    deg = (int)(__ldg(rp + 1) - a0);
                }
                tgt = A.in_s ? __ldg(A.in_s + x.base + x.u) != 0 : true;
            }
            const unsigned tm = __ballot_sync(FULL, tgt);
            sm.rowm[lane] = 0u;
            sm.ds[lane] = 0.0;
            __syncwarp();
            const SG* srow = sg + (int64_t)t * 1024;
            DT* crow = cc + (int64_t)t * 1024;
            bool no_ovf = false;
            tile_sums<false, WEIGHTED, MULT, false, DT, DT>(
                A, sm, lane, need, a0, deg, D, bd, x.rb, A.col, A.w, cc, 0, no_ovf,
                [&](bool ok, int r, int s, DT acc, unsigned first) {
                    double delta = 0.0;
                    if (ok) {
                        const SG sv = srow[r * 32 + s];
                        delta = (double)((DT)sv * acc);
                        crow[r * 32 + s] = (tm >> r) & 1u ? acc + recip_as<DT>(sv) : acc;
                    }
                    // sum of each row's run of lanes, then one lane per row adds it
                    const unsigned up = lane < 31 ? first >> (lane + 1) : 0u;
                    const int end = up ? lane + __ffs(up) : 32;   // first lane of the next row
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const bool in = lane + o < end;
                        if (!__any_sync(FULL, in)) break;
                        const double y = __shfl_down_sync(FULL, delta, o);
                        if (in) delta += y;
                    }
                    if (ok && (lane == 0 || (first >> lane) & 1u)) sm.ds[r] += delta;
                    __syncwarp();
                },
                [&](int r, uint32_t mask, DT acc) {
                    double delta = 0.0;
                    if ((mask >> lane) & 1u) {
                        const SG sv = srow[r * 32 + lane];
                        delta = (double)((DT)sv * acc);
                        crow[r * 32 + lane] = (tm >> r) & 1u ? acc + recip_as<DT>(sv) : acc;
                    }
                    delta = warp_sum(delta);
                    if (lane == 0) sm.ds[r] += delta;
                    __syncwarp();
                });
            __syncwarp();
            const uint32_t inner = sm.rowm[lane];
            const uint32_t leaf = tgt ? need & ~inner : 0u;   // no successor: c = 1 / sigma
            for_pairs<2>(leaf, lane, sm.idx, [&](const bool* ok, const int* r, const int* s, const unsigned*) {
                SG v[2];
#pragma unroll
                for (int g = 0; g < 2; g++) v[g] = ok[g] ? srow[r[g] * 32 + s[g]] : (SG)1;
#pragma unroll
                for (int g = 0; g < 2; g++)
                    if (ok[g]) crow[r[g] * 32 + s[g]] = recip_as<DT>(v[g]);
            });
            if ((inner | leaf) != need) *lrow = inner | leaf;
            const double ds = sm.ds[lane];
            if (ds != 0.0) A.dsum[row] += ds;
            __syncwarp();
        });
        if (D > 1 && !grid_barrier(A.ctl, A.flags)) return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && A.phase_ns) {
        unsigned long long t2;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t2));
        atomicAdd(&A.phase_ns[0], (t1 - t0) * (unsigned long long)A.nitems);
        atomicAdd(&A.phase_ns[1], (t2 - t1) * (unsigned long long)A.nitems);
    }
}

__global__ void lm_accumulate_kernel(const LmArgs A, const LmRun* __restrict__ runs, int nruns, int natiles, double* bcs,
                                     double* bcc) {
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    for (int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < natiles; q += nw) {
        int lo = 0, hi = nruns - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (runs[mid].atile0 <= q) lo = mid;
            else hi = mid - 1;
        }
        const LmRun r = runs[lo];
        const int64_t base = A.node_off[r.g];
        const int32_t n = (int32_t)(A.node_off[r.g + 1] - base);
        const int tpb = (n + 31) >> 5;
        const int tile0 = A.item_tile0 ? A.item_tile0[r.first] - A.tile_base : r.first * A.tpb;
        const int u = (q - r.atile0) * 32 + lane;
        if (u >= n) continue;
        const double* x = A.dsum + ((int64_t)tile0 * 32 + u);
        const int64_t step = (int64_t)(A.item_tile0 ? tpb : A.tpb) * 32;
        const int64_t ix = A.bc_map ? (int64_t)A.bc_map[base + u] : base + u;
        double s = bcs[ix], c = bcc[ix];
        int b = 0;
        for (; b + 8 <= r.count; b += 8) {
            double y[8];
#pragma unroll
            for (int i = 0; i < 8; i++) y[i] = x[(b + i) * step];
#pragma unroll
            for (int i = 0; i < 8; i++) neumaier_add(s, c, y[i]);
        }
        for (; b < r.count; b++) neumaier_add(s, c, x[b * step]);
        bcs[ix] = s;
        bcc[ix] = c;
    }
}

__global__ void lm_scatter_kernel(const LmArgs A, int32_t n, double* bc_sum, double* bc_cmp, int64_t cap_bc) {
    const int64_t stride = (int64_t)A.tpb * 32;
    const int i = blockIdx.y;
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
        const double x = A.dsum[i * stride + u];
        if (x == 0.0) continue;
        const int64_t ix = (int64_t)i * cap_bc + A.bc_map[u];
        double s = bc_sum[ix], c = bc_cmp[ix];
        neumaier_add(s, c, x);
        bc_sum[ix] = s;
        bc_cmp[ix] = c;
    }
}

// A block turns tiles of 32 rows x 32 sources around in shared memory (both sides coalesced).
__global__ void lm_paths_out_kernel(const LmArgs A, int32_t n, int32_t* dist, uint64_t* sigma) {
    __shared__ int32_t s_d[32][33];
    __shared__ uint64_t s_s[32][33];
    const int x = threadIdx.x & 31, y0 = threadIdx.x >> 5;
    const uint64_t* sg = static_cast<const uint64_t*>(A.sg);
    for (int t = blockIdx.x; t < A.ntiles; t += gridDim.x) {
        const int it = t / A.tpb;
        const LsItem I = A.items[it];
        const int u0 = (t - it * A.tpb) * 32;
        for (int y = y0; y < 32; y += LM_WARPS) {
            const int64_t o = ((int64_t)t * 32 + y) * 32 + x;
            const int32_t d = A.drow[o];
            s_d[y][x] = d;
            s_s[y][x] = d == DINF ? 0ull : sg[o];
        }
        __syncthreads();
        for (int y = y0; y < I.nsrc; y += LM_WARPS) {
            if (u0 + x < n) {
                const int64_t o = (int64_t)(I.src_off + y) * n + u0 + x;
                dist[o] = s_d[x][y];
                sigma[o] = s_s[x][y];
            }
        }
        __syncthreads();
    }
}

__global__ void lm_tile_items_kernel(const int32_t* __restrict__ item_tile0, int nitems, int32_t ntiles,
                                     int32_t* tile_item) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < ntiles; t += gridDim.x * blockDim.x) {
        int lo = 0, hi = nitems - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (item_tile0[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        tile_item[t] = lo;
    }
}

template <typename SG, bool WEIGHTED, bool MULT = false, bool TABLE = false, typename DT = double>
cudaError_t lm_go(const LmArgs& A, int num_sms, cudaStream_t st) {
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, lm_kernel<SG, DT, WEIGHTED, MULT, TABLE>, LM_THREADS, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorLaunchOutOfResources;
    // Parts of tiles until there are enough units: up to two per warp where rows are long (30 arcs on average:
    // 1.74 ms on whole tiles, 1.07 on halves, 0.93 on quarters, 0.87 on eighths), none where whole tiles nearly
    // fill the GPU and rows are short (6 arcs, 0.65 tiles per warp: 0.49 ms on whole tiles, 0.56 on halves, whose
    // units have to be fetched).
    const double warps = (double)per_sm * num_sms * LM_WARPS;
    const double goal = warps * std::min(2.0, std::max(0.5, A.mean_degree / 16.0));
    int sub_log = 0;
    while (sub_log < LM_MAX_SUB && (double)((int64_t)A.ntiles << sub_log) < goal) sub_log++;
    // And where single tiles hold far more arcs than a warp's share of a level, which would wait for their warps (with
    // many tiles the others go on meanwhile): 50,000 nodes on 60 hubs of neighbouring ids, 64 targets: 12.0 -> 5.0 ms.
    // (Not where one row holds most of them: star of 20,000, weights up to 30, 500 targets: 28.8 ms, in parts 35.9.)
    if (A.ntiles < 2 * warps && A.row_arcs < A.tile_arcs / 2) {
        const double share = 32.0 * A.mean_degree * A.ntiles / warps;
        while (sub_log < LM_MAX_SUB && (double)(A.tile_arcs >> sub_log) > std::max(4.0 * LM_CAP, 4.0 * share)) sub_log++;
    }
    const int64_t units = (int64_t)A.ntiles << sub_log;
    const int blocks = (int)std::min<int64_t>((int64_t)per_sm * num_sms, std::max<int64_t>(1, (units + LM_WARPS - 1) / LM_WARPS));
    LmArgs a = A;
    void* args[] = {&a, &sub_log};
    return cudaLaunchCooperativeKernel((const void*)lm_kernel<SG, DT, WEIGHTED, MULT, TABLE>, dim3(blocks), dim3(LM_THREADS), args, 0,
                                       st);
}

}  // namespace

int64_t lm_ctl_words(int lcap, int nitems) { return CTL_LVL + lcap + 1 + (int64_t)nitems * DEPTH_STRIDE + 2 * (int64_t)lcap + 2 * PROBE_WORDS; }

cudaError_t lm_launch(const LmArgs& A, bool narrow, bool fp32, int num_sms, cudaStream_t st) {
    if (A.nitems <= 0 || A.ntiles <= 0) return cudaSuccess;
    const bool weighted = A.w != nullptr;
    if (fp32) {
        if (!narrow || weighted || A.mud) return cudaErrorInvalidValue;
        return lm_go<uint32_t, false, false, false, float>(A, num_sms, st);
    }
    if (narrow) return weighted ? lm_go<uint32_t, true>(A, num_sms, st) : lm_go<uint32_t, false>(A, num_sms, st);
    if (A.mud) return weighted ? lm_go<uint64_t, true, true>(A, num_sms, st) : cudaErrorInvalidValue;
    return weighted ? lm_go<uint64_t, true>(A, num_sms, st) : lm_go<uint64_t, false>(A, num_sms, st);
}

cudaError_t lm_tables_launch(const LmArgs& A, int num_sms, cudaStream_t st) {
    if (A.nitems <= 0 || A.ntiles <= 0) return cudaSuccess;
    return A.w ? lm_go<uint32_t, true, false, true>(A, num_sms, st) : lm_go<uint32_t, false, false, true>(A, num_sms, st);
}

void lm_accumulate(const LmArgs& A, const LmRun* runs, int nruns, int natiles, double* bcs, double* bcc,
                   cudaStream_t st) {
    if (nruns <= 0 || natiles <= 0) return;
    const int blocks = std::min((natiles + 3) / 4, 152 * 16);
    lm_accumulate_kernel<<<blocks, 128, 0, st>>>(A, runs, nruns, natiles, bcs, bcc);
}

void lm_scatter(const LmArgs& A, int32_t n, double* bc_sum, double* bc_cmp, int64_t cap_bc, cudaStream_t st) {
    if (n <= 0) return;
    // at most 65,535 batches per launch (grid.y)
    for (int i0 = 0; i0 < A.nitems; i0 += 65535) {
        LmArgs a = A;
        a.dsum = A.dsum + (int64_t)i0 * A.tpb * 32;
        const dim3 grid((unsigned)std::min((n + 255) / 256, 1024), (unsigned)std::min(A.nitems - i0, 65535));
        lm_scatter_kernel<<<grid, 256, 0, st>>>(a, n, bc_sum + (int64_t)i0 * cap_bc, bc_cmp + (int64_t)i0 * cap_bc,
                                                cap_bc);
    }
}

void lm_paths_out(const LmArgs& A, int32_t n, int32_t* dist, uint64_t* sigma, cudaStream_t st) {
    if (n > 0 && A.ntiles > 0)
        lm_paths_out_kernel<<<std::min(A.ntiles, 152 * 16), LM_THREADS, 0, st>>>(A, n, dist, sigma);
}

void lm_tile_items(const int32_t* item_tile0, int nitems, int32_t ntiles, int32_t* tile_item, cudaStream_t st) {
    if (nitems <= 0 || ntiles <= 0) return;
    lm_tile_items_kernel<<<std::min((ntiles + 255) / 256, 152 * 16), 256, 0, st>>>(item_tile0, nitems, ntiles,
                                                                                  tile_item);
}

}  // namespace bcpp
