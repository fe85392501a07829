// CSR construction, validation, transposition and target-set checks.
#pragma once
#include "common.cuh"

namespace bcpp {

// Build by counting: arcs per tail (counts zeroed before), every arc's place in its row, and the longest rows; flags
// input errors.  place: one word per arc (undirected: 2i is u -> v, 2i + 1 is v -> u).
constexpr uint32_t CSR_LONG_ROW = 16384;
struct CsrLong {                 // zeroed before
    unsigned long long arcs;     // of the rows above CSR_LONG_ROW
    uint32_t rows;               // their number
    uint32_t longest;            // arcs of the longest row of all
};
// rows, len: list and lengths of the rows above CSR_LONG_ROW (room for all arcs / CSR_LONG_ROW)
void csr_count(int32_t n, int64_t m, const int32_t* eu, const int32_t* ev, const uint32_t* ew, int directed,
               uint32_t* counts, uint32_t* place, CsrLong* L, int32_t* rows, int64_t* len, uint32_t* flags,
               cudaStream_t st);
void csr_scatter(int64_t m, const int32_t* eu, const int32_t* ev, const uint32_t* ew, int directed, const int64_t* rp,
                 const uint32_t* place, int32_t* col, uint32_t* w, cudaStream_t st);
// sort every row of at most CSR_LONG_ROW arcs and flag repeated arcs; longrows: n words, nlong: one zeroed word
cudaError_t csr_sort_rows(int32_t n, uint32_t longest, const int64_t* rp, int32_t* col, uint32_t* w, int32_t* longrows,
                          uint32_t* nlong, uint32_t* flags, cudaStream_t st);
// the rows above: keys (row index * n + head) and weights of their arcs at off (prefix sums of len), and back when sorted
void csr_gather_rows(int32_t n, int32_t nrows, const int32_t* rows, const int64_t* off, const int64_t* rp, const int32_t* col,
                     const uint32_t* w, uint64_t* keys, uint32_t* vals, cudaStream_t st);
void csr_return_rows(int32_t n, int64_t arcs, const int32_t* rows, const int64_t* off, const int64_t* rp, const uint64_t* keys,
                     const uint32_t* vals, int32_t* col, uint32_t* w, uint32_t* flags, cudaStream_t st);
// checks of a CSR: *wmax (zeroed) = largest weight
void csr_check(int32_t n, int64_t na, const int64_t* rp, const int32_t* col, const uint32_t* w, int directed,
               uint32_t* flags, unsigned long long* wmax, cudaStream_t st, const int64_t* node_off = nullptr,
               int32_t ngraphs = 0);
// stats (two zeroed words) = most arcs of 32 consecutive rows and of one row
void csr_stats(int32_t n, const int64_t* rp, unsigned long long* stats, cudaStream_t st);
// graph-local heads of a disjoint union (flags arcs that leave their graph)
void csr_localize(int32_t n, const int64_t* rp, const int32_t* col, const int64_t* node_off, int32_t ngraphs,
                  int32_t* lcol, uint32_t* flags, cudaStream_t st);
void targets_check(const int32_t* S, int32_t nS, int32_t n, uint8_t* in_s, uint32_t* cnt, uint32_t* flags,
                   cudaStream_t st);
void csr_transpose_count(int32_t n, const int64_t* rp, const int32_t* col, int64_t* counts, cudaStream_t st);
void csr_transpose_fill(int32_t n, const int64_t* rp, const int32_t* col, const uint32_t* w, int64_t* cursor,
                        int32_t* tcol, uint32_t* tw, cudaStream_t st);

}  // namespace bcpp
