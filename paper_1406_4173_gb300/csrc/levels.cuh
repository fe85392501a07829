// Level-mask shortest paths with path counts and dependency accumulation over many source
// batches at once (see levels.cu for the method).
#pragma once
#include "common.cuh"
#include "lockstep.cuh"

namespace bcpp {

// Distance levels a launch provides for.  A batch that reaches a later one is given back (LmArgs::back, FLAG_MASKS), and
// the caller runs it on the lockstep kernel.
constexpr int LM_MAX_LEVELS = 256;
// Largest arc weight: every row that is not settled on all its sources looks at its in-arcs once per
// distance value, so the forward cost grows with the number of distance values.
constexpr uint64_t LM_MAX_WEIGHT = 32;

// One wave of batches (items) of up to 32 sources.  Batch i owns the rows [32 tile0(i), 32 tile0(i) +
// n) of the row arrays, one row per node of its graph, and whole tiles of 32 rows.
struct LmArgs {
    const int64_t* rp;          // out-arcs
    const int32_t* col;
    const int32_t* w;           // nullptr = unit weights
    const double* mud;          // multiplicities as doubles; nullptr = 1
    const int64_t* irp;         // in-arcs
    const int32_t* icol;
    const int32_t* iw;
    const uint64_t* imu;
    const int64_t* node_off;    // graph g: nodes [node_off[g], node_off[g + 1])
    const LsItem* items;        // the wave's batches
    const int32_t* item_tile0;  // first tile of each batch plus tile_base; nullptr: uniform, batch i at i * tpb
    const int32_t* tile_item;   // batch of tile t at [t + tile_base], plus item_base
    int32_t tile_base, item_base;
    int32_t tpb;                // tiles per batch (uniform layout)
    int32_t nitems, ntiles;
    const int32_t* srcs;        // graph-local sources
    const uint8_t* in_s;        // per global node: target flag; nullptr = every node
    uint32_t* lev;              // [lcap][rows]: sources that reach the row's node at that distance
    uint32_t* seen;             // [rows]: sources that reached it so far
    void* sg;                   // [rows][32] path counts (32- or 64-bit)
    void* cc;                   // [rows][32] (I + delta) / sigma, double or float; nullptr: forward pass only
    int32_t* drow;              // [rows][32] distances (DINF = unreached), or nullptr; with it cc is zero
                                // wherever it is not written
    double* dsum;               // [rows] dependencies summed over the batch's sources
    const int32_t* nfront;      // Dijkstra_SK tables: frontiers of each graph (its first nodes); nullptr: no tables
    const int64_t* toff;        // table offset of each graph
    int32_t* td;                // d_i[v][f], filled with DINF before
    uint64_t* ts;               // sigma_i[v][f], zeroed before
    const int32_t* bc_map;      // global node -> index of the sums over sources (nullptr = same)
    int64_t rows;               // 32 ntiles
    int32_t lcap;               // levels provided for
    bool bounded;               // no distance reaches lcap: a pass that ends there is complete
    bool few;                   // when more than a third of the batches are given back, all are
    bool probe;                 // no bound on the levels is known: give up early on a graph that looks too deep
    int32_t wmax;
    double mean_degree;         // arcs per node
    int64_t tile_arcs, row_arcs;   // most arcs of 32 consecutive rows, of one row (0: not known)
    uint32_t* back;             // [nitems], zeroed: set for the batches given back (their dsum stays 0)
    uint32_t* ctl;              // lm_ctl_words() zeroed words: barrier, level status, depth of each batch
    uint32_t* flags;
    unsigned long long* phase_ns;
};

int64_t lm_ctl_words(int lcap, int nitems);

// Forward and backward pass of every batch of the wave; one cooperative launch.  narrow: 32-bit path
// counts (a batch with a count of 2^32 or more is given back).  fp32: FP32 dependencies (unit weights, narrow).
cudaError_t lm_launch(const LmArgs& A, bool narrow, bool fp32, int num_sms, cudaStream_t st);

// Dijkstra_SK (Eq. 10): forward pass of every batch (sources: frontiers aux .. aux + nsrc - 1 of graph g, cc =
// nullptr) into the tables; 32-bit path counts as with narrow.
cudaError_t lm_tables_launch(const LmArgs& A, int num_sms, cudaStream_t st);

// A run of consecutive batches of one graph in a wave: dsum of its batches is summed per node.
struct LmRun {
    int32_t g, first, count;   // graph, first batch in the wave, batches
    int32_t atile0;            // tiles of the wave's earlier runs (one tile set per run)
};
// bcs / bcc (Neumaier sum and compensation per global node) += dsum over the runs' batches
void lm_accumulate(const LmArgs& A, const LmRun* runs, int nruns, int natiles, double* bcs, double* bcc,
                   cudaStream_t st);

// Partial sums of batch i at i * cap_bc (single graph, uniform layout): bc_sum / bc_cmp [bc_map[u]] += dsum
void lm_scatter(const LmArgs& A, int32_t n, double* bc_sum, double* bc_cmp, int64_t cap_bc, cudaStream_t st);

// Distances and counts of a forward-only wave with distance rows (single graph, uniform layout):
// dist / sigma [source position][n], DINF and 0 where unreached
void lm_paths_out(const LmArgs& A, int32_t n, int32_t* dist, uint64_t* sigma, cudaStream_t st);

// tile_item[t] = batch of tile t, for all batches
void lm_tile_items(const int32_t* item_tile0, int nitems, int32_t ntiles, int32_t* tile_item, cudaStream_t st);

}  // namespace bcpp
