// Breadth-first discovery order of all nodes (see order.cu).
#pragma once
#include "common.cuh"

namespace bcpp {

int64_t order_ctl_words(int num_sms);   // control block of order_bfs_launch, in 32-bit words

// queue[0 .. n) = the nodes in breadth-first discovery order from the node of largest degree (unit weights; smallest id
// on ties), the unreached ones behind them by id; depth[0] = the deepest level, depth[1] = unreached nodes with two arcs
// or more.  par: n words of scratch.
// Levels past ORDER_MAX_LEVELS count as unreached.
constexpr int ORDER_MAX_LEVELS = 4096;
cudaError_t order_bfs_launch(int32_t n, const int64_t* rp, const int32_t* col, int32_t* par, int32_t* queue,
                             uint32_t* ctl, int32_t* depth, uint32_t* flags, int num_sms, cudaStream_t st);

// mem[S[i]] = 1 (mem zeroed before); f[i] = mem[queue[i]]
void order_member(const int32_t* S, int64_t ns, const int32_t* queue, int32_t n, uint8_t* mem, int32_t* f,
                  cudaStream_t st);
// out[pos[i]] = queue[i] where f[i]
void order_compact(const int32_t* queue, const int32_t* f, const int64_t* pos, int32_t n, uint32_t* out, cudaStream_t st);

}  // namespace bcpp
