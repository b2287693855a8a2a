// core.cuh -- the dense core of the pair and wheel sweeps: what core.cu offers
// to the census (see core.cu for the counting).
#pragma once
#include "common.cuh"
#include "internal.h"

#include <vector>

namespace esc {

// Work cut into runs of centres whose operand blocks fit the scratch.  Centres
// are numbered s = 0 .. h - 1 from the highest rank down.
struct CoreChunks {
  std::vector<int64_t> start;      // centre numbers, ending with the first one that has no work
  int64_t max_blocks = 0, max_tiles = 0, max_tri = 0, max_row_blocks = 0;
};
struct CoreBuffers {
  void* blocks = nullptr;          // core_block_bytes(chunks)
  void* bits = nullptr;            // core_bit_bytes(chunks): the same matrices as bits
  void* tiles = nullptr;           // 16 bytes x max_tiles
  void* k4 = nullptr;              // zeroed u64 per slot from k4_0, the first one of rank h0
  int64_t k4_0 = 0;
  void* b = nullptr;               // max_tri counts as wide as W's; null when no vertex lies below the core
  unsigned long long wait_ns = 4000000000ull;   // limit of every wait of the contraction
  uint32_t give_up = 0;            // tile whose wait runs out at once (tests; 0: none)
};

// dh, and the prefix sums off (4 x (h + 1)); for a single graph also li and rowb
cudaError_t core_layout(const DevGraph& g, int64_t h0, bool single, int32_t* dh, int32_t* li, int64_t* rowb,
                        int64_t* off, int sms, cudaStream_t s);
// hl, hb, li, rowb of a union; wbase (num_graphs + 1) ends with the entries of W
cudaError_t core_union(const int32_t* vg, int num_graphs, int64_t h0, int64_t h, int32_t* hl, int64_t* hb, int32_t* li,
                       int64_t* rowb, int64_t* wbase, DeviceArena& arena, int sms, cudaStream_t s);
cudaError_t core_low(const DevGraph& g, const uint32_t* T, const int64_t* off, const int32_t* U, int64_t h0,
                     uint32_t* low, int sms, cudaStream_t s);
void core_chunks(const int64_t* off, int64_t h, int64_t cap_bytes, CoreChunks* ck);
size_t core_block_bytes(const CoreChunks& ck);
size_t core_bit_bytes(const CoreChunks& ck);
// every chunk's contraction; adds to ACC_N17H, ACC_N18H, ACC_N20H, ACC_K4H and k4
cudaError_t core_run(const DevGraph& g, const CoreView& cv, const uint32_t* T, const int64_t* offp, const int32_t* P,
                     const int64_t* d_off, const int64_t* off, const CoreChunks& ck, const CoreBuffers& cb,
                     const AccSet& acc, unsigned* status, int sms, int smem_optin, cudaStream_t s);

}  // namespace esc
