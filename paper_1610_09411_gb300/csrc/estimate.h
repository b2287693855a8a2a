// estimate.h -- work space of a batch chunk, estimated on the host (plain C++).
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace esc {

// The dense core (core.cu): least degree of its vertices, the most that its
// wedge counts W may take, and the operand blocks of one chunk of centres.
static constexpr int CORE_MIN_DEG = 48, CORE_CHUNK_MB = 2048;
static constexpr size_t CORE_W_BYTES = (size_t)24 << 30;

// Device bytes that the census of a union of graphs takes, from above:
//   per graph the common-neighbour lists (36 B per triangle, 12 more for the
//   packed lists of a core, and 3T <= wedges), per-entry and per-vertex arrays,
//   and per vertex the sweeps' per-CTA counters (32 B in 4 CTAs per SM);
//   for its core 2 or 4 B per pair of core vertices of one graph, and once per
//   union the operand blocks of a chunk (128 x 128 B each, (d + 127)^2 at most
//   for a centre of d core neighbours) with their bits and the below-core counts.
class ChunkEstimate {
 public:
  // graph of the rows [r0, r1) of rp
  void add(const int64_t* rp, int64_t r0, int64_t r1, int sms) {
    // whole numbers without a branch, for the compiler's vectors: a batch has many rows
    uint64_t wedges2 = 0, sq = 0, cores = 0;
    uint32_t top = 0;
    for (int64_t r = r0; r < r1; ++r) {
      const uint32_t d = (uint32_t)(rp[r + 1] - rp[r]);
      const uint64_t in = d >= (uint32_t)CORE_MIN_DEG ? ~0ull : 0ull;
      wedges2 += (uint64_t)d * (d - 1u);        // d = 0: 0 x (2^32 - 1)
      sq += ((uint64_t)(d + 127u) * (d + 127u)) & in;
      cores -= in;
      top = std::max(top, d);
    }
    const double big = (double)top + 127;
    sweeps_ += 8.0 * (double)wedges2 + 160.0 * (double)(rp[r1] - rp[r0]) + (260.0 + 32.0 * 4 * sms) * (double)(r1 - r0);
    w_ += 4.0 * (double)cores * (double)cores;
    wide_ = wide_ || top >= 65536;
    blocks_ += (double)sq;
    if (cores) block_ = std::max(block_, big * big);
  }
  double bytes() const {
    const double w = wide_ ? w_ : w_ / 2;
    if (w > (double)CORE_W_BYTES) return sweeps_;         // no core
    return sweeps_ + w + (wide_ ? 3.125 : 2.125) * std::min(blocks_, std::max((double)CORE_CHUNK_MB * (1 << 20), block_));
  }

 private:
  double sweeps_ = 0, w_ = 0, blocks_ = 0, block_ = 0;
  bool wide_ = false;
};

}  // namespace esc
