// core.cu -- the dense core of the pair and wheel sweeps (Thms 11, 12) on the
// tensor cores.
//
// The core H is the set of vertices from rank h0 on (the highest degrees).
// For a centre c in H let L be the d core vertices adjacent to c and B_c the
// 0/1 adjacency matrix of G[L].  (B_c B_c)(u, v) = M_c(u, v) is the number of
// common neighbours of u and v inside L, and with b_c(u, v) the number of
// neighbours of c below h0 that are adjacent to u and v,
//   N18, 4-cycles of G[N(c)] with opposite vertices u, v in H:
//       all four vertices in H ........ 1/2 sum_{u>v} C(M, 2)   (two diagonals)
//       exactly one below h0 .......... sum_{u>v} b M           (its neighbours on the cycle are u, v)
//       two opposite ones below h0 .... sum_{u>v} C(b, 2)
//   N17, diamonds with tips u, v in H and an edge at c:
//       edge inside H (seen from both ends) .... 1/2 sum_{u>v} (W(u,v) - 2) M
//       edge from c to below h0 ................ sum_{u>v} (W(u,v) - 2) b
// With Y = M + 2b that is 1/2 sum (W - 2) Y and 1/4 sum (Y^2 - Y - 2 b^2).
// For adjacent u and v, M + b is K4(t) of the triangle t = {c, u, v} (Thm 7), and
// M counts the 4-cliques of t inside H, so over the adjacent pairs
//   N20, triangles inside H ........ 1/3 sum C(M + b, 2)     (t is seen from three centres)
//   K4 inside H .................... 1/12 sum M
//   K4(c, u) inside H .............. 1/2 sum_v M
// and the clique pass leaves these to the core for lowest vertices in H.
// Every diamond and cycle not named here (a tip below h0; both ends of the edge
// below h0; two adjacent cycle vertices below h0; a centre below h0) is counted
// by the sweeps in census.cu, which skip the ones named here.
//
// What bounds it: enumerating the diamonds inside H one by one costs one
// scattered list read and one counter read each.  Most diamonds lie there
// (R-MAT scale 19: 90% within the top 16,384 ranks), and M_c has thousands of
// times fewer entries than there are diamonds, so the contraction B_c B_c goes
// to tcgen05 and only its d^2 / 2 entries per centre are touched by scalar code.
//
// Measured (GB300), the census without and with the core: R-MAT scale 19 726 and
// 380 ms, scale 16 50.6 and 24.2 ms, Chung-Lu 2.1 n = 262,144 53.2 and 39.8 ms.
//
// Operands are fp8 (e4m3: 0 and 1 are exact) with fp32 accumulation in tensor
// memory: every partial sum is a whole number below d, exact in fp32 below 2^24
// (a core of CORE_W_BYTES has d below 2^17; the epilogue reads up to 2^23).  The
// tests put odd sums of up to 65,000, reached in odd steps, through it.
// k_core_build writes B_c once as blocks of 128 rows x 128 bytes in the
// 128-byte-swizzled K-major layout the tensor cores read, 16 KB contiguous, so
// that a plain bulk copy (cp.async.bulk) moves an operand block to shared memory
// without a tensor map.
#include "core.cuh"

#include <algorithm>

namespace esc {

static constexpr int CORE_BLK = 128;                       // rows and columns of an operand block
static constexpr int CORE_BLK_BYTES = CORE_BLK * CORE_BLK;
static constexpr int CORE_BIT_WORDS = CORE_BLK * 4;        // words of bits per operand block
static constexpr int CORE_TN = 256;                        // columns of an output tile (two blocks)
static constexpr int CORE_STAGES = 4;
static constexpr int CORE_STAGE_BYTES = 3 * CORE_BLK_BYTES;   // one block of rows, two of columns
static constexpr int CORE_EPI_WARPS = 8;
static constexpr int CORE_THREADS = (CORE_EPI_WARPS + 2) * 32;

// ---------------------------------------------------------------- layout
// Core neighbours of every core vertex; its place in W for a single graph.
__global__ void k_core_dims(DevGraph g, int64_t h0, int32_t* dh, int32_t* li, int64_t* rowb) {
  const int64_t h = g.n - h0;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < h; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = h0 + t;
    dh[t] = (int32_t)(g.R[c + 1] - lower_bound_i32(g.C, g.R[c], g.R[c + 1], (int32_t)h0));
    if (li) {
      li[t] = (int32_t)t;
      rowb[t] = t * h;
    }
  }
}

// Exclusive prefix sums over the core vertices from the highest rank down
// (entry s belongs to rank n - 1 - s): row blocks, operand blocks, output
// tiles and pairs.  One CTA; h is at most a few hundred thousand.
__device__ __forceinline__ void core_sizes(int64_t d, int64_t* v) {
  const int64_t nb = d < 2 ? 0 : (d + CORE_BLK - 1) / CORE_BLK, nv = (nb + 1) / 2;
  v[0] = nb;
  v[1] = nb * nb;
  v[2] = nb * nv - (nb > 0 ? ((nb - 1) * (nb - 1)) / 4 : 0);   // sum over row blocks r of nv - floor(r / 2)
  v[3] = d < 2 ? 0 : (d * (d - 1) / 2 + 1) & ~(int64_t)1;
}
__global__ void __launch_bounds__(1024) k_core_scan(const int32_t* dh, int64_t h, int64_t* off) {
  __shared__ int64_t sh[4][32], carry[4];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x < 4) carry[threadIdx.x] = 0;
  __syncthreads();
  for (int64_t b = 0; b < h + 1; b += 1024) {
    const int64_t s = b + threadIdx.x;
    int64_t v[4] = {0, 0, 0, 0}, x[4];
    if (s < h) core_sizes(dh[h - 1 - s], v);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      x[k] = v[k];
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x[k], o);
        if (lane >= o) x[k] += y;
      }
      if (lane == 31) sh[k][wid] = x[k];
    }
    __syncthreads();
    if (wid < 4) {
      int64_t y = sh[wid][lane];
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t z = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= o) y += z;
      }
      sh[wid][lane] = y;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (s <= h) off[k * (h + 1) + s] = carry[k] + (wid ? sh[k][wid - 1] : 0) + x[k] - v[k];
    __syncthreads();
    if (threadIdx.x < 4) carry[threadIdx.x] += sh[threadIdx.x][31];
    __syncthreads();
  }
}

// last s in [s0, s1) with off[s] <= key
__device__ __forceinline__ int64_t core_find(const int64_t* off, int64_t s0, int64_t s1, int64_t key) {
  while (s1 - s0 > 1) {
    const int64_t mid = (s0 + s1) >> 1;
    if (off[mid] <= key) s0 = mid; else s1 = mid;
  }
  return s0;
}

// Places in W for a union of graphs: the core vertices sorted by graph (order,
// from a stable sort, so ascending ranks within a graph) and the start of every
// graph's group; W holds one square per graph.
__global__ void k_core_union_count(const int32_t* vg, int64_t h0, int64_t h, uint64_t* keys, uint32_t* vals,
                                   unsigned long long* cnt) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < h; t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t k = vg[h0 + t];
    keys[t] = (uint64_t)k;
    vals[t] = (uint32_t)t;
    atomicAdd(&cnt[k], 1ull);
  }
}
__global__ void k_core_union_squares(const int64_t* cnt, int num_graphs, int64_t* sq) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < num_graphs; k += gridDim.x * blockDim.x)
    sq[k] = cnt[k] * cnt[k];
}
__global__ void k_core_union_place(const uint64_t* keys, const uint32_t* vals, int64_t h0, int64_t h,
                                   const int64_t* start, const int64_t* wbase, int32_t* hl, int64_t* hb, int32_t* li,
                                   int64_t* rowb) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < h; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = (int64_t)keys[q], t = vals[q], g0 = start[k], hg = start[k + 1] - g0;
    hl[q] = (int32_t)(h0 + t);
    hb[t] = g0;
    li[t] = (int32_t)(q - g0);
    rowb[t] = wbase[k] + (q - g0) * hg;
  }
}

// low[p]: common neighbours of edge p below h0, for every slot whose entry is
// in the core (one binary search of the edge's sorted list).  rows: all of them.
__global__ void k_core_low(DevGraph g, const uint32_t* T, const int64_t* off, const int32_t* U, int64_t h0,
                           uint32_t* low) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t k = warp; k < g.n; k += nwarps) {
    const int64_t x = g.n - 1 - k, b = g.R[x];
    for (int64_t p = g.R[x + 1] - 1 - lane; p >= b; p -= 32) {
      if (g.C[p] < h0) break;
      const uint32_t len = T[p];
      uint32_t lo = 0, hi = len;
      const int32_t* L = U + off[p];
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (L[mid] < h0) lo = mid + 1; else hi = mid;
      }
      low[p] = lo;
    }
  }
}

// ---------------------------------------------------------------- b_c
// For every centre of the chunk and every neighbour k below h0, the core
// vertices adjacent to both (a suffix of the position list of slot c -> k) add
// one to b at each of their pairs.  b is a triangle of counts as wide as W's
// (16 bits, two to a word, when no degree reaches 2^16: b(u, v) < d_c).  One
// CTA per centre, one warp for 32 k's.
static constexpr int CORE_SHORT = 8;
template <typename WT>
__global__ void __launch_bounds__(256) k_core_mixed(DevGraph g, const uint32_t* T, const int64_t* offp,
                                                    const int32_t* P, int64_t h0, const int32_t* dh,
                                                    const int64_t* tri_off, int64_t s0, WT* b_all) {
  const int64_t s = s0 + blockIdx.x, c = g.n - 1 - s;
  const int d = dh[c - h0];
  if (d < 2) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t base = g.R[c], pc = g.R[c + 1] - d - base;
  uint32_t* b = reinterpret_cast<uint32_t*>(b_all + (tri_off[s] - tri_off[s0]));
  for (int64_t kb = (int64_t)wid * 32; kb < pc; kb += (int64_t)nw * 32) {
    const int64_t k = kb + lane;
    int64_t st_l = 0;
    int cnt_l = 0;
    if (k < pc) {
      const int len = (int)T[base + k];
      const int64_t o = offp[base + k];
      int lo = 0, hi = len;
      if (len >= 2 && P[o + len - 2] < pc) lo = len;       // fewer than two core entries
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (P[o + mid] < pc) lo = mid + 1; else hi = mid;
      }
      st_l = o + lo;
      cnt_l = len - lo;
    }
    // short suffixes: each lane its own pairs; long ones: the warp, one at a time
    auto add = [&](int64_t v, int64_t u) {
      const int64_t e = v * (v - 1) / 2 + u;
      if (sizeof(WT) == 2) atomicAdd(&b[e >> 1], 1u << (16 * (int)(e & 1)));
      else atomicAdd(&b[e], 1u);
    };
    if (cnt_l >= 2 && cnt_l <= CORE_SHORT) {
      const int32_t* L = P + st_l;
      int32_t e[CORE_SHORT];
#pragma unroll
      for (int y = 0; y < CORE_SHORT; ++y) e[y] = y < cnt_l ? L[y] - (int32_t)pc : 0;
#pragma unroll
      for (int y = 1; y < CORE_SHORT; ++y)
#pragma unroll
        for (int x = 0; x < y; ++x)
          if (y < cnt_l) add(e[y], e[x]);
    }
    unsigned m = __ballot_sync(0xffffffffu, cnt_l > CORE_SHORT);
    while (m) {
      const int q = __ffs(m) - 1;
      m &= m - 1;
      const int32_t* L = P + __shfl_sync(0xffffffffu, st_l, q);
      const int cnt = __shfl_sync(0xffffffffu, cnt_l, q);
      for (int x0 = 0; x0 < cnt; x0 += 32) {    // 32 entries x against every later y
        const int64_t u = x0 + lane < cnt ? L[x0 + lane] - pc : 0;
        for (int yb = x0; yb < cnt; yb += 32) {
          const int32_t v_l = yb + lane < cnt ? L[yb + lane] - (int32_t)pc : 0;
          const int ye = min(32, cnt - yb);
#pragma unroll 4
          for (int y = 0; y < ye; ++y) {
            const int64_t v = __shfl_sync(0xffffffffu, v_l, y);
            if (x0 + lane < yb + y) add(v, u);
          }
        }
      }
    }
  }
}

// ---------------------------------------------------------------- operand blocks
// One CTA per 128-row block of one centre's B_c: each warp marks the core
// neighbours of one row u (the positions of N(c) cap N(u) from the slot's
// position list) as bits and spreads them to bytes, 16 columns per store.  The
// CTA also writes the descriptors of the output tiles of its row block.
__global__ void __launch_bounds__(256) k_core_build(DevGraph g, const uint32_t* T, const int64_t* offp,
                                                    const int32_t* P, int64_t h0, int64_t h, const int32_t* dh,
                                                    const int64_t* off, int64_t s0, int64_t s1, int bit_words,
                                                    uint8_t* blocks, uint32_t* bitm, int4* tiles) {
  extern __shared__ uint32_t core_bits[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t *rb_off = off, *blk_off = off + (h + 1), *tile_off = off + 2 * (h + 1);
  const int64_t item = rb_off[s0] + blockIdx.x;
  const int64_t s = core_find(rb_off, s0, s1, item);
  const int64_t c = g.n - 1 - s;
  const int d = dh[c - h0];
  const int nb = (d + CORE_BLK - 1) / CORE_BLK, rb = (int)(item - rb_off[s]);
  const int64_t row0 = g.R[c + 1] - d;
  const int32_t pc = (int32_t)(row0 - g.R[c]);
  const int64_t blk0 = blk_off[s] - blk_off[s0];
  uint8_t* out = blocks + (blk0 + (int64_t)rb * nb) * CORE_BLK_BYTES;
  uint32_t* bits = core_bits + wid * bit_words;
  uint32_t* bout = bitm + (blk0 + (int64_t)rb * nb) * CORE_BIT_WORDS;   // rows of 4 nb words
  for (int r = wid; r < CORE_BLK; r += 8) {
    const int a = rb * CORE_BLK + r;
    for (int i = lane; i < nb * 4; i += 32) bits[i] = 0u;
    __syncwarp();
    if (a < d) {
      const uint32_t len = T[row0 + a];
      const int32_t* L = P + offp[row0 + a];
      for (uint32_t q = lane; q < len; q += 32) {
        const int32_t pos = L[q] - pc;
        if (pos >= 0) atomicOr(&bits[pos >> 5], 1u << (pos & 31));
      }
    }
    __syncwarp();
    for (int j = lane; j < nb * 4; j += 32) bout[r * (nb * 4) + j] = bits[j];
    for (int j = lane; j < nb * 8; j += 32) {
      const uint32_t x = bits[j >> 1] >> ((j & 1) * 16);
      uint4 o;                                  // bit -> byte 0x38 (1.0 in e4m3)
      o.x = (((x & 15u) * 0x00204081u) & 0x01010101u) * 0x38u;
      o.y = ((((x >> 4) & 15u) * 0x00204081u) & 0x01010101u) * 0x38u;
      o.z = ((((x >> 8) & 15u) * 0x00204081u) & 0x01010101u) * 0x38u;
      o.w = ((((x >> 12) & 15u) * 0x00204081u) & 0x01010101u) * 0x38u;
      *reinterpret_cast<uint4*>(out + (int64_t)(j >> 3) * CORE_BLK_BYTES + r * CORE_BLK +
                                (((j & 7) ^ (r & 7)) << 4)) = o;
    }
    __syncwarp();
  }
  const int nv = (nb + 1) / 2;
  int4* td = tiles + (tile_off[s] - tile_off[s0]) + (int64_t)rb * nv - (rb > 0 ? ((int64_t)(rb - 1) * (rb - 1)) / 4 : 0);
  for (int k = threadIdx.x; rb / 2 + k < nv; k += blockDim.x)
    td[k] = make_int4((int)blk0, (int)s, d, rb | ((rb / 2 + k) << 16));
}

// ---------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mb_init(uint32_t bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mb_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mb_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mb_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Waits at most limit_ns (0: not at all); false when the wait ran out.
static constexpr unsigned long long CORE_DRAIN_NS = 4000000000ull;
__device__ __forceinline__ bool mb_wait(uint32_t bar, uint32_t parity, unsigned long long limit_ns) {
  if (limit_ns == 0) return false;
  for (int k = 0; k < 16; ++k)
    if (mb_try(bar, parity)) return true;
  const unsigned long long t0 = now_ns();
  while (true) {
    for (int k = 0; k < 32; ++k)
      if (mb_try(bar, parity)) return true;
    if (now_ns() - t0 > limit_ns) return false;
  }
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// K-major operand in 128-byte swizzled rows: 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t core_desc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3fffu) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void core_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b), "r"(idesc),
               "r"(acc) : "memory");
}
__device__ __forceinline__ void core_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld(uint32_t (&r)[32], uint32_t addr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr));
}
__device__ __forceinline__ void tmem_ld(uint32_t (&r)[16], uint32_t addr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ---------------------------------------------------------------- contraction
// Persistent, one CTA per SM (shared memory): warp 8 streams operand blocks
// through CORE_STAGES stages, warp 9 issues the MMAs of a 128 x 256 output tile
// (rows u, columns v; only tiles with some u < v exist), warps 0-7 read the
// finished tile from tensor memory while the next one is accumulated in the
// other half of its 512 columns.  A lane holds one row u and walks the columns,
// so that the lanes of a warp read W(v, .) and b(v, .) along their rows.
// Every wait is bounded (wait_ns): a wait that runs out sets the status word and
// ends that role's work, after which the other roles' waits run out too.  A
// reading warp decides with all its lanes at once, as what follows the wait is
// warp-wide.  However it ends, the copying thread waits until its copies have
// landed and the issuing thread until its MMAs have finished (CORE_DRAIN_NS at
// most) before the tensor memory goes back and the CTA ends.  give_up: the
// reading warps take their wait for this tile (from 1; 0: none) as run out.
// One centre with d = 16,000 runs at 3.4 PFLOP/s; the many smaller
// centres of R-MAT 19 (3.3e13 multiply-adds in its triangle's tiles) take 42 ms
// and are bound by the scattered sectors of W (512 MB, beyond L2) that the
// entries read, not by the MMAs; the adjacency bits, N20 and the 4-clique sums
// cost 4 ms of it and save the clique pass 22 ms.  On R-MAT 22, with 32-bit
// counts, the contraction reads 3.54 TB in 0.62 s (5.7 TB/s, 0.84 of the measured
// copy rate).
template <typename WT> struct CoreSum { typedef uint32_t type; };   // 32 terms below 2^18
template <> struct CoreSum<uint32_t> { typedef unsigned long long type; };
// barrier of the eight reading warps; true when ok holds on every thread
__device__ __forceinline__ bool epi_all(bool ok) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.and.pred p, 1, 256, q;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(r) : "r"((uint32_t)ok) : "memory");
  return r != 0;
}
struct CoreBars {
  unsigned long long full[CORE_STAGES], empty[CORE_STAGES], accf[2], acce[2], drain;
};
static constexpr size_t CORE_SMEM = 1024 + (size_t)CORE_STAGES * CORE_STAGE_BYTES + 2 * CORE_TN * sizeof(void*);

template <typename WT, bool HASB>
__global__ void __launch_bounds__(CORE_THREADS, 1) k_core_mma(DevGraph g, CoreView cv, const int4* tiles,
                                                              int64_t ntiles, const uint8_t* blocks,
                                                              const uint32_t* bitm, unsigned long long* k4,
                                                              int64_t k4_0, const WT* b_all, const int64_t* tri_off, int64_t s0,
                                                              AccSet acc, unsigned* status,
                                                              unsigned long long wait_ns, uint32_t give_up) {
  extern __shared__ uint8_t core_smem_raw[];
  __shared__ CoreBars bars;
  __shared__ uint32_t s_tmem;
  __shared__ u128 sh[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t stage0 = (smem_u32(core_smem_raw) + 1023u) & ~1023u;
  const WT** wrow = reinterpret_cast<const WT**>(core_smem_raw + (stage0 - smem_u32(core_smem_raw)) +
                                                 (size_t)CORE_STAGES * CORE_STAGE_BYTES);   // [2][CORE_TN]
  if (threadIdx.x == 0) {
    for (int k = 0; k < CORE_STAGES; ++k) {
      mb_init(smem_u32(&bars.full[k]), 1);
      mb_init(smem_u32(&bars.empty[k]), 1);
    }
    for (int k = 0; k < 2; ++k) {
      mb_init(smem_u32(&bars.accf[k]), 1);
      mb_init(smem_u32(&bars.acce[k]), CORE_EPI_WARPS);
    }
    mb_init(smem_u32(&bars.drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (wid == CORE_EPI_WARPS + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const int ids[4] = {ACC_N17H, ACC_N18H, ACC_N20H, ACC_K4H};
  LocalAcc<4> la;
  la.zero();
  const int64_t step = gridDim.x;
  if (wid == CORE_EPI_WARPS) {                  // ------------ operand copies
    if (lane == 0) {
      uint32_t fill = 0;                        // stages filled so far
      bool ok = true;
      for (int64_t t = blockIdx.x; t < ntiles && ok; t += step) {
        const int4 td = tiles[t];
        const int d = td.z, ut = td.w & 0xffff, vt = td.w >> 16, nb = (d + CORE_BLK - 1) / CORE_BLK;
        const uint8_t* base = blocks + (int64_t)td.x * CORE_BLK_BYTES;
        const bool two = 2 * vt + 1 < nb;
        for (int kb = 0; kb < nb; ++kb, ++fill) {
          const uint32_t sl = fill % CORE_STAGES, ph = (fill / CORE_STAGES) & 1;
          if (!mb_wait(smem_u32(&bars.empty[sl]), ph ^ 1, wait_ns)) {
            ok = false;
            break;
          }
          const uint32_t full = smem_u32(&bars.full[sl]), dst = stage0 + sl * CORE_STAGE_BYTES;
          mb_expect(full, (two ? 3 : 2) * CORE_BLK_BYTES);
          bulk_g2s(dst, base + ((int64_t)ut * nb + kb) * CORE_BLK_BYTES, CORE_BLK_BYTES, full);
          bulk_g2s(dst + CORE_BLK_BYTES, base + ((int64_t)(2 * vt) * nb + kb) * CORE_BLK_BYTES, CORE_BLK_BYTES, full);
          if (two)
            bulk_g2s(dst + 2 * CORE_BLK_BYTES, base + ((int64_t)(2 * vt + 1) * nb + kb) * CORE_BLK_BYTES,
                     CORE_BLK_BYTES, full);
        }
      }
      // the copies in flight land before the CTA ends (the issuing thread may have given up on them)
      for (uint32_t k = fill > CORE_STAGES ? fill - CORE_STAGES : 0; k < fill; ++k)
        ok = mb_wait(smem_u32(&bars.full[k % CORE_STAGES]), (k / CORE_STAGES) & 1, CORE_DRAIN_NS) && ok;
      if (!ok) set_err(status, DEVERR_TIMEOUT);
    }
  } else if (wid == CORE_EPI_WARPS + 1) {       // ------------ MMA issue
    if (lane == 0) {
      uint32_t fill = 0, it = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < ntiles && ok; t += step, ++it) {
        const int4 td = tiles[t];
        const int d = td.z, vt = td.w >> 16, nb = (d + CORE_BLK - 1) / CORE_BLK;
        const int ncols = min(CORE_TN, (d - vt * CORE_TN + 31) & ~31);
        // D fp32, A and B e4m3, both K-major; N / 8 and M / 16
        const uint32_t idesc = (1u << 4) | ((uint32_t)(ncols >> 3) << 17) | ((CORE_BLK >> 4) << 24);
        const uint32_t buf = it & 1;
        if (!mb_wait(smem_u32(&bars.acce[buf]), ((it >> 1) & 1) ^ 1, wait_ns)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const int ksteps = (d + 31) / 32;       // columns beyond d are zero
        for (int kb = 0; kb < nb; ++kb, ++fill) {
          const uint32_t sl = fill % CORE_STAGES;
          if (!mb_wait(smem_u32(&bars.full[sl]), (fill / CORE_STAGES) & 1, wait_ns)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = stage0 + sl * CORE_STAGE_BYTES;
          const uint64_t da = core_desc(sa), db = core_desc(sa + CORE_BLK_BYTES);
          const int kn = min(4, ksteps - 4 * kb);
          for (int k = 0; k < kn; ++k)          // 32 bytes of K per MMA
            core_mma(tmem + buf * CORE_TN, da + 2 * k, db + 2 * k, idesc, kb > 0 || k > 0);
          core_commit(smem_u32(&bars.empty[sl]));
        }
        if (ok) core_commit(smem_u32(&bars.accf[buf]));
      }
      // every MMA issued, also of a tile given up on, ends before the tensor memory goes back
      core_commit(smem_u32(&bars.drain));
      ok = mb_wait(smem_u32(&bars.drain), 0, CORE_DRAIN_NS) && ok;
      if (!ok) set_err(status, DEVERR_TIMEOUT);
    }
  } else {                                      // ------------ finished tiles
    const int quad = wid & 3, half = wid >> 2, tid = threadIdx.x;
    const WT* Wm = (const WT*)cv.W;
    auto lists = [&](const int4& td, int32_t& lu, int32_t& lv) {   // core indices of this thread's u and v, or -1
      const int d = td.z, u = (td.w & 0xffff) * CORE_BLK + quad * 32 + lane, v = (td.w >> 16) * CORE_TN + tid;
      const int64_t r0 = g.R[g.n - td.y] - d;   // the row of rank n - 1 - s ends at R[n - s]
      lu = u < d ? (int32_t)(g.C[r0 + u] - cv.h0) : -1;
      lv = v < d ? (int32_t)(g.C[r0 + v] - cv.h0) : -1;
    };
    int4 td = make_int4(0, 0, 0, 0), td1 = td;
    int32_t lu = -1, lv = -1;
    int64_t t = blockIdx.x;
    if (t < ntiles) {
      td = tiles[t];
      lists(td, lu, lv);
      wrow[tid] = Wm + (lv >= 0 ? cv.rowb[lv] : 0);
      lu = lu >= 0 ? cv.li[lu] : 0;
      if (t + step < ntiles) td1 = tiles[t + step];
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    for (uint32_t it = 0; t < ntiles; t += step, ++it) {
      const uint32_t buf = it & 1;
      // the next tile's descriptor, list entries and W rows are fetched while this one is read
      int32_t lu1 = -1, lv1 = -1;
      int4 td2 = td1;
      const bool more = t + step < ntiles;
      if (more) {
        lists(td1, lu1, lv1);
        if (t + 2 * step < ntiles) td2 = tiles[t + 2 * step];
      }
      const int d = td.z, u = (td.w & 0xffff) * CORE_BLK + quad * 32 + lane, v0 = (td.w >> 16) * CORE_TN;
      const WT* bc = HASB ? b_all + (tri_off[td.y] - tri_off[s0]) : nullptr;
      // adjacency bits of the warp's 32 rows, one word per column; the slots from
      // pos on lead to vertices above c
      const int64_t c = g.n - 1 - td.y;
      const int nb = (d + CORE_BLK - 1) / CORE_BLK, pos = d - (int)(g.R[c + 1] - g.op[c]);
      const uint32_t* bw = bitm + (int64_t)td.x * CORE_BIT_WORDS + (td.w & 0xffff) * 4 + quad;
      unsigned long long* k4c = k4 + (g.R[c + 1] - d - k4_0);
      unsigned long long swy = 0, syy = 0, sy = 0, sbb = 0, s20 = 0, sk = 0;
      const bool ok = __all_sync(0xffffffffu, mb_wait(smem_u32(&bars.accf[buf]), (it >> 1) & 1,
                                                      it + 1 == give_up ? 0 : wait_ns));
      tc_fence_after();
      const WT* const* wr = wrow + buf * CORE_TN;
      constexpr int QC = HASB ? 16 : 32;        // columns in flight (registers)
#pragma unroll 1
      for (int q0 = half * 128; q0 < half * 128 + 128; q0 += QC) {
        const int vb = v0 + q0;
        if (vb >= d || !ok) break;
        if (vb + QC - 1 <= u - lane) continue;      // every pair of the warp has u >= v
        uint32_t m[QC];
        tmem_ld(m, tmem + buf * CORE_TN + q0 + ((uint32_t)(quad * 32) << 16));
        uint32_t w[QC], bb[HASB ? QC : 1];
        uint32_t adj = 0, col = 0;              // lane l: the bits and the M sum of column vb + l
        if (lane < QC) {
          const int v = vb + lane;              // padded rows are zero
          adj = __ldg(bw + (int64_t)(v / CORE_BLK) * nb * CORE_BIT_WORDS + (v % CORE_BLK) * (nb * 4));
        }
        const bool full = vb > u && vb + QC - 1 < d;
#pragma unroll
        for (int q = 0; q < QC; ++q) {
          const bool on = full || (vb + q > u && vb + q < d);
          w[q] = on ? (uint32_t)__ldg(wr[q0 + q] + lu) : 0u;
          if (HASB) {
            const int64_t v = vb + q;
            bb[HASB ? q : 0] = on ? (uint32_t)__ldg(bc + v * (v - 1) / 2 + u) : 0u;
          }
        }
        tmem_ld_wait();
        typename CoreSum<WT>::type sy32 = 0;
#pragma unroll
        for (int q = 0; q < QC; ++q) {
          const bool on = full || (vb + q > u && vb + q < d);
          // an integer below 2^23 in fp32: its low mantissa bits after adding 2^23
          uint32_t y = on ? __float_as_uint(__uint_as_float(m[q]) + 8388608.0f) & 0x7fffffu : 0u;
          const bool ad = ((__shfl_sync(0xffffffffu, adj, q) >> lane) & 1u) != 0;
          const uint32_t mk = ad ? y : 0u;
          const uint32_t cs = __reduce_add_sync(0xffffffffu, mk);
          if (lane == q) col = cs;
          sk += mk;
          uint32_t k = mk;
          if (HASB) {
            const uint32_t b = bb[HASB ? q : 0];
            y += 2 * b;
            sbb += (unsigned long long)b * b;
            if (ad) k += b;
          }
          s20 += (unsigned long long)k * (k - 1u);   // k = 0: 0 x (2^32 - 1)
          swy += (unsigned long long)w[q] * y;
          syy += (unsigned long long)y * y;
          sy32 += y;
        }
        sy += sy32;
        if (col && vb + lane >= pos) atomicAdd(&k4c[vb + lane], (unsigned long long)col);
      }
      if (sk && u >= pos) atomicAdd(&k4c[u], sk);
      tc_fence_before();
      __syncwarp();
      if (lane == 0 && ok) mb_arrive(smem_u32(&bars.acce[buf]));
      la.v[0] += swy - 2 * sy;                  // 2 x N17: W >= 2 wherever Y > 0
      la.v[1] += syy - sy - 2 * sbb;            // 4 x N18
      la.v[2] += s20 / 2;                       // 3 x N20
      la.v[3] += sk;                            // 12 x K4
      warp_item_flush(la, ids, acc, g.n - 1 - td.y);
      if (more) {
        wrow[(buf ^ 1) * CORE_TN + tid] = Wm + (lv1 >= 0 ? cv.rowb[lv1] : 0);
        lu = lu1 >= 0 ? cv.li[lu1] : 0;
      }
      td = td1;
      td1 = td2;
      if (!epi_all(ok)) {                       // one decision for all eight warps
        if (tid == 0) set_err(status, DEVERR_TIMEOUT);
        break;
      }
    }
  }
  __syncthreads();
  if (wid == CORE_EPI_WARPS + 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  final_flush(la, ids, acc, sh);
}

// ---------------------------------------------------------------- host side
static unsigned core_grid(int64_t work, int threads, int sms) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((work + threads - 1) / threads, (int64_t)sms * 8));
}

cudaError_t core_layout(const DevGraph& g, int64_t h0, bool single, int32_t* dh, int32_t* li, int64_t* rowb,
                        int64_t* off, int sms, cudaStream_t s) {
  const int64_t h = g.n - h0;
  (k_core_dims<<<core_grid(h, 256, sms), 256, 0, s>>>(g, h0, dh, single ? li : nullptr, rowb), note_launch());
  (k_core_scan<<<1, 1024, 0, s>>>(dh, h, off), note_launch());
  return cudaGetLastError();
}

cudaError_t core_union(const int32_t* vg, int num_graphs, int64_t h0, int64_t h, int32_t* hl, int64_t* hb, int32_t* li,
                       int64_t* rowb, int64_t* wbase, DeviceArena& arena, int sms, cudaStream_t s) {
  const size_t mark = arena.mark();
  uint64_t* keys = (uint64_t*)arena.alloc(sizeof(uint64_t) * (h + 1));
  uint64_t* tk = (uint64_t*)arena.alloc(sizeof(uint64_t) * (h + 1));
  uint32_t* vals = (uint32_t*)arena.alloc(sizeof(uint32_t) * (h + 1));
  uint32_t* tv = (uint32_t*)arena.alloc(sizeof(uint32_t) * (h + 1));
  int64_t* start = (int64_t*)arena.alloc(sizeof(int64_t) * (num_graphs + 1));
  if (!keys || !tk || !vals || !tv || !start) return cudaErrorMemoryAllocation;
  cudaError_t e = cudaMemsetAsync(start, 0, sizeof(int64_t) * (num_graphs + 1), s);
  if (e != cudaSuccess) return e;
  (k_core_union_count<<<core_grid(h, 256, sms), 256, 0, s>>>(vg, h0, h, keys, vals, (unsigned long long*)start),
   note_launch());
  (k_core_union_squares<<<core_grid(num_graphs, 256, sms), 256, 0, s>>>(start, num_graphs, wbase), note_launch());
  e = exclusive_scan_i64(start, start, num_graphs, true, arena, s);
  if (e == cudaSuccess) e = exclusive_scan_i64(wbase, wbase, num_graphs, true, arena, s);
  if (e == cudaSuccess) e = radix_sort(keys, vals, tk, tv, h, bits_for(num_graphs), arena, s);
  if (e != cudaSuccess) return e;
  (k_core_union_place<<<core_grid(h, 256, sms), 256, 0, s>>>(keys, vals, h0, h, start, wbase, hl, hb, li, rowb),
   note_launch());
  arena.release(mark);
  return cudaGetLastError();
}

cudaError_t core_low(const DevGraph& g, const uint32_t* T, const int64_t* off, const int32_t* U, int64_t h0,
                     uint32_t* low, int sms, cudaStream_t s) {
  (k_core_low<<<core_grid(g.n * 32, 256, sms), 256, 0, s>>>(g, T, off, U, h0, low), note_launch());
  return cudaGetLastError();
}

void core_chunks(const int64_t* off, int64_t h, int64_t cap_bytes, CoreChunks* ck) {
  const int64_t *rb = off, *blk = off + (h + 1), *til = off + 2 * (h + 1), *tri = off + 3 * (h + 1);
  ck->start.assign(1, 0);
  ck->max_blocks = ck->max_tiles = ck->max_tri = 0;
  ck->max_row_blocks = 0;
  for (int64_t s = 0; s < h; ++s) ck->max_row_blocks = std::max(ck->max_row_blocks, rb[s + 1] - rb[s]);
  int64_t s0 = 0;
  while (s0 < h && blk[s0] < blk[h]) {
    // as many centres as fit the byte limit, at least one
    int64_t s1 = std::upper_bound(blk + s0 + 1, blk + h + 1, blk[s0] + cap_bytes / CORE_BLK_BYTES) - blk - 1;
    s1 = std::max(s1, s0 + 1);
    if (blk[s1] == blk[h]) s1 = h;
    ck->max_blocks = std::max(ck->max_blocks, blk[s1] - blk[s0]);
    ck->max_tiles = std::max(ck->max_tiles, til[s1] - til[s0]);
    ck->max_tri = std::max(ck->max_tri, tri[s1] - tri[s0]);
    ck->start.push_back(s1);
    s0 = s1;
  }
}
size_t core_block_bytes(const CoreChunks& ck) { return (size_t)ck.max_blocks * CORE_BLK_BYTES; }
size_t core_bit_bytes(const CoreChunks& ck) { return (size_t)ck.max_blocks * CORE_BIT_WORDS * sizeof(uint32_t); }

template <typename WT>
static cudaError_t core_run_as(const DevGraph& g, const CoreView& cv, const uint32_t* T, const int64_t* offp,
                               const int32_t* P, const int64_t* d_off, const int64_t* off, const CoreChunks& ck,
                               const CoreBuffers& cb, const AccSet& acc, unsigned* status, int sms, int smem_optin,
                               cudaStream_t s) {
  const int64_t h = g.n - cv.h0;
  const int64_t *rb = off, *til = off + 2 * (h + 1), *tri = off + 3 * (h + 1);
  const int bit_words = (int)ck.max_row_blocks * 4;
  const size_t smem_b = sizeof(uint32_t) * 8 * (size_t)bit_words;
  cudaError_t e = cudaFuncSetAttribute((const void*)k_core_build, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       smem_optin - 1024);
  const void* km = cb.b ? (const void*)k_core_mma<WT, true> : (const void*)k_core_mma<WT, false>;
  if (e == cudaSuccess) e = cudaFuncSetAttribute(km, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CORE_SMEM);
  for (size_t k = 0; k + 1 < ck.start.size() && e == cudaSuccess; ++k) {
    const int64_t s0 = ck.start[k], s1 = ck.start[k + 1], nt = til[s1] - til[s0];
    if (nt == 0) continue;
    const int64_t* d_tri = d_off + 3 * (h + 1);
    WT* b = (WT*)cb.b;
    if (b) {
      e = cudaMemsetAsync(b, 0, sizeof(WT) * (size_t)(tri[s1] - tri[s0]), s);
      if (e != cudaSuccess) break;
      (k_core_mixed<WT><<<(unsigned)(s1 - s0), 256, 0, s>>>(g, T, offp, P, cv.h0, cv.dh, d_tri, s0, b), note_launch());
    }
    (k_core_build<<<(unsigned)(rb[s1] - rb[s0]), 256, smem_b, s>>>(g, T, offp, P, cv.h0, h, cv.dh, d_off, s0, s1,
                                                                   bit_words, (uint8_t*)cb.blocks, (uint32_t*)cb.bits,
                                                                   (int4*)cb.tiles),
     note_launch());
    const unsigned grid = (unsigned)std::min<int64_t>(sms, nt);
    if (b)
      (k_core_mma<WT, true><<<grid, CORE_THREADS, CORE_SMEM, s>>>(g, cv, (const int4*)cb.tiles, nt,
                                                                  (const uint8_t*)cb.blocks, (const uint32_t*)cb.bits,
                                                                  (unsigned long long*)cb.k4, cb.k4_0, b, d_tri, s0, acc,
                                                                  status, cb.wait_ns, cb.give_up),
       note_launch());
    else
      (k_core_mma<WT, false><<<grid, CORE_THREADS, CORE_SMEM, s>>>(g, cv, (const int4*)cb.tiles, nt,
                                                                   (const uint8_t*)cb.blocks, (const uint32_t*)cb.bits,
                                                                   (unsigned long long*)cb.k4, cb.k4_0, nullptr, d_tri,
                                                                   s0, acc, status, cb.wait_ns, cb.give_up),
       note_launch());
    e = cudaGetLastError();
  }
  return e;
}

cudaError_t core_run(const DevGraph& g, const CoreView& cv, const uint32_t* T, const int64_t* offp, const int32_t* P,
                     const int64_t* d_off, const int64_t* off, const CoreChunks& ck, const CoreBuffers& cb,
                     const AccSet& acc, unsigned* status, int sms, int smem_optin, cudaStream_t s) {
  return cv.wide ? core_run_as<uint32_t>(g, cv, T, offp, P, d_off, off, ck, cb, acc, status, sms, smem_optin, s)
                 : core_run_as<uint16_t>(g, cv, T, offp, P, d_off, off, ck, cb, acc, status, sms, smem_optin, s);
}

}  // namespace esc
