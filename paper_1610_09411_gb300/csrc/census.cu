// census.cu -- the enumeration and assembly kernels of the 5-vertex census.
//
// All vertices are ranks of the degree order (Sec. 3.2), so `a < b` is the
// order itself; N+(v) is the suffix of row v, N-(v) its prefix.  Counts are
// exact: per-element counters are 32/64-bit, global sums 128-bit.
//
// Kernel map (paper section -> kernel):
//   Thm 4, 8, 9 degree/edge closed forms ...... k_vertex_basic, k_edge_sums
//   Thm 7 triangles T(e), t(i) ................ k_tri_small / k_tri_large (pass A)
//   Thm 6/7 4-cliques K4(e), K4(t); Thm 10 N10,
//     N16, N20; Thm 14 5-cliques ............... k_clique_warp / k_clique_large (pass B)
//   Thm 13's directed tailed triangles ......... k_tri_small / k_tri_large (pass A)
//   Thm 5 4-cycles C4(e), C4(i) ................ k_cycles4_*
//   Thm 12 common-neighbour lists of edges ..... k_tri_lists
//   Thm 11/12 N13, N17 (pairs and diamonds) .... k_pairs_*, core.cu
//   Thm 11 N18 (wheels) ........................ k_wheels_warp / k_wheels_cta
//   Thm 13 5-cycles ............................ k_cycles5*
//   Thm 3 + App. B assembly .................... k_assemble
#include "common.cuh"
#include "core.cuh"
#include "estimate.h"
#include "internal.h"
#include "launch.h"

#include <algorithm>
#include <initializer_list>
#if defined(__has_include)
#if __has_include(<nvtx3/nvToolsExt.h>)
#include <nvtx3/nvToolsExt.h>          // header-only: no library to link
#define ESC_HAVE_NVTX 1
#endif
#endif
#ifndef ESC_HAVE_NVTX
#define ESC_HAVE_NVTX 0
#endif
#include <map>
#include <mutex>
#include <cstdio>
#include <cstdlib>
#include <vector>

namespace esc {

// ----------------------------------------------------------------------------
// Small device hash set of vertex ranks -> position (open addressing).
// ----------------------------------------------------------------------------
struct PosHash {
  int32_t* keys;     // EMPTY = -1
  int32_t* vals;
  int mask;
  __device__ __forceinline__ uint32_t h(int32_t k) const { return ((uint32_t)k * 0x9E3779B1u) >> 7; }
  __device__ __forceinline__ void insert(int32_t k, int32_t v) {
    uint32_t s = h(k) & mask;
    while (true) {
      int32_t old = atomicCAS(&keys[s], -1, k);
      if (old == -1 || old == k) { vals[s] = v; return; }
      s = (s + 1) & mask;
    }
  }
  __device__ __forceinline__ int32_t find(int32_t k) const {
    uint32_t s = h(k) & mask;
    while (true) {
      int32_t kk = keys[s];
      if (kk == k) return vals[s];
      if (kk == -1) return -1;
      s = (s + 1) & mask;
    }
  }
};

static __host__ __device__ __forceinline__ int pow2_at_least(int x) {
  int p = 1;
  while (p < x) p <<= 1;
  return p;
}

// ============================================================================
// Degree sums (Thm 4, Thm 8 N1/N3, Thm 9 N2, App. A P3+K2 terms).
// One warp per vertex.
// ============================================================================
__global__ void k_vertex_basic(DevGraph g, AccSet acc) {
  __shared__ u128 sh[32];
  int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int ids[9] = {ACC_W, ACC_S3, ACC_S4, ACC_D2D, ACC_DNBR, ACC_N2A, ACC_N3A, ACC_P4A, ACC_DP};
  LocalAcc<9> la;
  la.zero();
  for (int64_t v = warp; v < g.n; v += nwarps) {
    unsigned long long dv = (unsigned long long)dg_deg(g, v);
    unsigned long long dpv = (unsigned long long)dg_outdeg(g, v);
    u128 s1 = 0, s2 = 0, nb = 0, n2a = 0, p4a = 0, dp = 0;
    for (int64_t p = g.R[v] + lane; p < g.R[v + 1]; p += 32) {
      int32_t a = g.C[p];
      unsigned long long da = (unsigned long long)dg_deg(g, a);
      s1 += da - 1;
      s2 += (u128)(da - 1) * (da - 1);
      nb += da;
      n2a += ch2(dv - 1) * (da - 1);
      if (a > v) {
        p4a += (u128)(dv - 1) * (da - 1);
        dp += (u128)(dpv - 1) * (unsigned long long)dg_outdeg(g, a);   // the path's middle edge v -> a
      }
    }
    s1 = warp_sum_u128(s1);
    s2 = warp_sum_u128(s2);
    nb = warp_sum_u128(nb);
    n2a = warp_sum_u128(n2a);
    p4a = warp_sum_u128(p4a);
    dp = warp_sum_u128(dp);
    if (lane == 0) {
      la.v[8] += dp;
      la.v[0] += ch2(dv);
      la.v[1] += ch3(dv);
      la.v[2] += ch4(dv);
      la.v[3] += ch2(dv) * dv;
      la.v[4] += dv ? (u128)(dv - 1) * nb : 0;
      la.v[5] += n2a;
      la.v[6] += (s1 * s1 - s2) / 2;
      la.v[7] += p4a;
    }
    warp_item_flush(la, ids, acc, v);
  }
  final_flush(la, ids, acc, sh);
}

// ============================================================================
// Pass A: triangles.  Every triangle x < v < w is found once from its lowest
// vertex x as v in N+(x), w in N+(v) cap N+(x) (Thm 7).  It adds one to the
// triangle counts of its three edges (canonical slots in the lower endpoint's
// out-list) and contributes d+(x) + d+(v) + d+(w) - 3 to the directed
// tailed-triangle term of the 5-cycle count (Thm 13).
// ============================================================================
static constexpr int SMALL_DPLUS = 32;    // warp-per-vertex path up to this out-degree

// Warp per vertex with d+ <= 32: N+(x) in a per-warp shared-memory list,
// membership by binary search.
__global__ void k_tri_small(DevGraph g, const int32_t* items, int64_t nitems, uint32_t* T, AccSet acc) {
  __shared__ u128 sh[32];
  __shared__ int32_t lst[8][SMALL_DPLUS];
  __shared__ uint32_t cnt[8][SMALL_DPLUS];
  int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int ids[2] = {ACC_T, ACC_N8Z};
  LocalAcc<2> la;
  la.zero();
  for (int64_t it = warp; it < nitems; it += nwarps) {
    int64_t x = items[it];
    int64_t o = g.op[x];
    int d = (int)(g.R[x + 1] - o);
    if (lane < d) lst[wl][lane] = g.C[o + lane];
    cnt[wl][lane] = 0;
    __syncwarp();
    unsigned long long dpx = (unsigned long long)d;
    for (int a = 0; a < d; ++a) {
      int32_t v = lst[wl][a];
      int64_t vo = g.op[v], ve = g.R[v + 1];
      unsigned long long dpv = (unsigned long long)(ve - vo);
      for (int64_t q = vo + lane; q < ve; q += 32) {
        int32_t w = g.C[q];
        int lo = a + 1, hi = d;                 // w > v, so only positions after a
        while (lo < hi) { int mid = (lo + hi) >> 1; if (lst[wl][mid] < w) lo = mid + 1; else hi = mid; }
        if (lo < d && lst[wl][lo] == w) {
          atomicAdd(&T[q], 1u);
          atomicAdd(&cnt[wl][a], 1u);
          atomicAdd(&cnt[wl][lo], 1u);
          la.v[0] += 1;
          la.v[1] += dpx + dpv + (unsigned long long)(g.R[w + 1] - g.op[w]) - 3;
        }
      }
    }
    __syncwarp();
    if (lane < d && cnt[wl][lane]) atomicAdd(&T[o + lane], cnt[wl][lane]);
    __syncwarp();
    warp_item_flush(la, ids, acc, x);
  }
  final_flush(la, ids, acc, sh);
}

// CTA per vertex with d+ > 32: N+(x) in a shared-memory hash.
__global__ void k_tri_large(DevGraph g, const int32_t* items, int64_t nitems, unsigned long long* qctr,
                            uint32_t* T, AccSet acc, int hash_cap) {
  extern __shared__ int32_t smem[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  int32_t* hk = smem;
  int32_t* hv = hk + hash_cap;
  uint32_t* cnt = (uint32_t*)(hv + hash_cap);
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int ids[2] = {ACC_T, ACC_N8Z};
  LocalAcc<2> la;
  la.zero();
  while (true) {
    int64_t it = next_item(qctr, nitems, &sh_item);
    if (it < 0) break;
    int64_t x = items[it];
    int64_t o = g.op[x];
    int d = (int)(g.R[x + 1] - o);
    int hsz = pow2_at_least(2 * d);
    PosHash H{hk, hv, hsz - 1};
    for (int i = threadIdx.x; i < hsz; i += blockDim.x) hk[i] = -1;
    for (int i = threadIdx.x; i < d; i += blockDim.x) cnt[i] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < d; i += blockDim.x) H.insert(g.C[o + i], i);
    __syncthreads();
    unsigned long long dpx = (unsigned long long)d;
    for (int a = wid; a < d; a += nw) {
      int32_t v = g.C[o + a];
      int64_t vo = g.op[v], ve = g.R[v + 1];
      unsigned long long dpv = (unsigned long long)(ve - vo);
      unsigned on_xv = 0;
      for (int64_t q = vo + lane; q < ve; q += 32) {
        int32_t w = g.C[q];
        int b = H.find(w);
        if (b >= 0) {
          atomicAdd(&T[q], 1u);
          atomicAdd(&cnt[b], 1u);
          on_xv += 1;
          la.v[0] += 1;
          la.v[1] += dpx + dpv + (unsigned long long)(g.R[w + 1] - g.op[w]) - 3;
        }
      }
      on_xv = (unsigned)warp_sum_u64(on_xv);
      if (lane == 0 && on_xv) atomicAdd(&cnt[a], on_xv);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < d; i += blockDim.x)
      if (cnt[i]) atomicAdd(&T[o + i], cnt[i]);
    block_item_flush(la, ids, acc, x, sh);
    __syncthreads();
  }
  final_flush(la, ids, acc, sh);
}

// Copy canonical per-edge values to the reverse slot; per-vertex sums.
__global__ void k_sym_T(DevGraph g, uint32_t* T) {
  int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < g.n; v += nwarps)
    for (int64_t p = g.op[v] + lane; p < g.R[v + 1]; p += 32) T[g.rev[p]] = T[p];
}

__global__ void k_vertex_from_edges_T(DevGraph g, const uint32_t* T, unsigned long long* tv) {
  int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < g.n; v += nwarps) {
    unsigned long long s = 0;
    for (int64_t p = g.R[v] + lane; p < g.R[v + 1]; p += 32) s += T[p];
    s = warp_sum_u64(s);
    if (lane == 0) tv[v] = s / 2;
  }
}

// 4-cliques per edge: the canonical slot holds those whose lowest vertex lies
// below the core (all of them without one), H2 (slots from r0 on, or null) twice
// those inside the core; their sum goes to both slots.
__global__ void k_sym_K4(DevGraph g, unsigned long long* E, const unsigned long long* H2, int64_t r0) {
  int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < g.n; v += nwarps)
    for (int64_t p = g.op[v] + lane; p < g.R[v + 1]; p += 32) {
      unsigned long long e = E[p];
      if (H2 && p >= r0) {
        e += H2[p - r0] / 2;
        E[p] = e;
      }
      E[g.rev[p]] = e;
    }
}

// 4-cycle per-edge counts arrive in either slot of an edge: fold them.
__global__ void k_fold_u64(DevGraph g, unsigned long long* E) {
  int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < g.n; v += nwarps)
    for (int64_t p = g.op[v] + lane; p < g.R[v + 1]; p += 32) {
      int64_t r = g.rev[p];
      unsigned long long s = E[p] + E[r];
      E[p] = s;
      E[r] = s;
    }
}

__global__ void k_vertex_sum_div(DevGraph g, const unsigned long long* E, unsigned long long* V, unsigned div) {
  int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < g.n; v += nwarps) {
    unsigned long long s = 0;
    for (int64_t p = g.R[v] + lane; p < g.R[v + 1]; p += 32) s += E[p];
    s = warp_sum_u64(s);
    if (lane == 0) V[v] = s / div;
  }
}

// ============================================================================
// Pass B: 4-cliques, 5-cliques and the per-triangle sums.
//
// For the lowest vertex x, B holds the adjacency bit matrix of the graph
// induced on N+(x) (row a = the out-neighbours of N+(x)[a] that are also in
// N+(x)).  For an edge (a, b) of it -- the triangle {x, v_a, v_b} with x
// lowest --
//   alpha = |row_a & row_b|   apexes of the triangle above x (K4s x,a,b,c)
//   beta  = apexes below x: in-neighbours y of x adjacent to v_a and v_b.
//           With D_a = bit set over N-(x) of {y : v_a in N+(y)}, beta =
//           |D_a & D_b|.
// so K4(t) = alpha + beta (Thm 7), and
//   N20 += C(alpha + beta, 2)                                (Thm 10)
//   N10 += sum over the 3 vertices k of (T(opposite edge) - 1)(d_k - 2)
//   N16 += sum over the 3 vertices of (T(e1) - 1)(T(e2) - 1)  (Thm 10)
//   K4 total += alpha / 3; K4(v_a, v_b) += alpha; K4(x, v_a) += alpha / 2 summed
//   K5 += |row_a & row_b & row_c| above c for every c in row_a & row_b above b
//        (each 5-clique once, at its three lowest vertices: Thm 14)
// ============================================================================
struct CliqueScratch {
  uint64_t* D;         // per CTA: d+ x ceil(d-/64) words
  int64_t d_words;     // capacity per CTA in words
  uint64_t* G;         // per CTA: the bit matrix and its companions when they exceed shared memory
  int64_t g_words;     // capacity per CTA in words
};

// Bytes of the clique pass's work space for out-degree d (B, K4 accumulators,
// hash of 2 x pow2(2d) ints, T and degree of x's out-neighbours).  B rows are
// clique_stride(d) words apart: an odd stride, so the lanes of a warp reading
// word w of 32 different rows hit different shared-memory banks (an even stride
// of 2^k words puts them on 32 / 2^k banks).
static inline __host__ __device__ int clique_stride(int d) { return ((d + 63) >> 6) | 1; }
static constexpr int CLQ_MAX_WARPS = 16;         // warps of a CTA of the clique pass (512 threads)
static inline size_t clique_space(int d) {
  int h = 1;
  while (h < 2 * d) h <<= 1;
  return sizeof(uint64_t) * ((size_t)d * clique_stride(d) + d) + sizeof(int32_t) * (2 * (size_t)h) +
         sizeof(uint32_t) * 2 * (size_t)((d + 1) & ~1);
}
// per warp: a batch of CLQ_BATCH vertices b and their prefix sums (5-cliques);
// also the queue of edges waiting for a full warp (32 + 31 entries of two ints)
static constexpr int CLQ_BATCH_WORDS = 4, CLQ_BATCH = 64 * CLQ_BATCH_WORDS;
struct CliqueWarp {
  uint32_t pre[CLQ_BATCH];
  uint8_t b[CLQ_BATCH];            // from the first vertex of the batch
};

// Position of the k-th (0-based) set bit of m (k < popc(m)).
__device__ __forceinline__ int select32(unsigned m, int k) {
  int pos = 0, c = __popc(m & 0xffffu);
  if (k >= c) { k -= c; m >>= 16; pos += 16; }
  c = __popc(m & 0xffu);
  if (k >= c) { k -= c; m >>= 8; pos += 8; }
  c = __popc(m & 0xfu);
  if (k >= c) { k -= c; m >>= 4; pos += 4; }
  c = __popc(m & 0x3u);
  if (k >= c) { k -= c; m >>= 2; pos += 2; }
  if (k >= (int)(m & 1u)) pos += 1;
  return pos;
}
__device__ __forceinline__ int select64(uint64_t x, int k) {
  const int c = __popc((unsigned)x);
  return k < c ? select32((unsigned)x, k) : 32 + select32((unsigned)(x >> 32), k - c);
}
// bits above position b (of the word that holds position b + 1)
__device__ __forceinline__ uint64_t above_mask(int b) { return ~0ull << ((b + 1) & 63); }

// 5-cliques (Thm 14) whose two lowest vertices are x and v_a, by one warp: for
// every b above a in row a, the candidates c are the common neighbours of v_a
// and v_b above b, and each pair (b, c) adds the common neighbours of the three
// above c.  The b come in batches of CLQ_BATCH_WORDS words of row a; the pairs
// of a batch, numbered through by the prefix sums of |candidates|, are split
// evenly over the lanes, so every lane walks about the same number of pairs and
// nothing is shared per edge (one edge at a time for the whole warp cost some
// 150 warp instructions per edge before its first candidate: k_clique_large on
// R-MAT 19 149 -> 116 ms, on 96 graphs of up to 2,000 vertices 70 -> 41 ms; with
// the 4-cliques and N20 of the core taken from its contraction 94 and 28.5 ms).
// dbp += C(candidates, 2) per edge (directed bipyramids).
// A bit matrix in global memory (SPLIT false) has one b per lane instead, and the
// lanes go through the words of their candidates together: in the dense graphs
// that have such out-degrees they then read the same row c at a time, where an
// even split reads 32 rows (K_1500, clique phase 3,650 -> 2,110 ms; a lane's
// candidates without the other lanes' words 3,000 ms).
template <bool SPLIT>
__device__ __forceinline__ void k5_row(const uint64_t* B, int W, int RS, int a, CliqueWarp* cw, unsigned long long& k5,
                                       u128& dbp) {
  const int lane = threadIdx.x & 31;
  const uint64_t* ra = B + (int64_t)a * RS;
  for (int wb = (a + 1) >> 6; wb < W; wb += CLQ_BATCH_WORDS) {
    uint64_t m = 0;
    if (lane < CLQ_BATCH_WORDS && wb + lane < W) {
      m = ra[wb + lane];
      if (wb + lane == (a + 1) >> 6) m &= above_mask(a);
    }
    const int cnt = __popcll(m);
    const int c0 = __shfl_sync(0xffffffffu, cnt, 0), c1 = c0 + __shfl_sync(0xffffffffu, cnt, 1),
              c2 = c1 + __shfl_sync(0xffffffffu, cnt, 2), s = c2 + __shfl_sync(0xffffffffu, cnt, 3);
    unsigned total = 0;
    for (int t0 = 0; t0 < s; t0 += 32) {
      const int t = t0 + lane;
      const int wq = t < c0 ? 0 : (t < c1 ? 1 : (t < c2 ? 2 : 3));
      const uint64_t mw = __shfl_sync(0xffffffffu, m, wq);
      unsigned n = 0;
      int b = 0;
      if (t < s) {
        b = (wb + wq) * 64 + select64(mw, t - (wq == 0 ? 0 : (wq == 1 ? c0 : (wq == 2 ? c1 : c2))));
        const uint64_t* rb = B + (int64_t)b * RS;
        int u = (b + 1) >> 6;
        if (u < W) n = __popcll(ra[u] & rb[u] & above_mask(b));
        for (++u; u < W; ++u) n += __popcll(ra[u] & rb[u]);
        if (n >= 2) dbp += (unsigned long long)n * (n - 1) / 2;
        else n = 0;                             // a lone candidate closes no 5-clique
      }
      if (!SPLIT) {                             // the lanes go through the words together
        const uint64_t* rb = B + (int64_t)b * RS;
        const int wb0 = (b + 1) >> 6;
        for (int w = __shfl_sync(0xffffffffu, wb0, 0); w < W; ++w) {   // lane 0 holds the lowest b
          uint64_t cm = n && w >= wb0 ? ra[w] & rb[w] : 0;
          if (w == wb0) cm &= above_mask(b);
          while (cm) {
            const int c = w * 64 + __ffsll((long long)cm) - 1;
            cm &= cm - 1;
            const uint64_t* rc = B + (int64_t)c * RS;
            int u = (c + 1) >> 6;
            unsigned part = u < W ? __popcll(ra[u] & rb[u] & rc[u] & above_mask(c)) : 0u;
            for (++u; u + 4 <= W; u += 4)       // independent loads in flight
              part += __popcll(ra[u] & rb[u] & rc[u]) + __popcll(ra[u + 1] & rb[u + 1] & rc[u + 1]) +
                      __popcll(ra[u + 2] & rb[u + 2] & rc[u + 2]) + __popcll(ra[u + 3] & rb[u + 3] & rc[u + 3]);
            for (; u < W; ++u) part += __popcll(ra[u] & rb[u] & rc[u]);
            k5 += part;
          }
          __syncwarp();
        }
        continue;
      }
      unsigned incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (t < s) {
        cw->b[t] = (uint8_t)(b - wb * 64);
        cw->pre[t] = total + incl - n;
      }
      total += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (!SPLIT) continue;
    __syncwarp();
    const unsigned share = (total + 31) / 32, p0 = min(total, lane * share), p1 = min(total, p0 + share);
    if (p0 < p1) {
      int lo = 0, hi = s;                       // the b of pair p0: the last t with pre[t] <= p0
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (cw->pre[mid] <= p0) lo = mid; else hi = mid;
      }
      int t = lo, skip = (int)(p0 - cw->pre[t]);
      unsigned left = p1 - p0;
      while (true) {
        const int b = wb * 64 + cw->b[t];
        const uint64_t* rb = B + (int64_t)b * RS;
        unsigned here = min(left, (t + 1 < s ? cw->pre[t + 1] : total) - cw->pre[t] - (unsigned)skip);
        left -= here;
        int w = (b + 1) >> 6;
        uint64_t cm = here ? ra[w] & rb[w] & above_mask(b) : 0;
        while (here) {
          const int c_w = __popcll(cm);
          if (skip >= c_w) {                    // also: the word is used up
            skip -= c_w;
            ++w;
            cm = ra[w] & rb[w];
            continue;
          }
          if (skip) {
            cm &= ~0ull << select64(cm, skip);
            skip = 0;
          }
          const int c = w * 64 + __ffsll((long long)cm) - 1;
          cm &= cm - 1;
          --here;
          const uint64_t* rc = B + (int64_t)c * RS;
          int u = (c + 1) >> 6;
          unsigned part = u < W ? __popcll(ra[u] & rb[u] & rc[u] & above_mask(c)) : 0u;
          for (++u; u < W; ++u) part += __popcll(ra[u] & rb[u] & rc[u]);
          k5 += part;
        }
        if (!left) break;
        skip = 0;
        ++t;
      }
    }
    __syncwarp();                               // the batch is read before the next one is written
  }
}

// The same for rows of at most WW words: lane t of a warp takes the t-th of 32
// consecutive b and all its candidates, with the candidate set in registers, and
// every candidate adds the whole of its intersection with it, above and below
// (each pair of adjacent candidates twice): no masks and the same word loop in
// every lane, at six instructions a word instead of twelve.  k5x2 += 2 x the
// 5-cliques.
template <int WW>
__device__ __forceinline__ void k5_row_reg(const uint64_t* B, int W, int RS, int a, unsigned long long& k5x2, u128& dbp) {
  const int lane = threadIdx.x & 31;
  const uint64_t* ra = B + (int64_t)a * RS;
  uint64_t m = 0;                               // lane l: word l of row a above a
  if (lane < W) {
    m = ra[lane];
    const int w0 = (a + 1) >> 6;
    if (lane < w0) m = 0;
    else if (lane == w0) m &= above_mask(a);
  }
  const int cnt = __popcll(m);
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < WW; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int s = __shfl_sync(0xffffffffu, incl, WW - 1);
  for (int t0 = 0; t0 < s; t0 += 32) {
    const int t = t0 + lane;
    int wq = 0;
#pragma unroll
    for (int u = 0; u < WW - 1; ++u) wq += __shfl_sync(0xffffffffu, incl, u) <= t ? 1 : 0;
    const uint64_t mw = __shfl_sync(0xffffffffu, m, wq);
    const int before = __shfl_sync(0xffffffffu, incl - cnt, wq);
    const int b = t < s ? wq * 64 + select64(mw, t - before) : a;
    const int u0 = __shfl_sync(0xffffffffu, (b + 1) >> 6, 0);   // lane 0 holds the lowest b
    const uint64_t* rb = B + (int64_t)b * RS;
    uint64_t S[WW];
    int n = 0;
#pragma unroll
    for (int u = 0; u < WW; ++u) {
      S[u] = 0;
      if (u >= u0 && u < W) {
        const int wb = (b + 1) >> 6;
        uint64_t x = ra[u] & rb[u];
        if (u < wb || t >= s) x = 0;
        else if (u == wb) x &= above_mask(b);
        S[u] = x;
        n += __popcll(x);
      }
    }
    if (n >= 2) dbp += (unsigned long long)n * (n - 1) / 2;
    else n = 0;                                 // a lone candidate closes no 5-clique
    int w = (b + 1) >> 6;
    uint64_t cm = n ? ra[w] & rb[w] & above_mask(b) : 0;
    unsigned part = 0;                          // below 2^32: n <= 64 WW candidates of as many neighbours
    while (n > 0) {
      while (!cm) {
        ++w;
        cm = ra[w] & rb[w];
      }
      const uint64_t* rc = B + (int64_t)(w * 64 + __ffsll((long long)cm) - 1) * RS;
      cm &= cm - 1;
      --n;
#pragma unroll
      for (int u = 0; u < WW; ++u)
        if (u >= u0 && u < W) part += __popcll(S[u] & rc[u]);
    }
    k5x2 += part;
  }
}

// Work-space layout of the CTA path: B (d x RS u64, rows symmetric: row a = every
// neighbour of v_a inside N+(x)), K4 accumulators (d u64), hash (2 x hcap
// ints), T of x's out-edges and degree of its out-neighbours (d u32 each), in
// shared memory; for out-degrees whose bit matrix does not fit there (GLOBAL_B),
// the same layout in a per-CTA region of global memory (cs.G, cs.g_words words
// per CTA).  The per-warp batches follow in shared memory.
// A launch takes the items with dlo < d+ <= dmax and skips the others.
// five: also what only the 5-vertex counts need (beta, the triangle sums, the
// 5-cliques).  From rank core0 on, the 4-cliques and N20 come from the dense
// core (core.cu): no alpha, beta or D.
template <bool GLOBAL_B>
__global__ void __launch_bounds__(512, 1) k_clique_large(DevGraph g, const int32_t* items, int64_t nitems,
                                                         unsigned long long* qctr, const uint32_t* T,
                                                         unsigned long long* K4e, AccSet acc, CliqueScratch cs,
                                                         int hash_cap, int dlo, int dmax, unsigned* status, bool five,
                                                         int64_t core0) {
  extern __shared__ uint64_t smem64[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  __shared__ int sh_row;
  const int RS_cap = clique_stride(dmax);
  uint64_t* B = GLOBAL_B ? cs.G + (int64_t)blockIdx.x * cs.g_words : smem64;   // dmax * RS_cap
  unsigned long long* k4x = (unsigned long long*)(B + (int64_t)dmax * RS_cap);  // dmax
  int32_t* hk = (int32_t*)(k4x + dmax);                        // hash_cap
  int32_t* hv = hk + hash_cap;                                 // hash_cap
  uint32_t* Tx = (uint32_t*)(hv + hash_cap);                   // dmax, even
  uint32_t* dv = Tx + ((dmax + 1) & ~1);                       // dmax, even
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  CliqueWarp* cw = reinterpret_cast<CliqueWarp*>(GLOBAL_B ? (void*)smem64 : (void*)(dv + ((dmax + 1) & ~1))) + wid;
  uint64_t* D = cs.D + (int64_t)blockIdx.x * cs.d_words;
  const int ids[6] = {ACC_K4, ACC_N20, ACC_N10A, ACC_N16A, ACC_N21, ACC_DBP};
  LocalAcc<6> la;
  la.zero();
  while (true) {
    int64_t it = next_item(qctr, nitems, &sh_item);
    if (it < 0) break;
    int64_t x = items[it];
    int64_t o = g.op[x], ib = g.R[x];
    int d = (int)(g.R[x + 1] - o);
    int din = (int)(o - ib);
    if (d <= dlo || d > dmax) continue;        // the other launch's item
    int W = (d + 63) >> 6;
    const int RS = clique_stride(d);
    int DW = (din + 63) >> 6;
    const bool k4_here = x < core0;
    bool use_beta = five && k4_here && din > 0 && (int64_t)d * DW <= cs.d_words;
    if (five && k4_here && din > 0 && !use_beta && threadIdx.x == 0) set_err(status, DEVERR_SCRATCH);
    int hsz = pow2_at_least(2 * d);
    PosHash H{hk, hv, hsz - 1};
    for (int i = threadIdx.x; i < hsz; i += blockDim.x) hk[i] = -1;
    for (int64_t i = threadIdx.x; i < (int64_t)d * RS; i += blockDim.x) B[i] = 0;
    for (int i = threadIdx.x; i < d; i += blockDim.x) { k4x[i] = 0; Tx[i] = T[o + i]; }
    if (use_beta)
      for (int64_t i = threadIdx.x; i < (int64_t)d * DW; i += blockDim.x) D[i] = 0;
    if (threadIdx.x == 0) sh_row = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
      const int32_t v = g.C[o + i];
      H.insert(v, i);
      dv[i] = (uint32_t)(g.R[v + 1] - g.R[v]);
    }
    __syncthreads();
    unsigned long long dx = (unsigned long long)(g.R[x + 1] - g.R[x]);
    // build B; every hit (a, b) is the triangle {x, v_a, v_b}: its N10 and N16 terms
    for (int a = wid; a < d; a += nw) {
      int32_t v = g.C[o + a];
      const unsigned long long dva = dv[a], txa = Tx[a];
      for (int64_t q = g.op[v] + lane; q < g.R[v + 1]; q += 32) {
        int b = H.find(g.C[q]);
        if (b >= 0) {
          atomicOr((unsigned long long*)&B[(int64_t)a * RS + (b >> 6)], 1ull << (b & 63));
          atomicOr((unsigned long long*)&B[(int64_t)b * RS + (a >> 6)], 1ull << (a & 63));
          if (five) {
            const unsigned long long tab = T[q], txb = Tx[b], dvb = dv[b];
            la.v[2] += (u128)(tab - 1) * (dx - 2) + (u128)(txb - 1) * (dva - 2) + (u128)(txa - 1) * (dvb - 2);   // N10
            la.v[3] += (u128)(txa - 1) * (txb - 1) + (u128)(txa - 1) * (tab - 1) + (u128)(txb - 1) * (tab - 1);  // N16
          }
        }
      }
    }
    // build D: in-neighbour y (index k) sets bit k of D_a for every v_a in N+(y)
    if (use_beta) {
      for (int k = wid; k < din; k += nw) {
        int32_t y = g.C[ib + k];
        for (int64_t q = g.op[y] + lane; q < g.R[y + 1]; q += 32) {
          int a = H.find(g.C[q]);
          if (a >= 0) atomicOr((unsigned long long*)&D[(int64_t)a * DW + (k >> 6)], 1ull << (k & 63));
        }
      }
    }
    __syncthreads();
    // alpha and beta of the edges (a, b) of G[N+(x)]: N+(v_a) is scanned again
    // for the slot of (v_a, v_b); hits wait in the warp's queue until 32 of them
    // fill a warp (about a third of the entries are hits)
    int32_t* qb = reinterpret_cast<int32_t*>(cw);            // b of the waiting edges
    int32_t* qo = qb + 64;                                   // and their offsets in N+(v_a)
    for (int a = wid; a < (k4_here ? d : 0); a += nw) {
      int32_t v = g.C[o + a];
      const int64_t q0 = g.op[v];
      const int len = (int)(g.R[v + 1] - q0);
      const uint64_t* ra = B + (int64_t)a * RS;
      const uint64_t* Da = use_beta ? D + (int64_t)a * DW : nullptr;
      unsigned long long k4a = 0;
      int fill = 0;                                          // the same on every lane
      for (int e = 0; e < len || fill > 0; e += 32) {
        int b = -1;
        if (e + lane < len) b = H.find(g.C[q0 + e + lane]);
        const unsigned hm = __ballot_sync(0xffffffffu, b >= 0);
        if (b >= 0) {
          const int at = fill + __popc(hm & ((1u << lane) - 1u));
          qb[at] = b;
          qo[at] = e + lane;
        }
        fill += __popc(hm);
        if (fill < 32 && e + 32 < len) continue;
        __syncwarp();
        if (lane < fill) {
          const int bb = qb[lane];
          const int64_t q = q0 + qo[lane];
          const uint64_t* rb = B + (int64_t)bb * RS;
          unsigned long long alpha = 0, beta = 0;
#pragma unroll 4
          for (int w = 0; w < W; ++w) alpha += __popcll(ra[w] & rb[w]);
          if (use_beta) {
            const uint64_t* Db = D + (int64_t)bb * DW;
#pragma unroll 8
            for (int w = 0; w < DW; ++w) beta += __popcll(Da[w] & Db[w]);
          }
          la.v[0] += alpha;                                  // 3 x K4
          if (five) la.v[1] += ch2(alpha + beta);            // N20
          if (alpha) {
            atomicAdd(&K4e[q], alpha);
            atomicAdd(&k4x[bb], alpha);
            k4a += alpha;
          }
        }
        // the rest moves to the front
        const int rest = max(fill - 32, 0);
        int32_t mb = 0, mo = 0;
        if (lane < rest) {
          mb = qb[32 + lane];
          mo = qo[32 + lane];
        }
        __syncwarp();
        if (lane < rest) {
          qb[lane] = mb;
          qo[lane] = mo;
        }
        fill = rest;
      }
      k4a = warp_sum_u64(k4a);
      if (lane == 0 && k4a) atomicAdd(&k4x[a], k4a);
      __syncwarp();
    }
    if (five) {                                 // rows handed out one by one: low rows hold most of the work
      unsigned long long k5 = 0, k5x2 = 0;
      while (true) {
        int a = 0;
        if (lane == 0) a = atomicAdd(&sh_row, 1);
        a = __shfl_sync(0xffffffffu, a, 0);
        if (a >= d) break;
        if (!GLOBAL_B && W <= 4) k5_row_reg<4>(B, W, RS, a, k5x2, la.v[5]);
        else if (!GLOBAL_B && W <= 8) k5_row_reg<8>(B, W, RS, a, k5x2, la.v[5]);
        else if (!GLOBAL_B && W <= 12) k5_row_reg<12>(B, W, RS, a, k5x2, la.v[5]);
        else k5_row<!GLOBAL_B>(B, W, RS, a, cw, k5, la.v[5]);
      }
      la.v[4] += k5 + k5x2 / 2;                 // a lane's sum of two-fold counts is even
    }
    __syncthreads();
    for (int i = threadIdx.x; i < d; i += blockDim.x)
      if (k4x[i]) atomicAdd(&K4e[o + i], k4x[i] / 2);
    block_item_flush(la, ids, acc, x, sh);
    __syncthreads();
  }
  final_flush(la, ids, acc, sh);
}

// Small out-neighbourhoods (d+ <= 32 and d- <= CLQ_WARP_DIN): one warp per
// vertex x, everything in the warp's shared memory.  Lane a holds v_a, the
// a-th vertex of N+(x); row a of the bit matrix of G[N+(x)] is one 64-bit word
// and D_a (the in-neighbours of x adjacent to v_a) at most CLQ_WARP_DIN / 64.
// The sums and per-edge counts are those of k_clique_large.
static constexpr int CLQ_WARP_DIN = 512;
static constexpr int CLQ_WARPS = 8;            // warps per block
static constexpr int CLQ_ILP = 4;

__global__ void __launch_bounds__(CLQ_WARPS * 32, 4) k_clique_warp(DevGraph g, const int32_t* items, int64_t nitems,
                                                                unsigned long long* qctr, const uint32_t* T,
                                                                unsigned long long* K4e, AccSet acc, bool with_k5,
                                                                int64_t core0) {
  __shared__ u128 sh[32];
  __shared__ int32_t sL[CLQ_WARPS][32];
  __shared__ uint32_t sT[CLQ_WARPS][32];
  __shared__ unsigned long long sB[CLQ_WARPS][32], sK[CLQ_WARPS][32];
  __shared__ unsigned long long sD[CLQ_WARPS][32][CLQ_WARP_DIN / 64];
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  int32_t* L = sL[wl];
  unsigned long long* Bw = sB[wl];
  unsigned long long* K = sK[wl];
  const int ids[6] = {ACC_K4, ACC_N20, ACC_N10A, ACC_N16A, ACC_N21, ACC_DBP};
  LocalAcc<6> la;
  la.zero();
  // position of vertex key in N+(x) (sorted, padded with INT32_MAX), or -1
  auto find = [&](int32_t key) -> int {
    int lo = 0;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1)
      if (L[lo + st] <= key) lo += st;
    return L[lo] == key ? lo : -1;
  };
  while (true) {
    unsigned long long it_l = 0;
    if (lane == 0) it_l = atomicAdd(qctr, 1ull);
    int64_t it = (int64_t)__shfl_sync(0xffffffffu, it_l, 0);
    if (it >= nitems) break;
    int64_t x = items[it];
    int64_t o = g.op[x], ib = g.R[x];
    int d = (int)(g.R[x + 1] - o);
    int din = (int)(o - ib);
    const bool k4_here = x < core0;                   // else 4-cliques and N20 come from the core
    const int DW = with_k5 && k4_here ? (din + 63) >> 6 : 0;   // beta only feeds N20
    int32_t va = lane < d ? g.C[o + lane] : 0x7fffffff;
    L[lane] = va;
    sT[wl][lane] = lane < d ? T[o + lane] : 0u;
    Bw[lane] = 0;
    K[lane] = 0;
    for (int w = 0; w < DW; ++w) sD[wl][lane][w] = 0;
    __syncwarp();
    // rows of G[N+(x)]: lane a scans N+(v_a) (everything there is above v_a)
    int64_t qa0 = 0, qa1 = 0;
    if (lane < d) {
      qa0 = g.op[va];
      qa1 = g.R[va + 1];
    }
    for (int64_t q = qa0; q < qa1; q += CLQ_ILP) {
      int32_t ww[CLQ_ILP];
#pragma unroll
      for (int u = 0; u < CLQ_ILP; ++u) ww[u] = q + u < qa1 ? g.C[q + u] : 0x7fffffff;
#pragma unroll
      for (int u = 0; u < CLQ_ILP; ++u) {
        int b = ww[u] == 0x7fffffff ? -1 : find(ww[u]);
        if (b >= 0) {
          atomicOr(&Bw[lane], 1ull << b);
          atomicOr(&Bw[b], 1ull << lane);
        }
      }
    }
    // D: in-neighbour y (index k) marks bit k of D_a for every v_a in N+(y)
    for (int k = lane; k < (DW ? din : 0); k += 32) {
      int32_t y = g.C[ib + k];
      int64_t q1 = g.R[y + 1];
      for (int64_t q = g.op[y]; q < q1; q += CLQ_ILP) {
        int32_t ww[CLQ_ILP];
#pragma unroll
        for (int u = 0; u < CLQ_ILP; ++u) ww[u] = q + u < q1 ? g.C[q + u] : 0x7fffffff;
#pragma unroll
        for (int u = 0; u < CLQ_ILP; ++u) {
          int a = ww[u] == 0x7fffffff ? -1 : find(ww[u]);
          if (a >= 0) atomicOr(&sD[wl][a][k >> 6], 1ull << (k & 63));
        }
      }
    }
    __syncwarp();
    // edges (a, b) of G[N+(x)], a < b: lane a scans N+(v_a) again for the slot
    if (lane < d) {
      unsigned long long dx = (unsigned long long)(g.R[x + 1] - g.R[x]);
      unsigned long long dva = (unsigned long long)(g.R[va + 1] - g.R[va]);
      unsigned long long ra = Bw[lane], k4a = 0, txa = sT[wl][lane];
      for (int64_t q = qa0; q < qa1; ++q) {
        int32_t w = g.C[q];
        int b = find(w);
        if (b < 0) continue;
        unsigned long long cm = ra & Bw[b];
        unsigned long long alpha = (unsigned long long)__popcll(cm), beta = 0, k5 = 0;
        for (int t = 0; t < DW; ++t) beta += (unsigned long long)__popcll(sD[wl][lane][t] & sD[wl][b][t]);
        // 5-cliques at the three lowest vertices x, v_a, v_b: every c in the
        // common neighbourhood above b, then every l adjacent to a, b, c above c
        unsigned long long cm2 = with_k5 ? cm & (~0ull << (b + 1)) : 0ull;
        la.v[5] += ch2((unsigned long long)__popcll(cm2));        // directed bipyramids on this triangle
        while (cm2) {
          int c = __ffsll((long long)cm2) - 1;
          cm2 &= cm2 - 1;
          k5 += (unsigned long long)__popcll(cm & Bw[c] & (~0ull << (c + 1)));
        }
        unsigned long long dvb = (unsigned long long)(g.R[w + 1] - g.R[w]);
        unsigned long long tab = T[q], txb = sT[wl][b];
        if (k4_here) {
          la.v[0] += alpha;                                       // 3 x K4
          la.v[1] += ch2(alpha + beta);                           // N20
        }
        la.v[2] += (u128)(tab - 1) * (dx - 2) + (u128)(txb - 1) * (dva - 2) + (u128)(txa - 1) * (dvb - 2);   // N10
        la.v[3] += (u128)(txa - 1) * (txb - 1) + (u128)(txa - 1) * (tab - 1) + (u128)(txb - 1) * (tab - 1);  // N16
        la.v[4] += k5;                                            // N21
        if (alpha && k4_here) {
          atomicAdd(&K4e[q], alpha);
          atomicAdd(&K[b], alpha);
          k4a += alpha;
        }
      }
      if (k4a) atomicAdd(&K[lane], k4a);
    }
    __syncwarp();
    if (lane < d && K[lane]) atomicAdd(&K4e[o + lane], K[lane] / 2);
    warp_item_flush(la, ids, acc, x);
    __syncwarp();
  }
  final_flush(la, ids, acc, sh);
}

// Counters of the 4-cycle, pair and 5-cycle sweeps, tagged with the item they count
// for.  Before each increment a fire-and-forget atomicMax with the current tag
// turns an entry left by an earlier item into a zero count of the current one
// (a CTA's tags grow with the items it takes), so nothing is cleared between
// items and no list of touched entries is kept.  Every count at j (w(i,j),
// W(i,j) or w'(i,j)) is at most d(j), so the ranks below jbig, the first of degree
// >= 2^16, keep (tag << 16) | count in 32-bit words; the few ranks from jbig on
// keep (tag << 32) | count in a 64-bit side array.
struct TagScratch {
  uint32_t* w;              // per CTA: jbig words
  unsigned long long* wb;   // per CTA: n - jbig words
  int64_t jbig, n;
};

template <bool BIG>   // BIG: some rank has degree >= 2^16 (jbig < n)
struct TaggedCounters {
  static constexpr uint32_t TAG_MAX = 0xffffu;   // largest tag of the 32-bit words
  uint32_t* w;
  unsigned long long* wb;
  int32_t jbig;
  uint32_t tag;
  __device__ TaggedCounters(const TagScratch& ts) : TaggedCounters(ts, blockIdx.x) {}
  // the array of index `arr` (one per CTA, or one per cluster of CTAs)
  __device__ TaggedCounters(const TagScratch& ts, int64_t arr) {
    w = ts.w + arr * ts.jbig;
    wb = ts.wb + arr * (ts.n - ts.jbig);
    jbig = (int32_t)ts.jbig;
    tag = 0;
  }
  __device__ __forceinline__ uint32_t inc(int32_t j) const {
    if (!BIG || j < jbig) {
      atomicMax(&w[j], tag << 16);
      return atomicAdd(&w[j], 1u) & 0xffffu;
    }
    unsigned long long* p = &wb[j - jbig];
    atomicMax(p, (unsigned long long)tag << 32);
    return (uint32_t)atomicAdd(p, 1ull);
  }
  __device__ __forceinline__ void add(int32_t j) const {    // the same without the old value
    if (!BIG || j < jbig) {
      atomicMax(&w[j], tag << 16);
      atomicAdd(&w[j], 1u);
    } else {
      unsigned long long* p = &wb[j - jbig];
      atomicMax(p, (unsigned long long)tag << 32);
      atomicAdd(p, 1ull);
    }
  }
  __device__ __forceinline__ uint32_t get(int32_t j) const {
    if (!BIG || j < jbig) {
      uint32_t v = w[j];
      return (v >> 16) == tag ? (v & 0xffffu) : 0u;
    }
    unsigned long long v = wb[j - jbig];
    return (uint32_t)(v >> 32) == tag ? (uint32_t)v : 0u;
  }
  // get() for an array that CTAs of other SMs increment: read at L2 (the
  // increments are performed there; an L1 copy could be stale)
  __device__ __forceinline__ uint32_t get_l2(int32_t j) const {
    if (!BIG || j < jbig) {
      uint32_t v = __ldcg(&w[j]);
      return (v >> 16) == tag ? (v & 0xffffu) : 0u;
    }
    unsigned long long v = __ldcg(&wb[j - jbig]);
    return (uint32_t)(v >> 32) == tag ? (uint32_t)v : 0u;
  }
  // next item: a new tag, or zeroed counters once the tags are used up (all
  // threads of the CTA call it; returns true when it zeroed, and a barrier
  // must then publish the zeros before the next increment)
  __device__ __forceinline__ bool next(int64_t n) { return next_shared(n, 0, 1); }
  // the same for an array shared by the `parts` CTAs of a cluster: CTA
  // `part` zeroes its share, and a cluster barrier must follow a zeroing
  __device__ __forceinline__ bool next_shared(int64_t n, unsigned part, unsigned parts) {
    if (++tag <= TAG_MAX) return false;
    const int64_t t0 = (int64_t)part * blockDim.x + threadIdx.x, st = (int64_t)parts * blockDim.x;
    for (int64_t t = t0; t < jbig; t += st) w[t] = 0;
    if (BIG)
      for (int64_t t = t0; t < n - jbig; t += st) wb[t] = 0;
    tag = 1;
    return true;
  }
};

// ---------------------------------------------------------------- clusters
// Thread-block cluster helpers (PTX special registers and the hardware
// cluster barrier).  A kernel launched without a cluster dimension runs as
// clusters of one CTA, for which these reduce to the CTA itself.
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_index() {
  unsigned r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
// every thread of every CTA of the cluster; orders memory at cluster scope
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// 64-bit value at the address of `p` in the shared memory of cluster CTA `rank`
__device__ __forceinline__ long long ld_cluster_s64(const void* p, unsigned rank) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
  long long v;
  asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(v) : "r"(ra) : "memory");
  return v;
}

// ============================================================================
// Thm 5: 4-cycles.  For the highest vertex i and each j < i,
// w(i,j) = |{k in N(i) cap N(j) : k < i}| (out-wedges and in-out wedges);
// C4 = sum C(w,2), the sum of the values the increments return.  Per edge: every
// wedge i - k - j adds w-1 to edges (i,k) and (k,j); C4(v) is half the sum over
// the edges of v (a 4-cycle has two edges at each of its vertices), so no
// counter per vertex is touched.  Light and medium items count in a hash table
// (k_cycles4_hash), heavy ones in windows (k_cycles4_win) or, in a union of
// graphs, in tagged counters (k_cycles4_tag).
// ============================================================================
#ifndef ESC_SWEEP_ILP
#define ESC_SWEEP_ILP 8
#endif
static constexpr int SWEEP_ILP = ESC_SWEEP_ILP;   // independent accesses in flight per lane (4- and 5-cycles)
// Independent accesses in flight per lane of the pair sweep (8 at 64 registers: R-MAT 22 pairs 14.4 -> 13.8 s).
#ifndef ESC_PAIR_ILP
#define ESC_PAIR_ILP 8
#endif
static constexpr int PAIR_ILP = ESC_PAIR_ILP;
static_assert(PAIR_ILP >= 1 && PAIR_ILP <= 8, "pair_range sums at most 8 values of C(old, 2) in 64 bits");

struct SweepScratch {
  uint32_t* cnt2;      // per CTA: n counters of P2 (kept zero between items)
  int32_t* touched2;   // per CTA: n entries
  int64_t n;
};

// Per-edge common-neighbour lists (built by the triangle-list pass).
struct TriLists {
  const int64_t* off;    // per slot: start of the edge's id list (both slots of an edge share it)
  const int32_t* U;      // sorted common-neighbour ids
  const int64_t* offp;   // per slot: start of the slot's position list
  const int32_t* P;      // per slot (u -> v): positions in row u of the common neighbours, ascending
  const uint4* rec;      // per slot: the list the diamond pass reads (see k_list_records)
  const int32_t* UL;     // id lists of the slots to core vertices, entries below the core only
};
// What the diamond pass wants of a slot (x -> y), y above x, in one 16-byte
// record: it comes to the slots in no order, and the start, the length, the core
// length and the neighbour in arrays of their own are a sector each.
//   x, y: start of the list; z: its length; w: 1 for a slot to a core vertex
// From a list of an edge to a core vertex only the entries below the core are
// read (core.cu counts the other tips), so these are packed again, end to end: a
// fraction of the lists, and the pass is bound by their scattered sectors.
// R-MAT 19 census 417 -> 412 ms with the records, 400 -> 383 with the packed lists
// (R-MAT 16 24.8 -> 24.0, Chung-Lu 2.1 41.0 -> 39.9).
__global__ void k_low_counts(DevGraph g, const uint32_t* low, int64_t h0, int64_t* cnt) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < g.n; v += nwarps) {
    const int64_t o = g.op[v];
    for (int64_t p = g.R[v] + lane; p < g.R[v + 1]; p += 32) cnt[p] = p >= o && g.C[p] >= h0 ? (int64_t)low[p] : 0;
  }
}
__global__ void k_low_lists(int64_t nnz, const int64_t* off, const int32_t* U, const int64_t* off_l, int32_t* UL) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t pb = warp * 32; pb < nnz; pb += nwarps * 32) {
    const int64_t p = pb + lane;
    const long long to = p < nnz ? off_l[p] : 0, len = p < nnz ? off_l[p + 1] - to : 0;
    const long long from = len > 0 ? off[p] : 0;
    unsigned m = __ballot_sync(0xffffffffu, len > 0);
    while (m) {
      const int k = __ffs(m) - 1;
      m &= m - 1;
      const int32_t* src = U + __shfl_sync(0xffffffffu, from, k);
      int32_t* dst = UL + __shfl_sync(0xffffffffu, to, k);
      const long long cnt = __shfl_sync(0xffffffffu, len, k);
      for (long long q = lane; q < cnt; q += 32) dst[q] = src[q];
    }
  }
}
__global__ void k_list_records(DevGraph g, const uint32_t* T, const int64_t* off, const uint32_t* low,
                               const int64_t* off_l, int64_t h0, uint4* rec) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < g.nnz; p += (int64_t)gridDim.x * blockDim.x) {
    const bool core = off_l && g.C[p] >= h0;
    const unsigned long long o = (unsigned long long)(core ? off_l[p] : off[p]);
    rec[p] = make_uint4((uint32_t)o, (uint32_t)(o >> 32), core ? low[p] : T[p], core ? 1u : 0u);
  }
}

// ============================================================================
// Thm 11/12: N13 = sum_{j<i} C(W(i,j), 3) and
// N17 = sum_{j<i} (W(i,j) - 2) cc(i,j), cc = edges inside N(i) cap N(j).
// W(i,.) from every wedge i - c - j (c in N(i), j in N(c), j < i); C(W,3) is
// accumulated on the fly as the sum of C(old, 2) over the increments.  The cc
// term is gathered per diamond: for each triangle {i, x, y} (x < y, y reached
// through the position list of (x, i), so its slot in row x is direct) and each
// j in N(x) cap N(y) below i, add W(i,j) - 2 (Thm 12's enumeration through the
// per-edge triangle lists).
// ============================================================================


// Items of the pair, 4-cycle and 5-cycle sweeps are split by the number w_i of
// their counter increments, which with the size of the graph also bounds the
// distinct counters m_i = min(w_i, n):
//   light:   m_i <= IT_LIGHT_M and w_i <= 4 IT_LIGHT_M: one CTA of 64 threads
//   mid:     m_i <= half of medium's: one CTA of 256 threads
//   medium:  m_i <= IT_MEDIUM_M: one CTA of 512 threads
//   large:   m_i <= IT_LARGE_M, pair items of single graphs that take several
//            windows: one CTA of 1024 threads
//   heavy:   the rest
// Chung-Lu 2.3 n = 625,000 census 90.2 -> 82.5 ms with mid and large beside the
// others: an item waits for its chain of barriers and list reads, so what counts
// is how many are in flight and that their lists are walked once.
// Light and medium items count in a packed shared-memory hash table of 2 m_i
// words or more (a power of two), cleared for the item: small items clear
// little and keep many CTAs on an SM.  An item whose degree does not fit the
// count bits of a packed word is heavy.  What bounded the sweeps before: one
// 512-thread CTA per vertex with counters in global memory, most of whose time
// went to barriers and latency on vertices of a few dozen edges (alone, ms,
// before and after): Chung-Lu 2.3 n = 625,000 5-cycles 34.7 / 17.6, 4-cycles
// 16.7 / 6.2; Chung-Lu 2.1 n = 262,144 9.6 / 6.6 and 6.5 / 2.0; R-MAT 19 70 / 58
// and 56 / 20; 256 graphs of 20 to 200 vertices 1.03 / 0.36 and 0.40 / 0.14.
static constexpr int IT_LIGHT_LOG = 11, IT_MID_LOG = 13, IT_MEDIUM_LOG = 14, IT_LARGE_LOG = 15, IT_MIN_LOG = 7;
static constexpr int IT_LIGHT_THREADS = 64, IT_MID_THREADS = 256, IT_MEDIUM_THREADS = 512, IT_LARGE_THREADS = 1024;
static constexpr long long IT_LARGE_M = 3ll << (IT_LARGE_LOG - 2);
static constexpr long long IT_LIGHT_M = 1ll << (IT_LIGHT_LOG - 1);
static constexpr long long IT_MEDIUM_M = 1ll << (IT_MEDIUM_LOG - 1);
static constexpr long long IT5_MEDIUM_M = IT_MEDIUM_M / 2;   // the 5-cycle sweep has two tables

// A packed item: rank in the low 32 bits, log2 of the table size(s) above.
__host__ __device__ __forceinline__ int64_t item_rank(unsigned long long it) { return (int64_t)(it & 0xffffffffull); }
__host__ __device__ __forceinline__ int item_log(unsigned long long it) { return (int)((it >> 32) & 0xff); }
__host__ __device__ __forceinline__ int item_log2(unsigned long long it) { return (int)((it >> 40) & 0xff); }

// Open addressing in shared memory, key and count in one 32-bit word: key << cb
// | count, all ones = empty.  Half the space and half the accesses of separate
// key and count words.  Every key is below 2^(32 - cb) - 1 and every count
// below 2^cb - 1 (ranks below n, counts at most the item's degree: the host
// and the classification see to it), so no used word is all ones.
struct PackedHash {
  uint32_t* tab;
  int cb, log;
  static constexpr uint32_t EMPTY = 0xffffffffu;
  __device__ __forceinline__ uint32_t slot(int32_t j) const { return ((uint32_t)j * 0x9E3779B1u) >> (32 - log); }
  __device__ __forceinline__ void clear(int tid, int nthreads) const {
    uint4* t4 = reinterpret_cast<uint4*>(tab);
    for (int t = tid; t < (1 << log) / 4; t += nthreads) t4[t] = make_uint4(EMPTY, EMPTY, EMPTY, EMPTY);
  }
  // the count before; full: the table has no room (never: sized by m_i)
  __device__ __forceinline__ uint32_t inc(int32_t j, bool& full) const {
    const uint32_t m = (1u << log) - 1u, cm = (1u << cb) - 1u;
    uint32_t sl = slot(j);
    for (uint32_t probe = 0; probe <= m; ++probe) {
      uint32_t w = *(volatile uint32_t*)&tab[sl];
      if (w == EMPTY) {
        w = atomicCAS(&tab[sl], EMPTY, ((uint32_t)j << cb) | 1u);
        if (w == EMPTY) return 0u;
      }
      if ((w >> cb) == (uint32_t)j) return atomicAdd(&tab[sl], 1u) & cm;
      sl = (sl + 1u) & m;
    }
    full = true;
    return 0u;
  }
  // the count (0 when j was never counted)
  __device__ __forceinline__ uint32_t get(int32_t j) const {
    const uint32_t m = (1u << log) - 1u;
    uint32_t sl = slot(j);
    for (uint32_t probe = 0; probe <= m; ++probe) {
      const uint32_t w = tab[sl];
      if (w == EMPTY) return 0u;
      if ((w >> cb) == (uint32_t)j) return w & ((1u << cb) - 1u);
      sl = (sl + 1u) & m;
    }
    return 0u;
  }
};

// Places within the own graph.  A graph of up to DIRECT_N vertices has a counter
// for each of them in shared memory, and its medium items count without hashing
// (k_*_direct): of a single graph the place is the rank; of a union li gives
// it, and g.J holds the entries' places.
// A probe loop ends with the slowest of 32 lanes, and the 64 KB table left three
// CTAs on an SM.  Census of 96 graphs of 20 to 2,000 vertices 145 -> 107 ms (its
// 5-cycle items took 43 ms), of ER(800, 0.15) 1.39 -> 1.27 ms (5-cycles 0.21 ->
// 0.10).
struct LocalIds {
  const int32_t *li, *hl;                       // place of a rank; ranks by graph (null: one graph)
  const int64_t* hb;                            // first entry in hl of the graph of a rank
  const int32_t* vg;
  const unsigned long long* n_arr;
  int n;
  __device__ __forceinline__ int size(int64_t i) const { return li ? (int)n_arr[vg[i]] : n; }
  __device__ __forceinline__ int32_t place(int64_t j) const { return li ? li[j] : (int32_t)j; }
  __device__ __forceinline__ int64_t start(int64_t i) const { return li ? hb[i] : 0; }
  __device__ __forceinline__ int64_t rank(int64_t start, int32_t t) const { return li ? hl[start + t] : t; }
};
static constexpr int DIRECT_N = 8192;
__global__ void k_local_entries(const int32_t* C, int64_t nnz, const int32_t* li, int32_t* J) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x)
    J[p] = li[C[p]];
}
__device__ __forceinline__ void direct_clear(uint32_t* tab, int ng) {   // the table's size is a multiple of 4 words
  for (int t = threadIdx.x; t < (ng + 3) / 4; t += blockDim.x)
    reinterpret_cast<uint4*>(tab)[t] = make_uint4(0u, 0u, 0u, 0u);
}

// log2 of a table for m counters (load factor at most 1/2)
__device__ __forceinline__ int table_log(unsigned long long m) {
  const int l = m <= 1 ? 1 : 65 - __clzll((long long)(m - 1));   // ceil(log2(2 m))
  return max(l, IT_MIN_LOG);
}

// One sweep's item lists (light, medium, heavy, mid, large; n entries each) and
// counters: cnt[0..2] the first three lists' lengths, cnt[3..5] their queues,
// cnt[6] the largest heavy item, cnt[9..10] the last two's lengths, cnt[11..12]
// their queues.
static constexpr int IT_LISTS = 5, IT_CNT = 13;
struct ItemLists {
  unsigned long long* list;
  unsigned long long* cnt;
};
__device__ __forceinline__ void item_append(const ItemLists& il, int64_t n, int64_t i, unsigned long long w,
                                            unsigned long long m1, unsigned long long m2, long long light_m,
                                            long long medium_m, long long large_m, bool fits, bool direct) {
  const unsigned long long m = max(m1, m2);
  int cls = 2;
  if (!fits) cls = direct && (long long)m <= medium_m ? 1 : 2;   // no count bits in a direct counter
  else if ((long long)m <= light_m && (long long)w <= 4 * light_m) cls = 0;
  else if ((long long)m <= medium_m / 2 && !direct) cls = 3;
  else if ((long long)m <= medium_m) cls = 1;
  else if ((long long)m <= large_m) cls = 4;
  unsigned long long v = (unsigned long long)i;
  if (cls != 2) v |= ((unsigned long long)table_log(m1) << 32) | ((unsigned long long)table_log(m2) << 40);
  il.list[(int64_t)cls * n + (int64_t)atomicAdd(&il.cnt[cls < 3 ? cls : cls + 6], 1ull)] = v;
  if (cls == 2) atomicMax(&il.cnt[6], w);        // for the task buffers
}

// Pair items: w_i = sum_{c in N(i)} |N(c) below i| of every vertex with degree
// >= 2 (roughly by decreasing rank, so the heaviest items come first).
// Also the largest common-neighbour list (triangles on one edge) into cnt[7]
// and twice the number of diamonds, sum over slots of C(T, 2), into cnt[8].
__global__ void k_pair_classify(DevGraph g, const uint32_t* T, ItemLists il, long long light_m, long long medium_m,
                                long long large_m, int cb, const int32_t* vg, const unsigned long long* n_arr,
                                bool direct, Owner own) {
  int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  unsigned long long dia = 0;
  unsigned tmax = 0;
  for (int64_t k = warp; k < g.n; k += nwarps) {
    int64_t i = g.n - 1 - k;
    int64_t b0 = g.R[i], e0 = g.R[i + 1];
    unsigned long long w = 0;
    const bool mine = e0 - b0 >= 2 && own.owns(i);
    for (int64_t p = b0 + lane; p < e0; p += 32) {
      const uint32_t t = T[p];
      tmax = max(tmax, t);
      dia += t < 2 ? 0 : (unsigned long long)t * (t - 1) / 2;
      if (mine) w += (unsigned long long)(g.rev[p] - g.R[g.C[p]]);
    }
    w = warp_sum_u64(w);
    if (lane == 0 && w) {
      const unsigned long long m = min(w, min((unsigned long long)i, vg ? n_arr[vg[i]] : ~0ull));
      item_append(il, g.n, i, w, m, m, light_m, medium_m, large_m, (unsigned long long)(e0 - b0) < (1u << cb) - 1u, direct);
    }
  }
  dia = warp_sum_u64(dia);
  if (lane == 0 && dia) atomicAdd(&il.cnt[8], dia);
  tmax = __reduce_max_sync(0xffffffffu, tmax);
  if (lane == 0 && tmax) atomicMax(&il.cnt[7], (unsigned long long)tmax);
}

// 4-cycle items (w4_i = sum over k in N-(i) of |N(k) below i|) and, unless
// only4, 5-cycle items (the increments of w'(i, .) and of P2(i, .), see
// k_cycles5).
__global__ void k_cycle_classify(DevGraph g, ItemLists i4, ItemLists i5, bool only4, long long light_m,
                                 long long medium_m4, long long medium_m5, int cb, const int32_t* vg,
                                 const unsigned long long* n_arr, bool direct, Owner own) {
  int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t k = warp; k < g.n; k += nwarps) {
    const int64_t i = g.n - 1 - k;
    if (!own.owns(i)) continue;
    const int64_t b0 = g.R[i], o = g.op[i], e0 = g.R[i + 1];
    if (o == b0) continue;                      // no lower neighbour
    unsigned long long w4 = 0, w5 = 0, p2 = 0;
    for (int64_t p = b0 + lane; p < e0; p += 32) {
      const int32_t c = g.C[p];
      const int64_t cr = g.R[c], ce = g.R[c + 1];
      if (p < o) {
        w4 += (unsigned long long)(g.rev[p] - cr);
        w5 += (unsigned long long)(ce - cr);
        p2 += (unsigned long long)(ce - g.op[c]);
      } else {
        if (only4) break;
        w5 += (unsigned long long)(ce - g.op[c]);
      }
    }
    w4 = warp_sum_u64(w4);
    w5 = warp_sum_u64(w5);
    p2 = warp_sum_u64(p2);
    if (lane) continue;
    const unsigned long long ng = vg ? n_arr[vg[i]] : (unsigned long long)g.n;
    const bool fits = (unsigned long long)(e0 - b0) < (1u << cb) - 1u;
    if (w4) {
      const unsigned long long m = min(w4, min((unsigned long long)i, ng));
      item_append(i4, g.n, i, w4, m, m, light_m, medium_m4, 0, fits, direct);
    }
    // P2 counts the slot of i itself once per a: with nothing else, no path leaves it
    if (!only4 && p2 > (unsigned long long)(o - b0))
      item_append(i5, g.n, i, w5 + p2, min(w5, ng), min(p2, ng), light_m, medium_m5, 0, fits, direct);
  }
}

// The two passes of one item i, shared by both forms of the sweep.  Warp
// `gw` of `gnw` (the warps of a CTA, or of a whole cluster) takes its share:
//   inc(j) counts the wedge i - c - j and returns its term of the sum, a
//   function of the count before it (pair_c2 for N13, the count itself for C4);
//   get(j) returns W(i,j) after every increment.
// Pass 1: W(i,.) from every wedge i - c - j (c in N(i), j in N(c), j < i);
// C(W,3) is accumulated on the fly as the sum of C(old, 2).  The lists N(c) are
// fetched 32 per warp (lane k the k-th) and every lane keeps PAIR_ILP
// independent loads and counter operations in flight.
static constexpr int PAIR_TASK = 32 * 4 * 4;   // lists longer than this are shared as tasks of this size
#ifndef ESC_PAIR_SHORT
#define ESC_PAIR_SHORT 32
#endif
static constexpr int PAIR_SHORT = ESC_PAIR_SHORT;   // lists up to this long are walked by one lane (32: Chung-Lu pairs 40.8 -> 40.2 ms against 64)

// A 128-bit sum of 64-bit terms kept as a 64-bit word and a carry count:
// two 64-bit operations per term in the inner loops instead of a 128-bit add.
struct Sum128 {
  unsigned long long lo = 0;
  unsigned hi = 0;
  __device__ __forceinline__ void add(unsigned long long x) {
    lo += x;
    hi += lo < x ? 1u : 0u;
  }
  __device__ __forceinline__ u128 get() const { return ((u128)hi << 64) + lo; }
};

// C(old, 2) of a counter value below 2^32, exactly in 64 bits (zero for 0 and 1).
__device__ __forceinline__ unsigned long long pair_c2(uint32_t old) {
  return ((unsigned long long)old * (old - 1u)) >> 1;           // old = 0: 0 x (2^32 - 1)
}

// Increments for the entries C[cb .. ce) (one warp, PAIR_ILP loads per lane in
// flight).  Offsets within the list are 32-bit: a row has fewer than 2^31 entries.
template <class Inc>
__device__ __forceinline__ u128 pair_range(const DevGraph& g, int64_t cb, int64_t ce, Inc&& inc) {
  const int lane = threadIdx.x & 31;
  const int32_t* L = g.J + cb;
  const int len = (int)(ce - cb);
  Sum128 n13;
  // groups of 32 without a test per entry, then the rest (R-MAT 19 pairs 195 -> 190 ms, 4-cycles 20.0 -> 18.5)
  int q = 0;
  for (; q + 32 * PAIR_ILP <= len; q += 32 * PAIR_ILP) {
    int32_t jj[PAIR_ILP];
#pragma unroll
    for (int u = 0; u < PAIR_ILP; ++u) jj[u] = __ldcs(L + q + lane + 32 * u);
    unsigned long long blk = 0;                 // at most 8 terms below 2^61 (a count is below 2^31)
#pragma unroll
    for (int u = 0; u < PAIR_ILP; ++u) blk += inc(jj[u]);
    n13.add(blk);
  }
#pragma unroll
  for (int gsz = PAIR_ILP / 2; gsz >= 1; gsz >>= 1) {
    if (q + 32 * gsz <= len) {
      int32_t jj[PAIR_ILP / 2];
#pragma unroll
      for (int u = 0; u < gsz; ++u) jj[u] = __ldcs(L + q + lane + 32 * u);
      unsigned long long blk = 0;
#pragma unroll
      for (int u = 0; u < gsz; ++u) blk += inc(jj[u]);
      n13.add(blk);
      q += 32 * gsz;
    }
  }
  if (q + lane < len) n13.add(inc(__ldcs(L + q + lane)));
  return n13.get();
}

// defer(cb, ce) may take a long list off the warp (returning true) so that
// every warp shares it later; it is called by all 32 lanes with the same range.
template <class Inc, class Defer>
__device__ __forceinline__ u128 pair_wedges(const DevGraph& g, int64_t b0, int64_t e0, int64_t gw, int64_t gnw,
                                            Inc&& inc, Defer&& defer) {
  const int lane = threadIdx.x & 31;
  u128 n13 = 0;
  for (int64_t pbase = b0 + gw; pbase < e0; pbase += gnw * 32) {
    int64_t p = pbase + (int64_t)lane * gnw;
    int64_t cb_l = 0, ce_l = 0;
    if (p < e0) {
      int32_t c = g.C[p];
      cb_l = g.R[c];
      ce_l = g.rev[p];                          // N(c) below i ends at the slot of i
    }
    // short lists: each lane its own; the others one at a time by the warp
    if (ce_l - cb_l <= PAIR_SHORT) {
      const int32_t* L = g.J + cb_l;
      const int len = (int)(ce_l - cb_l);
      Sum128 sh13;
      for (int q = 0; q < len; q += 4) {
        int32_t jj[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) jj[u] = q + u < len ? __ldcs(L + q + u) : -1;
        unsigned long long blk = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (jj[u] >= 0) blk += inc(jj[u]);
        sh13.add(blk);
      }
      n13 += sh13.get();
    }
    unsigned longm = __ballot_sync(0xffffffffu, ce_l - cb_l > PAIR_SHORT);
    while (longm) {
      const int k = __ffs(longm) - 1;
      longm &= longm - 1;
      int64_t cb = __shfl_sync(0xffffffffu, cb_l, k), ce = __shfl_sync(0xffffffffu, ce_l, k);
      if (defer(cb, ce)) continue;
      n13 += pair_range(g, cb, ce, inc);
    }
  }
  return n13;
}

// Long lists split into tasks of PAIR_TASK entries, shared by all warps of a
// CTA or cluster: per work group a task array (entry ranges of C) and a count.
struct PairTasks {
  long long* q;             // per group: cap x (begin, end)
  unsigned long long* n;    // per group: number of tasks (zero between items)
  int64_t cap;              // tasks per group
};

// Appends the tasks of list [cb, ce) to group `grp`; false if they do not fit
// (the caller then counts the list itself).  All 32 lanes call it.
__device__ __forceinline__ bool pair_defer(const PairTasks& pt, int64_t grp, int64_t cb, int64_t ce) {
  const int lane = threadIdx.x & 31;
  const long long nt = (ce - cb + PAIR_TASK - 1) / PAIR_TASK;
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(&pt.n[grp], (unsigned long long)nt);
  base = __shfl_sync(0xffffffffu, base, 0);
  if ((long long)base + nt > pt.cap) return false;   // never: sized by the largest item
  long long* q = pt.q + 2 * (grp * pt.cap + (long long)base);
  for (long long t = lane; t < nt; t += 32) {
    long long a = cb + t * PAIR_TASK;
    q[2 * t] = a;
    q[2 * t + 1] = min((long long)ce, a + PAIR_TASK);
  }
  return true;
}

// The tasks of group `grp`, task t taken by warp t mod gnw.
// nt: the group's task count, read after the barrier that ends the appends
template <class Inc>
__device__ __forceinline__ u128 pair_run_tasks(const DevGraph& g, const PairTasks& pt, int64_t grp,
                                               unsigned long long nt, int64_t gw, int64_t gnw, Inc&& inc) {
  nt = min(nt, (unsigned long long)pt.cap);
  const long long* q = pt.q + 2 * grp * pt.cap;
  u128 n13 = 0;
  for (unsigned long long t = (unsigned long long)gw; t < nt; t += (unsigned long long)gnw)
    n13 += pair_range(g, __ldcg(&q[2 * t]), __ldcg(&q[2 * t + 1]), inc);
  return n13;
}

// Pass 2: the cc term per diamond with tip i.  For each x in N(i), the
// triangles {i, x, y} with y above x are a suffix of the position list of
// slot (x -> i); the common-neighbour list of (x, y) is sorted, so the j
// below i are a prefix of it; each adds W(i,j) - 2 (Thm 12's enumeration
// through the per-edge triangle lists).

// The diamonds of up to 32 triangles {i, x, y}, lane k with the k-th (`on`):
// entry r of the position lists is that of y in row x, which starts at xb.
// Short common-neighbour lists are walked by their lane, long ones by the warp.
template <class Get>
__device__ __forceinline__ u128 pair_diamond_chunk(const TriLists& tl3, const CoreView& cv, int64_t i, bool on,
                                                   int64_t xb, int64_t r, Get&& get) {
  const int lane = threadIdx.x & 31;
  const int32_t i32 = (int32_t)i;
  Sum128 n17;
  const int32_t* L_l = tl3.U;
  uint32_t len_l = 0;
  bool cut = false;
  if (on) {
    const uint4 e = __ldg(&tl3.rec[xb + tl3.P[r]]);   // slot (x -> y)
    cut = i >= cv.h0 && e.w != 0;               // every entry is below i
    len_l = e.z;
    L_l = (e.w ? tl3.UL : tl3.U) + (int64_t)(((unsigned long long)e.y << 32) | e.x);
  }
  // short lists: each lane walks its own, a few entries in flight, until it
  // passes i (no entry loaded beyond the next few); long ones: the whole warp
  // on one list at a time.  Each term W(i,j) - 2 is below 2^32; a lane adds at
  // most 2^26 of them per list into 64 bits before the carry-counted sum.
  if (on && len_l <= PAIR_SHORT) {
    const int32_t* L = L_l;
    const int len = (int)len_l;
    unsigned long long part = 0;
    for (int q = 0; q < len; q += 4) {
      int32_t jj[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) jj[u] = q + u < len ? __ldcs(L + q + u) : 0x7fffffff;
      bool past = false;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (jj[u] < i32) part += get(jj[u]) - 2u;
        else past = true;
      }
      if (past) break;
    }
    n17.add(part);
  }
  // long lists: each lane first finds how many entries of its list lie below
  // i (i is in the list: a binary search), then the warp reads exactly those,
  // one list at a time, in blocks of 32 x PAIR_ILP entries and then 4, 2, 1
  // and a last partial group of 32, so that no slot past the prefix is issued.
  const bool lng = on && len_l > PAIR_SHORT;
  int pre_l = lng && cut ? (int)len_l : 0;
  if (lng && !cut) {
    const int32_t* L = L_l;
    int lo = 0, hi = (int)len_l;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (__ldg(L + mid) < i32) lo = mid + 1;
      else hi = mid;
    }
    pre_l = lo;
  }
  unsigned longm = __ballot_sync(0xffffffffu, pre_l > 0);
  while (longm) {
    const int k = __ffs(longm) - 1;
    longm &= longm - 1;
    const int32_t* L = reinterpret_cast<const int32_t*>(
                           __shfl_sync(0xffffffffu, reinterpret_cast<uintptr_t>(L_l), k)) + lane;
    const int pre = __shfl_sync(0xffffffffu, pre_l, k);
    unsigned long long part = 0;             // x, y are common neighbours of i and every j read here
    int sb = 0;
    for (; sb + 32 * PAIR_ILP <= pre; sb += 32 * PAIR_ILP) {
      int32_t jj[PAIR_ILP];
#pragma unroll
      for (int u = 0; u < PAIR_ILP; ++u) jj[u] = __ldcs(L + sb + 32 * u);
#pragma unroll
      for (int u = 0; u < PAIR_ILP; ++u) part += get(jj[u]) - 2u;
    }
#pragma unroll
    for (int gsz = PAIR_ILP / 2; gsz >= 1; gsz >>= 1) {
      if (sb + 32 * gsz <= pre) {
        int32_t jj[PAIR_ILP / 2];
#pragma unroll
        for (int u = 0; u < gsz; ++u) jj[u] = __ldcs(L + sb + 32 * u);
#pragma unroll
        for (int u = 0; u < gsz; ++u) part += get(jj[u]) - 2u;
        sb += 32 * gsz;
      }
    }
    if (sb + lane < pre) part += get(__ldcs(L + sb)) - 2u;
    n17.add(part);
  }
  return n17.get();
}

// The triangles {i, x, y} with y above x of slot p = (i -> x): positions
// [r0, r1) of the position list of slot (x -> i); r0 = r1 if there are none.
__device__ __forceinline__ void pair_tri_range(const DevGraph& g, const TriLists& tl3, const uint32_t* T, int64_t p,
                                               int64_t& xb, int64_t& r0, int64_t& r1) {
  int32_t x = g.C[p];
  xb = g.R[x];
  int32_t xo = (int32_t)(g.op[x] - xb);         // positions >= xo in row x are above x
  int64_t rp_ = g.rev[p];                       // slot (x -> i)
  int64_t yb = tl3.offp[rp_];
  r1 = yb + T[rp_];
  r0 = lower_bound_i32(tl3.P, yb, r1, xo);
}

// 32 neighbours x per warp at once (lane l finds the l-th one's triangles), and
// their triangles as one sequence, 32 per step: most x have fewer than 32.  With
// one x at a time the warp waited for its binary search, then worked with the
// lanes that the x had triangles for (pairs alone: ER(800, 0.15) 0.31 -> 0.17 ms,
// R-MAT 16 10.6 -> 9.7, Chung-Lu 2.1 20.1 -> 19.8).
template <class Get>
__device__ __forceinline__ u128 pair_diamonds(const DevGraph& g, const TriLists& tl3, const uint32_t* T,
                                              const CoreView& cv, int64_t i, int64_t b0, int64_t e0, int64_t gw,
                                              int64_t gnw, Get&& get) {
  u128 n17 = 0;
  if (cv.h0 <= 0) return n17;                   // every vertex is in the core
  const int lane = threadIdx.x & 31;
  for (int64_t pbase = b0 + gw; pbase < e0; pbase += gnw * 32) {
    const int64_t p = pbase + (int64_t)lane * gnw;
    int64_t xb_l = 0, r0 = 0, r1 = 0;
    if (p < e0 && T[p] != 0) pair_tri_range(g, tl3, T, p, xb_l, r0, r1);
    long long end = r1 - r0;                    // triangles of lanes 0 .. lane
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += y;
    }
    const long long total = __shfl_sync(0xffffffffu, end, 31), at = r1 - end;   // triangle t of lane l: entry at + t
    for (long long t0 = 0; t0 < total; t0 += 32) {
      const long long t = t0 + lane;
      int o = 0;                                // lanes whose triangles end at or before t
#pragma unroll
      for (int h = 16; h >= 1; h >>= 1)
        if (__shfl_sync(0xffffffffu, end, o + h - 1) <= t) o += h;
      const long long base = __shfl_sync(0xffffffffu, at, o), xb = __shfl_sync(0xffffffffu, (long long)xb_l, o);
      n17 += pair_diamond_chunk(tl3, cv, i, t < total, xb, base + t, get);
    }
  }
  return n17;
}

// W(i, j) of a core item for the core vertices j below it in the same graph
// (thread tid of nthreads).  Entries whose W is zero may hold anything: no
// diamond reads them.
template <class Get>
__device__ __forceinline__ void core_store_row(const CoreView& cv, int64_t i, int64_t tid, int64_t nthreads, Get&& get) {
  if (i < cv.h0) return;
  const int64_t t = i - cv.h0, row = cv.rowb[t];
  const int32_t cnt = cv.li[t];
  const int32_t* hl = cv.hl ? cv.hl + cv.hb[t] : nullptr;
  for (int64_t k = tid; k < cnt; k += nthreads) cv.put(row + k, get(hl ? hl[k] : (int32_t)(cv.h0 + k)));
}

// Light and medium items: one CTA of THREADS threads per item, W(i, .) in a
// packed hash table.  An item of a few neighbours often has one hub among them
// whose list is nearly all of its wedges: lists longer than PH_PIECE are put
// aside and shared by all warps in pieces of that length (with one warp per
// list, 87% of the warps' time went to waiting for it: Chung-Lu 2.3
// n = 625,000, medium items 31.4 -> 8.9 ms; the census 117 -> 95.5 ms).
static constexpr int PH_PIECE = 128, PH_LONG = 64;
struct LongLists {
  longlong2 list[PH_LONG];
  unsigned n;                                   // zero before the barrier that precedes the item's wedges
};
template <class Inc>
__device__ __forceinline__ u128 pair_wedges_shared(const DevGraph& g, int64_t b0, int64_t e0, int wid, int nw,
                                                   LongLists& ll, Inc&& inc) {
  const int lane = threadIdx.x & 31;
  u128 sum = pair_wedges(g, b0, e0, wid, nw, inc, [&](int64_t cb, int64_t ce) {
    if (ce - cb <= PH_PIECE) return false;
    unsigned at = 0;
    if (lane == 0) at = atomicAdd(&ll.n, 1u);
    at = __shfl_sync(0xffffffffu, at, 0);
    if (at >= PH_LONG) return false;            // no room: the warp walks the list itself
    if (lane == 0) ll.list[at] = make_longlong2(cb, ce);
    return true;
  });
  __syncthreads();
  // the long lists in pieces of PH_PIECE entries, piece by piece over the warps
  const int nl = (int)min(ll.n, (unsigned)PH_LONG);
  for (int l = 0, w = wid; l < nl; ++l) {
    const longlong2 r = ll.list[l];
    const int np = (int)((r.y - r.x + PH_PIECE - 1) / PH_PIECE);
    for (; w < np; w += nw) {
      const int64_t a = r.x + (int64_t)w * PH_PIECE;
      sum += pair_range(g, a, min((int64_t)r.y, a + PH_PIECE), inc);
    }
    w -= np;
  }
  return sum;
}
template <int THREADS>
__global__ void __launch_bounds__(THREADS) k_pairs_hash(DevGraph g, const unsigned long long* items, int64_t nitems,
                                                       unsigned long long* qctr, int cb, int max_log, TriLists tl3,
                                                       const uint32_t* T, CoreView cv, AccSet acc, unsigned* status) {
  extern __shared__ uint4 hash_smem[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  __shared__ LongLists ll;
  const int wid = threadIdx.x >> 5, nw = THREADS / 32;
  PackedHash H{reinterpret_cast<uint32_t*>(hash_smem), cb, 0};
  const int ids[2] = {ACC_N13, ACC_N17};
  LocalAcc<2> la;
  la.zero();
  while (true) {
    int64_t it = next_item(qctr, nitems, &sh_item);     // its barriers end the last item's reads
    if (it < 0) break;
    const int64_t i = item_rank(items[it]);
    const int64_t b0 = g.R[i], e0 = g.R[i + 1];
    H.log = min(max_log, item_log(items[it]));
    H.clear(threadIdx.x, THREADS);
    if (threadIdx.x == 0) ll.n = 0;
    __syncthreads();
    bool full = false;
    auto inc = [&](int32_t j) -> unsigned long long { return pair_c2(H.inc(j, full)); };
    la.v[0] += pair_wedges_shared(g, b0, e0, wid, nw, ll, inc);
    if (full) set_err(status, DEVERR_SCRATCH);
    __syncthreads();
    la.v[1] += pair_diamonds(g, tl3, T, cv, i, b0, e0, wid, nw, [&](int32_t j) -> uint32_t { return H.get(j); });
    if (i >= cv.h0)
      for (int t = threadIdx.x; t < (1 << H.log); t += THREADS) {
        const uint32_t w = H.tab[t];
        const int64_t j = (int64_t)(w >> cb);
        if (w != PackedHash::EMPTY && j >= cv.h0)
          cv.put(cv.rowb[i - cv.h0] + cv.li[j - cv.h0], w & ((1u << cb) - 1u));
      }
    block_item_flush(la, ids, acc, i, sh);
  }
  final_flush(la, ids, acc, sh);
}

// Medium items of small graphs: a counter per vertex of the graph.
__global__ void __launch_bounds__(IT_MEDIUM_THREADS) k_pairs_direct(DevGraph g, const unsigned long long* items,
                                                                   int64_t nitems, unsigned long long* qctr,
                                                                   LocalIds lc, TriLists tl3, const uint32_t* T,
                                                                   CoreView cv, AccSet acc) {
  extern __shared__ uint4 hash_smem[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  __shared__ LongLists ll;
  uint32_t* tab = reinterpret_cast<uint32_t*>(hash_smem);
  const int wid = threadIdx.x >> 5, nw = IT_MEDIUM_THREADS / 32;
  const int ids[2] = {ACC_N13, ACC_N17};
  LocalAcc<2> la;
  la.zero();
  while (true) {
    const int64_t it = next_item(qctr, nitems, &sh_item);   // its barriers end the last item's reads
    if (it < 0) break;
    const int64_t i = item_rank(items[it]);
    const int64_t b0 = g.R[i], e0 = g.R[i + 1];
    const int ng = lc.size(i);
    direct_clear(tab, ng);
    if (threadIdx.x == 0) ll.n = 0;
    __syncthreads();
    la.v[0] += pair_wedges_shared(g, b0, e0, wid, nw, ll, [&](int32_t j) { return pair_c2(atomicAdd(&tab[j], 1u)); });
    __syncthreads();
    la.v[1] += pair_diamonds(g, tl3, T, cv, i, b0, e0, wid, nw, [&](int32_t j) -> uint32_t { return tab[lc.place(j)]; });
    if (i >= cv.h0) {
      const int64_t s0 = lc.start(i);
      for (int t = threadIdx.x; t < ng; t += IT_MEDIUM_THREADS) {
        const uint32_t w = tab[t];
        if (!w) continue;
        const int64_t j = lc.rank(s0, t);
        if (j >= cv.h0) cv.put(cv.rowb[i - cv.h0] + cv.li[j - cv.h0], w);
      }
    }
    block_item_flush(la, ids, acc, i, sh);
  }
  final_flush(la, ids, acc, sh);
}

// Heavy items: all CTAs of a cluster work on one item at a time, with one
// tagged counter array per cluster (index %clusterid.x).  CTA 0 of the
// cluster takes the next item from the queue and the others read it from its
// shared memory; two cluster barriers per item order the increments before
// the reads and the reads before the next item's increments.
// Lists longer than PAIR_TASK entries are cut into tasks that every warp of
// the cluster shares after a barrier, so one hub's list does not hold the
// cluster back.
//
// With clusters of one CTA, the counters of the ranks [wlo, jbig) -- the top
// ranks below the 64-bit side array, where nearly all the diamond reads and a
// good share of the increments land (measured: the top 16K ranks take 94% of
// the diamond reads on the Chung-Lu workload, the top 64K 98% on R-MAT scale
// 20) -- live in shared memory as 16-bit counts, two to a word, cleared for
// every item (a count there is at most the rank's degree, below 2^16).
template <bool BIG, int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) k_pairs_grp(DevGraph g, const unsigned long long* items,
                                                                         int64_t nitems, unsigned long long* qctr,
                                                                         TagScratch ts, TriLists tl3,
                                                                         const uint32_t* T, CoreView cv, AccSet acc,
                                                                         PairTasks pt, int64_t wlo, int win_words) {
  extern __shared__ uint32_t win[];
  __shared__ u128 sh[32];
  __shared__ long long sh_item;
  const unsigned crank = cluster_rank(), csize = cluster_size();
  const int64_t grp = (int64_t)cluster_index();
  TaggedCounters<BIG> w(ts, grp);
  const int wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t gw = (int64_t)crank * nw + wid, gnw = (int64_t)csize * nw;
  const int ids[2] = {ACC_N13, ACC_N17};
  const int64_t whi = win_words > 0 ? min(ts.jbig, wlo + 2 * (int64_t)win_words) : wlo;   // window [wlo, whi)
  LocalAcc<2> la;
  la.zero();
  while (true) {
    if (crank == 0 && threadIdx.x == 0) {
      sh_item = (long long)atomicAdd(qctr, 1ull);
      pt.n[grp] = 0;                           // every CTA is past the last item's tasks
    }
    cluster_barrier();                         // also: the last item's reads are done
    const long long it = ld_cluster_s64(&sh_item, 0);
    if (it >= nitems) break;
    const int64_t i = item_rank(items[it]);
    const int64_t b0 = g.R[i], e0 = g.R[i + 1];
    if (w.next_shared(ts.n, crank, csize)) cluster_barrier();
    if (win_words > 0) {
      for (int t = threadIdx.x; t < win_words; t += blockDim.x) win[t] = 0u;
      cluster_barrier();
    }
    auto inc = [&](int32_t j) -> unsigned long long {
      if (j >= wlo && j < whi) {
        const int64_t k = j - wlo;
        const unsigned sh16 = 16u * (unsigned)(k & 1);
        return pair_c2((atomicAdd(&win[k >> 1], 1u << sh16) >> sh16) & 0xffffu);
      }
      return pair_c2(w.inc(j));
    };
    u128 n13 = pair_wedges(g, b0, e0, gw, gnw, inc, [&](int64_t cb, int64_t ce) {
      return ce - cb > PAIR_TASK && pair_defer(pt, grp, cb, ce);
    });
    cluster_barrier();
    // the task count is read before the next barrier, after which CTA 0 may
    // clear it for the next item
    const unsigned long long nt1 = __ldcg(&pt.n[grp]);
    n13 += pair_run_tasks(g, pt, grp, nt1, gw, gnw, inc);
    cluster_barrier();
    auto get = [&](int32_t j) -> uint32_t {
      if (j >= wlo && j < whi) {
        const int64_t k = j - wlo;
        return (win[k >> 1] >> (16u * (unsigned)(k & 1))) & 0xffffu;
      }
      return w.get_l2(j);
    };
    u128 n17 = pair_diamonds(g, tl3, T, cv, i, b0, e0, gw, gnw, get);
    core_store_row(cv, i, (int64_t)crank * blockDim.x + threadIdx.x, (int64_t)csize * blockDim.x, get);
    la.v[0] += n13;
    la.v[1] += n17;
    block_item_flush(la, ids, acc, i, sh);
  }
  cluster_barrier();                           // CTA 0's shared memory stays until every CTA has read it
  final_flush(la, ids, acc, sh);
}

// ---------------------------------------------------------------- windowed heavy items
// Heavy items, default form: one 1024-thread CTA per SM and item.  The ranks
// below jbig are cut into windows of S = 2 * win_words ranks on a grid
// anchored at jbig (window k = [jbig - (k+1) S, jbig - k S)).  An item i
// counts its wedges window by window, from the lowest window that can hold a
// neighbour of a neighbour up to the one holding rank min(i, jbig) - 1, every
// increment a 16-bit shared-memory atomic.  For every c in N(i) a cursor marks
// how far N(c) has been walked; a window takes the entries below its upper
// end.  A finished window below the top one is written whole to the CTA's
// dense 16-bit array; the top window stays in shared memory.  Ranks from jbig
// on (degree >= 2^16, so counts may need more than 16 bits) go to tagged
// 64-bit counters.  The diamond pass then reads W(i,j) from shared memory
// (the top window, where most diamond tips lie), the dense array or the 64-bit
// counters.
// A count below jbig is at most d_j < 2^16.  The dense array needs no clearing:
// a window is written whole, and the diamond pass reads only windows this item
// wrote (a diamond tip j shares two neighbours with i, so W(i,j) >= 2 and its
// window took increments).
struct PairWin {
  uint32_t* g16;              // per CTA: rank j at bits 16 ((j + par) & 1) of word ((j + par) >> 1) + woff
  int64_t g16_words;          // a multiple of 4, >= (n + 2) / 2 + 4
  int woff;                   // 0..3: puts the first word of every window on a 16-byte boundary
  longlong2* curs;            // per CTA: (cursor, end) of the list N(c) of every c in N(i)
  int64_t curs_cap;           // >= the largest degree
  unsigned long long* side;   // per CTA: n - jbig counters (tag << 32) | count
  int64_t jbig, n, n0;        // n0: the first rank of degree >= 1
  int win_words;              // a multiple of 4
};

// First position q in [a, b) with C[q] >= key (C ascending there), or b; one
// warp, 32 probes per round.
__device__ __forceinline__ int64_t warp_lower_bound(const int32_t* C, int64_t a, int64_t b, int32_t key) {
  const int lane = threadIdx.x & 31;
  // C[q] < key for q < a, C[q] >= key for q >= b
  while (b - a > 32) {
    const int64_t step = (b - a + 31) / 32;
    const int64_t q = a + (int64_t)lane * step;
    const unsigned m = __ballot_sync(0xffffffffu, q >= b || C[q] >= key);
    if (m == 0) {
      a += 31 * step + 1;
    } else {
      const int f = __ffs(m) - 1;
      b = min(b, a + (int64_t)f * step);
      if (f > 0) a += (int64_t)(f - 1) * step + 1;
    }
  }
  const int64_t q = a + lane;
  const unsigned m = __ballot_sync(0xffffffffu, q >= b || C[q] >= key);
  return m ? min(b, a + (int64_t)(__ffs(m) - 1)) : b;
}

// Pass 1 of one window: for every c in N(i) (this warp's share), the entries
// of N(c) from its cursor that lie below `hi` (all remaining ones when `last`).
// `first`: the cursors start at the heads of the lists; unless `last`, the new
// cursors are stored.
template <class Inc, class Defer>
__device__ __forceinline__ u128 pair_wedges_win(const DevGraph& g, longlong2* curs, int64_t b0, int64_t e0,
                                                int64_t gw, int64_t gnw, bool first, bool last, int32_t hi,
                                                Inc&& inc, Defer&& defer) {
  const int lane = threadIdx.x & 31;
  u128 n13 = 0;
  for (int64_t pbase = b0 + gw; pbase < e0; pbase += gnw * 32) {
    const int64_t p = pbase + (int64_t)lane * gnw;
    int64_t cb_l = 0, ce_l = 0;
    if (p < e0) {
      if (first) {
        cb_l = g.R[g.C[p]];
        ce_l = g.rev[p];                        // N(c) below i ends at the slot of i
      } else {
        const longlong2 cu = curs[p - b0];
        cb_l = cu.x;
        ce_l = cu.y;
      }
    }
    int64_t cn_l = ce_l;                        // the lane's new cursor
    if (ce_l - cb_l <= PAIR_SHORT) {            // short: each lane walks its own list up to hi
      const int32_t* L = g.J + cb_l;
      const int len = (int)(ce_l - cb_l);
      Sum128 sh13;
      int q = 0;
      while (q < len) {
        int32_t jj[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) jj[u] = q + u < len ? __ldcs(L + q + u) : 0x7fffffff;
        int stop = 4;
#pragma unroll
        for (int u = 3; u >= 0; --u)
          if (jj[u] >= hi) stop = u;            // ascending: the first entry at or above hi
        unsigned long long blk = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (u < stop) blk += inc(jj[u]);
        sh13.add(blk);
        if (stop < 4) {
          q += stop;
          break;
        }
        q += 4;
      }
      n13 += sh13.get();
      cn_l = cb_l + min(q, len);
    }
    unsigned longm = __ballot_sync(0xffffffffu, ce_l - cb_l > PAIR_SHORT);
    while (longm) {                             // long: the warp takes them one at a time
      const int k = __ffs(longm) - 1;
      longm &= longm - 1;
      const int64_t cb = __shfl_sync(0xffffffffu, cb_l, k), ce = __shfl_sync(0xffffffffu, ce_l, k);
      const int64_t qe = last ? ce : warp_lower_bound(g.C, cb, ce, hi);
      if (lane == k) cn_l = qe;
      if (qe - cb > PAIR_TASK && defer(cb, qe)) continue;
      n13 += pair_range(g, cb, qe, inc);
    }
    if (!last && p < e0) curs[p - b0] = make_longlong2(cn_l, ce_l);
  }
  return n13;
}

// The windows of one item: every wedge i - c - j with c in C[b0 .. e0) is
// counted; term(old) is summed.  get(j) of the result reads the counts.
template <bool BIG>
struct WinItem {
  const PairWin& pw;
  uint32_t* win;
  uint32_t* g16;
  longlong2* curs;
  unsigned long long* side;
  uint32_t tag = 0;
  int64_t S, par, ktop = 0;
  bool top_touched = false;
  __device__ WinItem(const PairWin& p, uint32_t* w) : pw(p), win(w) {
    const int64_t grp = blockIdx.x;
    S = 2 * (int64_t)pw.win_words;
    par = pw.jbig & 1;
    g16 = pw.g16 + grp * pw.g16_words + pw.woff;
    curs = pw.curs + grp * pw.curs_cap;
    side = pw.side + grp * (pw.n - pw.jbig);
  }
  __device__ __forceinline__ void clear_window() {
    uint4* const win4 = reinterpret_cast<uint4*>(win);
    for (int t = threadIdx.x; t < (pw.win_words >> 2); t += blockDim.x) win4[t] = make_uint4(0u, 0u, 0u, 0u);
  }
  template <class Term>
  __device__ __forceinline__ u128 count(const DevGraph& g, const PairTasks& pt, int64_t i, int64_t b0, int64_t e0,
                                        int* sh_flag, Term&& term) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t grp = blockIdx.x;
    uint4* const win4 = reinterpret_cast<uint4*>(win);
    const int nv = pw.win_words >> 2;
    if (BIG && ++tag == 0xffffffffu) {          // tags used up: zero the 64-bit counters
      for (int64_t t = threadIdx.x; t < pw.n - pw.jbig; t += blockDim.x) side[t] = 0ull;
      tag = 1;
      __syncthreads();
    }
    const int64_t top = min(i, pw.jbig);        // ranks [0, top) are counted in windows
    ktop = (pw.jbig - top) / S;                 // the window of rank top - 1
    const int64_t kbot = max(ktop, (pw.jbig - 1 - pw.n0) / S);   // the window of rank n0
    u128 sum = 0;
    top_touched = false;
    for (int64_t k = kbot; k >= ktop; --k) {
      const int64_t lo = pw.jbig - (k + 1) * S;
      const uint32_t lo32 = (uint32_t)lo;       // -S <= lo < 2^31: 32-bit differences below
      const bool last = k == ktop;
      const int32_t hi = last ? 0x7fffffff : (int32_t)(pw.jbig - k * S);
      bool tch = false;
      auto inc = [&](int32_t j) -> unsigned long long {
        tch = true;
        if (BIG && j >= pw.jbig) {
          unsigned long long* q = &side[j - pw.jbig];
          atomicMax(q, (unsigned long long)tag << 32);
          return term((uint32_t)atomicAdd(q, 1ull));
        }
        const uint32_t q = (uint32_t)j - lo32;  // in [0, S)
        const unsigned s16 = (q & 1u) << 4;
        return term((atomicAdd(&win[q >> 1], 1u << s16) >> s16) & 0xffffu);
      };
      sum += pair_wedges_win(g, curs, b0, e0, wid, nw, k == kbot, last, hi, inc,
                             [&](int64_t cb, int64_t ce) { return pair_defer(pt, grp, cb, ce); });
      __syncthreads();                          // the window's long lists are appended as tasks
      const unsigned long long nt = __ldcg(&pt.n[grp]);
      sum += pair_run_tasks(g, pt, grp, nt, wid, nw, inc);
      if (__any_sync(0xffffffffu, tch) && lane == 0) sh_flag[k & 1] = 1;
      __syncthreads();                          // the window's counts are complete; every thread has read nt
      const bool touched = sh_flag[k & 1] != 0;
      if (threadIdx.x == 0) {
        pt.n[grp] = 0;                          // the next window appends after a later barrier
        sh_flag[(k - 1) & 1] = 0;               // the next window's flag (last read before the first barrier above)
      }
      if (last) {
        top_touched = touched;
      } else {
        if (touched) {                          // write the window whole and clear it, 4 words at a time
          const int64_t w0 = (lo + par) >> 1;   // lo + par is even; w0 + woff is a multiple of 4
          uint4* g4 = reinterpret_cast<uint4*>(g16 + w0);
          for (int t = threadIdx.x; t < nv; t += blockDim.x) {
            const uint4 v = win4[t];
            if (pw.woff + w0 + 4 * t >= 0) g4[t] = v;   // the lowest window may start below rank 0
            win4[t] = make_uint4(0u, 0u, 0u, 0u);
          }
        }
        __syncthreads();
      }
    }
    return sum;
  }
  __device__ __forceinline__ uint32_t get(int32_t j) const {
    // j < min(i, jbig) lies in the top window exactly when j - lo_top (mod 2^32) is below S
    const uint32_t q = (uint32_t)j - (uint32_t)(pw.jbig - (ktop + 1) * S);
    if (q < (uint32_t)S) return (win[q >> 1] >> ((q & 1u) << 4)) & 0xffffu;
    if (BIG && j >= pw.jbig) {
      const unsigned long long v = __ldcg(&side[j - pw.jbig]);
      return (uint32_t)(v >> 32) == tag ? (uint32_t)v : 0u;
    }
    const uint32_t t = (uint32_t)j + (uint32_t)par;
    return (__ldcg(&g16[t >> 1]) >> ((t & 1u) << 4)) & 0xffffu;
  }
  // after the last get (a barrier between)
  __device__ __forceinline__ void done(int* sh_flag) {
    if (top_touched) clear_window();
    if (threadIdx.x == 0) sh_flag[0] = sh_flag[1] = 0;
  }
};

template <bool BIG>
__global__ void __launch_bounds__(1024, 1) k_pairs_win(DevGraph g, const unsigned long long* items, int64_t nitems,
                                                        unsigned long long* qctr, PairWin pw, TriLists tl3,
                                                        const uint32_t* T, CoreView cv, AccSet acc, PairTasks pt,
                                                        unsigned* status) {
  extern __shared__ uint32_t win[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  __shared__ int sh_flag[2];                   // a window took increments (windows alternate)
  const int wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  WinItem<BIG> wi(pw, win);
  const int ids[2] = {ACC_N13, ACC_N17};
  LocalAcc<2> la;
  la.zero();
  wi.clear_window();
  if (threadIdx.x == 0) sh_flag[0] = sh_flag[1] = 0;
  while (true) {
    const int64_t it = next_item(qctr, nitems, &sh_item);   // its barriers publish the cleared window
    if (it < 0) break;
    const int64_t i = item_rank(items[it]);
    const int64_t b0 = g.R[i], e0 = g.R[i + 1];
    if (e0 - b0 > pw.curs_cap) {                // never: sized by the largest degree
      if (threadIdx.x == 0) set_err(status, DEVERR_SCRATCH);
      continue;
    }
    la.v[0] += wi.count(g, pt, i, b0, e0, sh_flag, [](uint32_t old) { return pair_c2(old); });
    auto get = [&](int32_t j) -> uint32_t { return wi.get(j); };
    la.v[1] += pair_diamonds(g, tl3, T, cv, i, b0, e0, wid, nw, get);
    core_store_row(cv, i, threadIdx.x, blockDim.x, get);
    __syncthreads();                            // the diamond reads of the window are done
    wi.done(sh_flag);
    block_item_flush(la, ids, acc, i, sh);
  }
  final_flush(la, ids, acc, sh);
}

// ---------------------------------------------------------------- 4-cycles
// Second pass of one item (Thm 5's rule): every wedge i - k - j adds
// w(i,j) - 1 to the edges (i,k) and (k,j).  Lists of up to PAIR_SHORT entries
// are walked by one lane each, longer ones by the warp.
template <class Get>
__device__ __forceinline__ void cycle4_edges(const DevGraph& g, int64_t b0, int64_t e0, int64_t gw, int64_t gnw,
                                             unsigned long long* C4raw, Get&& get) {
  const int lane = threadIdx.x & 31;
  for (int64_t pbase = b0 + gw; pbase < e0; pbase += gnw * 32) {
    const int64_t p = pbase + (int64_t)lane * gnw;
    int64_t kb_l = 0;
    int len_l = 0;
    if (p < e0) {
      kb_l = g.R[g.C[p]];
      len_l = (int)(g.rev[p] - kb_l);           // N(k) below i ends at the slot of i
    }
    if (len_l <= PAIR_SHORT) {
      unsigned long long sk = 0;
      for (int q = 0; q < len_l; q += 4) {
        int32_t jj[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) jj[u] = q + u < len_l ? g.J[kb_l + q + u] : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (jj[u] >= 0) {
            const unsigned long long c = get(jj[u]) - 1u;
            if (c) {
              atomicAdd(&C4raw[kb_l + q + u], c);
              sk += c;
            }
          }
      }
      if (sk) atomicAdd(&C4raw[p], sk);
    }
    unsigned longm = __ballot_sync(0xffffffffu, len_l > PAIR_SHORT);
    while (longm) {
      const int k = __ffs(longm) - 1;
      longm &= longm - 1;
      const int64_t kb = __shfl_sync(0xffffffffu, kb_l, k);
      const int len = __shfl_sync(0xffffffffu, len_l, k);
      const int32_t* L = g.J + kb;
      unsigned long long sk = 0;
      for (int q = lane; q < len; q += 32 * SWEEP_ILP) {
        int32_t jj[SWEEP_ILP];
#pragma unroll
        for (int u = 0; u < SWEEP_ILP; ++u) jj[u] = q + 32 * u < len ? L[q + 32 * u] : -1;
#pragma unroll
        for (int u = 0; u < SWEEP_ILP; ++u)
          if (jj[u] >= 0) {
            const unsigned long long c = get(jj[u]) - 1u;
            if (c) {
              atomicAdd(&C4raw[kb + q + 32 * u], c);
              sk += c;
            }
          }
      }
      sk = warp_sum_u64(sk);
      if (lane == 0 && sk) atomicAdd(&C4raw[pbase + (int64_t)k * gnw], sk);
    }
  }
}

// Heavy items of a single graph: the wedges to lower neighbours counted in the
// same windows as the pair sweep's.
template <bool BIG>
__global__ void __launch_bounds__(1024, 1) k_cycles4_win(DevGraph g, const unsigned long long* items, int64_t nitems,
                                                          unsigned long long* qctr, PairWin pw, PairTasks pt,
                                                          unsigned long long* C4raw, AccSet acc, unsigned* status) {
  extern __shared__ uint32_t win[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  __shared__ int sh_flag[2];
  const int wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  WinItem<BIG> wi(pw, win);
  const int ids[1] = {ACC_C4};
  LocalAcc<1> la;
  la.zero();
  wi.clear_window();
  if (threadIdx.x == 0) sh_flag[0] = sh_flag[1] = 0;
  while (true) {
    const int64_t it = next_item(qctr, nitems, &sh_item);
    if (it < 0) break;
    const int64_t i = item_rank(items[it]);
    const int64_t b0 = g.R[i], e0 = g.op[i];
    if (e0 - b0 > pw.curs_cap) {
      if (threadIdx.x == 0) set_err(status, DEVERR_SCRATCH);
      continue;
    }
    const u128 c4 = wi.count(g, pt, i, b0, e0, sh_flag, [](uint32_t old) { return (unsigned long long)old; });
    la.v[0] += c4;
    if (__syncthreads_or(c4 != 0)) cycle4_edges(g, b0, e0, wid, nw, C4raw, [&](int32_t j) { return wi.get(j); });
    __syncthreads();
    wi.done(sh_flag);
    block_item_flush(la, ids, acc, i, sh);
  }
  final_flush(la, ids, acc, sh);
}

// Heavy items of a union: dense tagged counters per CTA.
template <bool BIG>
__global__ void __launch_bounds__(512, 2) k_cycles4_tag(DevGraph g, const unsigned long long* items, int64_t nitems,
                                                        unsigned long long* qctr, TagScratch ts,
                                                        unsigned long long* C4raw, AccSet acc) {
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  TaggedCounters<BIG> w(ts);
  const int wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int ids[1] = {ACC_C4};
  LocalAcc<1> la;
  la.zero();
  while (true) {
    const int64_t it = next_item(qctr, nitems, &sh_item);
    if (it < 0) break;
    const int64_t i = item_rank(items[it]);
    const int64_t b0 = g.R[i], e0 = g.op[i];
    if (w.next(g.n)) __syncthreads();
    const u128 c4 = pair_wedges(g, b0, e0, wid, nw, [&](int32_t j) -> unsigned long long { return w.inc(j); },
                                [](int64_t, int64_t) { return false; });
    la.v[0] += c4;
    if (__syncthreads_or(c4 != 0)) cycle4_edges(g, b0, e0, wid, nw, C4raw, [&](int32_t j) { return w.get(j); });
    block_item_flush(la, ids, acc, i, sh);
    __syncthreads();                            // the next item's counts must not meet these reads
  }
  final_flush(la, ids, acc, sh);
}

// Light and medium items: one CTA of THREADS threads per item, w(i, .) in a
// packed hash table.
template <int THREADS>
__global__ void __launch_bounds__(THREADS) k_cycles4_hash(DevGraph g, const unsigned long long* items, int64_t nitems,
                                                         unsigned long long* qctr, int cb, int max_log,
                                                         unsigned long long* C4raw, AccSet acc, unsigned* status) {
  extern __shared__ uint4 hash_smem[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  const int wid = threadIdx.x >> 5, nw = THREADS / 32;
  PackedHash H{reinterpret_cast<uint32_t*>(hash_smem), cb, 0};
  const int ids[1] = {ACC_C4};
  LocalAcc<1> la;
  la.zero();
  while (true) {
    const int64_t it = next_item(qctr, nitems, &sh_item);
    if (it < 0) break;
    const int64_t i = item_rank(items[it]);
    const int64_t b0 = g.R[i], e0 = g.op[i];
    H.log = min(max_log, item_log(items[it]));
    H.clear(threadIdx.x, THREADS);
    __syncthreads();
    bool full = false;
    const u128 c4 = pair_wedges(g, b0, e0, wid, nw, [&](int32_t j) -> unsigned long long {
      return H.inc(j, full);
    }, [](int64_t, int64_t) { return false; });
    if (full) set_err(status, DEVERR_SCRATCH);
    la.v[0] += c4;
    if (__syncthreads_or(c4 != 0)) cycle4_edges(g, b0, e0, wid, nw, C4raw, [&](int32_t j) { return H.get(j); });
    block_item_flush(la, ids, acc, i, sh);
  }
  final_flush(la, ids, acc, sh);
}

// Medium items of small graphs: a counter per vertex of the graph.
__global__ void __launch_bounds__(IT_MEDIUM_THREADS) k_cycles4_direct(DevGraph g, const unsigned long long* items,
                                                                     int64_t nitems, unsigned long long* qctr,
                                                                     LocalIds lc, unsigned long long* C4raw,
                                                                     AccSet acc) {
  extern __shared__ uint4 hash_smem[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  uint32_t* tab = reinterpret_cast<uint32_t*>(hash_smem);
  const int wid = threadIdx.x >> 5, nw = IT_MEDIUM_THREADS / 32;
  const int ids[1] = {ACC_C4};
  LocalAcc<1> la;
  la.zero();
  while (true) {
    const int64_t it = next_item(qctr, nitems, &sh_item);
    if (it < 0) break;
    const int64_t i = item_rank(items[it]);
    const int64_t b0 = g.R[i], e0 = g.op[i];
    direct_clear(tab, lc.size(i));
    __syncthreads();
    const u128 c4 = pair_wedges(g, b0, e0, wid, nw,
                                [&](int32_t j) -> unsigned long long { return atomicAdd(&tab[j], 1u); },
                                [](int64_t, int64_t) { return false; });
    la.v[0] += c4;
    if (__syncthreads_or(c4 != 0)) cycle4_edges(g, b0, e0, wid, nw, C4raw, [&](int32_t j) { return tab[j]; });
    block_item_flush(la, ids, acc, i, sh);
  }
  final_flush(la, ids, acc, sh);
}

// ============================================================================
// Thm 11: N18 (wheels) = sum over centres c of the 4-cycles of G[N(c)],
// counted by the 4-cycle rule inside the neighbourhood: for u in N(c) and
// v < u, C(w_c(u,v), 2) with w_c(u,v) = |{k in N(c) cap N(u) cap N(v): k < u}|.
// Everything happens in the position space of row c: the lists of the slots
// (c -> u) hold positions in row c, so k < u is pk < pu and the counters are
// indexed by position.  sum_v C(w, 2) is the sum of the values each increment
// returns.
// ============================================================================
static constexpr int WHEEL_WARP_MAX = 1024;     // centres up to this degree: warp items

// Core centres (core.cu) leave the 4-cycles whose low vertices (below h0; the
// positions below pc) are none, one, or two opposite ones to the contraction.
// What is left has two adjacent low vertices.  For u low, everything below u is
// low and the rule above applies unchanged.  For u in the core, v is low and
// with wL (wH) the number of k that are low (in the core and below u),
// wL wH + C(wL, 2): the low k are counted first, then the core k read the counts.
//
// One of these walks for one u: for the k at entries [a0, a1) of the list Lu of
// slot c -> u that are below kmax (the warp takes a0 + w, a0 + w + step, ...,
// 32 at a time, lane l the l-th), every v below vmax in the list of slot
// c -> k: visit(pv).  LEN gives the entries of that list that can lie below
// vmax.  Lists of up to WHEEL_SHORT entries are walked by one lane each, longer
// ones by the warp, with WHEEL_ILP independent loads in flight per lane.
#ifndef ESC_WHEEL_ILP
#define ESC_WHEEL_ILP 8
#endif
static constexpr int WHEEL_ILP = ESC_WHEEL_ILP;
static constexpr uint32_t WHEEL_SHORT = 32;

template <class Visit>
__device__ __forceinline__ void wheel_walk(const TriLists& tl3, const uint32_t* LEN, int64_t base, const int32_t* Lu,
                                           uint32_t a0, uint32_t a1, int kmax, int vmax, uint32_t w, uint32_t step,
                                           Visit&& visit) {
  const int lane = threadIdx.x & 31;
  for (uint32_t ab = a0 + w; ab < a1; ab += 32 * step) {
    const uint32_t a = ab + lane * step;
    const int32_t* Lk_l = tl3.P;
    uint32_t lk_l = 0;
    const bool live = a < a1;
    bool in = false;
    if (live) {
      const int32_t pk = Lu[a];
      if (pk < kmax) {
        in = true;
        Lk_l = tl3.P + tl3.offp[base + pk];
        lk_l = LEN[base + pk];
      }
    }
    const bool done = __any_sync(0xffffffffu, live && !in);   // the k list is sorted: later rounds are above kmax
    if (lk_l <= WHEEL_SHORT) {
      for (uint32_t t = 0; t < lk_l; t += 4) {
        int32_t pv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) pv[u] = t + u < lk_l ? Lk_l[t + u] : 0x7fffffff;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (pv[u] < vmax) visit(pv[u]);
        if (pv[3] >= vmax) break;
      }
      lk_l = 0;
    }
    unsigned m = __ballot_sync(0xffffffffu, lk_l > 0);
    while (m) {
      const int k = __ffs(m) - 1;
      m &= m - 1;
      const int32_t* Lk = reinterpret_cast<const int32_t*>(
          __shfl_sync(0xffffffffu, reinterpret_cast<uintptr_t>(Lk_l), k));
      const uint32_t lk = __shfl_sync(0xffffffffu, lk_l, k);
      for (uint32_t tb = 0; tb < lk; tb += 32 * WHEEL_ILP) {
        int32_t pv[WHEEL_ILP];
        bool past = false;
#pragma unroll
        for (int u = 0; u < WHEEL_ILP; ++u) {
          const uint32_t t = tb + lane + 32 * u;
          pv[u] = t < lk ? Lk[t] : 0x7fffffff;
          if (pv[u] >= vmax) { pv[u] = -1; past = true; }
        }
#pragma unroll
        for (int u = 0; u < WHEEL_ILP; ++u)
          if (pv[u] >= 0) visit(pv[u]);
        if (__any_sync(0xffffffffu, past)) break;
      }
    }
    if (done) break;
  }
}

// Centres up to WHEEL_WARP_MAX: work items are (centre, block of WHEEL_WBLK
// positions u), pulled by whole warps from a queue, heaviest centres first.
// Each warp owns a counter array in shared memory whose entries are
// (tag << 16) | count for the u they were counted for; before each increment
// an atomicMax with the current u's tag turns an older entry into a zero
// count, so nothing is cleared between u's or items.
static constexpr int WHEEL_WBLK = 32;

// item_cnt[k] = number of items of centre c0 - 1 - k (position k in the queue)
__global__ void k_wheel_warp_counts(DevGraph g, int64_t c0, int64_t* item_cnt, Owner own) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < c0; k += (int64_t)gridDim.x * blockDim.x) {
    int64_t c = c0 - 1 - k;
    int64_t d = g.R[c + 1] - g.R[c];
    item_cnt[k] = d >= 4 && own.owns(c) ? (d + WHEEL_WBLK - 1) / WHEEL_WBLK : 0;
  }
}

__global__ void __launch_bounds__(256, 6) k_wheels_warp(DevGraph g, int64_t c0, const int64_t* item_off,
                                                        unsigned long long* qctr, TriLists tl3, const uint32_t* T,
                                                        CoreView cv, AccSet acc) {
  __shared__ u128 sh[32];
  __shared__ uint32_t scr_all[8][WHEEL_WARP_MAX];
  int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  uint32_t* scr = scr_all[wl];
  const int ids[1] = {ACC_N18};
  LocalAcc<1> la;
  la.zero();
  for (int i = lane; i < WHEEL_WARP_MAX; i += 32) scr[i] = 0;
  __syncwarp();
  uint32_t tag = 0;
  const int64_t nitems = item_off[c0];
  while (true) {
    unsigned long long it_l = 0;
    if (lane == 0) it_l = atomicAdd(qctr, 1ull);
    int64_t it = (int64_t)__shfl_sync(0xffffffffu, it_l, 0);
    if (it >= nitems) break;
    // queue position of the centre: the last k with item_off[k] <= it
    int64_t lo = 0, hi = c0;
    while (hi - lo > 1) {
      int64_t mid = (lo + hi) >> 1;
      if (item_off[mid] <= it) lo = mid; else hi = mid;
    }
    int64_t c = c0 - 1 - lo;
    int64_t base = g.R[c];
    int d = (int)(g.R[c + 1] - base);
    int u0 = (int)(it - item_off[lo]) * WHEEL_WBLK;
    int u1 = min(d, u0 + WHEEL_WBLK);
    const int pc = c >= cv.h0 ? d - cv.dh[c - cv.h0] : d;   // positions from pc on are in the core
    u128 n18 = 0;
    for (int pu = u0; pu < u1; ++pu) {
      uint32_t lenu = T[base + pu];
      if (lenu < 2) continue;
      const bool top = pu >= pc;
      const uint32_t lowu = top ? cv.low[base + pu] : lenu;
      if (lowu == 0) continue;
      if (++tag == 0x10000u) {                           // tags exhausted: start over from zeroed counters
        __syncwarp();
        for (int i = lane; i < WHEEL_WARP_MAX; i += 32) scr[i] = 0;
        __syncwarp();
        tag = 1;
      }
      const int32_t* Lu = tl3.P + tl3.offp[base + pu];
      unsigned long long part = 0;
      const uint32_t t16 = tag << 16;
      wheel_walk(tl3, T, base, Lu, 0u, lowu, pu, min(pu, pc), 0u, 1u, [&](int32_t pv) {
        atomicMax(&scr[pv], t16);               // an older u's entry becomes a zero count of this one
        part += atomicAdd(&scr[pv], 1u) & 0xffffu;
      });
      __syncwarp();                             // this u's increments before the next u's tag
      if (top && lowu < lenu) {
        wheel_walk(tl3, cv.low, base, Lu, lowu, lenu, pu, pc, 0u, 1u, [&](int32_t pv) {
          const uint32_t v = scr[pv];
          if ((v & 0xffff0000u) == t16) part += v & 0xffffu;
        });
        __syncwarp();
      }
      n18 += part;
    }
    la.v[0] += n18;
    warp_item_flush(la, ids, acc, c);
  }
  final_flush(la, ids, acc, sh);
}

// Centres above WHEEL_WARP_MAX: work items (centre, block of WHEEL_CHUNK
// positions u) taken by a CTA of WHEEL_THREADS threads (one per SM: its shared
// memory holds the counters).  The CTA's warps form groups that take different
// u's, as many groups as counter arrays of pc positions fit: a core centre
// leaves little work per u, so one warp per u (pc up to about 1,700) or four
// keep more u's in flight than the whole CTA on one.
static constexpr int WHEEL_CHUNK = 128;
static constexpr int WHEEL_THREADS = 1024;

// Counters are tagged with the u they count for, (tag << 16) | count in the
// 32-bit shared-memory words and (tag << 32) | count in the 64-bit global ones
// (counts there can pass 2^16); before each increment an atomicMax with the
// current tag turns an older entry into a zero count, so no clearing pass
// walks the lists a second time.  The tags of a CTA grow with its items and
// within an item with u, whatever array an item's groups use.
// win16: every count of the sweep stays below 2^16 (the largest common-
// neighbour list is shorter), so centres with more positions than the shared
// memory holds keep a shared-memory window over the last smem_cap of them (the
// highest ranks, where the common neighbours concentrate) and count the others
// in global memory.
__device__ __forceinline__ void wheel_group_sync(int gs, int grp) {
  if (gs == 1) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(gs * 32) : "memory");
}

__global__ void __launch_bounds__(WHEEL_THREADS, 1) k_wheels_cta(DevGraph g, int64_t c0, const int64_t* item_off,
                                                                int64_t nitems, unsigned long long* qctr, TriLists tl3,
                                                                const uint32_t* T, CoreView cv,
                                                                unsigned long long* gscr, int64_t gscr_stride,
                                                                int smem_cap, AccSet acc, bool win16) {
  extern __shared__ uint32_t sscr[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  const int wid = threadIdx.x >> 5;
  const int ids[1] = {ACC_N18};
  LocalAcc<1> la;
  la.zero();
  unsigned long long* g64 = gscr + (int64_t)blockIdx.x * gscr_stride;
  for (int i = threadIdx.x; i < smem_cap; i += blockDim.x) sscr[i] = 0;
  __syncthreads();
  uint32_t tag0 = 0;                            // tags used so far, the same in every thread of the CTA
  while (true) {
    int64_t it = next_item(qctr, nitems, &sh_item);   // its barriers also end the last item's reads
    if (it < 0) break;
    it = nitems - 1 - it;                     // heaviest centres first
    // centre of item `it`: the last k with item_off[k] <= it (item_off over centres c0..n-1)
    int64_t lo = 0, hi = g.n - c0;
    while (hi - lo > 1) { int64_t mid = (lo + hi) >> 1; if (item_off[mid] <= it) lo = mid; else hi = mid; }
    const int64_t c = c0 + lo;
    const int64_t base = g.R[c];
    const int d = (int)(g.R[c + 1] - base);
    const int u0 = (int)(it - item_off[lo]) * WHEEL_CHUNK;
    const int u1 = min(d, u0 + WHEEL_CHUNK);
    const int pc = c >= cv.h0 ? d - cv.dh[c - cv.h0] : d;   // positions from pc on are in the core
    if (tag0 + WHEEL_CHUNK > 0xffffu) {         // tags used up: zero both counter sets, start over
      for (int i = threadIdx.x; i < smem_cap; i += blockDim.x) sscr[i] = 0;
      for (int64_t i = threadIdx.x; i < gscr_stride; i += blockDim.x) g64[i] = 0;
      __syncthreads();
      tag0 = 0;
    }
    const bool in_smem = pc <= smem_cap;
    // warps per group: 1, 4, 8, 16 or 32 (groups of two would need more than the 15 named barriers)
    int gs = WHEEL_THREADS / 32;
    if ((int64_t)pc * 32 <= smem_cap) gs = 1;
    else if ((int64_t)pc * 8 <= smem_cap) gs = 4;
    else if ((int64_t)pc * 4 <= smem_cap) gs = 8;
    else if ((int64_t)pc * 2 <= smem_cap) gs = 16;
    const int grp = wid / gs, ngrp = WHEEL_THREADS / 32 / gs, gw = wid % gs;
    uint32_t* scr = sscr + (in_smem ? (int64_t)grp * pc : 0);
    for (int pu = u0 + grp; pu < u1; pu += ngrp) {
      const uint32_t lenu = T[base + pu];
      if (lenu < 2) continue;
      const bool top = pu >= pc;
      const uint32_t lowu = top ? cv.low[base + pu] : lenu;
      if (lowu == 0) continue;
      const int32_t* Lu = tl3.P + tl3.offp[base + pu];
      const uint32_t tag = tag0 + 1 + (uint32_t)(pu - u0), t16 = tag << 16;
      const unsigned long long t32 = (unsigned long long)tag << 32;
      const int wstart = in_smem ? 0 : (win16 ? pc - smem_cap : pc);
      unsigned long long part = 0;
      wheel_walk(tl3, T, base, Lu, 0u, lowu, pu, min(pu, pc), (uint32_t)gw, (uint32_t)gs, [&](int32_t pv) {
        if (pv >= wstart) {
          uint32_t* q = &scr[pv - wstart];
          atomicMax(q, t16);
          part += atomicAdd(q, 1u) & 0xffffu;
        } else {
          atomicMax(&g64[pv], t32);
          part += (uint32_t)atomicAdd(&g64[pv], 1ull);
        }
      });
      if (top && lowu < lenu) {
        wheel_group_sync(gs, grp);              // every low k is counted
        wheel_walk(tl3, cv.low, base, Lu, lowu, lenu, pu, pc, (uint32_t)gw, (uint32_t)gs, [&](int32_t pv) {
          if (pv >= wstart) {
            const uint32_t v = scr[pv - wstart];
            if ((v & 0xffff0000u) == t16) part += v & 0xffffu;
          } else {
            const unsigned long long v = __ldcg(&g64[pv]);
            if ((v >> 32) == tag) part += (uint32_t)v;
          }
        });
      }
      la.v[0] += part;
      wheel_group_sync(gs, grp);                // the next u's tag must not meet this u's counts
    }
    tag0 += WHEEL_CHUNK;
    block_item_flush(la, ids, acc, c, sh);
  }
  final_flush(la, ids, acc, sh);
}

// ============================================================================
// Thm 13: 5-cycles.  For every directed 3-path i <- a -> b -> j (a < i,
// a < b < j, b != i, j != i) add w'(i,j) = |{c in N(i) cap N(j) : c < max(i,j)}|.
// Grouped by the pair (i, b): sum_b P2(i,b) * sum_{j in N+(b)} w'(i,j) with
// P2(i,b) = |{a in N-(i) : b in N+(a)}| (each out-wedge pair visited once).
// The paths whose own a or b is counted by w' are the directed tailed
// triangles, subtracted through ACC_N8Z (pass A).
// ============================================================================
template <bool BIG> struct CountSum { typedef uint32_t type; };
template <> struct CountSum<true> { typedef unsigned long long type; };

// The lists N+(b) of up to 32 vertices b (lane l holds the l-th list [cb_l, ce_l)
// and its factor f_l; empty lists have cb_l = ce_l): sum of f * get(j) over
// their entries.  Lists of up to PAIR_SHORT entries are walked by one lane each.
// Blk holds the sum of SWEEP_ILP counts: 32 bits where a count is below 2^16.
template <typename Blk, class Get>
__device__ __forceinline__ u128 cycle5_lists(const DevGraph& g, int64_t cb_l, int64_t ce_l, uint32_t f_l, Get&& get) {
  const int lane = threadIdx.x & 31;
  const int len_l = (int)(ce_l - cb_l);
  u128 sum = 0;
  if (len_l <= PAIR_SHORT) {
    const int32_t* L = g.J + cb_l;
    unsigned long long s_ = 0;
    for (int q = 0; q < len_l; q += 4) {
      int32_t jj[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) jj[u] = q + u < len_l ? L[q + u] : -1;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (jj[u] >= 0) s_ += get(jj[u]);
    }
    sum += (u128)s_ * f_l;
  }
  unsigned longm = __ballot_sync(0xffffffffu, len_l > PAIR_SHORT);
  while (longm) {
    const int k = __ffs(longm) - 1;
    longm &= longm - 1;
    const int32_t* L = g.J + __shfl_sync(0xffffffffu, cb_l, k);
    const int len = __shfl_sync(0xffffffffu, len_l, k);
    const uint32_t f = __shfl_sync(0xffffffffu, f_l, k);
    // whole groups without a test per entry (R-MAT 19 5-cycles 57.3 -> 53.0 ms)
    unsigned long long s_ = 0;
    int q = 0;
    for (; q + 32 * SWEEP_ILP <= len; q += 32 * SWEEP_ILP) {
      int32_t jj[SWEEP_ILP];
#pragma unroll
      for (int u = 0; u < SWEEP_ILP; ++u) jj[u] = L[q + lane + 32 * u];
      Blk blk = 0;
#pragma unroll
      for (int u = 0; u < SWEEP_ILP; ++u) blk += get(jj[u]);
      s_ += blk;
    }
#pragma unroll
    for (int gsz = SWEEP_ILP / 2; gsz >= 1; gsz >>= 1) {
      if (q + 32 * gsz <= len) {
        int32_t jj[SWEEP_ILP / 2];
#pragma unroll
        for (int u = 0; u < gsz; ++u) jj[u] = L[q + lane + 32 * u];
        Blk blk = 0;
#pragma unroll
        for (int u = 0; u < gsz; ++u) blk += get(jj[u]);
        s_ += blk;
        q += 32 * gsz;
      }
    }
    if (q + lane < len) s_ += get(L[q + lane]);
    sum += (u128)s_ * f;
  }
  return sum;
}

// visit(j) for every entry of up to 32 lists (lane l holds the l-th), short
// ones by one lane each.
template <class Visit>
__device__ __forceinline__ void lists_each(const DevGraph& g, int64_t cb_l, int64_t ce_l, Visit&& visit) {
  const int lane = threadIdx.x & 31;
  const int len_l = (int)(ce_l - cb_l);
  if (len_l <= PAIR_SHORT) {
    const int32_t* L = g.J + cb_l;
    for (int q = 0; q < len_l; q += 4) {
      int32_t jj[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) jj[u] = q + u < len_l ? L[q + u] : -1;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (jj[u] >= 0) visit(jj[u]);
    }
  }
  unsigned longm = __ballot_sync(0xffffffffu, len_l > PAIR_SHORT);
  while (longm) {
    const int k = __ffs(longm) - 1;
    longm &= longm - 1;
    const int32_t* L = g.J + __shfl_sync(0xffffffffu, cb_l, k);
    const int len = __shfl_sync(0xffffffffu, len_l, k);
    for (int q = lane; q < len; q += 32 * SWEEP_ILP) {
      int32_t jj[SWEEP_ILP];
#pragma unroll
      for (int u = 0; u < SWEEP_ILP; ++u) jj[u] = q + 32 * u < len ? L[q + 32 * u] : -1;
#pragma unroll
      for (int u = 0; u < SWEEP_ILP; ++u)
        if (jj[u] >= 0) visit(jj[u]);
    }
  }
}

// The increments of one item: w'(i, .) from c < i (every j in N(c)) and c > i
// (j in N+(c)); P2(i, .) from a in N-(i) (b in N+(a)).  j = b = i (as g.J names
// the item) is left out.
template <class IncW, class IncP>
__device__ __forceinline__ void cycle5_counts(const DevGraph& g, int32_t i, int64_t b0, int64_t o, int64_t e0,
                                              int64_t gw, int64_t gnw, IncW&& incw, IncP&& incp) {
  const int lane = threadIdx.x & 31;
  for (int64_t pbase = b0 + gw; pbase < e0; pbase += gnw * 32) {
    const int64_t p = pbase + (int64_t)lane * gnw;
    int64_t cb_l = 0, ce_l = 0, cm_l = 0;       // the list; from cm_l on also P2
    if (p < e0) {
      const int32_t c = g.C[p];
      const int64_t co = g.op[c];
      ce_l = g.R[c + 1];
      cb_l = p < o ? g.R[c] : co;
      cm_l = p < o ? co : ce_l;
    }
    lists_each(g, cb_l, ce_l, [&](int32_t j) { if (j != i) incw(j); });
    lists_each(g, cm_l, ce_l, [&](int32_t j) { if (j != i) incp(j); });
  }
}

// Light and medium items: one CTA of THREADS threads per item, w'(i, .) and
// P2(i, .) in two packed hash tables; the distinct b are the used words of the
// second.
template <int THREADS>
__global__ void __launch_bounds__(THREADS) k_cycles5_hash(DevGraph g, const unsigned long long* items, int64_t nitems,
                                                         unsigned long long* qctr, int cb, int max_log, AccSet acc,
                                                         unsigned* status) {
  extern __shared__ uint4 hash_smem[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = THREADS / 32;
  PackedHash Hw{reinterpret_cast<uint32_t*>(hash_smem), cb, 0}, Hp = Hw;
  const int ids[1] = {ACC_N8M};
  LocalAcc<1> la;
  la.zero();
  while (true) {
    const int64_t it = next_item(qctr, nitems, &sh_item);   // its barriers end the last item's reads
    if (it < 0) break;
    const int64_t i = item_rank(items[it]);
    const int64_t b0 = g.R[i], o = g.op[i], e0 = g.R[i + 1];
    Hw.log = min(max_log, item_log(items[it]));
    Hp.log = min(max_log, item_log2(items[it]));
    Hp.tab = Hw.tab + (1 << Hw.log);
    Hw.clear(threadIdx.x, THREADS);
    Hp.clear(threadIdx.x, THREADS);
    __syncthreads();
    bool full = false;
    cycle5_counts(g, (int32_t)i, b0, o, e0, wid, nw, [&](int32_t j) { Hw.inc(j, full); }, [&](int32_t j) { Hp.inc(j, full); });
    if (full) set_err(status, DEVERR_SCRATCH);
    __syncthreads();
    for (int tb = wid * 32; tb < (1 << Hp.log); tb += THREADS) {
      const uint32_t w = Hp.tab[tb + lane];
      const bool used = w != PackedHash::EMPTY;
      if (!__any_sync(0xffffffffu, used)) continue;
      int64_t cb_l = 0, ce_l = 0;
      if (used) {
        const int32_t b = (int32_t)(w >> cb);
        cb_l = g.op[b];
        ce_l = g.R[b + 1];
      }
      la.v[0] += cycle5_lists<unsigned long long>(g, cb_l, ce_l, w & ((1u << cb) - 1u), [&](int32_t j) -> uint32_t { return Hw.get(j); });
    }
    block_item_flush(la, ids, acc, i, sh);
  }
  final_flush(la, ids, acc, sh);
}

// Medium items of small graphs: w'(i, .) in the low and P2(i, .) in the high 16
// bits of a counter per vertex of the graph (both below its size, at most
// DIRECT_N).  Each warp takes every 16th b, so that the long lists N+(b) of
// neighbouring ranks go to different warps.
__global__ void __launch_bounds__(IT_MEDIUM_THREADS) k_cycles5_direct(DevGraph g, const unsigned long long* items,
                                                                     int64_t nitems, unsigned long long* qctr,
                                                                     LocalIds lc, AccSet acc) {
  extern __shared__ uint4 hash_smem[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  uint32_t* tab = reinterpret_cast<uint32_t*>(hash_smem);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = IT_MEDIUM_THREADS / 32;
  const int ids[1] = {ACC_N8M};
  LocalAcc<1> la;
  la.zero();
  while (true) {
    const int64_t it = next_item(qctr, nitems, &sh_item);   // its barriers end the last item's reads
    if (it < 0) break;
    const int64_t i = item_rank(items[it]), s0 = lc.start(i);
    const int64_t b0 = g.R[i], o = g.op[i], e0 = g.R[i + 1];
    const int ng = lc.size(i);
    direct_clear(tab, ng);
    __syncthreads();
    cycle5_counts(g, lc.place(i), b0, o, e0, wid, nw, [&](int32_t j) { atomicAdd(&tab[j], 1u); },
                  [&](int32_t b) { atomicAdd(&tab[b], 1u << 16); });
    __syncthreads();
    for (int tb = wid; tb < ng; tb += nw * 32) {
      const int t = tb + lane * nw;
      const uint32_t f = t < ng ? tab[t] >> 16 : 0u;
      if (!__any_sync(0xffffffffu, f != 0)) continue;
      int64_t cb_l = 0, ce_l = 0;
      if (f) {
        const int64_t b = lc.rank(s0, t);
        cb_l = g.op[b];
        ce_l = g.R[b + 1];
      }
      la.v[0] += cycle5_lists<uint32_t>(g, cb_l, ce_l, f, [&](int32_t j) -> uint32_t { return tab[j] & 0xffffu; });
    }
    block_item_flush(la, ids, acc, i, sh);
  }
  final_flush(la, ids, acc, sh);
}

// Heavy items: one 1024-thread CTA per SM.  The counts of the ranks
// [wlo, jbig) -- the top ones below the 64-bit side array, where the j, two
// steps up the order from a, concentrate -- live in shared memory, w'(i, r) in
// the low and P2(i, r) in the high 16 bits of a word (both at most the rank's
// degree, below 2^16); lower ranks use tagged counters and a touched list in
// global memory.
template <bool BIG>
__global__ void __launch_bounds__(1024, 1) k_cycles5(DevGraph g, const unsigned long long* items, int64_t nitems,
                                                     unsigned long long* qctr, TagScratch ts, SweepScratch ss,
                                                     AccSet acc, int64_t wlo, int win_words) {
  extern __shared__ uint32_t win[];
  __shared__ u128 sh[32];
  __shared__ int64_t sh_item;
  __shared__ unsigned nt;
  TaggedCounters<BIG> wp(ts);                                                         // w'(i, .) outside the window
  uint32_t* p2 = ss.cnt2 + (int64_t)blockIdx.x * ss.n;                            // P2(i, .) there, with a list
  int32_t* tl2 = ss.touched2 + (int64_t)blockIdx.x * ss.n;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t wlo32 = (uint32_t)wlo, nwin = (uint32_t)win_words;
  const int ids[1] = {ACC_N8M};
  LocalAcc<1> la;
  la.zero();
  for (int t = threadIdx.x; t < win_words; t += blockDim.x) win[t] = 0u;
  while (true) {
    const int64_t it = next_item(qctr, nitems, &sh_item);
    if (it < 0) break;
    const int64_t i = item_rank(items[it]);
    const int64_t b0 = g.R[i], o = g.op[i], e0 = g.R[i + 1];
    wp.next(ts.n);
    if (threadIdx.x == 0) nt = 0;
    __syncthreads();
    cycle5_counts(g, (int32_t)i, b0, o, e0, wid, nw,
                  [&](int32_t j) {
                    const uint32_t q = (uint32_t)j - wlo32;
                    if (q < nwin) atomicAdd(&win[q], 1u);
                    else wp.add(j);
                  },
                  [&](int32_t b) {
                    const uint32_t q = (uint32_t)b - wlo32;
                    if (q < nwin) {
                      atomicAdd(&win[q], 1u << 16);
                    } else {
                      const bool first = atomicAdd(&p2[b], 1u) == 0;
                      if (first) tl2[atomicAdd(&nt, 1u)] = b;
                    }
                  });
    __syncthreads();
    auto get = [&](int32_t j) -> uint32_t {
      const uint32_t q = (uint32_t)j - wlo32;
      return q < nwin ? win[q] & 0xffffu : wp.get(j);
    };
    // sum over the distinct b of P2(i, b) * sum_{j in N+(b)} w'(i, j)
    const unsigned n2 = nt;
    for (uint32_t tb = (uint32_t)wid * 32; tb < nwin; tb += (uint32_t)nw * 32) {
      const uint32_t f = tb + lane < nwin ? win[tb + lane] >> 16 : 0u;
      if (!__any_sync(0xffffffffu, f != 0)) continue;
      int64_t cb_l = 0, ce_l = 0;
      if (f) {
        const int64_t b = wlo + tb + lane;
        cb_l = g.op[b];
        ce_l = g.R[b + 1];
      }
      la.v[0] += cycle5_lists<typename CountSum<BIG>::type>(g, cb_l, ce_l, f, get);
    }
    for (unsigned tb = (unsigned)wid * 32; tb < n2; tb += (unsigned)nw * 32) {
      const unsigned t = tb + lane;
      int64_t cb_l = 0, ce_l = 0;
      uint32_t f = 0;
      if (t < n2) {
        const int32_t b = tl2[t];
        cb_l = g.op[b];
        ce_l = g.R[b + 1];
        f = p2[b];
      }
      la.v[0] += cycle5_lists<typename CountSum<BIG>::type>(g, cb_l, ce_l, f, get);
    }
    __syncthreads();
    for (unsigned t = threadIdx.x; t < n2; t += blockDim.x) p2[tl2[t]] = 0;
    for (int t = threadIdx.x; t < win_words; t += blockDim.x) win[t] = 0u;
    block_item_flush(la, ids, acc, i, sh);
    __syncthreads();
  }
  final_flush(la, ids, acc, sh);
}

// ============================================================================
// Per-edge common-neighbour lists (the per-edge triangle lists of Thm 7),
// stored sorted: the id list once per undirected edge (addressed from both
// slots), and for each slot (u -> v) the positions in row u of the same
// vertices.  Edges without a triangle are skipped.  By the higher endpoint y:
//   degree <= TL_LIGHT: one thread per edge merges the two short rows;
//   above: one CTA per y, N(y) in a hash table (vertex -> position in row y); for
//     every lower neighbour x the row N(x) is filtered through it; a hit at
//     index q of row x has position q - R[x] there.
// One CTA for every y, with the offsets of each x fetched before its row, was
// bound by latency: R-MAT 19 41 ms, Chung-Lu 2.3 n = 625,000 6.4 ms.
// ============================================================================
static constexpr int TL_LIGHT = 64, TL_TILE = 2048, TL_ILP = 4;

// Slots [0, slots) are the rows of the vertices of degree <= TL_LIGHT.
__global__ void __launch_bounds__(256) k_tri_lists_light(DevGraph g, int64_t rows, int64_t slots, const int64_t* off,
                                                        const int64_t* offp, const uint32_t* T, int32_t* U, int32_t* P,
                                                        unsigned* status) {
  __shared__ int64_t sh_row[2];
  for (int64_t t0 = (int64_t)blockIdx.x * TL_TILE; t0 < slots; t0 += (int64_t)gridDim.x * TL_TILE) {
    const int64_t t1 = min(slots, t0 + TL_TILE);
    if (threadIdx.x < 2) {                      // rows of the first and last slot: the last y with R[y] <= p
      const int64_t p = threadIdx.x ? t1 - 1 : t0;
      int64_t lo = 0, hi = rows;
      while (hi - lo > 1) { const int64_t mid = (lo + hi) >> 1; if (g.R[mid] <= p) lo = mid; else hi = mid; }
      sh_row[threadIdx.x] = lo;
    }
    __syncthreads();
    const int64_t r0 = sh_row[0], r1 = sh_row[1];
    for (int64_t p = t0 + threadIdx.x; p < t1; p += blockDim.x) {
      const uint32_t expect = T[p];
      if (expect == 0) continue;
      int64_t lo = r0, hi = r1 + 1;
      while (hi - lo > 1) { const int64_t mid = (lo + hi) >> 1; if (g.R[mid] <= p) lo = mid; else hi = mid; }
      const int64_t y = lo;
      const int32_t x = g.C[p];
      if (x > y) continue;                      // once per edge, at its higher endpoint
      const int64_t yb = g.R[y], xb = g.R[x], cs = g.rev[p];
      const int dy = (int)(g.R[y + 1] - yb), dx = (int)(g.R[x + 1] - xb);
      const int64_t out = off[cs], outx = offp[cs], outy = offp[p];
      uint32_t k = 0;
      int i = 0, j = 0;
      while (i < dx && j < dy) {
        const int32_t a = g.C[xb + i], c = g.C[yb + j];
        if (a == c) {
          if (k < expect) {
            U[out + k] = a;
            P[outx + k] = i;
            P[outy + k] = j;
          }
          ++k;
        }
        i += a <= c ? 1 : 0;
        j += c <= a ? 1 : 0;
      }
      if (k != expect) set_err(status, DEVERR_BOUNDS);
    }
    __syncthreads();                            // the rows are read before the next tile's are written
  }
}

// Vertices n - 1 down to r0.
__global__ void __launch_bounds__(512) k_tri_lists(DevGraph g, int64_t r0, unsigned long long* qctr, const int64_t* off,
                                                  const int64_t* offp, const uint32_t* T, int32_t* U, int32_t* P,
                                                  int32_t* ghash, int64_t ghash_cap, int hash_cap, unsigned* status) {
  extern __shared__ int32_t smem[];
  __shared__ int64_t sh_item;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  int32_t* gk = ghash + (int64_t)blockIdx.x * 2 * ghash_cap;
  while (true) {
    int64_t it = next_item(qctr, g.n - r0, &sh_item);
    if (it < 0) break;
    int64_t y = g.n - 1 - it;
    int64_t yb = g.R[y], yo = g.op[y], ye = g.R[y + 1];
    if (yo == yb) continue;
    int dy = (int)(ye - yb);
    bool small = 2 * dy <= hash_cap;
    int hsz = pow2_at_least(2 * dy);
    if (!small && hsz > ghash_cap) {            // cannot happen: sized by the maximum degree
      if (threadIdx.x == 0) set_err(status, DEVERR_SCRATCH);
      continue;
    }
    PosHash H = small ? PosHash{smem, smem + hash_cap, hsz - 1} : PosHash{gk, gk + ghash_cap, hsz - 1};
    for (int i = threadIdx.x; i < hsz; i += blockDim.x) H.keys[i] = -1;
    __syncthreads();
    for (int i = threadIdx.x; i < dy; i += blockDim.x) H.insert(g.C[yb + i], i);
    __syncthreads();
    // x in N-(y), p = slot (y -> x): a warp fetches what it needs of 32 of them at
    // once (lane l the l-th), then filters their rows one by one
    for (int64_t pbase = yb + wid; pbase < yo; pbase += (int64_t)nw * 32) {
      const int64_t p = pbase + (int64_t)lane * nw;
      uint32_t expect_l = p < yo ? T[p] : 0u;
      int64_t xb_l = 0, out_l = 0, outx_l = 0, outy_l = 0;
      int len_l = 0;
      if (expect_l) {
        const int32_t x = g.C[p];
        const int64_t cs = g.rev[p];            // canonical slot (x -> y)
        xb_l = g.R[x];
        len_l = (int)(g.R[x + 1] - xb_l);
        out_l = off[cs];
        outx_l = offp[cs];
        outy_l = offp[p];
      }
      unsigned m = __ballot_sync(0xffffffffu, expect_l != 0);
      while (m) {
        const int k = __ffs(m) - 1;
        m &= m - 1;
        const uint32_t expect = __shfl_sync(0xffffffffu, expect_l, k);
        const int len = __shfl_sync(0xffffffffu, len_l, k);
        const int32_t* L = g.C + __shfl_sync(0xffffffffu, xb_l, k);
        const int64_t out = __shfl_sync(0xffffffffu, out_l, k), outx = __shfl_sync(0xffffffffu, outx_l, k),
                      outy = __shfl_sync(0xffffffffu, outy_l, k);
        uint32_t written = 0;
        for (int q = lane; q - lane < len && written < expect; q += 32 * TL_ILP) {
          int32_t z[TL_ILP], py[TL_ILP];
#pragma unroll
          for (int u = 0; u < TL_ILP; ++u) z[u] = q + 32 * u < len ? L[q + 32 * u] : -1;
#pragma unroll
          for (int u = 0; u < TL_ILP; ++u) py[u] = z[u] >= 0 ? H.find(z[u]) : -1;
#pragma unroll
          for (int u = 0; u < TL_ILP; ++u) {
            const unsigned hm = __ballot_sync(0xffffffffu, py[u] >= 0);
            const uint32_t at = written + __popc(hm & lt);
            if (py[u] >= 0 && at < expect) {
              U[out + at] = z[u];
              P[outx + at] = q + 32 * u;
              P[outy + at] = py[u];
            }
            written += __popc(hm);
          }
        }
        if (lane == 0 && written != expect) set_err(status, DEVERR_BOUNDS);
      }
    }
    __syncthreads();
  }
}

// list offsets: off[p] for canonical slots = scan of T; reverse slots share it
__global__ void k_canon_counts(DevGraph g, const uint32_t* T, int64_t* cnt) {
  int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < g.n; v += nwarps) {
    for (int64_t p = g.R[v] + lane; p < g.op[v]; p += 32) cnt[p] = 0;
    for (int64_t p = g.op[v] + lane; p < g.R[v + 1]; p += 32) cnt[p] = T[p];
  }
}
__global__ void k_all_counts(const uint32_t* T, int64_t nnz, int64_t* cnt) {
  int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += stride) cnt[p] = T[p];
}
__global__ void k_share_offsets(DevGraph g, int64_t* off) {
  int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < g.n; v += nwarps)
    for (int64_t p = g.op[v] + lane; p < g.R[v + 1]; p += 32) off[g.rev[p]] = off[p];
}

// ============================================================================
// Per-edge and per-vertex closed-form sums (Thms 4, 8, 9): one warp per row,
// canonical slots only for unordered sums.
// ============================================================================
__global__ void k_edge_sums(DevGraph g, const uint32_t* T, const unsigned long long* C4e,
                            const unsigned long long* K4e, const unsigned long long* tv,
                            const unsigned long long* C4v, const unsigned long long* K4v, AccSet acc) {
  __shared__ u128 sh[32];
  int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int ids[13] = {ACC_N5A, ACC_N11, ACC_D, ACC_N14, ACC_N6A, ACC_N12A, ACC_N19,
                       ACC_TT, ACC_N4, ACC_N9A, ACC_N7A, ACC_N15, ACC_TD};
  LocalAcc<13> la;
  la.zero();
  for (int64_t v = warp; v < g.n; v += nwarps) {
    unsigned long long dv = (unsigned long long)dg_deg(g, v), tvv = tv[v];
    for (int64_t p = g.R[v] + lane; p < g.R[v + 1]; p += 32) {
      int32_t u = g.C[p];
      unsigned long long du = (unsigned long long)dg_deg(g, u), te = T[p];
      // ordered (v -> u)
      la.v[0] += (u128)(tvv - te) * (du - 1);                       // N5 first term
      if (te >= 2) la.v[1] += ch2(te) * (dv - 3);                   // N11
      if (u > v) {                                                  // unordered
        la.v[2] += ch2(te);                                         // D
        la.v[3] += ch3(te);                                         // N14
        if (te) la.v[4] += (u128)te * (dv - 2) * (du - 2);          // N6 first term
        la.v[5] += (u128)C4e[p] * te;                               // N12 first term
        if (K4e[p]) la.v[6] += (u128)K4e[p] * (te - 2);             // N19
      }
    }
    if (lane == 0) {
      if (dv >= 2) la.v[7] += (u128)tvv * (dv - 2);                 // TT
      if (dv >= 2) la.v[8] += (u128)tvv * ch2(dv - 2);              // N4
      la.v[9] += ch2(tvv);                                          // N9 first term
      if (C4v[v]) la.v[10] += (u128)C4v[v] * (dv - 2);              // N7 first term
      if (K4v[v]) la.v[11] += (u128)K4v[v] * (dv - 3);              // N15
      la.v[12] += (u128)tvv * dv;                                   // P3+K2 / K3+K2 terms
    }
    warp_item_flush(la, ids, acc, v);
  }
  final_flush(la, ids, acc, sh);
}

// ============================================================================
// Assembly (Thm 3, App. A; Thms 4, 8-14; App. B).  All arithmetic
// modulo 2^128, which is exact because every final count is below 2^127.
// out: induced c3[4], c4[11], c5[34], then non-induced n3, n4, n5 (u128 each).
// ============================================================================
struct ConvTables {
  long long a3[4 * 4];
  long long a4[11 * 11];
  long long a5[34 * 34];
};

__device__ __forceinline__ u128 cnk(u128 n, int k) {
  // C(n, k) for k <= 5 with n < 2^64: exact in 128-bit (product of k terms / k!)
  if (n < (u128)k) return 0;
  u128 r = 1;
  for (int i = 0; i < k; ++i) r = r * (n - i) / (i + 1);
  return r;
}

// One CTA of ASM_THREADS threads per graph: graph k reads accumulator row k and
// writes result k.  Every non-induced count and every row of the conversion is
// one thread's (128-bit products and divisions by one thread took 54 us).
// basis_all (optional): per graph the four counts the runtime is linear in
// (Sec. 8's runtime fit): W, D, directed 3-paths, directed bipyramids.
static constexpr int ASM_THREADS = 64;
__global__ void __launch_bounds__(ASM_THREADS) k_assemble(const Acc128* acc_all, const unsigned long long* n_arr,
                                                         const unsigned long long* m_arr, int num_graphs,
                                                         ConvTables tabs, unsigned long long* out_all,
                                                         u128* basis_all) {
  __shared__ u128 A[ACC_COUNT], cnt[49];        // cnt: n3[4], n4[11], n5[34]
  const int t = threadIdx.x;
  for (int k = blockIdx.x; k < num_graphs; k += gridDim.x) {
    const Acc128* acc = acc_all + (int64_t)k * ACC_COUNT;
    __syncthreads();                            // the last graph's counts are read
    if (t < ACC_COUNT) A[t] = ((u128)acc[t].hi << 64) | acc[t].lo;
    __syncthreads();
    if (basis_all && t < 4)
      basis_all[(int64_t)k * 4 + t] = t == 0 ? A[ACC_W] : (t == 1 ? A[ACC_D] : (t == 2 ? A[ACC_DP] : A[ACC_DBP]));
    const u128 n = n_arr[k], m = m_arr[k];
    const u128 W = A[ACC_W], T = A[ACC_T], TT = A[ACC_TT], C4 = A[ACC_C4], D = A[ACC_D], S3 = A[ACC_S3];
    const u128 K4 = (A[ACC_K4] + A[ACC_K4H] / 4) / 3, P4 = A[ACC_P4A] - 3 * T;
    u128 v = 0;
    switch (t) {
      case 0: v = cnk(n, 3); break;
      case 1: v = n >= 2 ? m * (n - 2) : 0; break;
      case 2: v = W; break;
      case 3: v = T; break;
      case 4: v = S3; break;
      case 5: v = P4; break;
      case 6: v = TT; break;
      case 7: v = C4; break;
      case 8: v = D; break;
      case 9: v = K4; break;
      case 10: v = cnk(n, 4); break;
      case 11: v = n >= 2 ? m * cnk(n - 2, 2) : 0; break;
      case 12: v = cnk(m, 2) - W; break;
      case 13: v = n >= 3 ? W * (n - 3) : 0; break;
      case 14: v = n >= 3 ? T * (n - 3) : 0; break;
      // 5-vertex patterns 1 .. 34
      case 15: v = A[ACC_S4]; break;
      case 16: v = A[ACC_N2A] - 2 * TT; break;
      case 17: v = A[ACC_N3A] - 4 * C4 - 2 * TT - 3 * T; break;
      case 18: v = A[ACC_N4]; break;
      case 19: v = A[ACC_N5A] - 4 * D; break;
      case 20: v = A[ACC_N6A] - 2 * D; break;
      case 21: v = A[ACC_N7A] - 2 * D; break;
      case 22: v = A[ACC_N8M] - A[ACC_N8Z]; break;
      case 23: v = A[ACC_N9A] - 2 * D; break;
      case 24: v = A[ACC_N10A] - 12 * K4; break;
      case 25: v = A[ACC_N11]; break;
      case 26: v = A[ACC_N12A] - 4 * D; break;
      case 27: v = A[ACC_N13]; break;
      case 28: v = A[ACC_N14]; break;
      case 29: v = A[ACC_N15]; break;
      case 30: v = A[ACC_N16A] - 12 * K4; break;
      case 31: v = A[ACC_N17] + A[ACC_N17H] / 2; break;
      case 32: v = A[ACC_N18] + A[ACC_N18H] / 4; break;
      case 33: v = A[ACC_N19]; break;
      case 34: v = A[ACC_N20] + A[ACC_N20H] / 3; break;
      case 35: v = A[ACC_N21]; break;
      case 36: v = cnk(n, 5); break;
      case 37: v = n >= 2 ? m * cnk(n - 2, 3) : 0; break;
      case 38: v = n >= 4 ? (cnk(m, 2) - W) * (n - 4) : 0; break;
      case 39: v = n >= 3 ? W * cnk(n - 3, 2) : 0; break;
      case 40: v = n >= 3 ? T * cnk(n - 3, 2) : 0; break;
      case 41: v = n >= 4 ? S3 * (n - 4) : 0; break;
      case 42: v = n >= 4 ? P4 * (n - 4) : 0; break;
      case 43: v = n >= 4 ? TT * (n - 4) : 0; break;
      case 44: v = n >= 4 ? C4 * (n - 4) : 0; break;
      case 45: v = n >= 4 ? D * (n - 4) : 0; break;
      case 46: v = n >= 4 ? K4 * (n - 4) : 0; break;
      case 47: v = W * m - A[ACC_D2D] - A[ACC_DNBR] + 2 * W + 3 * T; break;
      case 48: v = T * m - A[ACC_TD] + 3 * T; break;
    }
    if (t < 49) cnt[t] = v;
    __syncthreads();
    // induced = A^-1 * non-induced (signed integer matrix, arithmetic mod 2^128)
    if (t < 49) {
      const int first = t < 4 ? 0 : (t < 15 ? 4 : 15), len = t < 4 ? 4 : (t < 15 ? 11 : 34);
      const long long* row = (t < 4 ? tabs.a3 : (t < 15 ? tabs.a4 : tabs.a5)) + (t - first) * len;
      u128 s = 0;
      for (int j = 0; j < len; ++j) s += (u128)(__int128)row[j] * cnt[first + j];
      u128* o = (u128*)(out_all + (int64_t)k * 2 * 98);
      o[t] = s;
      o[49 + t] = cnt[t];
    }
  }
}

// ============================================================================
// Host orchestration.
// ============================================================================
static unsigned grid_for(int64_t work, int threads, int sms) {
  int64_t b = (work + threads - 1) / threads;
  int64_t cap = (int64_t)sms * 8;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (unsigned)b;
}

// batch bookkeeping: graph of every rank-space vertex; vertices and edges per graph
__global__ void k_graph_of_vertex(const int64_t* voff, int num_graphs, const int32_t* rank, int64_t n, int32_t* vg) {
  int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += stride) {
    int lo = 0, hi = num_graphs;          // last k with voff[k] <= u
    while (hi - lo > 1) { int mid = (lo + hi) >> 1; if (voff[mid] <= u) lo = mid; else hi = mid; }
    vg[rank[u]] = lo;
  }
}
__global__ void k_graph_sizes(const int64_t* voff, const int64_t* rp, int num_graphs, unsigned long long* n_arr,
                              unsigned long long* m_arr) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= num_graphs) return;
  n_arr[k] = (unsigned long long)(voff[k + 1] - voff[k]);
  m_arr[k] = (unsigned long long)((rp[voff[k + 1]] - rp[voff[k]]) / 2);
}

__global__ void k_set_sizes(unsigned long long n, unsigned long long m, unsigned long long* n_arr,
                            unsigned long long* m_arr) {
  *n_arr = n;
  *m_arr = m;
}

// item lists of pass A/B: vertices by out-degree class
// small / large: d+ up to small_max or above (vertices with d+ >= 2); the
// small ones are also split by d- for the clique pass: up to warp_din in wsmall
// (one warp each), the rest in csmall (one CTA each).
// The clique pass takes only the owned vertices (wsmall, csmall, clarge);
// the triangle pass takes every vertex (small, large).
__global__ void k_split_items(DevGraph g, int32_t* small, int32_t* large, int32_t* wsmall, int32_t* csmall,
                              int32_t* clarge, unsigned long long* cnts, int small_max, int warp_din, Owner own) {
  int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < g.n; k += stride) {
    int64_t x = g.n - 1 - k;
    int64_t d = g.R[x + 1] - g.op[x];
    if (d < 2) continue;
    const bool mine = own.owns(x);
    if (d <= small_max) {
      small[atomicAdd(&cnts[0], 1ull)] = (int32_t)x;
      if (!mine) continue;
      if (g.op[x] - g.R[x] <= warp_din) wsmall[atomicAdd(&cnts[2], 1ull)] = (int32_t)x;
      else csmall[atomicAdd(&cnts[3], 1ull)] = (int32_t)x;
    } else {
      large[atomicAdd(&cnts[1], 1ull)] = (int32_t)x;
      if (mine) clarge[atomicAdd(&cnts[4], 1ull)] = (int32_t)x;
    }
  }
}

// max over vertices of d+ x ceil(d- / 64) (words of the D bit sets) and of d+;
// the largest graph's vertices
__global__ void k_clique_dims(DevGraph g, const unsigned long long* n_arr, int num_graphs, unsigned long long* out) {
  int64_t stride = (int64_t)gridDim.x * blockDim.x;
  unsigned long long mw = 0, md = 0;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < g.n; x += stride) {
    unsigned long long dp = (unsigned long long)(g.R[x + 1] - g.op[x]);
    unsigned long long dm = (unsigned long long)(g.op[x] - g.R[x]);
    if (dp >= 2) {
      unsigned long long wds = dp * ((dm + 63) / 64);
      if (wds > mw) mw = wds;
    }
    if (dp > md) md = dp;
  }
  unsigned long long mg = 0;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < num_graphs; k += stride)
    if (n_arr[k] > mg) mg = n_arr[k];
  if (mw) atomicMax(&out[0], mw);
  if (md) atomicMax(&out[1], md);
  if (mg) atomicMax(&out[2], mg);
}


// ---------------------------------------------------------------- buffers
// The device-buffer cache declared in internal.h.
static constexpr size_t kCacheCap = (size_t)8 << 30;

class BufCache {
 public:
  void* get(int dev, size_t b, size_t most, size_t* got) {
    std::lock_guard<std::mutex> lk(mu_);
    auto& m = free_[dev & 63];
    auto it = m.lower_bound(b);
    if (it == m.end() || it->first > most) return nullptr;
    void* p = it->second;
    *got = it->first;
    bytes_[dev & 63] -= it->first;
    m.erase(it);
    return p;
  }
  void put(int dev, void* p, size_t b, bool hold) {
    if (!hold || b < DevBuf::HOLD_BYTES) {
      std::lock_guard<std::mutex> lk(mu_);
      if (bytes_[dev & 63] + b <= kCacheCap) {
        free_[dev & 63].emplace(b, p);
        bytes_[dev & 63] += b;
        return;
      }
    }
    cudaFree(p);
  }
  void clear(int dev) {
    std::multimap<size_t, void*> m;
    {
      std::lock_guard<std::mutex> lk(mu_);
      m.swap(free_[dev & 63]);
      bytes_[dev & 63] = 0;
    }
    for (auto& kv : m) cudaFree(kv.second);
  }

 private:
  std::mutex mu_;
  std::multimap<size_t, void*> free_[64];
  size_t bytes_[64] = {};
};
// never destroyed: a handle freed during process exit may still come here
static BufCache& buf_cache() {
  static BufCache* c = new BufCache;
  return *c;
}

static thread_local CacheScope* t_scope = nullptr;
CacheScope::CacheScope(cudaStream_t st) : s(st), prev(t_scope) { t_scope = this; }
CacheScope::~CacheScope() {
  cudaStreamSynchronize(s);
  for (auto& b : pending) buf_cache().put(b.dev, b.p, b.bytes, b.hold);
  t_scope = prev;
}

void DevBuf::give_back() {
  if (p) buf_cache().put(dev, p, bytes, hold);
  p = nullptr;
  bytes = 0;
}
void DevBuf::release() {
  if (!p) return;
  if (t_scope) t_scope->pending.push_back({p, bytes, dev, hold});
  else buf_cache().put(dev, p, bytes, hold);
  p = nullptr;
  bytes = 0;
}
cudaError_t DevBuf::alloc(size_t b) {
  release();
  b = ((b > 0 ? b : 16) + 255) & ~(size_t)255;
  cudaGetDevice(&dev);
  size_t got = 0;
  if ((p = buf_cache().get(dev, b, hold ? b + b / 8 : 2 * b, &got)) != nullptr) {
    bytes = got;
    return cudaSuccess;
  }
  cudaError_t e = cudaMalloc(&p, b);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    buf_cache().clear(dev);
    e = cudaMalloc(&p, b);
  }
  if (e != cudaSuccess) {
    p = nullptr;
    return e;
  }
  bytes = b;
  return cudaSuccess;
}

#define ESC_TRY(x) do { cudaError_t _e = (x); if (_e != cudaSuccess) return _e; } while (0)

// Side streams and events for the concurrent phases; events order them after /
// before the caller's stream.  Creating them costs more than a small census
// computes (four streams, 0.1 ms), so sets are kept for later censuses, at most
// kStreamSets per device; a census holds one to itself.  A set goes back after
// its streams have drained: on an early error return the caller's stream may
// not have joined them, and the buffers their kernels use go back to the cache
// only after this destructor (they are declared before the StreamSet).
struct SideStreams {
  cudaStream_t st[4] = {nullptr, nullptr, nullptr, nullptr};
  cudaEvent_t fork = nullptr, join[4] = {nullptr, nullptr, nullptr, nullptr};
};
static constexpr size_t kStreamSets = 8;
static std::mutex g_sides_mu;
static std::vector<SideStreams>& side_pool(int dev) {
  static auto* pools = new std::vector<SideStreams>[64];
  return pools[dev & 63];
}
struct StreamSet {
  SideStreams ss;
  int count = 0, dev = 0;
  ~StreamSet() {
    if (!count) return;
    bool ok = count == 4;
    for (int i = 0; i < count; ++i) ok = cudaStreamSynchronize(ss.st[i]) == cudaSuccess && ok;
    if (ok) {
      std::lock_guard<std::mutex> lk(g_sides_mu);
      auto& pool = side_pool(dev);
      if (pool.size() < kStreamSets) {
        pool.push_back(ss);
        return;
      }
    }
    for (int i = 0; i < 4; ++i) {
      if (ss.st[i]) cudaStreamDestroy(ss.st[i]);
      if (ss.join[i]) cudaEventDestroy(ss.join[i]);
    }
    if (ss.fork) cudaEventDestroy(ss.fork);
  }
  // urgent[i] != 0: the device's greatest (most urgent) priority, else its least
  // (the same flags at every call)
  cudaError_t create(const int (&urgent)[4]) {
    cudaGetDevice(&dev);
    {
      std::lock_guard<std::mutex> lk(g_sides_mu);
      auto& pool = side_pool(dev);
      if (!pool.empty()) {
        ss = pool.back();
        pool.pop_back();
        count = 4;
        return cudaSuccess;
      }
    }
    int least = 0, greatest = 0;
    cudaDeviceGetStreamPriorityRange(&least, &greatest);
    cudaError_t e = cudaEventCreateWithFlags(&ss.fork, cudaEventDisableTiming);
    count = 0;
    for (int i = 0; i < 4 && e == cudaSuccess; ++i) {
      e = cudaEventCreateWithFlags(&ss.join[i], cudaEventDisableTiming);
      if (e == cudaSuccess)
        e = cudaStreamCreateWithPriority(&ss.st[i], cudaStreamNonBlocking, urgent[i] ? greatest : least);
      if (e == cudaSuccess) count = i + 1;
    }
    return e;
  }
  // the side streams wait for the work enqueued on `from` so far
  cudaError_t fork_from(cudaStream_t from) {
    cudaError_t r = cudaEventRecord(ss.fork, from);
    for (int i = 0; i < count && r == cudaSuccess; ++i) r = cudaStreamWaitEvent(ss.st[i], ss.fork, 0);
    return r;
  }
  // `into` waits for everything enqueued on the side streams
  cudaError_t join_into(cudaStream_t into) {
    cudaError_t r = cudaSuccess;
    for (int i = 0; i < count && r == cudaSuccess; ++i) {
      r = cudaEventRecord(ss.join[i], ss.st[i]);
      if (r == cudaSuccess) r = cudaStreamWaitEvent(into, ss.join[i], 0);
    }
    return r;
  }
};

// Lets kernel k use all of the device's opt-in shared memory (less its static
// shared memory) as dynamic shared memory.  Every call sets the same value, so
// censuses running on other host threads never lower the limit between this
// thread's setting and its launch.
static cudaError_t allow_max_smem(const void* k, int optin) {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, k);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

// Launch shape of the heavy pair items: CTAs of `threads` threads grouped in
// clusters of `cs`, `nclusters` clusters (one counter array each), as many
// clusters as the SMs hold.  ESC_PAIR_SHAPE, ESC_PAIR_CLUSTER and
// ESC_PAIR_CLUSTERS override the choice (tuning only; results are the same).
struct PairPlan {
  int cs = 1, threads = 512, nclusters = 0;
  int shape = 1;                               // kernel instance, see ESC_PAIR_SHAPES
  int win_words = 0;                           // shared-memory window (clusters of one CTA)
  int64_t wlo = 0;                             // its first rank
  bool windowed = false;                       // k_pairs_win: every rank below jbig in successive windows
};

static int env_int(const char* name, int dflt) {
  const char* v = getenv(name);
  if (!v || !*v) return dflt;
  int x = atoi(v);
  return x > 0 ? x : dflt;
}

// Launch shapes of the heavy-item kernel: (threads, CTAs per SM) = (512, 3)
// at 40 registers, (512, 2) at 64, (1024, 1) at 64.
#define ESC_PAIR_SHAPES(X) X(0, 512, 3) X(1, 512, 2) X(2, 1024, 1)
static const void* pairs_grp_fn(bool big, int shape) {
#define ESC_PG(k, t, b) if (shape == k) return big ? (const void*)k_pairs_grp<true, t, b> : (const void*)k_pairs_grp<false, t, b>;
  ESC_PAIR_SHAPES(ESC_PG)
#undef ESC_PG
  return nullptr;
}

// The windowed form (k_pairs_win, the default): one 1024-thread CTA per SM,
// the window as wide as shared memory allows, but no wider than the ranks
// [n0, jbig) need.
static cudaError_t plan_pair_windows(const void* k, int sms, int64_t n0, int64_t jbig, int smem_optin, PairPlan* plan) {
  cudaFuncAttributes fa;
  ESC_TRY(cudaFuncGetAttributes(&fa, k));
  ESC_TRY(allow_max_smem(k, smem_optin));     // the limit is the same for every graph
  const int bytes = (smem_optin - (int)fa.sharedSizeBytes - 1024) & ~15;
  const int64_t want = ((jbig - n0 + 2) / 2 + 3) & ~(int64_t)3;     // words covering [n0, jbig) in one window
  plan->windowed = true;
  plan->threads = 1024;
  plan->cs = 1;
  plan->shape = 0;
  plan->win_words = (int)std::min<int64_t>(bytes / 4, want);
  // ESC_PAIR_WIN_WORDS: narrower windows, so that small graphs take many (tests)
  plan->win_words = std::min(plan->win_words, env_int("ESC_PAIR_WIN_WORDS", plan->win_words));
  plan->win_words = std::max(4, plan->win_words & ~3);          // whole 16-byte vectors
  plan->wlo = jbig - 2 * (int64_t)plan->win_words;
  int per_sm = 0;
  ESC_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, plan->threads, plan->win_words * 4));
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  plan->nclusters = sms * per_sm;
  return cudaSuccess;
}

static cudaError_t plan_pair_clusters(bool big, int sms, size_t arr_bytes, int64_t n0, int64_t jbig, int smem_optin,
                                      bool union_of_graphs, PairPlan* plan) {
  // ESC_PAIR_WINDOW: 3 every rank in successive windows (k_pairs_win, the
  // default for one graph); 2 one window over the top ranks and tagged global
  // counters below it (the default for a batch: in a block-diagonal union the
  // ranks of one member are spread over the whole rank range, so an item
  // would walk and write nearly every window for a few hundred wedges); 1 no
  // window.  The single window takes one 1024-thread CTA per SM (its window
  // is twice as wide as two 512-thread CTAs' each); without the window,
  // (512, 2).
  const int wmode = env_int("ESC_PAIR_WINDOW", union_of_graphs ? 2 : 3);
  if (wmode >= 3 && env_int("ESC_PAIR_CLUSTER", 1) == 1) {
    const void* kw = big ? (const void*)k_pairs_win<true> : (const void*)k_pairs_win<false>;
    return plan_pair_windows(kw, sms, n0, jbig, smem_optin, plan);
  }
  const bool window = env_int("ESC_PAIR_CLUSTER", 1) == 1 && wmode != 1;
  plan->shape = std::min(2, env_int("ESC_PAIR_SHAPE", window ? 3 : 2) - 1);
  plan->threads = plan->shape == 2 ? 1024 : 512;
  const void* k = pairs_grp_fn(big, plan->shape);
  int dev = 0, l2 = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
  ESC_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  const size_t budget = (size_t)std::max(l2, 1 << 20) / 2;
  const int64_t kmax = std::max<int64_t>(1, (int64_t)(budget / std::max<size_t>(arr_bytes, 1)));
  // the window: what shared memory leaves per CTA, for clusters of one CTA
  // (ESC_PAIR_WINDOW=1 turns it off)
  plan->win_words = 0;
  plan->wlo = jbig;
  if (window) {
    cudaFuncAttributes fa;
    ESC_TRY(cudaFuncGetAttributes(&fa, k));
    const int per_sm_target = plan->threads == 1024 ? 1 : 2;
    int bytes = (smem_optin / per_sm_target - (int)fa.sharedSizeBytes - 1024) & ~15;
    int64_t want = std::max<int64_t>(0, (jbig - n0 + 1) / 2);        // words covering every countable rank
    plan->win_words = (int)std::max<int64_t>(0, std::min<int64_t>(bytes / 4, want));
    plan->wlo = std::max<int64_t>(n0, jbig - 2 * (int64_t)plan->win_words);
    if (plan->win_words > 0) ESC_TRY(allow_max_smem(k, smem_optin));   // the limit is the same for every graph
  }
  int per_sm = 1;
  ESC_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, plan->threads, plan->win_words * 4));
  const int64_t total = (int64_t)sms * std::max(1, per_sm);
  // clusters of one CTA with the shared-memory window by default; without
  // it, clusters of 4 CTAs were fastest on the Chung-Lu and R-MAT workloads,
  // ahead of the larger clusters whose fewer arrays stay in L2 (the items in
  // flight matter more than L2 hits); kmax, the cluster count that would fit
  // L2, is kept for the record of the plan
  int cs = env_int("ESC_PAIR_CLUSTER", plan->win_words > 0 ? 1 : 4);
  (void)kmax;
  plan->nclusters = (int)std::max<int64_t>(1, total / cs);
  // never more clusters than can be resident at once
  for (;; cs >>= 1) {
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    lc.gridDim = dim3((unsigned)(plan->nclusters * cs));
    lc.blockDim = dim3((unsigned)plan->threads);
    lc.dynamicSmemBytes = (size_t)plan->win_words * 4;
    lc.attrs = at;
    lc.numAttrs = 1;
    int active = 0;
    cudaError_t e = cudaOccupancyMaxActiveClusters(&active, k, &lc);
    if (e == cudaSuccess && active > 0) {
      plan->nclusters = std::min(plan->nclusters, active);
      break;
    }
    cudaGetLastError();
    if (cs == 1) return e == cudaSuccess ? cudaErrorInvalidConfiguration : e;
    plan->nclusters *= 2;                       // the same CTAs in half-size clusters
  }
  plan->cs = cs;
  plan->nclusters = std::min(plan->nclusters, env_int("ESC_PAIR_CLUSTERS", plan->nclusters));
  return cudaSuccess;
}

static cudaError_t launch_pairs_grp(bool big, const PairPlan& plan, const DevGraph& g, const unsigned long long* items,
                                    int64_t nitems, unsigned long long* qctr, const TagScratch& ts,
                                    const TriLists& tl3, const uint32_t* T, const CoreView& cv, const AccSet& accs,
                                    const PairTasks& pt, cudaStream_t s) {
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = plan.cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  lc.gridDim = dim3((unsigned)(plan.nclusters * plan.cs));
  lc.blockDim = dim3((unsigned)plan.threads);
  lc.dynamicSmemBytes = (size_t)plan.win_words * 4;
  lc.stream = s;
  lc.attrs = at;
  lc.numAttrs = 1;
  cudaError_t e = cudaErrorInvalidValue;
#define ESC_PG(k, t, b)                                                                                   \
  if (plan.shape == k)                                                                                    \
    e = big ? cudaLaunchKernelEx(&lc, k_pairs_grp<true, t, b>, g, items, nitems, qctr, ts, tl3, T, cv, accs, pt, \
                                 plan.wlo, plan.win_words)                                                      \
            : cudaLaunchKernelEx(&lc, k_pairs_grp<false, t, b>, g, items, nitems, qctr, ts, tl3, T, cv, accs, pt, \
                                 plan.wlo, plan.win_words);
  ESC_PAIR_SHAPES(ESC_PG)
#undef ESC_PG
  note_launch();
  return e;
}

// The dense core: vertices of degree CORE_MIN_DEG (estimate.h) or more, at most CORE_CAP
// of a single graph, in graphs (or unions) of at least CORE_MIN_D diamonds and
// CORE_D_PER_ENTRY per adjacency entry.  Below that the sweeps' diamonds cost
// less than the core's launches and passes over the graph (census, ms, without
// and with a core): ER(800, 0.15), 8e6 diamonds, 1.69 / 1.73; ER(500, 0.3),
// 4e7 (503 per entry), 2.22 / 1.83; R-MAT 11, 2e7 (387), 3.62 / 2.07;
// Chung-Lu n = 120,000, 5e8 (401), 18.2 / 16.4; Chung-Lu 2.3 n = 250,000, 5e8
// (134), 52.5 / 52.7; Chung-Lu 2.5 n = 500,000, 9e7 (11), 97.5 / 100.1.
// The degree limit hardly matters between 16 and 64 (R-MAT 16: 38.5 to 39.0 ms,
// 96: 45.2), the cap does on large graphs (R-MAT 19: 8,192 482 ms, 16,384 383,
// 32,768 384, 49,152 385; R-MAT 22: 16,384 15.0 s, 32,768 13.0 s); W takes 2 or 4
// bytes x cap^2.
static constexpr int CORE_CAP = 32768;
static constexpr unsigned long long CORE_MIN_D = 1ull << 24, CORE_D_PER_ENTRY = 160;

// App. B's matrices are constants of the pattern catalogue (the embedding
// counts take the host 0.85 ms): built once per process.
static const ConvTables& conversion_tables() {
  static const ConvTables tabs = [] {
    ConvTables t;
    conversion_inverse(3, t.a3);
    conversion_inverse(4, t.a4);
    conversion_inverse(5, t.a5);
    return t;
  }();
  return tabs;
}

cudaError_t run_census(const int64_t* rp, const int32_t* col, int64_t n, int64_t nnz, const CensusConfig& cfg,
                       unsigned long long* d_out, unsigned* d_status, PerElement* pe_out, Oriented* or_out,
                       cudaStream_t s) {
  CacheScope cache_scope(s);                    // destroyed last: the buffers below return after the stream drains
  const int sms = cfg.sms > 0 ? cfg.sms : 1;
  int smem_optin = 0;
  {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  }
  // phase k is timed by events 2k (begin) and 2k+1 (end) on the stream that runs it
  // Phase boundaries: CUDA events for the phase times, and NVTX ranges (a
  // profiler's timeline shows each phase's launches under its name).
  static const char* const kPhaseNames[9] = {"orient", "triangles", "cliques", "cycles4", "tri_lists",
                                             "pairs", "wheels", "cycles5", "assemble"};
  auto mark = [&](int k, int end, cudaStream_t st) {
    int i = 2 * k + end;
    if (cfg.phase_events && i < cfg.num_phase_events) cudaEventRecord(cfg.phase_events[i], st);
#if ESC_HAVE_NVTX
    if (!end) nvtxRangePushA(kPhaseNames[k]);
    else nvtxRangePop();
#else
    (void)kPhaseNames;
#endif
  };
  mark(0, 0, s);
  // ---------------- orientation (Sec. 3.2)
  DevBuf arena_buf;
  DeviceArena arena;
  int64_t nk = (n > nnz ? n : nnz) + 16;
  size_t arena_bytes = (size_t)nk * 8 * 2 + (size_t)(n + 16) * 8 + (size_t)(nk / 4096 + 2) * 256 * 8 * 2 + (1 << 22);
  ESC_TRY(arena_buf.alloc(arena_bytes));
  arena.base = arena_buf.as<char>();
  arena.cap = arena_bytes;

  DevBuf b_perm, b_rank, b_R, b_C, b_op, b_rev;
  for (DevBuf* b : {&b_perm, &b_rank, &b_R, &b_C, &b_op, &b_rev}) b->hold = or_out != nullptr;
  ESC_TRY(b_perm.alloc(sizeof(int32_t) * (n + 1)));
  ESC_TRY(b_rank.alloc(sizeof(int32_t) * (n + 1)));
  ESC_TRY(b_R.alloc(sizeof(int64_t) * (n + 1)));
  ESC_TRY(b_C.alloc(sizeof(int32_t) * (nnz + 1)));
  ESC_TRY(b_op.alloc(sizeof(int64_t) * (n + 1)));
  ESC_TRY(b_rev.alloc(sizeof(int64_t) * (nnz + 1)));
  Oriented o;
  o.perm = b_perm.as<int32_t>();
  o.rank = b_rank.as<int32_t>();
  o.R = b_R.as<int64_t>();
  o.C = b_C.as<int32_t>();
  o.op = b_op.as<int64_t>();
  o.rev = b_rev.as<int64_t>();
  ESC_TRY(orient(rp, col, n, nnz, o, arena, s, sms));
  mark(0, 1, s);

  DevGraph g{n, nnz, o.R, o.C, o.op, o.rev, o.C};
  const int TPB = 256;
  // ---------------- per-element arrays and accumulators
  DevBuf b_T, b_K4e, b_C4e, b_tv, b_C4v, b_K4v, b_acc, b_ctr;
  for (DevBuf* b : {&b_T, &b_C4e, &b_K4e, &b_tv, &b_C4v, &b_K4v}) b->hold = pe_out != nullptr;
  ESC_TRY(b_T.alloc(sizeof(uint32_t) * (nnz + 1)));
  ESC_TRY(b_K4e.alloc(sizeof(unsigned long long) * (nnz + 1)));
  ESC_TRY(b_C4e.alloc(sizeof(unsigned long long) * (nnz + 1)));
  ESC_TRY(b_tv.alloc(sizeof(unsigned long long) * (n + 1)));
  ESC_TRY(b_C4v.alloc(sizeof(unsigned long long) * (n + 1)));
  ESC_TRY(b_K4v.alloc(sizeof(unsigned long long) * (n + 1)));
  const int G = cfg.num_graphs > 1 ? cfg.num_graphs : 1;
  ESC_TRY(b_acc.alloc(sizeof(Acc128) * ACC_COUNT * G));
  ESC_TRY(b_ctr.alloc(sizeof(unsigned long long) * 16));
  uint32_t* T = b_T.as<uint32_t>();
  unsigned long long *K4e = b_K4e.as<unsigned long long>(), *C4e = b_C4e.as<unsigned long long>();
  unsigned long long *tv = b_tv.as<unsigned long long>(), *C4v = b_C4v.as<unsigned long long>(),
                     *K4v = b_K4v.as<unsigned long long>();
  Acc128* acc = b_acc.as<Acc128>();
  unsigned long long* ctr = b_ctr.as<unsigned long long>();
  cudaMemsetAsync(T, 0, sizeof(uint32_t) * (nnz + 1), s);
  cudaMemsetAsync(K4e, 0, sizeof(unsigned long long) * (nnz + 1), s);
  cudaMemsetAsync(C4e, 0, sizeof(unsigned long long) * (nnz + 1), s);
  cudaMemsetAsync(acc, 0, sizeof(Acc128) * ACC_COUNT * G, s);
  DevBuf b_vg, b_narr, b_marr;
  ESC_TRY(b_narr.alloc(sizeof(unsigned long long) * G));
  ESC_TRY(b_marr.alloc(sizeof(unsigned long long) * G));
  AccSet accs{acc, nullptr};
  if (G > 1) {
    ESC_TRY(b_vg.alloc(sizeof(int32_t) * (n + 1)));
    if (n > 0)
      (k_graph_of_vertex<<<grid_for(n, TPB, sms), TPB, 0, s>>>(cfg.d_vtx_offsets, G, o.rank, n, b_vg.as<int32_t>()),
       note_launch());
    (k_graph_sizes<<<(G + 127) / 128, 128, 0, s>>>(cfg.d_vtx_offsets, rp, G, b_narr.as<unsigned long long>(),
                                                   b_marr.as<unsigned long long>()), note_launch());
    accs.vg = b_vg.as<int32_t>();
  } else {
    (k_set_sizes<<<1, 1, 0, s>>>((unsigned long long)n, (unsigned long long)(nnz / 2), b_narr.as<unsigned long long>(),
                                 b_marr.as<unsigned long long>()), note_launch());
  }
  cudaMemsetAsync(ctr, 0, sizeof(unsigned long long) * 16, s);
  // a census split over parts: the sweeps take the owned items only, and the
  // sums of the phases every part repeats (degree sums, triangles) count on
  // part 0 alone (the others add them to a discarded row)
  const Owner own{cfg.part, std::max(1, cfg.parts)};
  AccSet acc_rep = accs;
  DevBuf b_junk;
  if (own.part != 0) {
    ESC_TRY(b_junk.alloc(sizeof(Acc128) * ACC_COUNT * G));
    acc_rep.base = b_junk.as<Acc128>();
  }

  if (n > 0) (k_vertex_basic<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(g, acc_rep), note_launch());

  // ---------------- item lists for the out-neighbourhood passes
  DevBuf b_small, b_large, b_wsmall, b_csmall, b_clarge, b_dims;
  ESC_TRY(b_small.alloc(sizeof(int32_t) * (n + 1)));
  ESC_TRY(b_large.alloc(sizeof(int32_t) * (n + 1)));
  ESC_TRY(b_wsmall.alloc(sizeof(int32_t) * (n + 1)));
  ESC_TRY(b_csmall.alloc(sizeof(int32_t) * (n + 1)));
  ESC_TRY(b_clarge.alloc(sizeof(int32_t) * (n + 1)));
  ESC_TRY(b_dims.alloc(sizeof(unsigned long long) * 3));
  cudaMemsetAsync(b_dims.p, 0, sizeof(unsigned long long) * 3, s);
  if (n > 0) {
    (k_split_items<<<grid_for(n, TPB, sms), TPB, 0, s>>>(g, b_small.as<int32_t>(), b_large.as<int32_t>(),
                                                          b_wsmall.as<int32_t>(), b_csmall.as<int32_t>(),
                                                          b_clarge.as<int32_t>(), ctr, SMALL_DPLUS,
                                                          std::min(CLQ_WARP_DIN, env_int("ESC_CLQ_WARP_DIN", CLQ_WARP_DIN)),
                                                          own), note_launch());
    (k_clique_dims<<<grid_for(n, TPB, sms), TPB, 0, s>>>(g, b_narr.as<unsigned long long>(), G,
                                                         b_dims.as<unsigned long long>()), note_launch());
  }
  unsigned long long hcnt[16] = {0}, dims[3] = {0, 0, 0};
  cudaMemcpyAsync(hcnt, ctr, sizeof(hcnt), cudaMemcpyDeviceToHost, s);
  cudaMemcpyAsync(dims, b_dims.p, sizeof(dims), cudaMemcpyDeviceToHost, s);
  ESC_TRY(cudaStreamSynchronize(s));
  int64_t nsmall = (int64_t)hcnt[0], nlarge = (int64_t)hcnt[1];
  int64_t nwsmall = (int64_t)hcnt[2], ncsmall = (int64_t)hcnt[3], nclarge = (int64_t)hcnt[4];
  int dmax = (int)dims[1];
  if (dmax < SMALL_DPLUS + 1) dmax = SMALL_DPLUS + 1;
  cudaMemsetAsync(ctr, 0, sizeof(unsigned long long) * 16, s);

  // ---------------- pass A: triangles
  mark(1, 0, s);
  int hcap_a = pow2_at_least(2 * dmax);
  size_t smem_a = sizeof(int32_t) * (2 * (size_t)hcap_a) + sizeof(uint32_t) * dmax;
  int grid_sweep = sms * (cfg.cta_per_sm > 0 ? cfg.cta_per_sm : 2);
  if (nsmall > 0)
    (k_tri_small<<<grid_for(nsmall * 32, TPB, sms), TPB, 0, s>>>(g, b_small.as<int32_t>(), nsmall, T, acc_rep),
     note_launch());
  if (nlarge > 0) {
    if (smem_a > 48 * 1024) ESC_TRY(allow_max_smem((const void*)k_tri_large, smem_optin));
    (k_tri_large<<<(unsigned)std::min<int64_t>(grid_sweep, nlarge), 512, smem_a, s>>>(
        g, b_large.as<int32_t>(), nlarge, ctr + 0, T, acc_rep, hcap_a), note_launch());
  }
  if (n > 0) {
    (k_sym_T<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(g, T), note_launch());
    (k_vertex_from_edges_T<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(g, T, tv), note_launch());
  }
  mark(1, 1, s);

  // ---------------- everything the concurrent phases need is sized and
  // allocated here, so no branch below waits on the host
  int dev = 0;
  cudaGetDevice(&dev);
  // pass B inputs
  // CTA items: every large out-neighbourhood, then the small ones with many
  // in-neighbours; the other small ones go to the warp kernel
  int64_t nitems_b = nclarge + ncsmall;
  DevBuf b_items, b_D;
  ESC_TRY(b_items.alloc(sizeof(int32_t) * (nitems_b + 1)));
  if (nclarge) cudaMemcpyAsync(b_items.p, b_clarge.p, sizeof(int32_t) * nclarge, cudaMemcpyDeviceToDevice, s);
  if (ncsmall)
    cudaMemcpyAsync(b_items.as<int32_t>() + nclarge, b_csmall.p, sizeof(int32_t) * ncsmall, cudaMemcpyDeviceToDevice,
                    s);
  // out-degrees up to dsplit keep the bit matrix in shared memory; the few
  // larger ones (dense graphs) use a per-CTA region of global memory
  int dsplit = dmax;
  while (dsplit > SMALL_DPLUS + 1 &&
         clique_space(dsplit) + 1024 + sizeof(CliqueWarp) * CLQ_MAX_WARPS > (size_t)smem_optin)
    --dsplit;
  const int dmax_s = std::min(dmax, dsplit);
  int hcap_b = pow2_at_least(2 * dmax_s);
  size_t smem_b = clique_space(dmax_s) + sizeof(CliqueWarp) * 8;
  ESC_TRY(allow_max_smem((const void*)k_clique_large<false>, smem_optin));
  // as many 256-thread CTAs per SM as registers and the bit matrix allow;
  // one 512-thread CTA per SM when fewer than two fit (large bit matrices)
  int clq_threads = 256, clq_per_sm = 1;
  ESC_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&clq_per_sm, k_clique_large<false>, clq_threads, smem_b));
  if (clq_per_sm < 2) {
    smem_b = clique_space(dmax_s) + sizeof(CliqueWarp) * CLQ_MAX_WARPS;
    clq_threads = 512;
    clq_per_sm = 1;
  }
  const int blocks_b = sms * std::min(clq_per_sm, 4);
  unsigned long long dwords = dims[0] > 0 ? dims[0] : 1;
  ESC_TRY(b_D.alloc(sizeof(uint64_t) * dwords * blocks_b));
  DevBuf b_Gq;
  int blocks_g = 0;
  int64_t gwords = 0;
  if (dmax > dsplit) {
    gwords = (int64_t)((clique_space(dmax) + 7) / 8);
    // at most one CTA per SM, and at most 8 GiB of work space in all
    blocks_g = (int)std::max<int64_t>(1, std::min<int64_t>(sms, ((int64_t)8 << 30) / (8 * gwords)));
    ESC_TRY(b_Gq.alloc(sizeof(uint64_t) * (size_t)gwords * blocks_g));
  }
  CliqueScratch cs{b_D.as<uint64_t>(), (int64_t)dwords, b_Gq.as<uint64_t>(), gwords};

  // sweep scratch: one set per concurrent sweep (4-cycles; pairs and the
  // tagged 5-cycle counters are sized below, once the largest degree is known)
  // With four_only, only the 4-cycle sweep runs; the lists, pairs, wheels and
  // 5-cycles (and their work space) are skipped.
  const bool five = !cfg.four_only;
  DevBuf b_cntA, b_cntB, b_cntC, b_cntD, b_tlD;

  // common-neighbour list offsets and sizes
  DevBuf b_off, b_offp, b_U, b_P, b_gh;
  ESC_TRY(b_off.alloc(sizeof(int64_t) * (nnz + 2)));
  ESC_TRY(b_offp.alloc(sizeof(int64_t) * (nnz + 2)));
  int64_t* off = b_off.as<int64_t>();
  int64_t* offp = b_offp.as<int64_t>();
  int64_t ulen = 0, plen = 0;
  if (five) {
    if (n > 0) (k_canon_counts<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(g, T, off), note_launch());
    ESC_TRY(exclusive_scan_i64(off, off, nnz, true, arena, s));
    if (n > 0) (k_all_counts<<<grid_for(nnz, TPB, sms), TPB, 0, s>>>(T, nnz, offp), note_launch());
    ESC_TRY(exclusive_scan_i64(offp, offp, nnz, true, arena, s));
    cudaMemcpyAsync(&ulen, off + nnz, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    cudaMemcpyAsync(&plen, offp + nnz, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
  }
  // items of the pair, 4-cycle and 5-cycle sweeps (light / medium / heavy lists)
  DevBuf b_plist, b_list4, b_list5, b_pctr;
  const size_t list_b = sizeof(unsigned long long) * IT_LISTS * (size_t)(n + 1);
  ESC_TRY(b_plist.alloc(five ? list_b : 16));
  ESC_TRY(b_list4.alloc(list_b));
  ESC_TRY(b_list5.alloc(five ? list_b : 16));
  ESC_TRY(b_pctr.alloc(sizeof(unsigned long long) * 3 * IT_CNT));
  cudaMemsetAsync(b_pctr.p, 0, sizeof(unsigned long long) * 3 * IT_CNT, s);
  ItemLists ilp{b_plist.as<unsigned long long>(), b_pctr.as<unsigned long long>()};
  ItemLists il4{b_list4.as<unsigned long long>(), ilp.cnt + IT_CNT}, il5{b_list5.as<unsigned long long>(), ilp.cnt + 2 * IT_CNT};
  // small graphs (a union's member for member): medium items count by place in
  // the graph; the places of a union take a sort of its vertices by graph
  // (ESC_DIRECT=1: never; tests)
  const bool direct = dims[2] <= (unsigned long long)DIRECT_N && (G == 1 || (nnz >= 4 * n && G <= n)) &&
                      env_int("ESC_DIRECT", 2) != 1;
  const size_t sm_direct = sizeof(uint32_t) * (((size_t)dims[2] + 3) & ~(size_t)3);
  DevBuf b_lli, b_lhl, b_lhb, b_lrow, b_lwb, b_lJ;
  LocalIds lc{nullptr, nullptr, nullptr, accs.vg, b_narr.as<unsigned long long>(), (int)std::min<int64_t>(n, DIRECT_N)};
  DevGraph gd = g;                              // entries by place
  if (direct && G > 1 && n > 0) {
    ESC_TRY(b_lli.alloc(sizeof(int32_t) * n));
    ESC_TRY(b_lhl.alloc(sizeof(int32_t) * n));
    ESC_TRY(b_lhb.alloc(sizeof(int64_t) * n));
    ESC_TRY(b_lrow.alloc(sizeof(int64_t) * n));
    ESC_TRY(b_lwb.alloc(sizeof(int64_t) * (G + 1)));
    ESC_TRY(b_lJ.alloc(sizeof(int32_t) * (nnz + 1)));
    ESC_TRY(core_union(accs.vg, G, 0, n, b_lhl.as<int32_t>(), b_lhb.as<int64_t>(), b_lli.as<int32_t>(),
                       b_lrow.as<int64_t>(), b_lwb.as<int64_t>(), arena, sms, s));
    (k_local_entries<<<grid_for(nnz, TPB, sms), TPB, 0, s>>>(o.C, nnz, b_lli.as<int32_t>(), b_lJ.as<int32_t>()),
     note_launch());
    lc.li = b_lli.as<int32_t>();
    lc.hl = b_lhl.as<int32_t>();
    lc.hb = b_lhb.as<int64_t>();
    gd.J = b_lJ.as<int32_t>();
  }
  unsigned long long cnts[3 * IT_CNT] = {0};
  const unsigned long long *pcnt = cnts, *cnt4 = cnts + IT_CNT, *cnt5 = cnts + 2 * IT_CNT;
  // a single graph of more ranks than a window: heavy items walk their lists once per window
  const bool large_pairs = G == 1 && n > 2 * (int64_t)std::min((smem_optin - 4096) / 4, env_int("ESC_PAIR_WIN_WORDS", 1 << 30));
  // count bits of a packed word: every rank is below 2^(32 - cb) - 1
  int cb = 31;
  while (cb > 1 && n >= ((int64_t)1 << (32 - cb)) - 1) --cb;
  if (n > 0) {
    // ESC_PAIR_SMALL_W / ESC_PAIR_LARGE_W and ESC_CYCLE_SMALL_W / ESC_CYCLE_LARGE_W lower the classes' limits (tests)
    const unsigned long long* n_arr = b_narr.as<unsigned long long>();
    auto limit = [](const char* name, long long m) { return std::min<long long>(m, env_int(name, (int)m + 1) - 1); };
    if (five)
      (k_pair_classify<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(
           g, T, ilp, limit("ESC_PAIR_SMALL_W", IT_LIGHT_M), limit("ESC_PAIR_LARGE_W", IT_MEDIUM_M),
           large_pairs ? limit("ESC_PAIR_LARGE_W", IT_LARGE_M) : 0, cb, accs.vg, n_arr, direct, own), note_launch());
    (k_cycle_classify<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(
         g, il4, il5, !five, limit("ESC_CYCLE_SMALL_W", IT_LIGHT_M), limit("ESC_CYCLE_LARGE_W", IT_MEDIUM_M),
         limit("ESC_CYCLE_LARGE_W", direct ? IT_MEDIUM_M : IT5_MEDIUM_M), cb, accs.vg, n_arr, direct, own), note_launch());
    cudaMemcpyAsync(cnts, b_pctr.p, sizeof(cnts), cudaMemcpyDeviceToHost, s);
  }
  std::vector<int64_t> hR(n + 1, 0);
  if (n > 0) cudaMemcpyAsync(hR.data(), o.R, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToHost, s);
  ESC_TRY(cudaStreamSynchronize(s));
  if (five && n > 0) (k_share_offsets<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(g, off), note_launch());
  ESC_TRY(b_U.alloc(sizeof(int32_t) * (ulen + 1)));
  ESC_TRY(b_P.alloc(sizeof(int32_t) * (plen + 1)));
  int64_t maxdeg = n > 0 ? hR[n] - hR[n - 1] : 0;   // the highest rank has the largest degree
  // 4-cycle, pair and 5-cycle sweeps: tagged counters, 32-bit words below the first
  // rank of degree >= 2^16, 64-bit words from there on
  int64_t jbig = n;
  {
    int64_t lo = 0, hi = n;
    while (lo < hi) { int64_t mid = (lo + hi) >> 1; if (hR[mid + 1] - hR[mid] >= 65536) hi = mid; else lo = mid + 1; }
    jbig = lo;
  }
  // the heavy pair items: clusters sharing one counter array each
  PairPlan pplan;
  int64_t n0 = 0;                               // first rank of degree >= 1 (lower ranks are never counted)
  if (n > 0) {
    {
      int64_t lo = 0, hi = n;
      while (lo < hi) { int64_t mid = (lo + hi) >> 1; if (hR[mid + 1] - hR[mid] >= 1) hi = mid; else lo = mid + 1; }
      n0 = lo;
    }
  }
  if (five && pcnt[2] > 0) {
    size_t arr_bytes = sizeof(uint32_t) * (size_t)std::max<int64_t>(jbig - n0, 0) +
                       sizeof(unsigned long long) * (size_t)(n - jbig);
    ESC_TRY(plan_pair_clusters(jbig < n, sms, arr_bytes, n0, jbig, smem_optin, cfg.num_graphs > 1, &pplan));
  }
  // task buffers of the heavy pair items: the largest item has at most
  // w_max / PAIR_TASK + d_max tasks
  DevBuf b_ptq, b_ptn;
  PairTasks ptasks{nullptr, nullptr, 0};
  if (five && pcnt[2] > 0) {
    ptasks.cap = (int64_t)(pcnt[6] / PAIR_TASK) + maxdeg + 1;
    ESC_TRY(b_ptq.alloc(sizeof(long long) * 2 * (size_t)ptasks.cap * pplan.nclusters));
    ESC_TRY(b_ptn.alloc(sizeof(unsigned long long) * (size_t)pplan.nclusters));
    cudaMemsetAsync(b_ptn.p, 0, sizeof(unsigned long long) * (size_t)pplan.nclusters, s);
    ptasks.q = b_ptq.as<long long>();
    ptasks.n = b_ptn.as<unsigned long long>();
  }
  // heavy 4-cycle items: windows for a single graph, tagged counters for a union
  const bool win4 = cnt4[2] > 0 && G == 1, tag4 = cnt4[2] > 0 && G > 1;
  PairPlan plan4;
  DevBuf b_ptq4, b_ptn4;
  PairTasks ptasks4{nullptr, nullptr, 0};
  if (win4) {
    ESC_TRY(plan_pair_windows(jbig < n ? (const void*)k_cycles4_win<true> : (const void*)k_cycles4_win<false>, sms, n0,
                              jbig, smem_optin, &plan4));
    ptasks4.cap = (int64_t)(cnt4[6] / PAIR_TASK) + maxdeg + 1;
    ESC_TRY(b_ptq4.alloc(sizeof(long long) * 2 * (size_t)ptasks4.cap * plan4.nclusters));
    ESC_TRY(b_ptn4.alloc(sizeof(unsigned long long) * (size_t)plan4.nclusters));
    cudaMemsetAsync(b_ptn4.p, 0, sizeof(unsigned long long) * (size_t)plan4.nclusters, s);
    ptasks4.q = b_ptq4.as<long long>();
    ptasks4.n = b_ptn4.as<unsigned long long>();
  }
  // heavy 5-cycle items: a shared-memory window over the top ranks, one CTA per SM
  // (ESC_CYCLE_WIN_WORDS: a narrower one, so that small graphs count outside it too; tests)
  const int win5_words = (int)std::min<int64_t>(
      std::min((smem_optin - 4096) / 4, env_int("ESC_CYCLE_WIN_WORDS", 1 << 30)), std::max<int64_t>(jbig - n0, 1));
  const int64_t wlo5 = jbig - win5_words;
  const bool heavy5 = five && cnt5[2] > 0, below5 = heavy5 && (wlo5 > n0 || jbig < n);   // some counters outside it
  size_t sw32 = tag4 ? sizeof(uint32_t) * (size_t)jbig * grid_sweep + 16 : 16;
  size_t sw64 = tag4   ? sizeof(unsigned long long) * (size_t)(n - jbig) * grid_sweep + 16
                : win4 ? sizeof(unsigned long long) * (size_t)(n - jbig) * plan4.nclusters + 16
                       : 16;
  size_t sw32p = five && !pplan.windowed ? sizeof(uint32_t) * (size_t)jbig * pplan.nclusters + 16 : 16;
  size_t sw64p = five ? sizeof(unsigned long long) * (size_t)(n - jbig) * pplan.nclusters + 16 : 16;
  size_t sw32c = below5 ? sizeof(uint32_t) * (size_t)jbig * sms + 16 : 16;
  size_t sw64c = below5 ? sizeof(unsigned long long) * (size_t)(n - jbig) * sms + 16 : 16;
  size_t swp2 = below5 ? sizeof(uint32_t) * (size_t)n * sms + 16 : 16;
  DevBuf b_bigA, b_bigB, b_bigC;
  ESC_TRY(b_cntA.alloc(sw32)); ESC_TRY(b_bigA.alloc(sw64));
  ESC_TRY(b_cntB.alloc(sw32p)); ESC_TRY(b_bigB.alloc(sw64p));
  ESC_TRY(b_cntC.alloc(sw32c)); ESC_TRY(b_bigC.alloc(sw64c));
  ESC_TRY(b_cntD.alloc(swp2)); ESC_TRY(b_tlD.alloc(swp2));
  auto zero = [&](const DevBuf& b, size_t bytes) {
    if (bytes > 16) cudaMemsetAsync(b.p, 0, bytes, s);
  };
  zero(b_cntA, sw32); zero(b_bigA, sw64);
  zero(b_cntB, sw32p); zero(b_bigB, sw64p);
  zero(b_cntC, sw32c); zero(b_bigC, sw64c);
  zero(b_cntD, swp2);
  TagScratch tsA{b_cntA.as<uint32_t>(), b_bigA.as<unsigned long long>(), jbig, n};
  TagScratch tsB{b_cntB.as<uint32_t>(), b_bigB.as<unsigned long long>(), jbig, n};
  // the windowed heavy items: per CTA the dense 16-bit counts and the list cursors
  DevBuf b_g16, b_curs, b_g16_4, b_curs4;
  PairWin pwin{}, pwin4{};
  auto windows = [&](const PairPlan& pl, DevBuf& bg, DevBuf& bc, unsigned long long* side, PairWin* pw) -> cudaError_t {
    pw->g16_words = ((n + 2) / 2 + 4 + 3) & ~(int64_t)3;
    pw->curs_cap = std::max<int64_t>(maxdeg, 1);
    ESC_TRY(bg.alloc(sizeof(uint32_t) * (size_t)pw->g16_words * pl.nclusters));
    ESC_TRY(bc.alloc(sizeof(longlong2) * (size_t)pw->curs_cap * pl.nclusters));
    pw->g16 = bg.as<uint32_t>();
    pw->curs = bc.as<longlong2>();
    pw->side = side;                            // zeroed above
    pw->jbig = jbig;
    pw->n = n;
    pw->n0 = n0;
    pw->win_words = pl.win_words;
    pw->woff = (int)((4 - (((jbig + (jbig & 1)) >> 1) & 3)) & 3);
    return cudaSuccess;
  };
  if (five && pplan.windowed) ESC_TRY(windows(pplan, b_g16, b_curs, b_bigB.as<unsigned long long>(), &pwin));
  if (win4) ESC_TRY(windows(plan4, b_g16_4, b_curs4, b_bigA.as<unsigned long long>(), &pwin4));
  // with every counted rank in the window nothing is kept outside it (no array, so none to zero)
  TagScratch tsC{b_cntC.as<uint32_t>(), b_bigC.as<unsigned long long>(), below5 ? jbig : 0, below5 ? n : 0};
  SweepScratch ssC{b_cntD.as<uint32_t>(), b_tlD.as<int32_t>(), below5 ? n : 0};
  const int hcap_l = 8192;
  int64_t ghash_cap = pow2_at_least((int)std::max<int64_t>(2 * maxdeg, 2));
  if (2 * maxdeg <= hcap_l) ghash_cap = 2;
  ESC_TRY(b_gh.alloc(five ? sizeof(int32_t) * 2 * (size_t)ghash_cap * grid_sweep + 16 : 16));
  size_t smem_l = sizeof(int32_t) * 2 * (size_t)hcap_l;
  ESC_TRY(allow_max_smem((const void*)k_tri_lists, smem_optin));
  TriLists tl3{off, b_U.as<int32_t>(), offp, b_P.as<int32_t>(), nullptr, nullptr};

  // wheel work items: ranks are in degree order, so the large centres are a suffix
  int64_t c0 = n;
  {
    // first rank with degree > the warp items' limit (WHEEL_WARP_MAX, or lower
    // with ESC_WHEEL_WARP_MAX)
    const int64_t wmax = std::min(WHEEL_WARP_MAX, env_int("ESC_WHEEL_WARP_MAX", WHEEL_WARP_MAX));
    int64_t lo = 0, hi = n;
    while (lo < hi) { int64_t mid = (lo + hi) >> 1; if (hR[mid + 1] - hR[mid] > wmax) hi = mid; else lo = mid + 1; }
    c0 = lo;
  }
  DevBuf b_io, b_gs;
  int64_t nitems_w = 0;
  // counters in shared memory: one CTA per SM, and no more than eight arrays of
  // the largest degree (small graphs leave room for the other sweeps' CTAs)
  int smem_cap = (int)std::min<int64_t>(std::max(0, (smem_optin - 4096) / 4), 8 * maxdeg);
  int64_t gstride = maxdeg > smem_cap ? maxdeg : 1;
  size_t smem_w = sizeof(uint32_t) * (size_t)std::max(smem_cap, 1);
  std::vector<int64_t> item_off(n - c0 + 1, 0);
  if (five && c0 < n) {
    for (int64_t c = c0; c < n; ++c)
      item_off[c - c0 + 1] = item_off[c - c0] + (own.owns(c) ? (hR[c + 1] - hR[c] + WHEEL_CHUNK - 1) / WHEEL_CHUNK : 0);
    nitems_w = item_off[n - c0];
    ESC_TRY(b_io.alloc(sizeof(int64_t) * (n - c0 + 1)));
    cudaMemcpyAsync(b_io.p, item_off.data(), sizeof(int64_t) * (n - c0 + 1), cudaMemcpyHostToDevice, s);
    ESC_TRY(b_gs.alloc(sizeof(unsigned long long) * (size_t)gstride * sms + 16));
    cudaMemsetAsync(b_gs.p, 0, sizeof(unsigned long long) * (size_t)gstride * sms + 16, s);
    ESC_TRY(allow_max_smem((const void*)k_wheels_cta, smem_optin));
  }
  DevBuf b_wo;                                 // warp wheel items: offsets over centres c0-1 .. 0
  if (five && c0 > 0) {
    ESC_TRY(b_wo.alloc(sizeof(int64_t) * (size_t)(c0 + 1)));
    (k_wheel_warp_counts<<<grid_for(c0, TPB, sms), TPB, 0, s>>>(g, c0, b_wo.as<int64_t>(), own), note_launch());
    ESC_TRY(exclusive_scan_i64(b_wo.as<int64_t>(), b_wo.as<int64_t>(), c0, true, arena, s));
  }

  // ---------------- the dense core
  // It saves time and nothing else, so it comes after the buffers that the census
  // cannot do without, and a core whose buffers do not fit the device (or whose W
  // would pass CORE_W_BYTES) is left out.  ESC_CORE_MAX_MB: a smaller limit (tests).
  DevBuf b_cdh, b_cli, b_crow, b_coff, b_chl, b_chb, b_cwb, b_low, b_W, b_cblk, b_ctile, b_cb, b_cbits, b_ck4, b_offl,
      b_UL;
  CoreView cv{n, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0};
  CoreChunks cchunks;
  CoreBuffers cbuf;
  std::vector<int64_t> coff;
  int64_t ch = 0, wlen = 0;
  const size_t core_max = (size_t)env_int("ESC_CORE_MAX_MB", 1 << 30) << 20;
  size_t core_held = 0;
  struct Want { DevBuf* b; size_t bytes; };
  auto no_core = [&] {
    ch = 0;
    cv = CoreView{n, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0};
    cbuf = CoreBuffers{};
  };
  // all of them or none (a buffer given back here has not been used yet)
  auto reserve = [&](std::initializer_list<Want> wants) -> cudaError_t {
    size_t sum = 0;
    for (const Want& w : wants) sum += w.bytes;
    cudaError_t e = core_held + sum > core_max ? cudaErrorMemoryAllocation : cudaSuccess;
    for (const Want& w : wants)
      if (e == cudaSuccess && w.bytes) e = w.b->alloc(w.bytes);
    core_held += sum;
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    for (const Want& w : wants) w.b->give_back();
    no_core();
    return cudaSuccess;
  };
  const int core_min_d = env_int("ESC_CORE_MIN_D", 0);
  if (five && own.parts <= 1 && env_int("ESC_CORE", 2) != 1 &&
      pcnt[8] / 2 >= (core_min_d ? (unsigned long long)core_min_d
                                 : std::max(CORE_MIN_D, CORE_D_PER_ENTRY * (unsigned long long)nnz))) {
    const int64_t min_deg = env_int("ESC_CORE_MIN_DEG", CORE_MIN_DEG);
    int64_t lo = 0, hi = n;                     // first rank of degree >= min_deg
    while (lo < hi) { int64_t mid = (lo + hi) >> 1; if (hR[mid + 1] - hR[mid] >= min_deg) hi = mid; else lo = mid + 1; }
    ch = n - lo;
    if (G == 1) ch = std::min<int64_t>(ch, env_int("ESC_CORE_CAP", CORE_CAP));
  }
  if (ch > 0)
    ESC_TRY(reserve({{&b_cdh, sizeof(int32_t) * ch}, {&b_cli, sizeof(int32_t) * ch}, {&b_crow, sizeof(int64_t) * ch},
                     {&b_coff, sizeof(int64_t) * 4 * (ch + 1)}, {&b_chl, G > 1 ? sizeof(int32_t) * ch : 0},
                     {&b_chb, G > 1 ? sizeof(int64_t) * ch : 0}, {&b_cwb, G > 1 ? sizeof(int64_t) * (G + 1) : 0}}));
  if (ch > 0) {
    // core neighbours, places in W and the prefix sums of the work
    cv.h0 = n - ch;
    ESC_TRY(core_layout(g, cv.h0, G == 1, b_cdh.as<int32_t>(), b_cli.as<int32_t>(), b_crow.as<int64_t>(),
                        b_coff.as<int64_t>(), sms, s));
    if (G > 1) {
      const cudaError_t e = core_union(accs.vg, G, cv.h0, ch, b_chl.as<int32_t>(), b_chb.as<int64_t>(),
                                       b_cli.as<int32_t>(), b_crow.as<int64_t>(), b_cwb.as<int64_t>(), arena, sms, s);
      if (e == cudaErrorMemoryAllocation) no_core();   // more graphs than the arena, sized by the entries, has room for
      else ESC_TRY(e);
    } else {
      wlen = ch * ch;
    }
  }
  if (ch > 0) {
    if (G > 1) cudaMemcpyAsync(&wlen, b_cwb.as<int64_t>() + G, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    coff.resize(4 * (size_t)(ch + 1));
    cudaMemcpyAsync(coff.data(), b_coff.p, sizeof(int64_t) * 4 * (ch + 1), cudaMemcpyDeviceToHost, s);
    ESC_TRY(cudaStreamSynchronize(s));
    cv.wide = jbig < n ? 1 : 0;
    const size_t word = cv.wide ? sizeof(uint32_t) : sizeof(uint16_t), wb = word * (size_t)(wlen + 1);
    core_chunks(coff.data(), ch, (int64_t)env_int("ESC_CORE_CHUNK_MB", CORE_CHUNK_MB) << 20, &cchunks);
    cbuf.k4_0 = hR[cv.h0];
    const size_t k4b = sizeof(unsigned long long) * (size_t)(nnz - cbuf.k4_0 + 1);
    if (wb > CORE_W_BYTES || cchunks.max_tiles == 0) {
      no_core();
    } else {
      ESC_TRY(reserve({{&b_low, sizeof(uint32_t) * (size_t)(nnz + 1)}, {&b_W, wb}, {&b_cblk, core_block_bytes(cchunks)},
                       {&b_ctile, sizeof(int4) * (size_t)cchunks.max_tiles}, {&b_cbits, core_bit_bytes(cchunks)},
                       {&b_ck4, k4b}, {&b_cb, cv.h0 > 0 ? word * (size_t)(cchunks.max_tri + 2) : 0},
                       {&b_offl, sizeof(int64_t) * (size_t)(nnz + 2)}}));
    }
    if (ch > 0) {
      cudaMemsetAsync(b_ck4.p, 0, k4b, s);
      cbuf.k4 = b_ck4.p;
      cbuf.bits = b_cbits.p;
      cbuf.blocks = b_cblk.p;
      cbuf.tiles = b_ctile.p;
      cbuf.b = cv.h0 > 0 ? b_cb.p : nullptr;
      // ESC_CORE_WAIT_US, ESC_CORE_GIVE_UP: a shorter limit, a wait that runs out (tests)
      cbuf.wait_ns = 1000ull * (unsigned long long)env_int("ESC_CORE_WAIT_US", 4000000);
      cbuf.give_up = (uint32_t)env_int("ESC_CORE_GIVE_UP", 0);
      cv.low = b_low.as<uint32_t>();
      cv.dh = b_cdh.as<int32_t>();
      cv.li = b_cli.as<int32_t>();
      cv.rowb = b_crow.as<int64_t>();
      cv.hl = G > 1 ? b_chl.as<int32_t>() : nullptr;
      cv.hb = G > 1 ? b_chb.as<int64_t>() : nullptr;
      cv.W = b_W.p;
    }
  }

  // ---------------- concurrent phases on forked streams
  // The common-neighbour lists come first (short when alone); then
  //   s3 (most urgent): wheels      s : pairs
  //   s1, s2, s4 (least urgent): cliques, 4-cycles, 5-cycles; s joins all.
  mark(4, 0, s);
  if (five && n > 0)
  {
    int64_t lo = 0, hi = n;                     // first rank of degree > TL_LIGHT
    while (lo < hi) { int64_t mid = (lo + hi) >> 1; if (hR[mid + 1] - hR[mid] > TL_LIGHT) hi = mid; else lo = mid + 1; }
    if (lo < n)
      (k_tri_lists<<<(unsigned)std::min<int64_t>(grid_sweep, n - lo), 512, smem_l, s>>>(
           g, lo, ctr + 3, off, offp, T, b_U.as<int32_t>(), b_P.as<int32_t>(), b_gh.as<int32_t>(), ghash_cap, hcap_l,
           d_status), note_launch());
    if (hR[lo] > 0)
      (k_tri_lists_light<<<(unsigned)std::min<int64_t>((hR[lo] + TL_TILE - 1) / TL_TILE, (int64_t)sms * 8), 256, 0, s>>>(
           g, lo, hR[lo], off, offp, T, b_U.as<int32_t>(), b_P.as<int32_t>(), d_status), note_launch());
  }
  if (ch > 0) ESC_TRY(core_low(g, T, off, b_U.as<int32_t>(), cv.h0, b_low.as<uint32_t>(), sms, s));
  if (ch > 0) {                                 // the core's short lists
    int64_t total = 0;
    (k_low_counts<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(g, b_low.as<uint32_t>(), cv.h0, b_offl.as<int64_t>()),
     note_launch());
    ESC_TRY(exclusive_scan_i64(b_offl.as<int64_t>(), b_offl.as<int64_t>(), nnz, true, arena, s));
    cudaMemcpyAsync(&total, b_offl.as<int64_t>() + nnz, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    ESC_TRY(cudaStreamSynchronize(s));
    ESC_TRY(reserve({{&b_UL, sizeof(int32_t) * (size_t)(total + 1)}}));
  }
  if (ch > 0) {
    (k_low_lists<<<grid_for(nnz, TPB, sms), TPB, 0, s>>>(nnz, off, b_U.as<int32_t>(), b_offl.as<int64_t>(),
                                                        b_UL.as<int32_t>()), note_launch());
    tl3.UL = b_UL.as<int32_t>();
  }
  // the slots' records take the place of the arena, which no later phase uses: 16
  // bytes per entry are its size, and buffers of their own would be a quarter more
  // than a graph without triangles needs
  arena.release(0);
  uint4* rec = (uint4*)arena.alloc(sizeof(uint4) * (size_t)nnz);
  if (!rec) return cudaErrorMemoryAllocation;
  tl3.rec = rec;
  if (five && nnz > 0)
    (k_list_records<<<grid_for(nnz, TPB, sms), TPB, 0, s>>>(g, T, off, b_low.as<uint32_t>(),
                                                          ch > 0 ? b_offl.as<int64_t>() : nullptr, cv.h0,
                                                          rec), note_launch());
  mark(4, 1, s);
  StreamSet ss_all;
  cudaStream_t s1 = s, s2 = s, s3 = s, s4 = s;
  if (!cfg.serial_phases) {
    const int urgent[4] = {0, 0, 1, 0};
    ESC_TRY(ss_all.create(urgent));
    s1 = ss_all.ss.st[0]; s2 = ss_all.ss.st[1]; s3 = ss_all.ss.st[2]; s4 = ss_all.ss.st[3];
    ESC_TRY(ss_all.fork_from(s));
  }

  // wheels (Thm 11), on the most urgent stream: few CTAs of long items
  mark(6, 0, s3);
  if (five && c0 < n)
    (k_wheels_cta<<<(unsigned)std::min<int64_t>(sms, std::max<int64_t>(nitems_w, 1)), WHEEL_THREADS, smem_w, s3>>>(
                                            g, c0, b_io.as<int64_t>(), nitems_w, ctr + 5, tl3, T, cv,
                                            b_gs.as<unsigned long long>(), gstride, smem_cap, accs,
                                            pcnt[7] < 65536 && env_int("ESC_WHEEL_WINDOW", 2) != 1), note_launch());
  if (five && c0 > 0) {
    int per_sm = 1;
    ESC_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_wheels_warp, 256, 0));
    (k_wheels_warp<<<(unsigned)std::max(1, per_sm) * sms, 256, 0, s3>>>(g, c0, b_wo.as<int64_t>(), ctr + 7, tl3, T,
                                                                          cv, accs), note_launch());
  }
  mark(6, 1, s3);
  // pairs (Thms 11, 12); 16-bit counters when no degree reaches 2^16 (then no W(i,j) can)
  mark(5, 0, s);
  // CTAs that fit the device at once, at most one per item (launch.h)
  const int cta = cfg.cta_per_sm;
  auto fill = [&](const void* k, int threads, size_t smem, int64_t items, unsigned* grid,
                  int cta_per_sm = 0) -> cudaError_t {
    ESC_TRY(allow_max_smem(k, smem_optin));
    int per_sm = 1;
    ESC_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem));
    *grid = persistent_grid(per_sm, threads, cta_per_sm, sms, items);
    return cudaSuccess;
  };
  const size_t sm_light = sizeof(uint32_t) << IT_LIGHT_LOG, sm_mid = sizeof(uint32_t) << IT_MID_LOG,
               sm_medium = sizeof(uint32_t) << IT_MEDIUM_LOG, sm_large = sizeof(uint32_t) << IT_LARGE_LOG;
  unsigned grid_i = 1;
  if (five && n > 0) {
    unsigned long long* pq = ilp.cnt + 3;       // queue counters of the first three lists
    const unsigned long long* pl = ilp.list;
    if (pcnt[0] > 0) {
      ESC_TRY(fill((const void*)k_pairs_hash<IT_LIGHT_THREADS>, IT_LIGHT_THREADS, sm_light, (int64_t)pcnt[0], &grid_i));
      (k_pairs_hash<IT_LIGHT_THREADS><<<grid_i, IT_LIGHT_THREADS, sm_light, s>>>(
           g, pl, (int64_t)pcnt[0], pq + 0, cb, IT_LIGHT_LOG, tl3, T, cv, accs, d_status), note_launch());
    }
    if (pcnt[9] > 0) {
      ESC_TRY(fill((const void*)k_pairs_hash<IT_MID_THREADS>, IT_MID_THREADS, sm_mid, (int64_t)pcnt[9], &grid_i));
      (k_pairs_hash<IT_MID_THREADS><<<grid_i, IT_MID_THREADS, sm_mid, s>>>(
           g, pl + 3 * n, (int64_t)pcnt[9], ilp.cnt + 11, cb, IT_MID_LOG, tl3, T, cv, accs, d_status), note_launch());
    }
    if (pcnt[10] > 0) {
      ESC_TRY(fill((const void*)k_pairs_hash<IT_LARGE_THREADS>, IT_LARGE_THREADS, sm_large, (int64_t)pcnt[10], &grid_i));
      (k_pairs_hash<IT_LARGE_THREADS><<<grid_i, IT_LARGE_THREADS, sm_large, s>>>(
           g, pl + 4 * n, (int64_t)pcnt[10], ilp.cnt + 12, cb, IT_LARGE_LOG, tl3, T, cv, accs, d_status), note_launch());
    }
    if (pcnt[1] > 0 && direct) {
      ESC_TRY(fill((const void*)k_pairs_direct, IT_MEDIUM_THREADS, sm_direct, (int64_t)pcnt[1], &grid_i));
      (k_pairs_direct<<<grid_i, IT_MEDIUM_THREADS, sm_direct, s>>>(gd, pl + n, (int64_t)pcnt[1], pq + 1, lc, tl3, T, cv,
                                                                 accs), note_launch());
    } else if (pcnt[1] > 0) {
      ESC_TRY(fill((const void*)k_pairs_hash<IT_MEDIUM_THREADS>, IT_MEDIUM_THREADS, sm_medium, (int64_t)pcnt[1], &grid_i));
      (k_pairs_hash<IT_MEDIUM_THREADS><<<grid_i, IT_MEDIUM_THREADS, sm_medium, s>>>(
           g, pl + n, (int64_t)pcnt[1], pq + 1, cb, IT_MEDIUM_LOG, tl3, T, cv, accs, d_status), note_launch());
    }
    if (pcnt[2] > 0 && pplan.windowed) {
      const size_t smw = sizeof(uint32_t) * (size_t)pplan.win_words;
      if (jbig < n)
        (k_pairs_win<true><<<pplan.nclusters, pplan.threads, smw, s>>>(g, pl + 2 * n, (int64_t)pcnt[2], pq + 2, pwin,
                                                                      tl3, T, cv, accs, ptasks, d_status), note_launch());
      else
        (k_pairs_win<false><<<pplan.nclusters, pplan.threads, smw, s>>>(g, pl + 2 * n, (int64_t)pcnt[2], pq + 2, pwin,
                                                                       tl3, T, cv, accs, ptasks, d_status), note_launch());
    } else if (pcnt[2] > 0) {
      ESC_TRY(launch_pairs_grp(jbig < n, pplan, g, pl + 2 * n, (int64_t)pcnt[2], pq + 2, tsB, tl3, T, cv, accs, ptasks,
                               s));
    }
    if (ch > 0)
      ESC_TRY(core_run(g, cv, T, offp, b_P.as<int32_t>(), b_coff.as<int64_t>(), coff.data(), cchunks, cbuf, accs,
                       d_status, sms, smem_optin, s));
  }
  mark(5, 1, s);
  // cliques and per-triangle sums (Thms 6, 7, 10, 14)
  mark(2, 0, s1);
  if (nitems_b > 0)
    (k_clique_large<false><<<(unsigned)std::min<int64_t>(blocks_b, nitems_b), clq_threads, smem_b, s1>>>(
        g, b_items.as<int32_t>(), nitems_b, ctr + 1, T, K4e, accs, cs, hcap_b, -1, dmax_s, d_status, five, cv.h0),
     note_launch());
  if (nitems_b > 0 && blocks_g > 0)
    (k_clique_large<true><<<(unsigned)std::min<int64_t>(blocks_g, nitems_b), 512, sizeof(CliqueWarp) * CLQ_MAX_WARPS,
                            s1>>>(
        g, b_items.as<int32_t>(), nitems_b, ctr + 9, T, K4e, accs, cs, pow2_at_least(2 * dmax), dsplit, dmax,
        d_status, five, cv.h0), note_launch());
  if (nwsmall > 0) {
    int per_sm = 1;
    ESC_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_clique_warp, CLQ_WARPS * 32, 0));
    unsigned grid_w = (unsigned)std::min<int64_t>((int64_t)std::max(1, per_sm) * sms, (nwsmall + CLQ_WARPS - 1) / CLQ_WARPS);
    (k_clique_warp<<<grid_w, CLQ_WARPS * 32, 0, s1>>>(g, b_wsmall.as<int32_t>(), nwsmall, ctr + 8, T, K4e, accs,
                                                      five, cv.h0), note_launch());
  }
  mark(2, 1, s1);
  // 4-cycles (Thm 5)
  mark(3, 0, s2);
  if (n > 0) {
    unsigned long long* q4 = il4.cnt + 3;
    const unsigned long long* l4 = il4.list;
    if (win4) {
      const size_t smw = sizeof(uint32_t) * (size_t)plan4.win_words;
      if (jbig < n)
        (k_cycles4_win<true><<<plan4.nclusters, plan4.threads, smw, s2>>>(
             g, l4 + 2 * n, (int64_t)cnt4[2], q4 + 2, pwin4, ptasks4, C4e, accs, d_status), note_launch());
      else
        (k_cycles4_win<false><<<plan4.nclusters, plan4.threads, smw, s2>>>(
             g, l4 + 2 * n, (int64_t)cnt4[2], q4 + 2, pwin4, ptasks4, C4e, accs, d_status), note_launch());
    } else if (tag4) {
      if (jbig < n)
        (k_cycles4_tag<true><<<grid_sweep, 512, 0, s2>>>(g, l4 + 2 * n, (int64_t)cnt4[2], q4 + 2, tsA, C4e, accs),
         note_launch());
      else
        (k_cycles4_tag<false><<<grid_sweep, 512, 0, s2>>>(g, l4 + 2 * n, (int64_t)cnt4[2], q4 + 2, tsA, C4e, accs),
         note_launch());
    }
    if (cnt4[1] > 0 && direct) {
      ESC_TRY(fill((const void*)k_cycles4_direct, IT_MEDIUM_THREADS, sm_direct, (int64_t)cnt4[1], &grid_i, cta));
      (k_cycles4_direct<<<grid_i, IT_MEDIUM_THREADS, sm_direct, s2>>>(gd, l4 + n, (int64_t)cnt4[1], q4 + 1, lc, C4e,
                                                                    accs), note_launch());
    } else if (cnt4[1] > 0) {
      ESC_TRY(fill((const void*)k_cycles4_hash<IT_MEDIUM_THREADS>, IT_MEDIUM_THREADS, sm_medium, (int64_t)cnt4[1], &grid_i, cta));
      (k_cycles4_hash<IT_MEDIUM_THREADS><<<grid_i, IT_MEDIUM_THREADS, sm_medium, s2>>>(
           g, l4 + n, (int64_t)cnt4[1], q4 + 1, cb, IT_MEDIUM_LOG, C4e, accs, d_status), note_launch());
    }
    if (cnt4[9] > 0) {
      ESC_TRY(fill((const void*)k_cycles4_hash<IT_MID_THREADS>, IT_MID_THREADS, sm_mid, (int64_t)cnt4[9], &grid_i, cta));
      (k_cycles4_hash<IT_MID_THREADS><<<grid_i, IT_MID_THREADS, sm_mid, s2>>>(
           g, l4 + 3 * n, (int64_t)cnt4[9], il4.cnt + 11, cb, IT_MID_LOG, C4e, accs, d_status), note_launch());
    }
    if (cnt4[0] > 0) {
      ESC_TRY(fill((const void*)k_cycles4_hash<IT_LIGHT_THREADS>, IT_LIGHT_THREADS, sm_light, (int64_t)cnt4[0], &grid_i, cta));
      (k_cycles4_hash<IT_LIGHT_THREADS><<<grid_i, IT_LIGHT_THREADS, sm_light, s2>>>(
           g, l4, (int64_t)cnt4[0], q4 + 0, cb, IT_LIGHT_LOG, C4e, accs, d_status), note_launch());
    }
    (k_fold_u64<<<grid_for(n * 32, TPB, sms), TPB, 0, s2>>>(g, C4e), note_launch());
    (k_vertex_sum_div<<<grid_for(n * 32, TPB, sms), TPB, 0, s2>>>(g, C4e, C4v, 2), note_launch());
  }
  mark(3, 1, s2);
  // 5-cycles (Thm 13)
  mark(7, 0, s4);
  if (five && n > 0) {
    unsigned long long* q5 = il5.cnt + 3;
    const unsigned long long* l5 = il5.list;
    if (heavy5) {
      const size_t smw = sizeof(uint32_t) * (size_t)win5_words;
      const void* k5 = jbig < n ? (const void*)k_cycles5<true> : (const void*)k_cycles5<false>;
      ESC_TRY(allow_max_smem(k5, smem_optin));
      const unsigned grid5 = (unsigned)std::min<int64_t>(sms, (int64_t)cnt5[2]);
      if (jbig < n)
        (k_cycles5<true><<<grid5, 1024, smw, s4>>>(g, l5 + 2 * n, (int64_t)cnt5[2], q5 + 2, tsC, ssC, accs, wlo5,
                                                   win5_words), note_launch());
      else
        (k_cycles5<false><<<grid5, 1024, smw, s4>>>(g, l5 + 2 * n, (int64_t)cnt5[2], q5 + 2, tsC, ssC, accs, wlo5,
                                                    win5_words), note_launch());
    }
    if (cnt5[1] > 0 && direct) {
      ESC_TRY(fill((const void*)k_cycles5_direct, IT_MEDIUM_THREADS, sm_direct, (int64_t)cnt5[1], &grid_i, cta));
      (k_cycles5_direct<<<grid_i, IT_MEDIUM_THREADS, sm_direct, s4>>>(gd, l5 + n, (int64_t)cnt5[1], q5 + 1, lc, accs),
       note_launch());
    } else if (cnt5[1] > 0) {                   // two tables of half the size
      ESC_TRY(fill((const void*)k_cycles5_hash<IT_MEDIUM_THREADS>, IT_MEDIUM_THREADS, sm_medium, (int64_t)cnt5[1], &grid_i, cta));
      (k_cycles5_hash<IT_MEDIUM_THREADS><<<grid_i, IT_MEDIUM_THREADS, sm_medium, s4>>>(
           g, l5 + n, (int64_t)cnt5[1], q5 + 1, cb, IT_MEDIUM_LOG - 1, accs, d_status), note_launch());
    }
    if (cnt5[9] > 0) {
      ESC_TRY(fill((const void*)k_cycles5_hash<IT_MID_THREADS>, IT_MID_THREADS, sm_mid, (int64_t)cnt5[9], &grid_i, cta));
      (k_cycles5_hash<IT_MID_THREADS><<<grid_i, IT_MID_THREADS, sm_mid, s4>>>(
           g, l5 + 3 * n, (int64_t)cnt5[9], il5.cnt + 11, cb, IT_MID_LOG - 1, accs, d_status), note_launch());
    }
    if (cnt5[0] > 0) {
      ESC_TRY(fill((const void*)k_cycles5_hash<IT_LIGHT_THREADS>, IT_LIGHT_THREADS, 2 * sm_light, (int64_t)cnt5[0], &grid_i, cta));
      (k_cycles5_hash<IT_LIGHT_THREADS><<<grid_i, IT_LIGHT_THREADS, 2 * sm_light, s4>>>(
           g, l5, (int64_t)cnt5[0], q5 + 0, cb, IT_LIGHT_LOG, accs, d_status), note_launch());
    }
  }
  mark(7, 1, s4);
  ESC_TRY(ss_all.join_into(s));

  // ---------------- closed forms over vertices and edges, then assembly
  mark(8, 0, s);
  if (n > 0) {
    (k_sym_K4<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(g, K4e, (const unsigned long long*)cbuf.k4, cbuf.k4_0),
     note_launch());
    if (!cfg.partial)                          // a part's K4 sums are divided once every part's are in
      (k_vertex_sum_div<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(g, K4e, K4v, 3), note_launch());
  }
  if (cfg.partial) {
    // one part of a split census: its raw sums; the closed forms need every
    // part's per-element counts and run in run_census_finish
    ESC_TRY(cudaMemcpyAsync(cfg.d_acc_out, acc, sizeof(Acc128) * ACC_COUNT, cudaMemcpyDeviceToDevice, s));
  } else {
    if (n > 0)
      (k_edge_sums<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(g, T, C4e, K4e, tv, C4v, K4v, accs), note_launch());
    const ConvTables& tabs = conversion_tables();
    (k_assemble<<<(unsigned)std::min(G, 65535), ASM_THREADS, 0, s>>>(acc, b_narr.as<unsigned long long>(), b_marr.as<unsigned long long>(),
                                            G, tabs, d_out, (u128*)cfg.d_basis), note_launch());
  }
  mark(8, 1, s);

  if (pe_out) {
    // hand the per-element arrays over to the caller (ownership moves)
    pe_out->Te = T;
    pe_out->C4e = C4e;
    pe_out->K4e = K4e;
    pe_out->tv = tv;
    pe_out->C4v = C4v;
    pe_out->K4v = K4v;
    for (DevBuf* b : {&b_T, &b_C4e, &b_K4e, &b_tv, &b_C4v, &b_K4v}) pe_out->own.push_back(std::move(*b));
  }
  if (or_out) {
    or_out->perm = o.perm;
    or_out->rank = o.rank;
    or_out->R = o.R;
    or_out->C = o.C;
    or_out->op = o.op;
    or_out->rev = o.rev;
    for (DevBuf* b : {&b_perm, &b_rank, &b_R, &b_C, &b_op, &b_rev}) or_out->own.push_back(std::move(*b));
  }
  ESC_TRY(cudaStreamSynchronize(s));   // scratch buffers are freed on return
  return cudaGetLastError();
}

// The end of a split census: every part's sums added (d_acc, ACC_COUNT
// 128-bit words) and every part's per-element counts added into pe (K4e, C4e,
// C4v; T and tv are whole on every part).  K4 per vertex, the closed forms
// over vertices and edges, and the assembly.
cudaError_t run_census_finish(const Oriented& o, int64_t n, int64_t nnz, const PerElement& pe,
                              const unsigned long long* d_acc, unsigned long long* d_out, int sms, cudaStream_t s) {
  CacheScope cache_scope(s);
  const int TPB = 256;
  DevGraph g{n, nnz, o.R, o.C, o.op, o.rev, o.C};
  DevBuf b_acc, b_nm;
  ESC_TRY(b_acc.alloc(sizeof(Acc128) * ACC_COUNT));
  ESC_TRY(b_nm.alloc(sizeof(unsigned long long) * 2));
  ESC_TRY(cudaMemcpyAsync(b_acc.p, d_acc, sizeof(Acc128) * ACC_COUNT, cudaMemcpyDeviceToDevice, s));
  unsigned long long nm[2] = {(unsigned long long)n, (unsigned long long)(nnz / 2)};
  ESC_TRY(cudaMemcpyAsync(b_nm.p, nm, sizeof(nm), cudaMemcpyHostToDevice, s));
  AccSet accs{b_acc.as<Acc128>(), nullptr};
  if (n > 0) {
    (k_vertex_sum_div<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(g, pe.K4e, pe.K4v, 3), note_launch());
    (k_edge_sums<<<grid_for(n * 32, TPB, sms), TPB, 0, s>>>(g, pe.Te, pe.C4e, pe.K4e, pe.tv, pe.C4v, pe.K4v, accs),
     note_launch());
  }
  const ConvTables& tabs = conversion_tables();
  (k_assemble<<<1, ASM_THREADS, 0, s>>>(b_acc.as<Acc128>(), b_nm.as<unsigned long long>(), b_nm.as<unsigned long long>() + 1,
                               1, tabs, d_out, nullptr), note_launch());
  ESC_TRY(cudaStreamSynchronize(s));   // nm lives on this stack frame
  return cudaGetLastError();
}

int census_sum_count() { return ACC_COUNT; }

}  // namespace esc
