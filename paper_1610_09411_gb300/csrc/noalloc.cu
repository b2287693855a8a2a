// noalloc.cu -- per-vertex 4-cycle counts without any device allocation.
//
// Some callers cannot allocate device memory at the time they want a count:
// a serving loop that has handed all of the GPU's memory to its own pool, or
// a latency-critical path that must not let cudaMalloc/cudaFree synchronise
// the device behind other streams' backs.  escape_cycles4_noalloc serves them:
// the caller passes device inputs and outputs, and the only work space is the
// fixed array below, which lives as long as the library is loaded.
//
// The counting is the 4-cycle rule of the main library (for the highest
// vertex i of a 4-cycle and the opposite vertex j, the number of middles
// below i), run here directly on the caller's CSR: the degree order is a key per
// vertex, (row length, id) in one 32-bit word.
//
// All counters are in shared memory: a vertex of at most 32 neighbours has at
// most 32 x 32 wedges to lower vertices (a middle has no more neighbours than
// it), counted by one warp in a packed hash table; the others take one CTA with
// a counter and a place in the touched list for every vertex (6 bytes x 32,768).
// Both are bound by the latency of row -> entry -> order key -> counter.  A warp
// therefore fetches 32 rows at a time and walks their entries as one sequence
// (na_flat), rows of more than NA_PIECE entries are shared by the CTA's warps,
// and the heavy kernel starts beside the light one.
// Chung-Lu n = 30,011 (232,000 edges) 0.46 ms, n = 719 48 us.  With a lane per
// row in the light kernel, a warp per row in the heavy one and the two in turn
// 0.62 ms and about 115 us; with 32 CTAs counting in global memory and two row
// lengths read per comparison 4.85 ms and 86 us.
#include "../../include/escape.h"
#include "common.cuh"
#include "internal.h"

#include <algorithm>
#include <mutex>

namespace {

constexpr int64_t NA_MAX_N = ESCAPE_NOALLOC_MAX_N;  // vertices
constexpr int NA_LIGHT_DEG = 32, NA_LIGHT_WARPS = 8, NA_LIGHT_LOG = 11, NA_HEAVY_THREADS = 1024;
constexpr int NA_ILP = 4, NA_PIECE = 256, NA_LONG = 128, NA_HUB_DEG = 256;
// Work space shared by every call on this device (256 KiB): a header of 64
// words (heavy items, queue, status), the order keys and the list of heavy
// vertices: those of more than NA_HUB_DEG neighbours from the front, so that
// they are taken first, the others from the back.
constexpr int64_t NA_WORDS = 64 + 2 * NA_MAX_N;
static __device__ __align__(256) unsigned int g_noalloc_scratch[NA_WORDS];
struct NaSpace {
  unsigned int *hubs, *queue, *status, *others, *key;
  int32_t* heavy;
};
NaSpace na_space(unsigned int* base) {
  return NaSpace{base, base + 1, base + 2, base + 3, base + 64, (int32_t*)(base + 64 + NA_MAX_N)};
}

std::mutex g_mu;
void* g_addr[64] = {nullptr};     // device address of g_noalloc_scratch, per device

// Row v's entry range, clamped: an offset outside [0, rp[n]] or a row that
// ends before it starts sets the status word and reads as an empty row, so no
// access leaves col[0 .. rp[n]).
__device__ __forceinline__ void na_row(const int64_t* rp, int64_t n, int64_t v, int64_t& b, int64_t& e,
                                       unsigned int* status) {
  b = rp[v];
  e = rp[v + 1];
  int64_t lim = rp[n];
  if (b < 0 || e < b || e > lim) {
    atomicOr(status, 1u);
    b = e = 0;
  }
}

// Order keys, the heavy list and zeroed outputs.  A row is at most n - 1 < 2^15 entries long in a
// simple graph; longer ones (malformed) share the largest length.
__global__ void k_na_prep(const int64_t* rp, int64_t n, NaSpace ns, unsigned long long* c4v,
                          unsigned long long* c4_total) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v == 0) *c4_total = 0;
  if (v >= n) return;
  int64_t b, e;
  na_row(rp, n, v, b, e, ns.status);
  ns.key[v] = ((unsigned int)min(e - b, (int64_t)0x1ffff) << 15) | (unsigned int)v;
  c4v[v] = 0;
  if (e - b > NA_HUB_DEG) ns.heavy[atomicAdd(ns.hubs, 1u)] = (int32_t)v;
  else if (e - b > NA_LIGHT_DEG) ns.heavy[NA_MAX_N - 1 - atomicAdd(ns.others, 1u)] = (int32_t)v;
}

__device__ __forceinline__ int na_len(unsigned int key) { return (int)(key >> 15); }

// The entries of up to 32 rows (lane l holds col[b_l .. b_l + len_l)) as one
// sequence, 32 * NA_ILP of them per round: visit(o, j, on) with the lane o of
// the row and the entry j; on: there is an entry, it names a vertex, and that
// one's key is below ki.  All lanes call visit together, and o does not
// decrease from lane to lane.
template <class Visit>
__device__ __forceinline__ void na_flat(const int32_t* col, int64_t n, const NaSpace& ns, unsigned int ki, int64_t b_l,
                                        int64_t len_l, Visit&& visit) {
  const int lane = threadIdx.x & 31;
  while (__any_sync(0xffffffffu, len_l > 0)) {
    const int take = (int)min(len_l, (int64_t)1 << 20);   // 32 of them fit 32 bits; one round for any simple graph
    int end = take;                             // entries of rows 0 .. lane
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += y;
    }
    const int total = __shfl_sync(0xffffffffu, end, 31);
    const long long at = (long long)b_l - (end - take);   // entry t of the sequence is col[at + t] of its row's lane
    for (int t0 = 0; t0 < total; t0 += 32 * NA_ILP) {
      int own[NA_ILP];
      int32_t j[NA_ILP];
      unsigned int kj[NA_ILP];
#pragma unroll
      for (int u = 0; u < NA_ILP; ++u) {
        const int t = t0 + 32 * u + lane;
        int o = 0;                              // rows that end at or before t
#pragma unroll
        for (int h = 16; h >= 1; h >>= 1)
          if (__shfl_sync(0xffffffffu, end, o + h - 1) <= t) o += h;
        const long long base = __shfl_sync(0xffffffffu, at, o);
        own[u] = o;
        j[u] = t < total ? col[base + t] : 0;
      }
#pragma unroll
      for (int u = 0; u < NA_ILP; ++u) {
        kj[u] = ~0u;
        if (j[u] < 0 || j[u] >= n) atomicOr(ns.status, 1u);
        else if (t0 + 32 * u + lane < total) kj[u] = ns.key[j[u]];
      }
#pragma unroll
      for (int u = 0; u < NA_ILP; ++u) {
        if (t0 + 32 * u >= total) break;
        visit(own[u], j[u], kj[u] < ki);
      }
    }
    b_l += take;
    len_l -= take;
  }
}

// sk[o] += x for the lanes' (o, x), o not decreasing from lane to lane.
__device__ __forceinline__ void na_add(unsigned int* sk, int o, unsigned int x) {
  if (__shfl_sync(0xffffffffu, o, 0) == __shfl_sync(0xffffffffu, o, 31)) {
    x = __reduce_add_sync(0xffffffffu, x);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(&sk[o], x);
  } else if (x) {
    atomicAdd(&sk[o], x);
  }
}

// One warp per vertex of at most NA_LIGHT_DEG neighbours (lane l takes the l-th
// one's row); the heavy kernel's work.
__global__ void __launch_bounds__(NA_LIGHT_WARPS * 32) k_na_light(const int64_t* rp, const int32_t* col, int64_t n,
                                                                 NaSpace ns, unsigned long long* c4v,
                                                                 unsigned long long* c4_total) {
  extern __shared__ uint4 na_smem[];
  __shared__ unsigned int sk_all[NA_LIGHT_WARPS][32];
  cudaTriggerProgrammaticLaunchCompletion();    // k_na_heavy reads nothing that this kernel writes
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  uint32_t* tab = reinterpret_cast<uint32_t*>(na_smem) + (wl << NA_LIGHT_LOG);
  unsigned int* sk = sk_all[wl];
  const int64_t nwarps = (int64_t)gridDim.x * NA_LIGHT_WARPS;
  unsigned long long total = 0;
  sk[lane] = 0;
  for (int64_t i = (int64_t)blockIdx.x * NA_LIGHT_WARPS + wl; i < n; i += nwarps) {
    const unsigned int ki = ns.key[i];
    const int d = na_len(ki);
    if (d > NA_LIGHT_DEG) continue;
    int64_t b, e, kb = 0, ke = 0;
    na_row(rp, n, i, b, e, ns.status);
    int32_t k = -1;
    if (lane < d && b + lane < e) {
      k = col[b + lane];
      if (k < 0 || k >= n) {
        atomicOr(ns.status, 1u);
        k = -1;
      } else if (ns.key[k] < ki) {
        na_row(rp, n, k, kb, ke, ns.status);
      }
    }
    if (d < 2) continue;
    // key << 16 | count: ids below 2^15 and counts of at most 2^10, so no used word is all ones
    const int log = max(7, 32 - __clz(2 * d * d - 1));
    const uint32_t mask = (1u << log) - 1u;
    for (int t = lane; t < (1 << log) / 4; t += 32)
      reinterpret_cast<uint4*>(tab)[t] = make_uint4(~0u, ~0u, ~0u, ~0u);
    __syncwarp();
    auto slot_of = [&](int32_t j, bool insert) -> int {
      uint32_t sl = ((uint32_t)j * 0x9E3779B1u) >> (32 - log);
      for (uint32_t probe = 0; probe <= mask; ++probe) {
        uint32_t w = *(volatile uint32_t*)&tab[sl];
        if (w == ~0u) {
          if (!insert) return -1;
          w = atomicCAS(&tab[sl], ~0u, (uint32_t)j << 16);
          if (w == ~0u) return (int)sl;
        }
        if ((w >> 16) == (uint32_t)j) return (int)sl;
        sl = (sl + 1u) & mask;
      }
      return -1;
    };
    na_flat(col, n, ns, ki, kb, ke - kb, [&](int, int32_t j, bool on) {
      if (!on) return;
      const int sl = slot_of(j, true);
      if (sl >= 0) atomicAdd(&tab[sl], 1u);
    });
    __syncwarp();
    na_flat(col, n, ns, ki, kb, ke - kb, [&](int o, int32_t j, bool on) {
      const int sl = on ? slot_of(j, false) : -1;
      if (sl >= 0 && (tab[sl] & 0xffffu) > 1u) atomicAdd(&sk[o], (tab[sl] & 0xffffu) - 1u);
    });
    __syncwarp();
    if (sk[lane]) {
      atomicAdd(&c4v[k], (unsigned long long)sk[lane]);
      sk[lane] = 0;
    }
    unsigned long long mine = 0;
    for (int t = lane; t <= (int)mask; t += 32) {
      const uint32_t w = tab[t];
      if (w == ~0u) continue;
      const unsigned long long c = (unsigned long long)(w & 0xffffu) * ((w & 0xffffu) - 1u) / 2;
      if (c) {
        atomicAdd(&c4v[w >> 16], c);
        mine += c;
      }
    }
    mine = warp_sum_u64(mine);
    if (lane == 0 && mine) atomicAdd(&c4v[i], mine);
    total += mine;                              // valid on lane 0
    __syncwarp();                               // the table is read before the next item clears it
  }
  // each 4-cycle is counted once, at its highest vertex
  if (lane == 0 && total) atomicAdd(c4_total, total);
}

// One CTA per heavy vertex: counters of every vertex and the touched list in
// shared memory.
__global__ void __launch_bounds__(NA_HEAVY_THREADS, 1) k_na_heavy(const int64_t* rp, const int32_t* col, int64_t n,
                                                                 NaSpace ns, unsigned long long* c4v,
                                                                 unsigned long long* c4_total) {
  extern __shared__ uint4 na_smem[];
  __shared__ u128 sh[32];
  __shared__ unsigned int sh_item, nt, nl;
  __shared__ unsigned int sk_all[NA_HEAVY_THREADS / 32][32];
  __shared__ longlong2 s_long[NA_LONG];         // rows of more than NA_PIECE entries, and their vertices
  __shared__ int32_t s_longk[NA_LONG];
  uint32_t* w = reinterpret_cast<uint32_t*>(na_smem);
  uint16_t* tl = reinterpret_cast<uint16_t*>(w + n);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned int* sk = sk_all[wid];
  const unsigned int hubs = *ns.hubs, items = hubs + *ns.others;
  u128 total = 0;
  for (int64_t t = threadIdx.x; t < n; t += blockDim.x) w[t] = 0;   // any CTA may take an item
  sk[lane] = 0;
  while (true) {
    if (threadIdx.x == 0) {
      sh_item = atomicAdd(ns.queue, 1u);
      nt = nl = 0;
    }
    __syncthreads();
    const unsigned int it = sh_item;
    if (it >= items) break;
    const int64_t i = it < hubs ? ns.heavy[it] : ns.heavy[NA_MAX_N - 1 - (it - hubs)];
    const unsigned int ki = ns.key[i];
    int64_t ib, ie;
    na_row(rp, n, i, ib, ie, ns.status);
    auto count = [&](int, int32_t j, bool on) {
      const bool fresh = on && atomicAdd(&w[j], 1u) == 0;
      const unsigned m = __ballot_sync(0xffffffffu, fresh);
      if (!m) return;
      unsigned at = 0;
      if (lane == 0) at = atomicAdd(&nt, (unsigned)__popc(m));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
      if (fresh) tl[at] = (uint16_t)j;
    };
    auto middle = [&](int o, int32_t j, bool on) { na_add(sk, o, on ? w[j] - 1u : 0u); };
    // this warp's sums go to the middles' vertices (lane l: k)
    auto flush = [&](int32_t k) {
      __syncwarp();
      if (sk[lane]) {
        atomicAdd(&c4v[k], (unsigned long long)sk[lane]);
        sk[lane] = 0;
      }
      __syncwarp();
    };
    // one pass over the wedges i - k - j with k, j below i; `first` counts them
    auto wedges = [&](bool first) {
      for (int64_t pb = ib + wid; pb < ie; pb += 32 * nw) {
        const int64_t p = pb + (int64_t)lane * nw;
        int64_t kb = 0, ke = 0;
        int32_t k = -1;
        if (p < ie) {
          k = col[p];
          if (k < 0 || k >= n) {
            atomicOr(ns.status, 1u);
            k = -1;
          } else if (ns.key[k] < ki) {
            na_row(rp, n, k, kb, ke, ns.status);
          }
        }
        if (ke - kb > NA_PIECE) {
          const unsigned at = atomicAdd(&nl, 1u);
          if (at < NA_LONG) {                   // else: walked here like the others
            s_long[at] = make_longlong2(kb, ke);
            s_longk[at] = k;
            ke = kb;
          }
        }
        if (first) {
          na_flat(col, n, ns, ki, kb, ke - kb, count);
        } else {
          na_flat(col, n, ns, ki, kb, ke - kb, middle);
          flush(k);
        }
      }
      __syncthreads();
      const int nlc = (int)min(nl, (unsigned)NA_LONG);
      int64_t pc = wid;                         // piece by piece over the warps
      for (int l = 0; l < nlc; ++l) {
        const longlong2 r = s_long[l];
        const int64_t np = (r.y - r.x + NA_PIECE - 1) / NA_PIECE;
        for (; pc < np; pc += nw) {
          const int64_t a = r.x + pc * NA_PIECE;
          const int64_t len = lane == 0 ? min((int64_t)NA_PIECE, (int64_t)r.y - a) : 0;
          if (first) {
            na_flat(col, n, ns, ki, a, len, count);
          } else {
            na_flat(col, n, ns, ki, a, len, middle);
            flush(s_longk[l]);                  // only lane 0's row had entries
          }
        }
        pc -= np;
      }
      __syncthreads();
    };
    wedges(true);
    const unsigned int ntc = nt;
    if (threadIdx.x == 0) nl = 0;
    __syncthreads();
    wedges(false);                              // w - 1 to every middle k
    u128 mine = 0;                              // C(w, 2) to i and j
    for (unsigned int t = threadIdx.x; t < ntc; t += blockDim.x) {
      const int32_t j = tl[t];
      const unsigned long long c = (unsigned long long)w[j] * (w[j] - 1) / 2;
      w[j] = 0;
      if (c) {
        atomicAdd(&c4v[j], c);
        mine += c;
      }
    }
    const u128 s = block_sum_u128(mine, sh);    // its barriers also end the reads of nt and sh_item
    if (threadIdx.x == 0) {
      if (s) atomicAdd(&c4v[i], (unsigned long long)s);
      total += s;
    }
  }
  if (threadIdx.x == 0 && total) atomicAdd(c4_total, (unsigned long long)total);
  cudaGridDependencySynchronize();              // what follows this kernel on the stream follows k_na_light too
}

}  // namespace

extern "C" escape_status escape_cycles4_noalloc(int64_t n, const int64_t* row_ptr, const int32_t* col,
                                                uint64_t* c4_v, uint64_t* c4_total, void* stream) {
  if (n < 0 || (n > 0 && (!row_ptr || !col || !c4_v)) || !c4_total) return ESCAPE_EINVAL;
  if (n > NA_MAX_N) return ESCAPE_EOVERFLOW;     // beyond the fixed work space
  cudaStream_t s = (cudaStream_t)stream;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 64) {
    esc::note_cuda_error(e);
    return ESCAPE_ECUDA;
  }
  void* base = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_addr[dev]) {
      e = cudaGetSymbolAddress(&g_addr[dev], g_noalloc_scratch);
      if (e != cudaSuccess) { g_addr[dev] = nullptr; cudaGetLastError(); esc::note_cuda_error(e); return ESCAPE_ECUDA; }
    }
    base = g_addr[dev];
  }
  const NaSpace ns = na_space((unsigned int*)base);
  int sms = 1;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // the header starts at zero; keys, lists and outputs are written by the kernels
  e = cudaMemsetAsync(base, 0, sizeof(unsigned int) * 64, s);
  if (n == 0 && e == cudaSuccess) e = cudaMemsetAsync(c4_total, 0, sizeof(uint64_t), s);
  const size_t sm_light = (sizeof(uint32_t) << NA_LIGHT_LOG) * NA_LIGHT_WARPS;
  const size_t sm_heavy = (sizeof(uint32_t) + sizeof(uint16_t)) * (size_t)NA_MAX_N;
  if (n > 0) {                                  // the same limits at every call
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_na_light, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_light);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_na_heavy, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_heavy);
  }
  if (e != cudaSuccess) { cudaGetLastError(); esc::note_cuda_error(e); return ESCAPE_ECUDA; }
  if (n > 0) {
    unsigned long long *v = (unsigned long long*)c4_v, *tot = (unsigned long long*)c4_total;
    const unsigned warps_grid = (unsigned)std::min<int64_t>((n + NA_LIGHT_WARPS - 1) / NA_LIGHT_WARPS, (int64_t)sms * 3);
    k_na_prep<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(row_ptr, n, ns, v, tot);
    k_na_light<<<warps_grid, NA_LIGHT_WARPS * 32, sm_light, s>>>(row_ptr, col, n, ns, v, tot);
    // k_na_heavy may start once every CTA of k_na_light has: both need k_na_prep only
    cudaLaunchAttribute beside{};
    beside.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    beside.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)std::min<int64_t>(sms, n));
    cfg.blockDim = dim3(NA_HEAVY_THREADS);
    cfg.dynamicSmemBytes = (sizeof(uint32_t) + sizeof(uint16_t)) * (size_t)((n + 1) & ~1ll);
    cfg.stream = s;
    cfg.attrs = &beside;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_na_heavy, row_ptr, col, n, ns, v, tot);
  }
  unsigned int status = 0;
  const cudaError_t le = cudaGetLastError();
  if (e == cudaSuccess) e = le;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&status, ns.status, sizeof(unsigned int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    cudaStreamSynchronize(s);                   // what was queued writes the outputs and the work space
    cudaGetLastError();
    esc::note_cuda_error(e);
    return ESCAPE_ECUDA;
  }
  return status ? ESCAPE_EINVAL : ESCAPE_OK;
}
