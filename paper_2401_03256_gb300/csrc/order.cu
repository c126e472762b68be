// order.cu - the internal vertex numbering of single-graph handles.
//
// The sweeps gather one contribution per in-edge, and their cost is the number of distinct
// 32-byte sectors those gathers touch.  A breadth-first numbering (over out- and in-edges
// together) gives the vertices discovered from one vertex consecutive numbers, so the
// short rows that a warp sweeps side by side gather from nearby contributions.  Two are
// computed, from different first levels:
//  kOrderFromMax: the vertex of largest degree (graphs with hubs, such as R-MAT: its
//    neighbourhood is most of the graph within a few levels);
//  kOrderFromSeeds: max(kSeeds, n / kSeedCell) vertices evenly spaced in the caller's
//    numbering (graphs of large diameter, such as chains of k-mers, which one seed would
//    cover only at one level per few dozen vertices).
//  kOrderPerGraph (batched handles): the vertex of largest degree of every graph, then a
//    stable sort by graph, so that each graph keeps its id range and within it the order
//    of its own breadth-first search from that vertex.
// Level by level, a newly reached vertex takes its place after the vertices reached from
// earlier-numbered vertices of the previous level (the earliest adjacent one decides),
// ties by vertex id; vertices not reached within kMaxLevels levels follow in id order.
// Each level costs a few launches and one host synchronisation.  A handle keeps the
// numbering whose modelled short-row gathers (order_cost) touch the fewest sectors, if
// that is at least 5% fewer than under the caller's numbering: a grid numbered row by row
// already gathers consecutive contributions.  (Putting the vertices of largest out-degree
// side by side was measured slower: a fifth of the gathers then fall in one 64 KB run,
// whose few L2 slices serve them while the others wait.)  Ranks, results and the update
// semantics do not depend on the numbering: ids are translated at the boundary (batches,
// ranks in and out, affected sets, CSR export).
#include <algorithm>
#include <cstdint>
#include <vector>

#include "prdf_graph.cuh"

namespace prdf {

#define CK(call)                                            \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) return cuda_fail(g, e_, #call);  \
  } while (0)

namespace {

constexpr uint32_t kUnset = 0xFFFFFFFFu;
constexpr int kMaxLevels = 1024;
constexpr uint32_t kSeeds = 8192;     // at least this many seeds,
constexpr uint32_t kSeedCell = 2048;  // and one per this many vertices (a cell of a few hundred levels at most)

__global__ void k_order_init(uint32_t n, uint32_t *label, uint32_t *cand) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) {
    label[v] = kUnset;
    cand[v] = kUnset;
  }
}

// the vertex of largest out + in degree (smallest id on ties): a max of (degree << 32 | ~v)
__global__ void k_order_seed(const uint2 *out_rd, const uint2 *in_rd, uint32_t n, unsigned long long *best) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long key = 0;
  if (v < n) key = ((unsigned long long)(out_rd[v].y + in_rd[v].y) << 32) | (unsigned long long)(~v);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, key, o);
    key = y > key ? y : key;
  }
  if ((threadIdx.x & 31) == 0 && key) atomicMax(best, key);
}

__global__ void k_order_start(const unsigned long long *best, uint32_t *label, uint32_t *perm) {
  const uint32_t s = ~(uint32_t)(*best & 0xFFFFFFFFull);
  label[s] = 0;
  perm[0] = s;
}

// graph of vertex v (first[c] <= v < first[c + 1]; nc <= kMaxComponents)
__device__ __forceinline__ uint32_t graph_of(const uint32_t *first, uint32_t nc, uint32_t v) {
  uint32_t lo = 0, hi = nc;  // last c with first[c] <= v
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (first[mid] <= v) lo = mid; else hi = mid;
  }
  return lo;
}

__global__ void k_order_graph_of(const uint32_t *first, uint32_t nc, uint32_t n, uint32_t *gid) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) gid[v] = graph_of(first, nc, v);
}

// every graph's vertex of largest out + in degree (smallest id on ties)
__global__ void k_order_graph_seed(const uint2 *out_rd, const uint2 *in_rd, const uint32_t *gid, uint32_t n,
                                   unsigned long long *best) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) atomicMax(best + gid[v], ((unsigned long long)(out_rd[v].y + in_rd[v].y) << 32) | (unsigned long long)(~v));
}

// level 0 of kOrderPerGraph: the graphs' seeds in graph order (graphs without vertices
// have none); one thread
__global__ void k_order_graph_start(const unsigned long long *best, uint32_t nc, uint32_t *label, uint32_t *perm,
                                    uint32_t *count) {
  uint32_t k = 0;
  for (uint32_t c = 0; c < nc; c++) {
    if (!best[c]) continue;
    const uint32_t s = ~(uint32_t)(best[c] & 0xFFFFFFFFull);
    label[s] = k;
    perm[k++] = s;
  }
  *count = k;
}

// sort keys of the final order: graph, then breadth-first number
__global__ void k_order_graph_keys(const uint32_t *gid, const uint32_t *label, uint32_t n, unsigned long long *keys) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) keys[v] = ((unsigned long long)gid[v] << 32) | label[v];
}

__global__ void k_order_graph_perm(const unsigned long long *sorted, const uint32_t *rank_perm, uint32_t n,
                                   uint32_t *perm, uint32_t *inv) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    const uint32_t v = rank_perm[(uint32_t)(sorted[i] & 0xFFFFFFFFull)];
    perm[i] = v;
    inv[v] = i;
  }
}

// level 0 of kOrderFromSeeds: seed i is vertex i * step
__global__ void k_order_seeds(uint32_t k, uint32_t step, uint32_t *label, uint32_t *perm) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < k) {
    label[i * step] = i;
    perm[i] = i * step;
  }
}

// One level: every vertex of the frontier (perm[lo, hi), numbered lo..hi-1) offers its
// number to its unnumbered neighbours (out- and in-rows, one warp per frontier vertex); a
// neighbour keeps the smallest offer, and its first offer lists it (the warp's new ones with
// one atomic).  Rows longer than kOrderRow are queued (long_v: 2 k + direction; long_base: first
// segment) for a second launch: with a warp to every row, two levels of an R-MAT graph of scale
// 20 took 9 ms (now 1.8 ms in all).
constexpr uint32_t kOrderRow = 1024, kOrderSeg = 256;
__device__ __forceinline__ void order_offer(const uint32_t *col, uint32_t len, uint32_t k, uint32_t lane,
                                            const uint32_t *label, uint32_t *cand, uint32_t *next, uint32_t *cnt) {
  for (uint32_t j0 = 0; j0 < len; j0 += 32) {  // the same rounds for the whole warp
    const uint32_t j = j0 + lane;
    uint32_t w = 0;
    bool fresh = false;
    if (j < len) {
      w = col[j];
      // an earlier offer seen here or one that arrives later: the smallest stays either way
      if (label[w] == kUnset && *(volatile uint32_t *)&cand[w] > k) fresh = atomicMin(&cand[w], k) == kUnset;
    }
    const uint32_t mask = __ballot_sync(0xffffffffu, fresh);
    if (mask) {
      const uint32_t leader = __ffs(mask) - 1, me = threadIdx.x & 31;
      uint32_t base = 0;
      if (me == leader) base = atomicAdd(cnt, (uint32_t)__popc(mask));
      base = __shfl_sync(0xffffffffu, base, leader);
      if (fresh) next[base + __popc(mask & ((1u << me) - 1u))] = w;
    }
  }
}

__global__ void k_order_expand(const uint2 *out_rd, const uint32_t *out_col, const uint2 *in_rd,
                               const uint32_t *in_col, const uint32_t *perm, uint32_t lo, uint32_t hi,
                               const uint32_t *label, uint32_t *cand, uint32_t *next, uint32_t *cnt,
                               unsigned long long *queue, uint32_t *long_v, uint32_t *long_base) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t k = lo + ((blockIdx.x * blockDim.x + threadIdx.x) >> 5); k < hi; k += nwarps) {
    const uint32_t u = perm[k];
    for (uint32_t dir = 0; dir < 2; dir++) {
      const uint2 d = dir ? in_rd[u] : out_rd[u];
      if (d.y > kOrderRow) {
        if (lane == 0) {  // entry and first segment from one atomic, so bases ascend
          const unsigned long long old = atomicAdd(queue, (1ull << 32) | ((d.y + kOrderSeg - 1) / kOrderSeg));
          long_v[old >> 32] = 2 * (k - lo) + dir;
          long_base[old >> 32] = (uint32_t)old;
        }
        continue;
      }
      order_offer((dir ? in_col : out_col) + d.x, d.y, k, lane, label, cand, next, cnt);
    }
  }
}

// The long rows of a level, in segments dealt to the warps of the grid.
__global__ void k_order_expand_long(const uint2 *out_rd, const uint32_t *out_col, const uint2 *in_rd,
                                    const uint32_t *in_col, const uint32_t *perm, uint32_t lo, const uint32_t *label,
                                    uint32_t *cand, uint32_t *next, uint32_t *cnt, const unsigned long long *queue,
                                    const uint32_t *long_v, const uint32_t *long_base) {
  const uint32_t lane = threadIdx.x & 31, nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t n_long = (uint32_t)(*queue >> 32), n_seg = (uint32_t)*queue;
  for (uint32_t s = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < n_seg; s += nwarps) {
    uint32_t a = 0, b = n_long;  // the row: last with long_base <= s
    while (b - a > 1) {
      const uint32_t mid = (a + b) >> 1;
      if (long_base[mid] <= s) a = mid; else b = mid;
    }
    const uint32_t x = long_v[a], k = lo + (x >> 1), u = perm[k], at = (s - long_base[a]) * kOrderSeg;
    const uint2 d = (x & 1) ? in_rd[u] : out_rd[u];
    order_offer(((x & 1) ? in_col : out_col) + d.x + at, min(kOrderSeg, d.y - at), k, lane, label, cand, next, cnt);
  }
}

__global__ void k_order_keys(const uint32_t *next, uint32_t cnt, const uint32_t *cand, unsigned long long *keys) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < cnt) keys[i] = ((unsigned long long)cand[next[i]] << 32) | next[i];
}

__global__ void k_order_assign(const unsigned long long *keys, uint32_t cnt, uint32_t base, uint32_t *label,
                               uint32_t *perm) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < cnt) {
    const uint32_t w = (uint32_t)(keys[i] & 0xFFFFFFFFull);
    label[w] = base + i;
    perm[base + i] = w;
  }
}

__global__ void k_order_unset_flags(const uint32_t *label, uint32_t n, uint32_t *flags) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) flags[v] = label[v] == kUnset ? 1u : 0u;
}

__global__ void k_order_rest(const uint32_t *flags, const uint32_t *pos, uint32_t n, uint32_t base, uint32_t *label,
                             uint32_t *perm) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n && flags[v]) {
    label[v] = base + pos[v];
    perm[base + pos[v]] = v;
  }
}

// The gather cost model that decides whether the new numbering is kept: the rows of at
// most kScoreRowMax in-edges are swept 32 consecutive rows a warp, one in-edge per lane per
// step, as the short-row tiers do; each step costs one request per distinct 32-byte sector
// among the lanes' contributions.  cnt[0] sums those sectors under the caller's
// numbering, cnt[1] under the new one.  (Long rows gather about one sector per in-edge in
// any numbering: their in-neighbours are spread over the graph.)
constexpr uint32_t kScoreRowMax = 64;

__global__ void k_order_score(const uint2 *in_rd, const uint32_t *in_col, const uint32_t *perm,
                              const uint32_t *inv, uint32_t n, int sec_shift, unsigned long long *cnt) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t ngroups = (uint32_t)(((uint64_t)n + 31) / 32);
  unsigned long long sec[2] = {0, 0};
  for (uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < ngroups; w += nwarps) {
    const uint32_t pos = w * 32 + lane;
    for (int mode = 0; mode < 2; mode++) {
      uint2 d = make_uint2(0, 0);
      if (pos < n) {
        d = in_rd[mode ? perm[pos] : pos];
        if (d.y > kScoreRowMax) d.y = 0;
      }
      uint32_t dmax = d.y;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dmax = max(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
      for (uint32_t k = 0; k < dmax; k++) {
        const bool act = k < d.y;
        const unsigned am = __ballot_sync(0xffffffffu, act);
        if (act) {
          uint32_t c = in_col[d.x + k];
          if (mode) c = inv[c];
          const unsigned peers = __match_any_sync(am, c >> sec_shift);
          if ((uint32_t)(__ffs(peers) - 1) == lane) sec[mode]++;
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sec[0] += __shfl_xor_sync(0xffffffffu, sec[0], o);
    sec[1] += __shfl_xor_sync(0xffffffffu, sec[1], o);
  }
  if (lane == 0) {
    if (sec[0]) atomicAdd(&cnt[0], sec[0]);
    if (sec[1]) atomicAdd(&cnt[1], sec[1]);
  }
}

__global__ void k_map_ids(const uint32_t *inv, uint32_t *a, uint64_t m) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) a[i] = inv[a[i]];
}

// Out-degrees by graph, counted by degree (kHotBins and above together; below kHotLeast not at
// all: such vertices are never put first).  Graphs of at most hot_max vertices are left out.
constexpr uint32_t kHotBins = 2048, kHotLeast = 4;
__global__ void k_hot_hist(const uint2 *out_rd, const uint32_t *first, uint32_t nc, uint32_t hot_max, uint32_t n,
                           uint32_t *hist) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const uint32_t d = out_rd[v].y;
  if (d < kHotLeast) return;
  const uint32_t c = graph_of(first, nc, v);
  if (first[c + 1] - first[c] > hot_max) atomicAdd(&hist[c * kHotBins + min(d, kHotBins - 1)], 1u);
}

// flags of the hot vertices by place in the numbering, and the sum of their out-degrees
__global__ void k_hot_flags(const uint2 *out_rd, const uint32_t *perm, const uint32_t *first, const uint32_t *least,
                            uint32_t nc, uint32_t n, uint32_t *flags, unsigned long long *edges) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long d = 0;
  if (i < n) {
    const uint32_t y = out_rd[perm[i]].y;
    const bool f = y >= least[graph_of(first, nc, i)];
    flags[i] = f ? 1u : 0u;
    d = f ? y : 0u;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
  if ((threadIdx.x & 31) == 0 && d) atomicAdd(edges, d);
}

// the numbering with every graph's flagged places (the first hot[c] of them) at its front
__global__ void k_hot_perm(const uint32_t *flags, const uint32_t *pos, const uint32_t *first, const uint32_t *hots,
                           uint32_t nc, uint32_t n, const uint32_t *old, uint32_t *perm, uint32_t *inv, uint32_t *lab,
                           uint32_t *at) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t c = graph_of(first, nc, i), b = first[c], hot = hots[c];
  const uint32_t p = pos[i] - pos[b];  // flagged places of the graph before this one
  const bool f = flags[i] && p < hot;
  const uint32_t k = f ? b + p : b + hot + (i - b - min(p, hot));
  perm[k] = old[i];
  inv[old[i]] = k;
  if (lab) {
    lab[k] = i;
    at[i] = k;
  }
}

unsigned grid_of(uint64_t n) { return (unsigned)std::max<uint64_t>(1, (n + 255) / 256); }

}  // namespace

pr_status vertex_order(Graph *g, int kind, uint32_t *perm, uint32_t *inv, const std::vector<uint32_t> *comp_n) {
  const uint32_t n = g->n;
  cudaStream_t st = g->st;
  pr_status rc = apply_scratch(g, n);
  if (rc != PR_OK) return rc;
  ApplyScratch &s = g->sc;
  // a level's counters, side by side: chains have a thousand levels, and each clears and reads them
  struct Level {
    uint32_t cnt, pad;
    unsigned long long queue;
  };
  static_assert(offsetof(ApplyCtl, reloc_out) - offsetof(ApplyCtl, n_seg_out) == offsetof(Level, queue),
                "the counters' place in the control block of updates");
  uint32_t *cand = s.flags, *next = s.pos, *cnt = (uint32_t *)&g->actl->n_seg_out;
  uint32_t *long_v = s.seg, *long_base = s.tagpref;  // 2 (cap + 2) words: both rows of every vertex
  unsigned long long *queue = &g->actl->reloc_out;
  unsigned long long *keys = (unsigned long long *)s.kd;
  k_order_init<<<grid_of(n), 256, 0, st>>>(n, inv, cand);
  count_launch();
  int b = 0;
  while (b < 32 && (1ull << b) < (uint64_t)n) b++;
  uint32_t lo = 0, hi;
  uint32_t *gid = nullptr;
  if (kind == kOrderPerGraph) {
    // graphs of a batched handle: one seed each
    const uint32_t nc = comp_n ? (uint32_t)comp_n->size() : 0u;
    if (!nc || nc > kMaxComponents) {
      g->err = "per-graph numbering needs the graphs' sizes";
      return PR_ERR_INVALID_ARG;
    }
    std::vector<uint32_t> first(nc + 1, 0);
    for (uint32_t c = 0; c < nc; c++) first[c + 1] = first[c] + (*comp_n)[c];
    uint32_t *first_d = g->gen_tmp;  // needed only until every vertex has its graph
    unsigned long long *best = (unsigned long long *)s.tmp2;
    CK(cudaMemcpyAsync(first_d, first.data(), 4ull * (nc + 1), cudaMemcpyHostToDevice, st));
    k_order_graph_of<<<grid_of(n), 256, 0, st>>>(first_d, nc, n, s.vals);
    count_launch();
    gid = s.vals;
    CK(cudaMemsetAsync(best, 0, 8ull * nc, st));
    k_order_graph_seed<<<grid_of(n), 256, 0, st>>>(g->out.rd, g->in.rd, gid, n, best);
    count_launch();
    k_order_graph_start<<<1, 1, 0, st>>>(best, nc, inv, perm, cnt);
    count_launch();
    CK(cudaMemcpyAsync(&hi, cnt, 4, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
  } else if (kind == kOrderFromSeeds) {
    const uint32_t k = std::min(n, std::max(kSeeds, n / kSeedCell)), step = n / k;
    k_order_seeds<<<grid_of(k), 256, 0, st>>>(k, step, inv, perm);
    count_launch();
    hi = k;
  } else {
    unsigned long long *best = (unsigned long long *)s.tmp2;
    CK(cudaMemsetAsync(best, 0, 8, st));
    k_order_seed<<<grid_of(n), 256, 0, st>>>(g->out.rd, g->in.rd, n, best);
    count_launch();
    k_order_start<<<1, 1, 0, st>>>(best, inv, perm);
    count_launch();
    hi = 1;
  }
  const unsigned egrid = (unsigned)std::max(1, g->sm_count * 8);
  for (int level = 0; hi > lo && level < kMaxLevels; level++) {
    CK(cudaMemsetAsync(cnt, 0, sizeof(Level), st));
    k_order_expand<<<egrid, 256, 0, st>>>(g->out.rd, g->out.col, g->in.rd, g->in.col, perm, lo, hi, inv, cand,
                                          next, cnt, queue, long_v, long_base);
    count_launch();
    Level h{};
    CK(cudaMemcpyAsync(&h, cnt, sizeof(Level), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    uint32_t c = h.cnt;
    if (h.queue) {
      k_order_expand_long<<<egrid, 256, 0, st>>>(g->out.rd, g->out.col, g->in.rd, g->in.col, perm, lo, inv, cand,
                                                 next, cnt, queue, long_v, long_base);
      count_launch();
      CK(cudaMemcpyAsync(&c, cnt, 4, cudaMemcpyDeviceToHost, st));
      CK(cudaStreamSynchronize(st));
    }
    if (c) {
      k_order_keys<<<grid_of(c), 256, 0, st>>>(next, c, cand, keys);
      count_launch();
      // keys: (offering number < n: b bits) << 32 | vertex id
      uint64_t *sorted = sort_u64((uint64_t *)keys, s.tmp, c, 32 + b, s.radix_hist, s.scan_tmp, st);
      k_order_assign<<<grid_of(c), 256, 0, st>>>((const unsigned long long *)sorted, c, hi, inv, perm);
      count_launch();
    }
    lo = hi;
    hi += c;
  }
  if (hi < n) {
    // vertices no edge path reaches from the first level, or none within kMaxLevels, in id order
    k_order_unset_flags<<<grid_of(n), 256, 0, st>>>(inv, n, g->gen_tmp);
    count_launch();
    exclusive_scan_u32(g->gen_tmp, g->gen_tmp2, n, g->scan_tmp, st);
    k_order_rest<<<grid_of(n), 256, 0, st>>>(g->gen_tmp, g->gen_tmp2, n, hi, inv, perm);
    count_launch();
  }
  if (kind == kOrderPerGraph) {
    // stable by graph: each graph keeps its id range, ordered by its own search
    const uint32_t nc = (uint32_t)comp_n->size();
    int cb = 1;
    while ((1u << cb) < nc) cb++;
    k_order_graph_keys<<<grid_of(n), 256, 0, st>>>(gid, inv, n, keys);
    count_launch();
    const unsigned long long *sorted =
        (const unsigned long long *)sort_u64((uint64_t *)keys, s.tmp, n, 32 + cb, s.radix_hist, s.scan_tmp, st);
    CK(cudaMemcpyAsync(next, perm, 4ull * n, cudaMemcpyDeviceToDevice, st));
    k_order_graph_perm<<<grid_of(n), 256, 0, st>>>(sorted, next, n, perm, inv);
    count_launch();
  }

  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(st));
  return PR_OK;
}

pr_status order_cost(Graph *g, const uint32_t *perm, const uint32_t *inv, uint64_t cost[2]) {
  cudaStream_t st = g->st;
  const uint32_t n = g->n;
  unsigned long long *cnt = (unsigned long long *)g->sc.tmp2, h[2] = {0, 0};
  CK(cudaMemsetAsync(cnt, 0, 16, st));
  const unsigned grid = (unsigned)std::max(1, g->sm_count * 8);
  // 8-byte contributions: 4 to a sector; 4-byte: 8
  k_order_score<<<grid, 256, 0, st>>>(g->in.rd, g->in.col, perm, inv, n, g->f32 ? 3 : 2, cnt);
  count_launch();
  CK(cudaMemcpyAsync(h, cnt, 16, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  cost[0] = h[0];
  cost[1] = h[1];
  return PR_OK;
}

// Every graph's first vertices, hot_max at most, become those of largest out-degree: the
// sweeps keep their contributions in shared memory.  R-MAT graphs take 16 K (64-bit) or 32 K (FP32) of
// them: 38% and 50% of the gathers at scale 22, 54% and 66% at scale 20 (edge factor 16), 70%
// and 80% at scale 18 (edge factor 8); graphs of at most hot_max vertices are copied whole, in any order.  Where the
// hot vertices have less than a tenth of the out-edges (grids, chains) the numbering is left
// as it is: a gather that can be hot costs two predicated loads.
pr_status hot_order(Graph *g, const std::vector<uint32_t> &comp_n, uint32_t hot_max, uint32_t *perm, uint32_t *inv,
                    std::vector<uint32_t> &hot, uint32_t *lab, uint32_t *at) {
  hot.clear();
  const uint32_t n = g->n, nc = (uint32_t)comp_n.size();
  cudaStream_t st = g->st;
  bool any = false;
  for (uint32_t k : comp_n) any = any || k > hot_max;
  if (!any) return PR_OK;
  pr_status rc = apply_scratch(g, std::max<uint64_t>(n, (uint64_t)nc * kHotBins));
  if (rc != PR_OK) return rc;
  ApplyScratch &s = g->sc;
  uint32_t *hist = s.vals, *flags = s.flags, *pos = s.pos, *old = s.vals2;
  uint32_t *first_d = s.seg, *least_d = s.seg + (nc + 1), *hot_d = least_d + nc;  // seg: 2 (cap + 2) words
  unsigned long long *edges = (unsigned long long *)s.tmp2;
  std::vector<uint32_t> first(nc + 1, 0), least(nc, kHotLeast);
  for (uint32_t c = 0; c < nc; c++) first[c + 1] = first[c] + comp_n[c];
  CK(cudaMemcpyAsync(first_d, first.data(), 4ull * (nc + 1), cudaMemcpyHostToDevice, st));
  CK(cudaMemsetAsync(hist, 0, 4ull * nc * kHotBins, st));
  CK(cudaMemsetAsync(edges, 0, 8, st));
  k_hot_hist<<<grid_of(n), 256, 0, st>>>(g->out.rd, first_d, nc, hot_max, n, hist);
  count_launch();
  std::vector<uint32_t> h((size_t)nc * kHotBins);
  CK(cudaMemcpyAsync(h.data(), hist, 4ull * h.size(), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  std::vector<uint32_t> counts(nc);
  for (uint32_t c = 0; c < nc; c++) {
    // the least degree of at most hot_max vertices (the bin of the largest degrees may hold
    // more: the first of them in the numbering are taken)
    const uint32_t *b = h.data() + (size_t)c * kHotBins;
    uint32_t d = kHotBins - 1, k = b[d];
    while (d > kHotLeast && k + b[d - 1] <= hot_max) k += b[--d];
    least[c] = comp_n[c] > hot_max ? d : 0xFFFFFFFFu;
    counts[c] = comp_n[c] > hot_max ? std::min(k, hot_max) : 0u;
  }
  CK(cudaMemcpyAsync(least_d, least.data(), 4ull * nc, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(hot_d, counts.data(), 4ull * nc, cudaMemcpyHostToDevice, st));
  k_hot_flags<<<grid_of(n), 256, 0, st>>>(g->out.rd, perm, first_d, least_d, nc, n, flags, edges);
  count_launch();
  unsigned long long he = 0;
  CK(cudaMemcpyAsync(&he, edges, 8, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  if (he * 10 < g->m) return PR_OK;
  exclusive_scan_u32(flags, pos, n, s.scan_tmp, st);
  CK(cudaMemcpyAsync(old, perm, 4ull * n, cudaMemcpyDeviceToDevice, st));
  k_hot_perm<<<grid_of(n), 256, 0, st>>>(flags, pos, first_d, hot_d, nc, n, old, perm, inv, lab, at);
  count_launch();
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(st));
  for (uint32_t c = 0; c < nc; c++) hot.push_back(comp_n[c] > hot_max ? counts[c] : comp_n[c]);
  return PR_OK;
}

// The three affected lists of a call one after another, in the caller's numbering.
struct IdLists {
  const uint32_t *ids[3];
  uint32_t count[3];
};
__global__ void k_gather_lists(const uint32_t *perm, const IdLists l, uint32_t *out, uint64_t k) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= k) return;
  uint64_t j = i;
  int b = 0;
  for (; b < 2 && j >= l.count[b]; b++) j -= l.count[b];
  const uint32_t v = l.ids[b][j];
  out[i] = perm ? perm[v] : v;
}

void gather_lists(const Graph *g, uint32_t *out, uint64_t k) {
  if (k == 0) return;
  IdLists l;
  for (int b = 0; b < 3; b++) {
    l.ids[b] = g->list[b];
    l.count[b] = g->last_list_cnt[b];
  }
  k_gather_lists<<<grid_of(k), 256, 0, g->st>>>(g->perm, l, out, k);
  count_launch();
}

void map_ids(const uint32_t *inv, uint32_t *a, uint64_t m, cudaStream_t st) {
  if (m == 0) return;
  k_map_ids<<<grid_of(m), 256, 0, st>>>(inv, a, m);
  count_launch();
}

}  // namespace prdf
