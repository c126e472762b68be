// graph.cu - device graph store: build from pairs, repack, export (batch updates: apply.cu).
//
// Section 3.2 of the paper defines a batch update as E^t = (E^{t-1} \ D) U I with
// effective deletions Delta^- = E^{t-1} \ E^t and insertions Delta^+ = E^t \ E^{t-1};
// Section 3.1 / 5.1.4 add a self-loop to every vertex (kept fixed across updates).
#include <algorithm>
#include <vector>

#include "prdf_graph.cuh"

namespace prdf {

#define CK(call)                                            \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) return cuda_fail(g, e_, #call);  \
  } while (0)

pr_status cuda_fail(Graph *g, cudaError_t e, const char *what) {
  g->err = std::string(what) + ": " + cudaGetErrorString(e);
  cudaGetLastError();
  return e == cudaErrorMemoryAllocation ? PR_ERR_OUT_OF_MEMORY : PR_ERR_CUDA;
}

template <class T>
static cudaError_t dalloc(T **p, uint64_t count) {
  *p = nullptr;
  if (alloc_fault()) return cudaErrorMemoryAllocation;
  return cudaMalloc((void **)p, sizeof(T) * (count ? count : 1));
}

cudaError_t alloc_pieces(std::initializer_list<Piece> pieces) {
  auto room = [](uint64_t bytes) { return (bytes + 255) & ~255ull; };  // 256-byte aligned, as cudaMalloc's
  uint64_t total = 0;
  for (const Piece &x : pieces) {
    *x.p = nullptr;
    total += room(x.bytes);
  }
  if (alloc_fault()) return cudaErrorMemoryAllocation;
  char *base = nullptr;
  const cudaError_t e = cudaMalloc((void **)&base, total);
  if (e != cudaSuccess) return e;
  for (const Piece &x : pieces) {
    *x.p = base;
    base += room(x.bytes);
  }
  return cudaSuccess;
}

static inline unsigned grid_for(uint64_t n, int threads = 256) {
  uint64_t g = (n + threads - 1) / threads;
  return (unsigned)std::max<uint64_t>(1, g);
}

// ------------------------------------------------------------------- kernels ----

__global__ void k_validate_pairs(const uint32_t *src, const uint32_t *dst, uint64_t m, uint32_t n, uint32_t *bad) {
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m && (src[i] >= n || dst[i] >= n)) atomicOr(bad, 1u);
}

// Keys (u << b | v) of the input pairs (self pairs become the sentinel), followed by the
// n self-loop keys when self_loops is set.
__global__ void k_make_keys(const uint32_t *src, const uint32_t *dst, uint64_t m_in, uint32_t n, int b,
                            int self_loops, uint64_t *keys) {
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m_in) {
    uint64_t u = src[i], v = dst[i];
    keys[i] = u == v ? kSentinel : ((u << b) | v);
  } else if (self_loops && i < m_in + n) {
    uint64_t v = i - m_in;
    keys[i] = (v << b) | v;
  }
}

__device__ __forceinline__ uint32_t unique_flag(const uint64_t *keys, uint64_t i) {
  uint64_t k = keys[i];
  return (k != kSentinel && (i == 0 || keys[i - 1] != k)) ? 1u : 0u;
}

__global__ void k_unique_flags(const uint64_t *keys, uint64_t m, uint32_t *flags) {
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) flags[i] = unique_flag(keys, i);
}

__global__ void k_compact_unique(const uint64_t *keys, const uint32_t *pos, uint64_t m, uint64_t *out,
                                 uint32_t *count) {
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  uint32_t f = unique_flag(keys, i);
  if (f) out[pos[i]] = keys[i];
  if (i == m - 1) *count = pos[i] + f;
}

// (v, u) keys; u by its place in the in-rows' order (lab), where that is another than by id
__global__ void k_transpose_keys(const uint64_t *keys, uint64_t m, int b, const uint32_t *lab, uint64_t *out) {
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  uint64_t k = keys[i], mask = (1ull << b) - 1;
  out[i] = ((k & mask) << b) | (lab ? (uint64_t)lab[k >> b] : k >> b);
}

// off[r] = index of the first key of row r (rows are key >> b); off[n] = m.
__global__ void k_row_bounds(const uint64_t *keys, uint64_t m, int b, uint32_t n, uint32_t *off) {
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i > m) return;
  int64_t prev = i == 0 ? -1 : (int64_t)(keys[i - 1] >> b);
  int64_t cur = i == m ? (int64_t)n : (int64_t)(keys[i] >> b);
  for (int64_t r = prev + 1; r <= cur; r++) off[r] = (uint32_t)i;
}

__global__ void k_row_caps(const uint32_t *off, uint32_t n, uint32_t *cap) {
  uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) cap[v] = slack_cap(off[v + 1] - off[v]);
}

__global__ void k_row_desc(const uint32_t *start, const uint32_t *off, uint32_t n, uint2 *rd) {
  uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) rd[v] = make_uint2(start[v], off[v + 1] - off[v]);
}

__global__ void k_scatter_cols(const uint64_t *keys, uint64_t m, int b, const uint32_t *off, const uint2 *rd,
                               uint32_t *col, const uint32_t *at) {
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  uint64_t k = keys[i];
  uint32_t r = (uint32_t)(k >> b);
  const uint32_t c = (uint32_t)(k & ((1ull << b) - 1));
  col[rd[r].x + (uint32_t)(i - off[r])] = at ? at[c] : c;
}

template <bool F32>
__global__ void k_init_rank(const uint2 *out_rd, uint32_t n, double alpha, typename Store<F32>::A *adeg,
                            typename Store<F32>::R *R0, typename Store<F32>::R *R1, typename Store<F32>::C *C0,
                            typename Store<F32>::C *C1) {
  using S = Store<F32>;
  uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  typename S::A a = S::factor(alpha, out_rd[v].y);
  typename S::R r = S::from_double(1.0 / (double)n);
  typename S::C c = S::contrib(r, a);
  adeg[v] = a;
  R0[v] = r;
  R1[v] = r;
  C0[v] = c;
  C1[v] = c;
}

// ---- repack / export / bins ----

__global__ void k_len_caps(const uint2 *rd, uint32_t n, uint32_t *cap) {
  uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) cap[v] = slack_cap(rd[v].y);
}

// One warp per row: copies the row to new_col + start[v] and points rd at it.
__global__ void k_repack_rows(uint2 *rd, uint32_t n, const uint32_t *old_col, uint32_t *new_col,
                              const uint32_t *start) {
  uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  uint32_t lane = threadIdx.x & 31;
  if (w >= n) return;
  uint2 d = rd[w];
  uint32_t s = start[w];
  for (uint32_t j = lane; j < d.y; j += 32) new_col[s + j] = old_col[d.x + j];
  __syncwarp();
  if (lane == 0) rd[w] = make_uint2(s, d.y);
}

__global__ void k_row_len(const uint2 *rd, uint32_t n, uint32_t *len) {
  uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) len[v] = rd[v].y;
  else if (v == n) len[v] = 0;
}

__global__ void k_pack_rows(const uint2 *rd, uint32_t n, const uint32_t *col, const uint32_t *off, uint32_t *packed) {
  uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  uint32_t lane = threadIdx.x & 31;
  if (w >= n) return;
  uint2 d = rd[w];
  uint32_t o = off[w];
  for (uint32_t j = lane; j < d.y; j += 32) packed[o + j] = col[d.x + j];
}

__global__ void k_dead_flags(const uint2 *rd, uint32_t n, uint32_t *flags) {
  uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) flags[v] = rd[v].y == 0;
}

// Stable compaction of the ids whose flag is set; count = total.
// Sweep-item rebuild in two passes over the vertices (tile of kIdentTile per block): the
// first counts each tile's vertices per tier and the chunk items of its tier-2 rows; after
// one exclusive scan of those counts (tier 0, 1, 2 tiles back to back, then the chunk
// counts), the second writes every vertex's item(s) at its place, in ascending vertex order
// within each tier.
constexpr uint32_t kIdentTile = 4096;

__global__ void k_tier_counts(const uint2 *rd, uint32_t n, uint32_t lo, uint32_t gmax, uint32_t chunk,
                              uint32_t nblk, uint32_t *bcnt, uint32_t *over) {
  __shared__ uint32_t s[4][8];
  const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint32_t base = blockIdx.x * kIdentTile;
  uint32_t c[4] = {0u, 0u, 0u, 0u};
  for (uint32_t k = tid; k < kIdentTile; k += 256) {
    const uint32_t v = base + k;
    if (v < n) {
      const uint32_t d = rd[v].y;
      const int t = sweep_tier(d, lo, gmax);
      c[t]++;
      if (t == 2) {
        const uint32_t ch = (d + chunk - 1) / chunk;
        c[3] += ch;
        if (ch > (1u << 21)) *over = 1u;  // a chunk's index within its row has 21 bits
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 4; j++) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c[j] += __shfl_xor_sync(0xffffffffu, c[j], o);
    if (lane == 0) s[j][w] = c[j];
  }
  __syncthreads();
  if (tid < 4) {
    uint32_t t = 0;
    for (int k = 0; k < 8; k++) t += s[tid][k];
    // tiers 0-2 back to back, a zero, the chunk counts, a zero
    bcnt[tid < 3 ? tid * nblk + blockIdx.x : 3 * nblk + 1 + blockIdx.x] = t;
  }
  if (blockIdx.x == 0 && tid == 0) {
    bcnt[3 * nblk] = 0u;
    bcnt[4 * nblk + 1] = 0u;
  }
}

__global__ void k_items_write(const uint2 *rd, uint32_t n, uint32_t lo, uint32_t gmax, uint32_t chunk,
                              uint32_t nblk, const uint32_t *bpos, uint4 *items, uint32_t *item_pos) {
  __shared__ uint32_t s[4][8];
  __shared__ uint32_t s_at[4];
  const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint32_t base = blockIdx.x * kIdentTile;
  // item positions of this tile's first vertex of tiers 0 and 1, and of its first chunk item
  // (the chunk items follow the items of tiers 0 and 1, bpos[2 * nblk] of them)
  const uint32_t c01 = bpos[2 * nblk];
  if (tid < 3) s_at[tid] = bpos[tid * nblk + blockIdx.x];
  if (tid == 3) s_at[3] = c01 + bpos[3 * nblk + 1 + blockIdx.x] - bpos[3 * nblk + 1];
  __syncthreads();
  for (uint32_t r0 = 0; r0 < kIdentTile; r0 += 256) {
    const uint32_t v = base + r0 + tid;
    uint2 d = make_uint2(0u, 0u);
    int t = -1;
    uint32_t ch = 0;
    if (v < n) {
      d = rd[v];
      t = sweep_tier(d.y, lo, gmax);
      if (t == 2) ch = (d.y + chunk - 1) / chunk;
    }
    // rank within the warp per tier, chunk prefix within the warp
    uint32_t m[3], incl = ch;
#pragma unroll
    for (int j = 0; j < 3; j++) m[j] = __ballot_sync(0xffffffffu, t == j);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    if (lane == 31) s[3][w] = incl;
    if (lane < 3) s[lane][w] = __popc(m[lane]);
    __syncthreads();
    uint32_t before[4] = {0u, 0u, 0u, 0u}, all[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int j = 0; j < 4; j++)
      for (int k = 0; k < 8; k++) {
        before[j] += k < (int)w ? s[j][k] : 0u;
        all[j] += s[j][k];
      }
    if (t >= 0 && t < 2) {
      const uint32_t pos = s_at[t] + before[t] + __popc(m[t] & ((1u << lane) - 1u));
      items[pos] = make_uint4(v, d.x, d.y, 0u);
      item_pos[v] = pos;
    } else if (t == 2) {
      const uint32_t first = s_at[3] + before[3] + incl - ch;  // index of the row's first chunk item
      const uint32_t number = first - c01;                     // its chunk number
      for (uint32_t c = 0; c < ch; c++) {
        const uint32_t len = min(chunk, d.y - c * chunk);
        items[first + c] = make_uint4(v, d.x + c * chunk, len | (c << 10) | (ch > 1 ? 0x80000000u : 0u), number + c);
      }
      item_pos[v] = first;
    }
    __syncthreads();
    if (tid < 4) s_at[tid] += all[tid];
    __syncthreads();
  }
}

__global__ void k_compact_ids(const uint32_t *flags, const uint32_t *pos, uint32_t n, uint32_t *out, uint32_t *count) {
  uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  if (flags[v]) out[pos[v]] = v;
  if (v == n - 1) *count = pos[v] + flags[v];
}

// ------------------------------------------------------------------ host side ---

static pr_status build_adj(Graph *g, const uint64_t *keys, uint64_t m, Adj &A, uint32_t *off, uint32_t *tmp,
                           uint32_t *scan_tmp, const uint32_t *at) {
  const uint32_t n = g->n;
  cudaStream_t st = g->st;
  CK(alloc_pieces({piece(&A.rd, n), piece(&A.cap, n)}));
  k_row_bounds<<<grid_for(m + 1), 256, 0, st>>>(keys, m, g->b, n, off); count_launch();
  k_row_caps<<<grid_for(n), 256, 0, st>>>(off, n, A.cap); count_launch();
  exclusive_scan_u32(A.cap, tmp, n, scan_tmp, st);
  uint32_t last[2];
  CK(cudaMemcpyAsync(&last[0], tmp + (n - 1), 4, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(&last[1], A.cap + (n - 1), 4, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  uint64_t total = (uint64_t)last[0] + last[1];
  uint64_t reserve = std::max<uint64_t>(total / 4, 1024);
  reserve = (reserve + 3) & ~3ull;
  if (total + reserve > 0xFFFFFFFFull) {
    g->err = "graph too large: more than 2^32 - 1 column slots";
    return PR_ERR_CAPACITY;
  }
  A.col_cap = total + reserve;
  CK(dalloc(&A.col, A.col_cap));
  CK(cudaMemsetAsync(A.col, 0xFF, sizeof(uint32_t) * A.col_cap, st));  // free slots: kNoCol
  k_row_desc<<<grid_for(n), 256, 0, st>>>(tmp, off, n, A.rd); count_launch();
  k_scatter_cols<<<grid_for(m), 256, 0, st>>>(keys, m, g->b, off, A.rd, A.col, at); count_launch();
  A.used = total;
  A.garbage = 0;
  CK(cudaGetLastError());
  return PR_OK;
}

pr_status graph_build(Graph *g, uint64_t m_in, const uint32_t *src_d, const uint32_t *dst_d) {
  const uint32_t n = g->n;
  cudaStream_t st = g->st;
  g->b = bits_for(n);
  const bool sl = !g->teleport;
  const uint64_t mk = m_in + (sl ? n : 0);
  // validation before anything else
  uint32_t *flag = nullptr;
  CK(dalloc(&flag, 1));
  CK(cudaMemsetAsync(flag, 0, 4, st));
  if (m_in) {
    k_validate_pairs<<<grid_for(m_in), 256, 0, st>>>(src_d, dst_d, m_in, n, flag);
    count_launch();
  }
  uint32_t bad = 0;
  CK(cudaMemcpyAsync(&bad, flag, 4, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  cudaFree(flag);
  if (bad) {
    g->err = "vertex id out of range";
    return PR_ERR_VERTEX_RANGE;
  }
  if ((double)mk * 1.13 + 6.0 * n > 4.0e9) {
    g->err = "graph too large: more than 2^32 - 1 column slots";
    return PR_ERR_CAPACITY;
  }
  // scratch for the build
  uint64_t *keys = nullptr, *alt = nullptr;
  uint32_t *flags = nullptr, *pos = nullptr, *hist = nullptr, *stmp = nullptr, *cnt = nullptr;
  const uint64_t mk1 = std::max<uint64_t>(mk, 1);
  const uint64_t big = std::max<uint64_t>(mk1 + 1, (uint64_t)n + 1);
  pr_status rc = PR_OK;
  auto cleanup = [&]() { cudaFree(keys); };
  cudaError_t e = alloc_pieces(
      {piece(&keys, mk1), piece(&alt, mk1), piece(&flags, big), piece(&pos, big),
       piece(&hist, std::max(radix_hist_words(mk1), scan_tmp_words(big)) + 1),
       piece(&stmp, scan_tmp_words(std::max<uint64_t>(big, radix_hist_words(mk1))) + 1), piece(&cnt, 1)});
  if (e != cudaSuccess) return cuda_fail(g, e, "graph build scratch");
  do {
    if (mk) {
    k_make_keys<<<grid_for(mk), 256, 0, st>>>(src_d, dst_d, m_in, n, g->b, sl ? 1 : 0, keys);
    count_launch();
  }
    uint64_t *sorted = sort_u64(keys, alt, mk, 2 * g->b, hist, stmp, st);
    uint64_t *other = sorted == keys ? alt : keys;
    uint32_t m = 0;
    if (mk) {
      k_unique_flags<<<grid_for(mk), 256, 0, st>>>(sorted, mk, flags); count_launch();
      exclusive_scan_u32(flags, pos, mk, stmp, st);
      k_compact_unique<<<grid_for(mk), 256, 0, st>>>(sorted, pos, mk, other, cnt); count_launch();
      if ((e = cudaMemcpyAsync(&m, cnt, 4, cudaMemcpyDeviceToHost, st)) != cudaSuccess) break;
      if ((e = cudaStreamSynchronize(st)) != cudaSuccess) break;
    }
    g->m = m;
    // out-adjacency from keys sorted by (u, v)
    rc = build_adj(g, other, m, g->out, flags, pos, stmp, nullptr);
    if (rc != PR_OK) break;
    // in-adjacency from transposed keys sorted by (v, u)
    if (m) {
    k_transpose_keys<<<grid_for(m), 256, 0, st>>>(other, m, g->b, g->lab, sorted);
    count_launch();
  }
    // the keys are in (u, v) order: a stable sort by v alone puts them in (v, u) order, unless
    // the in-rows are ordered by another key than u
    uint64_t *tsorted = sort_u64(sorted, other, m, 2 * g->b, hist, stmp, st, g->lab ? 0 : g->b);
    rc = build_adj(g, tsorted, m, g->in, flags, pos, stmp, g->at);
    if (rc != PR_OK) break;
    e = cudaStreamSynchronize(st);
  } while (0);
  cleanup();
  if (e != cudaSuccess) return cuda_fail(g, e, "graph build");
  if (rc != PR_OK) return rc;

  // scratch (gen_tmp also holds the sweep-item rebuild's 4 ceil(n / 4096) + 2 tile counts): all
  // that the vertex numbering needs of a transient build
  const uint64_t scan_words = scan_tmp_words((uint64_t)n + 8) + 1;
  if (g->transient) {
    CK(alloc_pieces({piece(&g->gen_tmp, (uint64_t)n + 8), piece(&g->gen_tmp2, (uint64_t)n + 8),
                     piece(&g->scan_tmp, scan_words), piece(&g->actl, 1)}));
    return PR_OK;
  }
  // ... and the rank state
  const uint64_t rank_bytes = (uint64_t)(g->f32 ? 4 : 8) * n;
  const uint32_t words = (n + 31) / 32;
  g->pend_cap = std::max<uint32_t>(1u << 16, std::min<uint32_t>(n, 1u << 22));
  // (a vertex is queued once per iteration, but initially once for every update of its row)
  const uint32_t hubs = std::max(n, g->pend_cap);
  CK(alloc_pieces({piece(&g->gen_tmp, (uint64_t)n + 8), piece(&g->gen_tmp2, (uint64_t)n + 8),
                   piece(&g->scan_tmp, scan_words), piece(&g->actl, 1), piece(&g->ctl, 1),
                   piece(&g->dpart, 2ull * kRankBlocksPerSm * g->sm_count),
                   Piece{&g->R[0], rank_bytes}, Piece{&g->R[1], rank_bytes}, Piece{&g->C[0], rank_bytes},
                   Piece{&g->C[1], rank_bytes}, Piece{&g->adeg, rank_bytes}, piece(&g->bitmap, words),
                   piece(&g->xbits, words), piece(&g->stamp, n), piece(&g->emap, 2ull * n), piece(&g->chunk_done, n),
                   piece(&g->item_pos, n), piece(&g->hub_v, hubs), piece(&g->hub_base, hubs), piece(&g->list[0], n),
                   piece(&g->list[1], n), piece(&g->list[2], n), piece(&g->xlist, n), piece(&g->dead, n),
                   piece(&g->pend_src, g->pend_cap), piece(&g->pend_tgt, g->pend_cap)}));
  CK(cudaMemsetAsync(g->bitmap, 0, 4ull * words, st));
  CK(cudaMemsetAsync(g->xbits, 0, 4ull * words, st));
  CK(cudaMemsetAsync(g->stamp, 0xFF, 2ull * n, st));
  CK(cudaMemsetAsync(g->emap, 0, 2ull * n, st));
  CK(cudaMemsetAsync(g->chunk_done, 0, 4ull * n, st));
  char *host = nullptr;
  const size_t actl_room = (sizeof(ApplyCtl) + 255) & ~(size_t)255;
  const size_t ctl_room = (sizeof(RankCtl) + 255) & ~(size_t)255;
  CK(cudaMallocHost((void **)&host, actl_room + ctl_room + 4ull * kPinnedIds));
  g->actl_h = (ApplyCtl *)host;
  g->ctl_h = (RankCtl *)(host + actl_room);
  g->ids_h = (uint32_t *)(host + actl_room + ctl_room);
  if (g->f32) {
    using S = Store<true>;
    k_init_rank<true><<<grid_for(n), 256, 0, st>>>(g->out.rd, n, g->p.alpha, (S::A *)g->adeg, (S::R *)g->R[0],
                                                   (S::R *)g->R[1], (S::C *)g->C[0], (S::C *)g->C[1]);
  } else {
    using S = Store<false>;
    k_init_rank<false><<<grid_for(n), 256, 0, st>>>(g->out.rd, n, g->p.alpha, (S::A *)g->adeg, (S::R *)g->R[0],
                                                    (S::R *)g->R[1], (S::C *)g->C[0], (S::C *)g->C[1]);
  }
  count_launch();
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(st));
  g->ident_dirty = true;
  g->dead_dirty = true;
  return graph_refresh_ident(g);
}

pr_status apply_scratch(Graph *g, uint64_t N) {
  ApplyScratch &s = g->sc;
  if (N <= s.cap && s.pairs) return PR_OK;
  uint64_t cap = std::max<uint64_t>(N, 4096);
  uint32_t *boff = s.boff;
  const int32_t boff_cap = s.boff_cap;
  cudaFree(s.pairs);
  s = ApplyScratch{};
  s.boff = boff;
  s.boff_cap = boff_cap;
  // (the plan of an update in one launch keeps 256 + 8 words a block there)
  s.radix_hist_cap = std::max<uint64_t>(radix_hist_words(cap) + 256, 264ull * g->sm_count);
  s.scan_tmp_cap = scan_tmp_words(std::max<uint64_t>(cap + 2, s.radix_hist_cap)) + 1;
  CK(alloc_pieces({piece(&s.pairs, 2 * cap), piece(&s.kd, cap), piece(&s.vals, cap), piece(&s.vals2, cap),
                   piece(&s.tmp, cap), piece(&s.tmp2, cap), piece(&s.chg, cap), piece(&s.chg_t, cap),
                   piece(&s.flags, cap + 2), piece(&s.pos, cap + 2), piece(&s.seg, 2 * (cap + 2)),
                   piece(&s.tagpref, 2 * (cap + 2)), piece(&s.radix_hist, s.radix_hist_cap),
                   piece(&s.scan_tmp, s.scan_tmp_cap)}));
  s.cap = cap;
  return PR_OK;
}

// Rebuilds adjacency A with fresh slack and at least `reserve` free tail words.  The sweep items
// hold the in-rows' starts, so they are rebuilt before the next sweep.
pr_status repack_adj(Graph *g, Adj &A, uint64_t reserve) {
  const uint32_t n = g->n;
  cudaStream_t st = g->st;
  // (the rows' own capacities change only once there is room: a failure leaves them as they are)
  uint32_t *caps = g->gen_tmp2;
  k_len_caps<<<grid_for(n), 256, 0, st>>>(A.rd, n, caps); count_launch();
  exclusive_scan_u32(caps, g->gen_tmp, n, g->scan_tmp, st);
  uint32_t last[2];
  CK(cudaMemcpyAsync(&last[0], g->gen_tmp + (n - 1), 4, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(&last[1], caps + (n - 1), 4, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  uint64_t total = (uint64_t)last[0] + last[1];
  reserve = std::max<uint64_t>(reserve, std::max<uint64_t>(total / 4, 1024));
  reserve = (reserve + 3) & ~3ull;
  if (total + reserve > 0xFFFFFFFFull) {
    g->err = "graph too large: more than 2^32 - 1 column slots";
    return PR_ERR_CAPACITY;
  }
  uint32_t *nc = nullptr;
  CK(dalloc(&nc, total + reserve));
  cudaError_t e = cudaMemsetAsync(nc, 0xFF, sizeof(uint32_t) * (total + reserve), st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(A.cap, caps, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) {
    cudaFree(nc);
    return cuda_fail(g, e, "repack");
  }
  k_repack_rows<<<grid_for((uint64_t)n * 32), 256, 0, st>>>(A.rd, n, A.col, nc, g->gen_tmp); count_launch();
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(st));
  cudaFree(A.col);
  A.col = nc;
  A.col_cap = total + reserve;
  A.used = total;
  A.garbage = 0;
  if (&A == &g->in) g->ident_dirty = true;
  return PR_OK;
}

pr_status graph_export(Graph *g, int dir, uint64_t *offs_h, uint32_t *cols_h) {
  const uint32_t n = g->n;
  cudaStream_t st = g->st;
  Adj &A = dir ? g->in : g->out;
  k_row_len<<<grid_for((uint64_t)n + 1), 256, 0, st>>>(A.rd, n, g->gen_tmp); count_launch();
  exclusive_scan_u32(g->gen_tmp, g->gen_tmp2, (uint64_t)n + 1, g->scan_tmp, st);
  uint32_t *packed = nullptr;
  CK(dalloc(&packed, std::max<uint64_t>(g->m, 1)));
  k_pack_rows<<<grid_for((uint64_t)n * 32), 256, 0, st>>>(A.rd, n, A.col, g->gen_tmp2, packed); count_launch();
  std::vector<uint32_t> off(n + 1);
  std::vector<uint32_t> icols;
  if (g->perm) icols.resize(g->m);
  uint32_t *dst_cols = g->perm ? icols.data() : cols_h;
  cudaError_t e = cudaMemcpyAsync(off.data(), g->gen_tmp2, 4ull * (n + 1), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(dst_cols, packed, 4ull * g->m, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(packed);
  if (e != cudaSuccess) return cuda_fail(g, e, "export csr");
  if (!g->perm) {
    for (uint32_t v = 0; v <= n; v++) offs_h[v] = off[v];
    return PR_OK;
  }
  // rows and columns back in the caller's numbering, each row sorted
  std::vector<uint32_t> perm(n), inv(n);
  CK(cudaMemcpyAsync(perm.data(), g->perm, 4ull * n, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  for (uint32_t r = 0; r < n; r++) inv[perm[r]] = r;
  uint64_t at = 0;
  for (uint32_t v = 0; v < n; v++) {
    offs_h[v] = at;
    const uint32_t r = inv[v];
    for (uint32_t j = off[r]; j < off[r + 1]; j++) cols_h[at++] = perm[icols[j]];
    std::sort(cols_h + offs_h[v], cols_h + at);
  }
  offs_h[n] = at;
  return PR_OK;
}

pr_status graph_refresh_ident(Graph *g) {
  if (!g->ident_dirty) return PR_OK;
  const uint32_t n = g->n;
  cudaStream_t st = g->st;
  uint32_t *over = (uint32_t *)&g->actl->n_seg_out;  // reuse a device word
  const uint32_t lo = (uint32_t)g->p.bin_lo, gmax = g->group_max, chunk = g->chunk_len;
  const uint32_t nblk = (uint32_t)(((uint64_t)n + kIdentTile - 1) / kIdentTile);
  const uint64_t len = 4ull * nblk + 2;  // tiers 0-2, 0, chunk counts, 0 (<= n + 8: fits gen_tmp)
  CK(cudaMemsetAsync(over, 0, 4, st));
  k_tier_counts<<<nblk, 256, 0, st>>>(g->in.rd, n, lo, gmax, chunk, nblk, g->gen_tmp, over);
  count_launch();
  exclusive_scan_u32(g->gen_tmp, g->gen_tmp2, len, g->scan_tmp, st);
  uint32_t h[4] = {0, 0, 0, 0};  // tier-0 count, tiers 0+1, n + chunk items, over
  CK(cudaMemcpyAsync(&h[0], g->gen_tmp2 + nblk, 4, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(&h[1], g->gen_tmp2 + 2 * nblk, 4, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(&h[2], g->gen_tmp2 + len - 1, 4, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(&h[3], over, 4, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  if (h[3]) {
    g->err = "a vertex has more in-edges than 2^21 sweep chunks hold (raise chunk_len)";
    return PR_ERR_CAPACITY;
  }
  const uint32_t c01 = h[1], total = h[2] - n;
  if ((uint64_t)c01 + total > g->items_cap || total > g->chunk_cap) {  // items, and partials by chunk number
    cudaFree(g->items);
    g->items = g->items_cmp = nullptr;
    g->partials = nullptr;
    g->items_cap = g->chunk_cap = 0;
    uint64_t chunks = (uint64_t)total + total / 4 + 1024;
    uint64_t cap = (uint64_t)n + chunks;
    CK(alloc_pieces({piece(&g->items, cap), piece(&g->items_cmp, cap), Piece{&g->partials, 8 * chunks}}));
    g->items_cap = cap;
    g->chunk_cap = chunks;
  }
  k_items_write<<<nblk, 256, 0, st>>>(g->in.rd, n, lo, gmax, chunk, nblk, g->gen_tmp2, g->items, g->item_pos);
  count_launch();
  CK(cudaGetLastError());
  g->item_cnt[0] = h[0];
  g->item_cnt[1] = c01 - h[0];
  g->item_cnt[2] = total;
  g->ident_dirty = false;
  return g->comp_item ? batch_items(g) : PR_OK;
}

pr_status graph_refresh_dead(Graph *g) {
  if (!g->dead_dirty) return PR_OK;
  const uint32_t n = g->n;
  cudaStream_t st = g->st;
  uint32_t *cnt = (uint32_t *)&g->actl->n_seg_in;
  k_dead_flags<<<grid_for(n), 256, 0, st>>>(g->out.rd, n, g->gen_tmp); count_launch();
  exclusive_scan_u32(g->gen_tmp, g->gen_tmp2, n, g->scan_tmp, st);
  k_compact_ids<<<grid_for(n), 256, 0, st>>>(g->gen_tmp, g->gen_tmp2, n, g->dead, cnt); count_launch();
  uint32_t c = 0;
  CK(cudaMemcpyAsync(&c, cnt, 4, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  g->n_dead = c;
  g->dead_dirty = false;
  return PR_OK;
}

__global__ void k_fill_comp(uint16_t *comp, uint32_t first, uint32_t count, uint16_t c) {
  uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) comp[first + i] = c;
}

// One thread per vertex: flags an out-edge that leaves the vertex's graph.
__global__ void k_check_comp(const uint2 *rd, const uint32_t *col, const uint16_t *comp, uint32_t n, uint32_t *bad) {
  uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= n) return;
  uint2 d = rd[u];
  for (uint32_t j = 0; j < d.y; j++)
    if (comp[col[d.x + j]] != comp[u]) {
      atomicOr(bad, 1u);
      return;
    }
}

template <bool F32>
__global__ void k_init_comp_rank(const uint16_t *comp, uint32_t n, const typename Store<F32>::R *init,
                                 const typename Store<F32>::A *adeg, typename Store<F32>::R *R0,
                                 typename Store<F32>::R *R1, typename Store<F32>::C *C0, typename Store<F32>::C *C1) {
  using S = Store<F32>;
  uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  typename S::R r = init[comp[v]];
  typename S::C c = S::contrib(r, adeg[v]);
  R0[v] = r;
  R1[v] = r;
  C0[v] = c;
  C1[v] = c;
}

template <bool F32>
__global__ void k_comp_consts(const uint32_t *first, uint32_t ncomp, double alpha, typename Store<F32>::R *base,
                              typename Store<F32>::R *init) {
  using S = Store<F32>;
  uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncomp) return;
  double nc = (double)(first[c + 1] - first[c]);
  base[c] = S::from_double((1.0 - alpha) / nc);
  init[c] = S::from_double(1.0 / nc);
}

pr_status components_setup(Graph *g, const std::vector<uint32_t> &comp_n) {
  const uint32_t n = g->n, nc = (uint32_t)comp_n.size();
  cudaStream_t st = g->st;
  g->ncomp = nc;
  g->comp_first.assign(nc + 1, 0);
  for (uint32_t c = 0; c < nc; c++) g->comp_first[c + 1] = g->comp_first[c] + comp_n[c];
  CK(dalloc(&g->comp, n));
  for (uint32_t c = 0; c < nc; c++) {
    k_fill_comp<<<grid_for(comp_n[c]), 256, 0, st>>>(g->comp, g->comp_first[c], comp_n[c], (uint16_t)c);
    count_launch();
  }
  uint32_t *bad = nullptr, *first_d = nullptr;
  CK(dalloc(&bad, 1));
  CK(dalloc(&first_d, nc + 1));
  CK(cudaMemsetAsync(bad, 0, 4, st));
  CK(cudaMemcpyAsync(first_d, g->comp_first.data(), 4ull * (nc + 1), cudaMemcpyHostToDevice, st));
  k_check_comp<<<grid_for(n), 256, 0, st>>>(g->out.rd, g->out.col, g->comp, n, bad);
  count_launch();
  uint32_t hbad = 0;
  CK(cudaMemcpyAsync(&hbad, bad, 4, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  cudaFree(bad);
  if (hbad) {
    cudaFree(first_d);
    g->err = "an edge joins two different graphs of a batched handle";
    return PR_ERR_INVALID_ARG;
  }
  CK(cudaMalloc(&g->comp_base, 8ull * nc));
  CK(cudaMalloc(&g->comp_init, 8ull * nc));
  CK(dalloc(&g->dRc, 3ull * nc));
  CK(dalloc(&g->comp_x, 3ull * nc));
  CK(dalloc(&g->comp_hot, nc));
  CK(dalloc(&g->comp_item, 3ull * (nc + 1)));
  // a graph's first vertices, as many as fit an SM's shared copy: numbered by out-degree where
  // the graph is larger and the handle has an internal numbering
  std::vector<uint32_t> hot(nc);
  for (uint32_t c = 0; c < nc; c++)
    hot[c] = g->comp_hot_h.empty() ? std::min(comp_n[c], hot_limit(g->f32)) : g->comp_hot_h[c];
  CK(cudaMemcpyAsync(g->comp_hot, hot.data(), 4ull * nc, cudaMemcpyHostToDevice, st));
  CK(dalloc(&g->comp_out, 4ull * nc));
  CK(dalloc(&g->comp_last, nc));
  if (g->f32) {
    using S = Store<true>;
    k_comp_consts<true><<<grid_for(nc), 256, 0, st>>>(first_d, nc, g->p.alpha, (S::R *)g->comp_base, (S::R *)g->comp_init);
    count_launch();
    k_init_comp_rank<true><<<grid_for(n), 256, 0, st>>>(g->comp, n, (const S::R *)g->comp_init, (const S::A *)g->adeg,
                                                        (S::R *)g->R[0], (S::R *)g->R[1], (S::C *)g->C[0],
                                                        (S::C *)g->C[1]);
  } else {
    using S = Store<false>;
    k_comp_consts<false><<<grid_for(nc), 256, 0, st>>>(first_d, nc, g->p.alpha, (S::R *)g->comp_base,
                                                       (S::R *)g->comp_init);
    count_launch();
    k_init_comp_rank<false><<<grid_for(n), 256, 0, st>>>(g->comp, n, (const S::R *)g->comp_init,
                                                         (const S::A *)g->adeg, (S::R *)g->R[0], (S::R *)g->R[1],
                                                         (S::C *)g->C[0], (S::C *)g->C[1]);
  }
  count_launch();
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(st));
  g->comp_first_d = first_d;
  g->comp_stats.assign(nc, pr_stats{});
  return PR_OK;
}

void graph_free(Graph *g) {
  for (auto &at : g->served) {
    std::lock_guard<std::mutex> lk(at->mu);
    at->g = nullptr;
  }
  sweep_free(g);
  Adj *adjs[2] = {&g->out, &g->in};
  // (what alloc_pieces gave is owned by the first array of each group)
  for (Adj *A : adjs) {
    cudaFree(A->rd);
    cudaFree(A->col);
  }
  cudaFree(g->gen_tmp);
  cudaFree(g->items);
  cudaFree(g->sc.pairs);
  cudaFree(g->sc.boff);
  cudaFree(g->comp);
  cudaFree(g->comp_base);
  cudaFree(g->comp_init);
  cudaFree(g->dRc);
  cudaFree(g->comp_x);
  cudaFree(g->comp_first_d);
  cudaFree(g->comp_hot);
  cudaFree(g->comp_item);
  cudaFree(g->comp_out);
  cudaFree(g->comp_last);
  if (g->actl_h) cudaFreeHost(g->actl_h);
  cudaFree(g->big);
  cudaFree(g->longs);
  cudaFree(g->perm);
  cudaFree(g->lab);
  if (g->cg_exec) cudaGraphExecDestroy(g->cg_exec);
  if (g->cg) cudaGraphDestroy(g->cg);
  if (g->ev0) cudaEventDestroy(g->ev0);
  if (g->ev1) cudaEventDestroy(g->ev1);
}

}  // namespace prdf
