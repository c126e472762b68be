// apply.cu - batch updates of the device graph store (Section 3.2).
//
// E^t = (E^{t-1} \ D) U I; the effective changes are Delta^- = E^{t-1} \ E^t and
// Delta^+ = E^t \ E^{t-1}.  Two stages, a host synchronisation after each:
//   plan    keys (u << b | v) of the requested pairs in sequence order -> stable sort -> the
//           last request on each edge decides its state, and the edges whose state changes are
//           the effective changes (self pairs, duplicates, deletions of absent edges, deletions
//           that are re-inserted and insertions of present edges drop out) -> tagged change
//           list in (u, v) order and a transposed copy in (v, u) order -> segments = touched
//           rows, with the room they need.  One cooperative launch (k_plan).
//   merge   every touched row of both adjacencies with its changes, in place if the row's
//           slots suffice, else into freshly allocated tail slots: a warp a row, the long
//           rows in slices dealt to all blocks.  The out-row merge also refreshes the row's
//           contribution alpha R[u] / |out(u)| and records the pending marks (sources and
//           deleted targets) for the next Dynamic Frontier call; the in-row merge keeps the
//           row's sweep items current.
#include <algorithm>
#include <cstring>
#include <vector>

#include "prdf_graph.cuh"

namespace prdf {

#define CK(call)                                            \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) return cuda_fail(g, e_, #call);  \
  } while (0)

namespace {

inline unsigned grid_for(uint64_t n, int threads = 256) {
  return (unsigned)std::max<uint64_t>(1, (n + threads - 1) / threads);
}

constexpr uint32_t kAllLanes = 0xffffffffu;

// ------------------------------------------------------------- per-request steps ----

__device__ __forceinline__ bool row_has(const uint2 *rd, const uint32_t *col, uint32_t u, uint32_t v) {
  uint2 d = rd[u];
  const uint32_t *c = col + d.x;
  uint32_t lo = 0, hi = d.y;
  while (lo < hi) {
    uint32_t mid = (lo + hi) >> 1;
    if (c[mid] < v) lo = mid + 1; else hi = mid;
  }
  return lo < d.y && c[lo] == v;
}

// Batch k of a sequence holding op x of one kind: the last k with off[k] <= x.
__device__ __forceinline__ uint32_t batch_of(const uint32_t *off, int nb, uint64_t x) {
  uint32_t lo = 0, hi = (uint32_t)nb;  // off[0] = 0 <= x
  while (hi - lo > 1) {
    uint32_t mid = (lo + hi) >> 1;
    if (off[mid] <= x) lo = mid; else hi = mid;
  }
  return lo;
}

// The requests of a sequence of batches: off = [del offsets (nb + 1), ins offsets (nb + 1)], or
// null for a single batch.
struct Requests {
  const uint32_t *ds, *dd, *is, *id;
  uint64_t nd, ni;
  int nb;
  const uint32_t *off;
  uint32_t n;
  int b;
  const uint16_t *comp;
  const uint32_t *inv, *lab;  // internal numbering; in-rows' order (see the graph handle)
  const uint2 *out_rd;
  const uint32_t *out_col;
};

// Key (u << b | v) of request i, written at its place in the order D_0, I_0, D_1, I_1, ...
// (deletions before insertions inside a batch, Section 3.2), with the payload
// (place << 1) | is_insertion.
__device__ __forceinline__ void request_key(const Requests &q, uint64_t i, uint64_t *keys, uint32_t *vals,
                                            ApplyCtl *actl) {
  uint64_t u, v, at;
  uint32_t kind;
  if (i < q.nd) {
    u = q.ds[i];
    v = q.dd[i];
    kind = 0;
    at = q.off ? q.off[q.nb + 1 + batch_of(q.off, q.nb, i)] + i : i;
  } else {
    const uint64_t j = i - q.nd;
    u = q.is[j];
    v = q.id[j];
    kind = 1;
    at = q.off ? q.off[batch_of(q.off + q.nb + 1, q.nb, j) + 1] + j : q.nd + j;
  }
  uint64_t key;
  if (u >= q.n || v >= q.n) {
    atomicOr(&actl->bad_id, 1u);
    key = kSentinel;
  } else if (q.comp && q.comp[u] != q.comp[v]) {
    atomicOr(&actl->bad_comp, 1u);
    key = kSentinel;
  } else {
    if (q.inv) {  // the handle's internal numbering
      u = q.inv[u];
      v = q.inv[v];
    }
    key = u == v ? kSentinel : ((u << q.b) | v);
  }
  keys[at] = key;
  vals[at] = (uint32_t)(at << 1) | kind;
}

// After the stable sort every key's requests sit together in sequence order, so the last
// one fixes the edge's final state; true where that state differs from the graph's
// (an effective deletion or insertion).  Self pairs and repeated requests never count.
__device__ __forceinline__ bool is_change(const Requests &q, uint64_t k, uint64_t next, uint32_t val) {
  if (k == kSentinel || next == k) return false;
  const bool was = row_has(q.out_rd, q.out_col, (uint32_t)(k >> q.b), (uint32_t)(k & ((1ull << q.b) - 1)));
  return ((val & 1u) != 0) != was;
}

// Tagged change keys: (key << 1) | is_insertion, in row-major (u, v) order and a
// transposed (v, u) copy, u by its place in the in-rows' order.
__device__ __forceinline__ void emit_change(const Requests &q, uint64_t k, uint32_t val, uint32_t at, uint64_t *chg,
                                            uint64_t *chg_t) {
  const uint64_t tag = val & 1u, mask = (1ull << q.b) - 1;
  const uint64_t kt = ((k & mask) << q.b) | (q.lab ? (uint64_t)q.lab[k >> q.b] : k >> q.b);
  chg[at] = (k << 1) | tag;
  chg_t[at] = (kt << 1) | tag;
}

__device__ __forceinline__ uint32_t chg_row(uint64_t c, int b) { return (uint32_t)((c >> 1) >> b); }
__device__ __forceinline__ uint32_t chg_col(uint64_t c, int b) { return (uint32_t)((c >> 1) & ((1ull << b) - 1)); }

// Touched rows are merged by a warp if they have at most kWarpRow entries and kWarpChanges
// changes (8 warps stage both in 20 KB of shared memory, so the registers, not that, limit
// the warps in flight), in slices of kSlice entries otherwise.  The merge is bound by the
// latency of a row's few dependent reads, so what counts is rows in flight: a block of 256
// threads for every row, and one block of 1024 per row above 8192 entries, took 2.83 + 0.89
// ms for 263,427 pairs on an R-MAT graph of 16.8 M vertices, and rows by warps and slices take
// 0.44 + 1.05 ms (652 pairs on 4.2 M vertices: 0.15 to 0.034 ms, the hubs' rows no longer one
// block's work).
constexpr uint32_t kWarpRow = 512, kWarpChanges = 64, kSlice = 2048;
__device__ __forceinline__ bool long_row(uint32_t len, uint32_t changes) {
  return len > kWarpRow || changes > kWarpChanges;
}

// Room the merge of segment s of a change list needs: tail words of a row that must move, and
// staging words of a long row.
__device__ __forceinline__ void plan_row(const uint2 *rd, const uint32_t *cap, const uint64_t *chg, int b,
                                         const uint32_t *seg, const uint32_t *tagpref, uint32_t s,
                                         unsigned long long *reloc, ApplyCtl *actl) {
  const uint32_t s0 = __ldcg(seg + s), e = __ldcg(seg + s + 1);
  const uint32_t r = chg_row(__ldcg(chg + s0), b);
  const uint32_t nI = __ldcg(tagpref + e) - __ldcg(tagpref + s0), nD = (e - s0) - nI;
  const uint32_t len = rd[r].y, new_len = len - nD + nI;
  if (new_len > cap[r]) atomicAdd(reloc, (unsigned long long)move_cap(new_len));
  if (long_row(len, e - s0)) {
    atomicAdd(&actl->big_need, (unsigned long long)len);
    atomicAdd(&actl->n_long, 1u);
  }
}

// ----------------------------------------------------------------------- plan ----
//
// One cooperative launch of 1024-thread blocks, one per 1024 pairs up to one per SM; up to
// kPlanBlockSort pairs a single block, which needs no grid barriers and sorts in shared memory.
// Small and ordinary updates are bound by launches and dependent passes: a launch for every
// step (three and a scan per sort pass, two sorts) made 17 launches for 12 pairs, 58 for
// 4200 and 90 for 20,000, and a whole update (host to host) of an R-MAT graph went from 0.16
// to 0.10 ms at 12 pairs (16 K vertices), 0.36 to 0.29 at 652 (4.2 M), 0.70 to 0.42 at 20,287
// (1.3 M), 2.58 to 2.35 at 263,427 (16.8 M); at 8 M pairs, bound by the passes' traffic, the one
// launch is still 2% ahead (48.3 and 47.7 ms on 4.2 M vertices), so there is no other path.

constexpr int kPlanThreads = 1024;
constexpr int kPlanWarps = kPlanThreads / 32;
constexpr int kPlanItems = 2;
constexpr uint32_t kPlanTile = kPlanThreads * kPlanItems;  // keys a block ranks together
constexpr uint32_t kPlanBlockSort = 2048;                  // at most this many pairs: one block, sorted in shared memory
constexpr unsigned long long kPlanBarrierNs = 4000000000ull;

struct PlanArgs {
  Requests q;
  uint64_t *keys, *keys2;
  uint32_t *vals, *vals2;
  uint32_t *flags;
  uint64_t *chg, *chg_t, *chg_t2;
  uint32_t *seg_o, *seg_i, *tp_o, *tp_i;
  uint32_t *hist;  // [gridDim.x][256]
  uint32_t *part;  // [gridDim.x][8]
  const uint2 *in_rd;
  const uint32_t *out_cap, *in_cap;
  ApplyCtl *actl;
};

struct PlanShared {
  union {
    uint32_t wcnt[kPlanWarps][256];
    struct {
      uint64_t key[kPlanBlockSort];
      uint32_t val[kPlanBlockSort];
    } sort;
  };
  uint32_t tot[4][256], mine[4][256], gbase[256];
  unsigned long long wsum[kPlanWarps];
  uint32_t sums[8];
  uint32_t err;
};

// Grid barrier, its wait bounded (a single block needs none beyond the block barrier).
__device__ __forceinline__ bool plan_barrier(ApplyCtl *actl, uint32_t &epoch, PlanShared &sh) {
  __syncthreads();
  if (gridDim.x == 1) return true;
  epoch++;
  if (threadIdx.x == 0) {
    __threadfence();
    red_release_add_u32(&actl->bar, 1u);
    const uint32_t target = epoch * gridDim.x;
    const unsigned long long lim = *(volatile unsigned long long *)&actl->bar_limit_ns;
    const uint32_t every = lim ? 0u : 127u;  // (a short limit, set for tests: looked at every time)
    unsigned long long t0 = 0;
    for (uint32_t spins = 1; ld_acquire_u32(&actl->bar) < target; spins++) {
      if (*(volatile uint32_t *)&actl->err) break;
      if ((spins & every) == 0) {
        const unsigned long long t = globaltimer_ns();
        if (t0 == 0) t0 = t;
        else if (t - t0 > (lim ? lim : kPlanBarrierNs)) atomicExch(&actl->err, 1u);
      }
    }
    sh.err = *(volatile uint32_t *)&actl->err;
  }
  __syncthreads();
  return sh.err == 0;
}

// Exclusive scan over the block's threads of a packed word; *total = the block's sum.
__device__ __forceinline__ unsigned long long plan_scan(unsigned long long x, PlanShared &sh,
                                                        unsigned long long *total) {
  const uint32_t lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  unsigned long long incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(kAllLanes, incl, o);
    if (lane >= (uint32_t)o) incl += y;
  }
  __syncthreads();
  if (lane == 31) sh.wsum[wib] = incl;
  __syncthreads();
  unsigned long long before = 0, all = 0;
  for (uint32_t w = 0; w < (uint32_t)kPlanWarps; w++) {
    const unsigned long long y = sh.wsum[w];
    before += w < wib ? y : 0ull;
    all += y;
  }
  *total = all;
  return before + incl - x;
}

// Bitonic sort of n <= kPlanBlockSort keys (by key, then value: stable) by one block, in place.
template <bool KV>
__device__ void plan_block_sort(uint64_t *keys, uint32_t *vals, uint32_t n, PlanShared &sh) {
  uint32_t p = 2;
  while (p < n) p <<= 1;
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < p; i += kPlanThreads) {
    sh.sort.key[i] = i < n ? __ldcg(keys + i) : kSentinel;
    if (KV) sh.sort.val[i] = i < n ? __ldcg(vals + i) : 0xFFFFFFFFu;
  }
  __syncthreads();
  for (uint32_t k = 2; k <= p; k <<= 1) {
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      for (uint32_t t = threadIdx.x; t < p / 2; t += kPlanThreads) {
        const uint32_t i = ((t & ~(j - 1)) << 1) | (t & (j - 1)), l = i | j;  // a pair per thread
        const uint64_t a = sh.sort.key[i], c = sh.sort.key[l];
        bool gt = a > c;
        uint32_t va = 0, vc = 0;
        if (KV) {
          va = sh.sort.val[i];
          vc = sh.sort.val[l];
          gt = gt || (a == c && va > vc);
        }
        if (gt == ((i & k) == 0)) {
          sh.sort.key[i] = c;
          sh.sort.key[l] = a;
          if (KV) {
            sh.sort.val[i] = vc;
            sh.sort.val[l] = va;
          }
        }
      }
      __syncthreads();
    }
  }
  for (uint32_t i = threadIdx.x; i < n; i += kPlanThreads) {
    keys[i] = sh.sort.key[i];
    if (KV) vals[i] = sh.sort.val[i];
  }
  __syncthreads();
}

// Stable LSD radix sort on bits [first, bits) by the whole grid: every block owns a run of
// the input of each pass, counts its digits, and after a barrier adds up all blocks' counts
// itself (no separate scan).  src ends up pointing at the sorted keys.
template <bool KV>
__device__ bool plan_radix(uint64_t *&src, uint32_t *&sv, uint64_t *&dst, uint32_t *&dv, uint32_t n, int first,
                           int bits, uint32_t *hist, ApplyCtl *actl, uint32_t &epoch, PlanShared &sh) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, wib = tid >> 5, nblk = gridDim.x, blk = blockIdx.x;
  const uint32_t per = (n + nblk - 1) / nblk, c0 = min(n, blk * per), c1 = min(n, c0 + per);
  for (int shift = first; shift < bits; shift += 8) {
    uint32_t *cnt = sh.tot[0];
    if (tid < 256) cnt[tid] = 0;
    __syncthreads();
    for (uint32_t i = c0 + tid; i < c1; i += kPlanThreads) atomicAdd(&cnt[(__ldcg(src + i) >> shift) & 0xFF], 1u);
    __syncthreads();
    if (tid < 256) hist[blk * 256 + tid] = cnt[tid];
    if (!plan_barrier(actl, epoch, sh)) return false;
    {
      const uint32_t d = tid & 255, part = tid >> 8;
      uint32_t tot = 0, mine = 0;
#pragma unroll 4
      for (uint32_t k = part; k < nblk; k += 4) {
        const uint32_t x = __ldcg(hist + k * 256 + d);
        tot += x;
        mine += k < blk ? x : 0u;
      }
      sh.tot[part][d] = tot;
      sh.mine[part][d] = mine;
    }
    __syncthreads();
    uint32_t tot = 0, mine = 0;
    if (tid < 256) {
      for (int part = 0; part < 4; part++) {
        tot += sh.tot[part][tid];
        mine += sh.mine[part][tid];
      }
    }
    unsigned long long all;
    const uint32_t before = (uint32_t)plan_scan(tid < 256 ? tot : 0u, sh, &all);
    if (tid < 256) sh.gbase[tid] = before + mine;
    for (uint32_t t0 = c0; t0 < c1; t0 += kPlanTile) {
      for (uint32_t k = tid; k < kPlanWarps * 256; k += kPlanThreads) (&sh.wcnt[0][0])[k] = 0;
      __syncthreads();
      const uint32_t base = t0 + wib * 32 * kPlanItems;
      uint64_t k[kPlanItems];
      uint32_t v[kPlanItems], local[kPlanItems];
#pragma unroll
      for (int r = 0; r < kPlanItems; r++) {
        const uint32_t i = base + r * 32 + lane;
        k[r] = i < c1 ? __ldcg(src + i) : 0ull;
        if (KV) v[r] = i < c1 ? __ldcg(sv + i) : 0u;
      }
#pragma unroll
      for (int r = 0; r < kPlanItems; r++) {
        const bool valid = base + r * 32 + lane < c1;
        const uint32_t d = valid ? (uint32_t)((k[r] >> shift) & 0xFF) : 0xFFFFu;
        const uint32_t peers = __match_any_sync(kAllLanes, d), rank = __popc(peers & lanemask_lt());
        const uint32_t x = valid ? sh.wcnt[wib][d] : 0u;
        __syncwarp();
        if (valid && rank == 0) sh.wcnt[wib][d] = x + __popc(peers);
        __syncwarp();
        local[r] = x + rank;
      }
      __syncthreads();
      if (tid < 256) {  // places of this tile's digits by warp; the next tile's follow
        uint32_t run = sh.gbase[tid];
        for (int w = 0; w < kPlanWarps; w++) {
          const uint32_t x = sh.wcnt[w][tid];
          sh.wcnt[w][tid] = run;
          run += x;
        }
        sh.gbase[tid] = run;
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < kPlanItems; r++) {
        if (base + r * 32 + lane < c1) {
          const uint32_t at = sh.wcnt[wib][(k[r] >> shift) & 0xFF] + local[r];
          dst[at] = k[r];
          if (KV) dv[at] = v[r];
        }
      }
      __syncthreads();
    }
    if (!plan_barrier(actl, epoch, sh)) return false;
    uint64_t *tk = src;
    src = dst;
    dst = tk;
    uint32_t *tv = sv;
    sv = dv;
    dv = tv;
  }
  return true;
}

__global__ void __launch_bounds__(kPlanThreads, 1) k_plan(const PlanArgs p) {
  __shared__ PlanShared sh;
  const Requests &q = p.q;
  ApplyCtl *actl = p.actl;
  const uint32_t tid = threadIdx.x, nblk = gridDim.x, blk = blockIdx.x;
  const uint32_t gtid = blk * kPlanThreads + tid, nthreads = nblk * kPlanThreads;
  const uint32_t N = (uint32_t)(q.nd + q.ni);
  uint32_t epoch = 0;
  for (uint32_t i = gtid; i < N; i += nthreads) request_key(q, i, p.keys, p.vals, actl);
  if (!plan_barrier(actl, epoch, sh)) return;
  if (*(volatile uint32_t *)&actl->bad_id || *(volatile uint32_t *)&actl->bad_comp) return;  // the same in every block
  uint64_t *keys = p.keys, *keys2 = p.keys2;
  uint32_t *vals = p.vals, *vals2 = p.vals2;
  if (nblk == 1) plan_block_sort<true>(keys, vals, N, sh);
  else if (!plan_radix<true>(keys, vals, keys2, vals2, N, 0, 2 * q.b, p.hist, actl, epoch, sh)) return;

  // effective changes: counted by block, then written in order
  const uint32_t per = (N + nblk - 1) / nblk, c0 = min(N, blk * per), c1 = min(N, c0 + per);
  if (tid < 8) sh.sums[tid] = 0;
  __syncthreads();
  uint32_t mine = 0;
  for (uint32_t i = c0 + tid; i < c1; i += kPlanThreads) {
    const uint64_t k = __ldcg(keys + i), next = i + 1 < N ? __ldcg(keys + i + 1) : kSentinel;
    const bool f = is_change(q, k, next, __ldcg(vals + i));
    p.flags[i] = f ? 1u : 0u;
    mine += f ? 1u : 0u;
  }
  if (mine) atomicAdd(&sh.sums[0], mine);
  __syncthreads();
  if (tid == 0) p.part[blk * 8] = sh.sums[0];
  if (!plan_barrier(actl, epoch, sh)) return;
  for (uint32_t k = tid; k < nblk; k += kPlanThreads) {
    const uint32_t x = __ldcg(p.part + k * 8);
    atomicAdd(&sh.sums[1], x);
    if (k < blk) atomicAdd(&sh.sums[2], x);
  }
  __syncthreads();
  const uint32_t K = sh.sums[1];
  if (gtid == 0) actl->n_eff = K;
  if (K == 0) return;
  uint32_t at = sh.sums[2];
  for (uint32_t t0 = c0; t0 < c1; t0 += kPlanThreads) {
    const uint32_t i = t0 + tid;
    const bool f = i < c1 && p.flags[i];
    unsigned long long all;
    const uint32_t x = (uint32_t)plan_scan(f ? 1u : 0u, sh, &all);
    if (f) emit_change(q, __ldcg(keys + i), __ldcg(vals + i), at + x, p.chg, p.chg_t);
    at += (uint32_t)all;
  }
  if (!plan_barrier(actl, epoch, sh)) return;

  // the change list is in (u, v) order already; the transposed copy follows it by a stable sort
  // on v alone, unless the in-rows are ordered by another key than u
  uint64_t *ct = p.chg_t, *ct2 = p.chg_t2;
  if (nblk == 1) {
    plan_block_sort<false>(ct, nullptr, K, sh);
  } else {
    uint32_t *none = nullptr, *none2 = nullptr;
    if (!plan_radix<false>(ct, none, ct2, none2, K, q.lab ? 1 : q.b + 1, 2 * q.b + 1, p.hist, actl, epoch, sh)) return;
  }

  // segments (touched rows) and insertion counts of both lists: by block, then written in order.
  // Four counts a thread in one word (a tile has at most 1024 of each)
  const uint32_t per2 = (K + nblk - 1) / nblk, k0 = min(K, blk * per2), k1 = min(K, k0 + per2);
  auto counts = [&](uint32_t j) -> unsigned long long {
    const uint64_t o = __ldcg(p.chg + j), i = __ldcg(ct + j);
    const bool fo = j == 0 || chg_row(o, q.b) != chg_row(__ldcg(p.chg + j - 1), q.b);
    const bool fi = j == 0 || chg_row(i, q.b) != chg_row(__ldcg(ct + j - 1), q.b);
    return (fo ? 1ull : 0ull) | ((o & 1ull) << 16) | (fi ? 1ull << 32 : 0ull) | ((i & 1ull) << 48);
  };
  if (tid < 8) sh.sums[tid] = 0;
  __syncthreads();
  uint32_t m4[4] = {0, 0, 0, 0};
  for (uint32_t j = k0 + tid; j < k1; j += kPlanThreads) {
    const unsigned long long x = counts(j);
    for (int c = 0; c < 4; c++) m4[c] += (uint32_t)(x >> (16 * c)) & 0xFFFFu;
  }
  for (int c = 0; c < 4; c++)
    if (m4[c]) atomicAdd(&sh.sums[c], m4[c]);
  __syncthreads();
  if (tid < 4) p.part[blk * 8 + 4 + tid] = sh.sums[tid];
  if (!plan_barrier(actl, epoch, sh)) return;
  if (tid < 8) sh.sums[tid] = 0;
  __syncthreads();
  for (uint32_t k = tid; k < nblk * 4; k += kPlanThreads) {
    const uint32_t x = __ldcg(p.part + (k >> 2) * 8 + 4 + (k & 3));
    atomicAdd(&sh.sums[k & 3], x);
    if ((k >> 2) < blk) atomicAdd(&sh.sums[4 + (k & 3)], x);
  }
  __syncthreads();
  const uint32_t n_o = sh.sums[0], ins = sh.sums[1], n_i = sh.sums[2];
  uint32_t a_o = sh.sums[4], t_o = sh.sums[5], a_i = sh.sums[6], t_i = sh.sums[7];
  for (uint32_t t0 = k0; t0 < k1; t0 += kPlanThreads) {
    const uint32_t j = t0 + tid;
    const unsigned long long x = j < k1 ? counts(j) : 0ull;
    unsigned long long all;
    const unsigned long long ex = plan_scan(x, sh, &all);
    if (j < k1) {
      p.tp_o[j] = t_o + ((uint32_t)(ex >> 16) & 0xFFFFu);
      p.tp_i[j] = t_i + ((uint32_t)(ex >> 48) & 0xFFFFu);
      if (x & 0xFFFFu) p.seg_o[a_o + ((uint32_t)ex & 0xFFFFu)] = j;
      if ((x >> 32) & 0xFFFFu) p.seg_i[a_i + ((uint32_t)(ex >> 32) & 0xFFFFu)] = j;
    }
    a_o += (uint32_t)all & 0xFFFFu;
    t_o += (uint32_t)(all >> 16) & 0xFFFFu;
    a_i += (uint32_t)(all >> 32) & 0xFFFFu;
    t_i += (uint32_t)(all >> 48) & 0xFFFFu;
  }
  if (gtid == 0) {
    p.seg_o[n_o] = K;
    p.seg_i[n_i] = K;
    p.tp_o[K] = ins;
    p.tp_i[K] = ins;
    actl->n_seg_out = n_o;
    actl->n_seg_in = n_i;
    actl->n_eff_del = K - ins;
  }
  if (!plan_barrier(actl, epoch, sh)) return;
  for (uint32_t s = gtid; s < n_o + n_i; s += nthreads) {
    if (s < n_o) plan_row(q.out_rd, p.out_cap, p.chg, q.b, p.seg_o, p.tp_o, s, &actl->reloc_out, actl);
    else plan_row(p.in_rd, p.in_cap, ct, q.b, p.seg_i, p.tp_i, s - n_o, &actl->reloc_in, actl);
  }
}

// ... and again, after a repack.
__global__ void k_plan_rows(const uint2 *rd, const uint32_t *cap, const uint64_t *chg, int b, const uint32_t *seg,
                            const uint32_t *nseg, const uint32_t *tagpref, unsigned long long *reloc, ApplyCtl *actl) {
  uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < *nseg) plan_row(rd, cap, chg, b, seg, tagpref, s, reloc, actl);
}

// -------------------------------------------------------------------------- merge ----

// One adjacency's side of a merge.
struct MergeAdj {
  uint2 *rd;
  uint32_t *cap, *col;
  const uint64_t *chg;
  const uint32_t *seg, *tagpref;
  uint32_t nseg;
  unsigned long long *tail, *garbage;
  uint64_t col_cap;
};

// A long row: what its slices need after the row's descriptor has changed.
struct LongRow {
  uint32_t dir, seg, row, start, len, cap, new_len, dest, slice0, moves;
  unsigned long long big;  // its entries' staging, from big + this
};

template <bool F32>
struct MergeArgs {
  using S = Store<F32>;
  MergeAdj adj[2];  // out-rows, in-rows
  int b;
  // out-rows: contribution refresh and pending marks (each touched row is a source, each
  // effective deletion a target: both have a place by their number)
  double alpha;
  typename S::A *adeg;
  const typename S::R *R0;
  typename S::C *C0, *C1;
  uint32_t *pend_src, *pend_tgt;
  uint32_t pend_cap, n_src, n_tgt;
  // in-rows: sweep items (patched where tier and chunk count stay; null: rebuilt in any case,
  // out of date since a repack, or an earlier call found no room for them), the rows' order
  uint32_t bin_lo, gmax, chunk;
  uint4 *items;
  const uint32_t *item_pos;
  const uint32_t *lab, *at;
  uint32_t *big;
  uint64_t big_cap;
  LongRow *longs;
  uint32_t long_cap;
  ApplyCtl *actl;
};

// Chunk items of the tier-2 rows; chunk c of a row covers edges [c chunk, (c+1) chunk).
__device__ __forceinline__ uint4 chunk_item(uint32_t v, uint2 d, uint32_t c, uint32_t nch, uint32_t number,
                                            uint32_t chunk) {
  uint32_t len = min(chunk, d.y - c * chunk);
  return make_uint4(v, d.x + c * chunk, len | (c << 10) | (nch > 1 ? 0x80000000u : 0u), number);
}

// The new row's descriptor and what follows from its length, by nt threads (t of them): lane 0
// of a warp's row, or a block.
template <bool F32>
__device__ __forceinline__ void finish_row(const MergeArgs<F32> &p, uint32_t dir, uint32_t s, uint32_t r,
                                           uint32_t dest, uint32_t len, uint32_t new_len, uint32_t cap_r, bool moves,
                                           uint32_t t, uint32_t nt) {
  using S = Store<F32>;
  const MergeAdj &A = p.adj[dir];
  const uint2 nd = make_uint2(dest, new_len);
  if (t == 0) {
    A.rd[r] = nd;
    if (moves) {
      A.cap[r] = move_cap(new_len);
      atomicAdd(A.garbage, (unsigned long long)cap_r);
    }
    if (dir == 0) {
      const typename S::A a = S::factor(p.alpha, new_len);
      p.adeg[r] = a;
      const typename S::C c = S::contrib(p.R0[r], a);
      p.C0[r] = c;
      p.C1[r] = c;
      if ((len == 0) != (new_len == 0)) p.actl->dead_changed = 1;
      if ((uint64_t)p.n_src + s < p.pend_cap) p.pend_src[p.n_src + s] = r;
    }
  }
  // free slots of the row's last 16 bytes (the sweeps read rows by 16 bytes)
  for (uint32_t k = new_len + t; k < ((new_len + 3) & ~3u); k += nt) A.col[dest + k] = kNoCol;
  if (dir == 1 && p.items) {
    const int tier = sweep_tier(new_len, p.bin_lo, p.gmax);
    const uint32_t nch = (new_len + p.chunk - 1) / p.chunk;
    if (sweep_tier(len, p.bin_lo, p.gmax) != tier || (tier == 2 && (len + p.chunk - 1) / p.chunk != nch)) {
      if (t == 0) p.actl->bins_changed = 1;  // the sweep items are rebuilt after this update
      return;
    }
    const uint32_t pos = p.item_pos[r];
    if (tier < 2) {
      if (t == 0) p.items[pos] = make_uint4(r, nd.x, nd.y, 0u);
    } else {
      for (uint32_t c = t; c < nch; c += nt) {  // (a chunk's number is its own: .w stays)
        uint4 it = chunk_item(r, nd, c, nch, 0u, p.chunk);
        it.w = p.items[pos + c].w;
        p.items[pos + c] = it;
      }
    }
  }
}

constexpr int kMergeWarps = 8;

// A warp a touched row of either adjacency (the long ones queued): entries and changes staged
// in shared memory; an entry's new place is its old one less the deletions and plus the
// insertions before it, found by a binary search over the row's changes.
template <bool F32>
__global__ void __launch_bounds__(kMergeWarps * 32) k_merge_rows(const MergeArgs<F32> p) {
  __shared__ uint32_t s_row[kMergeWarps][kWarpRow], s_col[kMergeWarps][kWarpChanges], s_ins[kMergeWarps][kWarpChanges];
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t s = blockIdx.x * kMergeWarps + w;
  if (s >= p.adj[0].nseg + p.adj[1].nseg) return;
  const uint32_t dir = s < p.adj[0].nseg ? 0u : 1u;
  if (dir) s -= p.adj[0].nseg;
  const MergeAdj &A = p.adj[dir];
  const int b = p.b;
  const uint32_t s0 = A.seg[s], e = A.seg[s + 1], c = e - s0;
  const uint32_t r = chg_row(A.chg[s0], b);
  const uint2 d = A.rd[r];
  const uint32_t len = d.y, cap_r = A.cap[r], ins0 = A.tagpref[s0];
  const uint32_t nI = A.tagpref[e] - ins0, new_len = len - (c - nI) + nI;
  const bool moves = new_len > cap_r;
  unsigned long long dest = d.x;
  if (lane == 0 && moves) dest = atomicAdd(A.tail, (unsigned long long)move_cap(new_len));
  dest = __shfl_sync(kAllLanes, dest, 0);
  bool room = !moves || dest + move_cap(new_len) <= A.col_cap;
  if (long_row(len, c)) {
    if (lane == 0) {
      const unsigned long long bg = atomicAdd(&p.actl->big_cursor, (unsigned long long)len);
      room = room && bg + len <= p.big_cap;
      // number and first slice from one atomic, so first slices ascend with the number; a row
      // without room keeps its place in the queue but has no slices
      const uint32_t ns = room ? max(1u, (len + kSlice - 1) / kSlice) : 0u;
      const unsigned long long q = atomicAdd(&p.actl->longq, (1ull << 32) | ns);
      if (!room || (uint32_t)(q >> 32) >= p.long_cap) atomicOr(&p.actl->overflow, 1u);
      else
        p.longs[q >> 32] = LongRow{dir, s, r, d.x, len, cap_r, new_len, (uint32_t)dest, (uint32_t)q, moves ? 1u : 0u, bg};
    }
    return;
  }
  if (!room) {  // the row is left as it was and the host reports the failure
    if (lane == 0) atomicOr(&p.actl->overflow, 1u);
    return;
  }
  const uint32_t *lab = dir ? p.lab : nullptr, *at = dir ? p.at : nullptr;
  uint32_t *row = s_row[w], *cc = s_col[w], *ci = s_ins[w];
  for (uint32_t j = lane; j < len; j += 32) {
    const uint32_t x = A.col[d.x + j];
    row[j] = lab ? lab[x] : x;
  }
  for (uint32_t q = lane; q < c; q += 32) {
    const uint64_t k = A.chg[s0 + q];
    cc[q] = chg_col(k, b);
    ci[q] = ((A.tagpref[s0 + q] - ins0) << 1) | (uint32_t)(k & 1);  // insertions before it, its own kind
  }
  __syncwarp();
  uint32_t *dst = A.col + dest;
  for (uint32_t j = lane; j < len; j += 32) {
    const uint32_t x = row[j];
    uint32_t lo = 0, hi = c;  // first change with column >= x
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (cc[mid] < x) lo = mid + 1; else hi = mid;
    }
    if (lo < c && cc[lo] == x) continue;  // deleted
    const uint32_t ib = lo < c ? ci[lo] >> 1 : nI;
    dst[j - (lo - ib) + ib] = at ? at[x] : x;
  }
  for (uint32_t q = lane; q < c; q += 32) {
    const uint32_t y = cc[q], ib = ci[q] >> 1;
    if (ci[q] & 1u) {
      uint32_t lo = 0, hi = len;  // old entries below y
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (row[mid] < y) lo = mid + 1; else hi = mid;
      }
      dst[lo - (q - ib) + ib] = at ? at[y] : y;
    } else if (dir == 0) {
      const uint64_t t = (uint64_t)p.n_tgt + (s0 + q) - (ins0 + ib);  // deletions before it in the whole list
      if (t < p.pend_cap) p.pend_tgt[t] = y;
    }
  }
  finish_row<F32>(p, dir, s, r, (uint32_t)dest, len, new_len, cap_r, moves, lane, 32u);
}

// The queued row that slice k belongs to: the last with slice0 <= k.
__device__ __forceinline__ uint32_t long_of(const LongRow *longs, uint32_t n, uint32_t k) {
  uint32_t lo = 0, hi = n;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (longs[mid].slice0 <= k) lo = mid; else hi = mid;
  }
  return lo;
}

// Long rows, by slices of their old entries.  First every slice is copied to the staging area
// (the new row may overlap the old one) ...
template <bool F32>
__global__ void __launch_bounds__(256) k_long_copy(const MergeArgs<F32> p) {
  const unsigned long long q = p.actl->longq;
  const uint32_t n = min((uint32_t)(q >> 32), p.long_cap), ns = (uint32_t)q;
  if (p.actl->overflow) return;
  for (uint32_t k = blockIdx.x; k < ns; k += gridDim.x) {
    const LongRow L = p.longs[long_of(p.longs, n, k)];
    const uint32_t a = (k - L.slice0) * kSlice, e = min(L.len, a + kSlice);
    const uint32_t *src = p.adj[L.dir].col + L.start;
    const uint32_t *lab = L.dir ? p.lab : nullptr;
    uint32_t *dst = p.big + L.big;
    for (uint32_t j = a + threadIdx.x; j < e; j += 256) {
      const uint32_t x = src[j];
      dst[j] = lab ? lab[x] : x;
    }
  }
}

// ... then each slice's entries, and the changes that fall among them, go to their places; the
// block of a row's first slice finishes the row.
template <bool F32>
__global__ void __launch_bounds__(256) k_long_merge(const MergeArgs<F32> p) {
  __shared__ uint32_t s_cut[2], s_col[kSlice], s_ins[kSlice];
  const unsigned long long qn = p.actl->longq;
  const uint32_t n = min((uint32_t)(qn >> 32), p.long_cap), ns = (uint32_t)qn, tid = threadIdx.x;
  const int b = p.b;
  if (p.actl->overflow) return;
  for (uint32_t k = blockIdx.x; k < ns; k += gridDim.x) {
    const LongRow L = p.longs[long_of(p.longs, n, k)];
    const MergeAdj &A = p.adj[L.dir];
    const uint32_t s0 = A.seg[L.seg], e = A.seg[L.seg + 1], ins0 = A.tagpref[s0];
    const uint32_t a = (k - L.slice0) * kSlice, z = min(L.len, a + kSlice);
    const uint32_t *row = p.big + L.big;
    if (tid < 2) {  // the slice's changes: from the first >= its first entry to the first >= the next slice's
      const uint32_t j = tid == 0 ? a : z;
      uint32_t lo = s0, hi = e;
      if (tid == 0 && a == 0) hi = s0;
      else if (tid == 1 && z == L.len) lo = e;
      else {
        const uint32_t x = row[j];
        while (lo < hi) {
          const uint32_t mid = (lo + hi) >> 1;
          if (chg_col(A.chg[mid], b) < x) lo = mid + 1; else hi = mid;
        }
      }
      s_cut[tid] = lo;
    }
    __syncthreads();
    const uint32_t f = s_cut[0], c = s_cut[1] - f;
    const bool staged = c <= kSlice;
    if (staged) {
      for (uint32_t q = tid; q < c; q += 256) {
        const uint64_t x = A.chg[f + q];
        s_col[q] = chg_col(x, b);
        s_ins[q] = A.tagpref[f + q];
      }
    }
    __syncthreads();
    const uint32_t *at = L.dir ? p.at : nullptr;
    const uint32_t ins_end = A.tagpref[f + c];
    uint32_t *dst = A.col + L.dest;
    for (uint32_t j = a + tid; j < z; j += 256) {
      const uint32_t x = row[j];
      uint32_t lo = 0, hi = c;
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if ((staged ? s_col[mid] : chg_col(A.chg[f + mid], b)) < x) lo = mid + 1; else hi = mid;
      }
      if (lo < c && (staged ? s_col[lo] : chg_col(A.chg[f + lo], b)) == x) continue;  // deleted
      const uint32_t ib = (lo < c ? (staged ? s_ins[lo] : A.tagpref[f + lo]) : ins_end) - ins0;
      const uint32_t db = f + lo - s0 - ib;
      dst[j - db + ib] = at ? at[x] : x;
    }
    for (uint32_t q = tid; q < c; q += 256) {
      const uint64_t x = A.chg[f + q];
      const uint32_t y = chg_col(x, b), ib = A.tagpref[f + q] - ins0, db = f + q - s0 - ib;
      if (x & 1) {
        uint32_t lo = a, hi = z;  // old entries below y
        while (lo < hi) {
          const uint32_t mid = (lo + hi) >> 1;
          if (row[mid] < y) lo = mid + 1; else hi = mid;
        }
        dst[lo - db + ib] = at ? at[y] : y;
      } else if (L.dir == 0) {
        const uint64_t t = (uint64_t)p.n_tgt + (f + q) - (ins0 + ib);
        if (t < p.pend_cap) p.pend_tgt[t] = y;
      }
    }
    if (a == 0) finish_row<F32>(p, L.dir, L.seg, L.row, L.dest, L.len, L.new_len, L.cap, L.moves != 0, tid, 256u);
    __syncthreads();  // the staged changes are read until here
  }
}

}  // namespace

// ------------------------------------------------------------------ host side ---

template <class T>
static cudaError_t grow(T **p, uint64_t count) {
  cudaFree(*p);
  *p = nullptr;
  if (alloc_fault()) return cudaErrorMemoryAllocation;
  return cudaMalloc((void **)p, sizeof(T) * count);
}

template <bool F32>
static pr_status run_merge(Graph *g, const MergeAdj &out, const MergeAdj &in, uint32_t n_long, uint64_t big_need) {
  using S = Store<F32>;
  cudaStream_t st = g->st;
  MergeArgs<F32> p{};
  p.adj[0] = out;
  p.adj[1] = in;
  p.b = g->b;
  p.alpha = g->p.alpha;
  p.adeg = (typename S::A *)g->adeg;
  p.R0 = (const typename S::R *)g->R[0];
  p.C0 = (typename S::C *)g->C[0];
  p.C1 = (typename S::C *)g->C[1];
  p.pend_src = g->pend_src;
  p.pend_tgt = g->pend_tgt;
  p.pend_cap = g->pend_cap;
  p.n_src = g->n_pend_src;
  p.n_tgt = g->n_pend_tgt;
  p.bin_lo = (uint32_t)g->p.bin_lo;
  p.gmax = g->group_max;
  p.chunk = g->chunk_len;
  p.items = g->ident_dirty ? nullptr : g->items;
  p.item_pos = g->item_pos;
  p.lab = g->lab;
  p.at = g->at;
  p.big = g->big;
  p.big_cap = g->big_cap;
  p.longs = (LongRow *)g->longs;
  p.long_cap = g->long_cap;
  p.actl = g->actl;
  k_merge_rows<F32><<<grid_for((uint64_t)out.nseg + in.nseg, kMergeWarps), kMergeWarps * 32, 0, st>>>(p);
  count_launch();
  if (n_long) {
    const unsigned grid = (unsigned)std::min<uint64_t>(big_need / kSlice + n_long, (uint64_t)g->sm_count * 8);
    k_long_copy<F32><<<grid, 256, 0, st>>>(p);
    count_launch();
    k_long_merge<F32><<<grid, 256, 0, st>>>(p);
    count_launch();
  }
  CK(cudaGetLastError());
  return PR_OK;
}

pr_status graph_apply(Graph *g, uint64_t nd, const uint32_t *ds, const uint32_t *dd, uint64_t ni, const uint32_t *is,
                      const uint32_t *id, int nb, const uint32_t *off) {
  const uint64_t N = nd + ni;
  if (N == 0) return PR_OK;
  cudaStream_t st = g->st;
  pr_status rc = apply_scratch(g, N);
  if (rc != PR_OK) return rc;
  ApplyScratch &s = g->sc;
  const int b = g->b;
  ApplyCtl *dctl = g->actl;
  ApplyCtl &h = *g->actl_h;
  std::memset(&h, 0, sizeof(ApplyCtl));
  h.tail_out = g->out.used;
  h.tail_in = g->in.used;
  h.bar_limit_ns = 1000ull * (unsigned long long)g->barrier_us;
  CK(cudaMemcpyAsync(dctl, &h, sizeof(ApplyCtl), cudaMemcpyHostToDevice, st));

  const Requests q{ds, dd, is, id, nd, ni, nb, off, g->n, b, g->comp, g->inv, g->lab, g->out.rd, g->out.col};
  uint32_t *seg_o = s.seg, *seg_i = s.seg + (s.cap + 2);
  uint32_t *tp_o = s.tagpref, *tp_i = s.tagpref + (s.cap + 2);
  uint64_t *co = s.chg, *ci = s.chg_t;
  const int first = g->lab ? 1 : b + 1;  // lowest bit the transposed list is sorted by
  auto read_ctl = [&]() -> pr_status {
    CK(cudaMemcpyAsync(&h, dctl, sizeof(ApplyCtl), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (h.err) {
      g->err = "batch update: a grid barrier wait timed out (graph unchanged)";
      return PR_ERR_DEVICE_TIMEOUT;
    }
    if (h.bad_id) {
      g->err = "vertex id out of range";
      return PR_ERR_VERTEX_RANGE;
    }
    if (h.bad_comp) {
      g->err = "a pair joins two different graphs of a batched handle";
      return PR_ERR_INVALID_ARG;
    }
    return PR_OK;
  };
  PlanArgs p{};
  p.q = q;
  p.keys = s.kd;
  p.keys2 = s.tmp;
  p.vals = s.vals;
  p.vals2 = s.vals2;
  p.flags = s.flags;
  p.chg = s.chg;
  p.chg_t = s.chg_t;
  p.chg_t2 = s.tmp2;
  p.seg_o = seg_o;
  p.seg_i = seg_i;
  p.tp_o = tp_o;
  p.tp_i = tp_i;
  const unsigned grid =
      N <= kPlanBlockSort ? 1u
                          : (unsigned)std::min<uint64_t>((N + kPlanThreads - 1) / kPlanThreads,
                                                         (uint64_t)std::max(2, g->share_grid));
  p.hist = s.radix_hist;
  p.part = s.radix_hist + 256ull * grid;
  p.in_rd = g->in.rd;
  p.out_cap = g->out.cap;
  p.in_cap = g->in.cap;
  p.actl = dctl;
  void *args[] = {(void *)&p};
  if (grid == 1) k_plan<<<1, kPlanThreads, 0, st>>>(p);
  else CK(cudaLaunchCooperativeKernel((const void *)k_plan, dim3(grid), dim3(kPlanThreads), args, 0, st));
  count_launch();
  CK(cudaGetLastError());
  // the radix passes swap the transposed list's buffers
  if (grid > 1 && ((2 * b + 1 - first + 7) / 8) % 2 == 1) ci = s.tmp2;
  if ((rc = read_ctl()) != PR_OK) return rc;
  if (h.n_eff == 0) return PR_OK;
  const uint32_t K = h.n_eff, K_del = h.n_eff_del, n_o = h.n_seg_out, n_i = h.n_seg_in;

  // room for moved rows and staging of long rows; a repack gives rows fresh (possibly
  // smaller) slack, so the plan is redone after one
  for (int round = 0; round < 4; round++) {
    bool again = false;
    if (g->out.used + h.reloc_out > g->out.col_cap) {
      if ((rc = repack_adj(g, g->out, 2 * h.reloc_out)) != PR_OK) return rc;
      again = true;
    }
    if (g->in.used + h.reloc_in > g->in.col_cap) {
      if ((rc = repack_adj(g, g->in, 2 * h.reloc_in)) != PR_OK) return rc;
      again = true;
    }
    if (!again) break;
    h.reloc_out = h.reloc_in = 0;
    h.tail_out = g->out.used;
    h.tail_in = g->in.used;
    h.big_need = 0;
    h.n_long = 0;
    CK(cudaMemcpyAsync(dctl, &h, sizeof(ApplyCtl), cudaMemcpyHostToDevice, st));
    k_plan_rows<<<grid_for(n_o), 256, 0, st>>>(g->out.rd, g->out.cap, co, b, seg_o, &dctl->n_seg_out, tp_o,
                                               &dctl->reloc_out, dctl);
    count_launch();
    k_plan_rows<<<grid_for(n_i), 256, 0, st>>>(g->in.rd, g->in.cap, ci, b, seg_i, &dctl->n_seg_in, tp_i,
                                               &dctl->reloc_in, dctl);
    count_launch();
    CK(cudaGetLastError());
    if ((rc = read_ctl()) != PR_OK) return rc;
  }
  if (h.big_need > g->big_cap) {
    const uint64_t c = std::max<uint64_t>(h.big_need * 2, 1u << 18);
    g->big_cap = 0;
    CK(grow(&g->big, c));
    g->big_cap = c;
  }
  if (h.n_long > g->long_cap) {
    const uint32_t c = std::max<uint32_t>(h.n_long * 2, 1024);
    g->long_cap = 0;
    CK(grow((LongRow **)&g->longs, c));
    g->long_cap = c;
  }
  const MergeAdj out{g->out.rd, g->out.cap, g->out.col, co, seg_o, tp_o, n_o, &dctl->tail_out, &dctl->garbage_out,
                     g->out.col_cap};
  const MergeAdj in{g->in.rd, g->in.cap, g->in.col, ci, seg_i, tp_i, n_i, &dctl->tail_in, &dctl->garbage_in,
                    g->in.col_cap};
  rc = g->f32 ? run_merge<true>(g, out, in, h.n_long, h.big_need) : run_merge<false>(g, out, in, h.n_long, h.big_need);
  if (rc != PR_OK) return rc;
  if ((rc = read_ctl()) != PR_OK) return rc;
  if (h.overflow) {
    g->err = "internal error: no room for a moved row (graph rows partly updated)";
    return PR_ERR_CUDA;
  }

  g->m = g->m + (uint64_t)(K - K_del) - (uint64_t)K_del;
  g->out.used = h.tail_out;
  g->in.used = h.tail_in;
  g->out.garbage += h.garbage_out;
  g->in.garbage += h.garbage_in;
  const uint64_t n_src = (uint64_t)g->n_pend_src + n_o, n_tgt = (uint64_t)g->n_pend_tgt + K_del;
  g->n_pend_src = (uint32_t)std::min<uint64_t>(n_src, g->pend_cap);
  g->n_pend_tgt = (uint32_t)std::min<uint64_t>(n_tgt, g->pend_cap);
  if (n_src > g->pend_cap || n_tgt > g->pend_cap) g->pend_all = true;
  if (h.dead_changed) g->dead_dirty = true;
  if (h.bins_changed) g->ident_dirty = true;
  // The update is in place: where there is no room to give abandoned slots back once they dominate,
  // or for larger sweep items, the call has not failed; later ones try again
  const std::string err = g->err;
  for (Adj *A : {&g->out, &g->in}) {
    if (A->garbage <= A->used / 2 || A->garbage <= 1024) continue;
    rc = repack_adj(g, *A, 0);
    if (rc != PR_OK && rc != PR_ERR_OUT_OF_MEMORY) return rc;
  }
  // the degree-binned vertex order used by full and dense sweeps follows the graph
  rc = graph_refresh_ident(g);
  if (rc != PR_OK && rc != PR_ERR_OUT_OF_MEMORY) return rc;
  g->err = err;
  return PR_OK;
}

}  // namespace prdf
