// sweep_dev.cuh - one iteration of Eq. 1 over sweep items by the whole grid, shared by the
// iterations of single graphs (sweep.cu) and of batched handles (batch.cu): contribution gathers with
// a shared-memory copy of the hot ones, the three tiers, the marking of dense iterations.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstring>

#include "rank_dev.cuh"

namespace prdf {

// One block of 32 warps per SM, so that the SM holds one copy of the hot contributions.  The
// sweep waits on memory: R-MAT scale 22, 64-bit, full sweep 0.235 ms with 32 warps of 64
// registers, 0.248 with 28 of 72, 0.270 with 24 of 80, 0.286 with 16; two blocks of 20 warps and
// 48 registers (spills, two copies of 64 KB) 0.234.
constexpr int kSweepBlock = 1024;
constexpr int kSweepWarps = kSweepBlock / 32;
// Kernel parameters of a sweep (fixed for a handle until a buffer moves; the per-call
// sizes travel in the control block).
template <bool F32>
struct SweepArgs {
  using S = Store<F32>;
  typename S::R *R0, *R1;
  typename S::C *C0, *C1;
  const typename S::A *adeg;
  const uint32_t *in_col;
  const uint2 *in_rd;
  const uint4 *items;      // all sweep items, tier order
  uint4 *items_cmp;        // the affected vertices' items (dense Dynamic Frontier); .w of a
                           // tier-0/1 item caches "out-row already marked"
  typename S::C *partials;
  uint32_t *chunk_done;
  uint16_t *stamp;
  uint32_t *bitmap;
  uint32_t *list0;
  uint32_t *xbits;
  uint32_t *xlist;
  uint8_t *emap;
  const uint2 *out_rd;     // out-row descriptors (the compacted iterations' expansion path reads lengths)
  RankCtl *ctl;
  uint32_t hot;            // contributions of vertices [0, hot) are kept in shared memory
  typename S::R base;      // (1 - alpha) / n
  typename Num<F32>::B ftol;
  unsigned long long tol_key;
  uint32_t n;
  uint32_t chunk;          // edges per chunk of a tier-2 row
  int max_iter;
  cudaGraphConditionalHandle h_loop, h_pro, h_mode, h_fin;
};

// First expansions found by a dense sweep, appended to the expansion list (one atomic per
// warp round) until the iteration's entries reach cap (cap_end = the cursor where they
// would); past it a pull follows and the warp only counts them (xloc, added at the end).
__device__ __forceinline__ void note_expansion(RankCtl *ctl, uint32_t *xlist, bool push, uint32_t v, uint32_t lane,
                                               uint32_t cap_end, bool &xfull, uint32_t &xloc) {
  const uint32_t mask = __ballot_sync(kFull, push);
  if (!mask) return;
  if (xfull) {
    xloc += __popc(mask);
    return;
  }
  const uint32_t leader = __ffs(mask) - 1;
  uint32_t base = 0;
  if (lane == leader) base = atomicAdd(&ctl->xcnt, (uint32_t)__popc(mask));
  base = __shfl_sync(kFull, base, leader);
  const uint32_t at = base + __popc(mask & lanemask_lt());
  if (push && at < cap_end) xlist[at] = v;
  if (base + __popc(mask) >= cap_end) xfull = true;
}

// Compacted iterations: v changed by more than tau_f and its cache says it may not have
// expanded yet (no bit on its tier-0/1 item, no expanded bit in the stamp of a tier-2
// row).  The stamp's expanded bit or the marking launch's bitmap decides; a first
// expansion sets the stamp bit and is appended to the expansion list (the lanes that get
// here together share one atomic; past the iteration's cap only counted), and a tier-0/1
// item gets its cache bit either way.  Out of line: after the first iteration over a
// compaction it is rare, and the sweep loops keep the registers of a full sweep.
[[maybe_unused]] static __device__ __noinline__ void expand_cmp(RankCtl *ctl, uint16_t *stamp, const uint32_t *xbits, uint32_t *xlist,
                                        uint4 *items_cmp, const uint2 *out_rd, uint32_t v, uint32_t ci,
                                        bool has_item, uint32_t *grew) {
  const uint16_t s2 = __ldcg(reinterpret_cast<const unsigned short *>(stamp + v));
  const bool was = (s2 & kStampExp) || ((__ldcg(xbits + (v >> 5)) >> (v & 31)) & 1u);
  if (!was) {
    stamp[v] = (uint16_t)(s2 | kStampExp);
    if (__ldg(&out_rd[v]).y > kInlineOut) atomicOr(&ctl->x_long, 1u);  // the next push needs the grid
  }
  if (has_item) items_cmp[ci].w = 1u;
  const uint32_t mask = __activemask();
  const uint32_t want = __ballot_sync(mask, !was);
  if (!want) return;
  const uint32_t lane = threadIdx.x & 31, leader = __ffs(want) - 1;
  uint32_t base = 0;
  if (lane == leader) {
    base = atomicAdd(&ctl->xcnt, (uint32_t)__popc(want));
    *grew = 1;  // ends a run of iterations after this one
  }
  base = __shfl_sync(mask, base, leader);
  if (!was) {
    const uint32_t x0 = __ldcg(&ctl->xdone), xc = __ldcg(&ctl->xcap);
    const uint32_t cap_end = xc > 0xFFFFFFFFu - x0 ? 0xFFFFFFFFu : x0 + xc;
    const uint32_t at = base + __popc(want & lanemask_lt());
    if (at < cap_end) xlist[at] = v;
  }
}

// ------------------------------------------------------------ contribution gathers ----
// The sweep's cost is its gathers: 32 random contributions a warp instruction are 32 lines
// to look up, one per clock and SM (L1 and L2 both about 75% busy).  A handle's internal
// numbering puts the vertices of largest out-degree first, and every SM keeps the
// contributions of the first `hot` vertices in shared memory for the iteration, where 32
// random reads take a few clocks.  The copy takes part of the SM's L1, which also holds the
// lines of loads in flight.  Full sweep of R-MAT scale 22 (69 M edges) in 64-bit mode: 0.318 ms with
// every gather through L1; 0.246 with 64 KB hot (31% of the gathers), 0.238 with 96 KB, 0.234
// with 128 KB (38%), 0.239 with 160 KB; of 1.3 M vertices and 21.6 M edges in FP32: 0.128;
// 0.071, 0.068, 0.067, 0.067.
constexpr uint32_t kHotBytes = 131072;
static_assert(kHotBytes % 128 == 0, "copied in eight pieces of a multiple of 16 bytes");

// Volatile: the contributions change between the iterations of one launch.
__device__ __forceinline__ void cold_load(long long &r, const long long *p, bool on, unsigned long long pol) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p ld.global.ca.L2::cache_hint.b64 %0, [%1], %3;\n}\n"
               : "+l"(r)
               : "l"(p), "r"((uint32_t)on), "l"(pol));
}
__device__ __forceinline__ void cold_load(float &r, const float *p, bool on, unsigned long long pol) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p ld.global.ca.L2::cache_hint.f32 %0, [%1], %3;\n}\n"
               : "+f"(r)
               : "l"(p), "r"((uint32_t)on), "l"(pol));
}
__device__ __forceinline__ void hot_load(long long &r, uint32_t p, bool on) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p ld.shared.b64 %0, [%1];\n}\n"
               : "+l"(r)
               : "r"(p), "r"((uint32_t)on));
}
__device__ __forceinline__ void hot_load(float &r, uint32_t p, bool on) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p ld.shared.f32 %0, [%1];\n}\n"
               : "+f"(r)
               : "r"(p), "r"((uint32_t)on));
}
__device__ __forceinline__ void hot_load(long long &r, uint32_t p) {
  asm volatile("ld.shared.b64 %0, [%1];" : "=l"(r) : "r"(p));
}
__device__ __forceinline__ void hot_load(float &r, uint32_t p) {
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(r) : "r"(p));
}
// s plus the contributions of RUNS runs of four columns, in order.  The hot ones (of vertices
// [hfirst, hfirst + hot), copied to shared memory from sbase on) come from there, into
// the registers that the others are then loaded into, all in flight together.  A column is
// cold if w - (hfirst + hot) < kNoCol - (hfirst + hot), which no hot one and no free slot
// (kNoCol) is.  MOSTLY: every lane reads the copy, the other columns the zero behind it, which saves
// the tests where most columns are hot: 256 batched graphs FP32 0.529 ms an iteration against
// 0.541; the full sweep of scale 22 (64-bit, 38% hot) 0.228 against 0.223.
template <int RUNS, bool MOSTLY, class C>
__device__ __forceinline__ C gather_runs(C s, const C *Cv, const uint4 *q, uint32_t sbase, uint32_t hfirst,
                                         uint32_t hot, unsigned long long pol) {
  C x[RUNS][4];
#pragma unroll
  for (int k = 0; k < RUNS; k++) {
    const uint32_t w[4] = {q[k].x, q[k].y, q[k].z, q[k].w};
#pragma unroll
    for (int e = 0; e < 4; e++) {
      const uint32_t i = w[e] - hfirst;
      if constexpr (MOSTLY) {
        hot_load(x[k][e], sbase + min(i, hot) * (uint32_t)sizeof(C));
      } else {
        x[k][e] = (C)0;
        hot_load(x[k][e], sbase + i * (uint32_t)sizeof(C), i < hot);
      }
    }
  }
  const uint32_t end = hfirst + hot;
#pragma unroll
  for (int k = 0; k < RUNS; k++) {
    const uint32_t w[4] = {q[k].x, q[k].y, q[k].z, q[k].w};
#pragma unroll
    for (int e = 0; e < 4; e++) cold_load(x[k][e], Cv + w[e], w[e] - end < kNoCol - end, pol);
  }
#pragma unroll
  for (int k = 0; k < RUNS; k++) s += ((x[k][0] + x[k][1]) + x[k][2]) + x[k][3];
  return s;
}

__device__ __forceinline__ uint4 ld_cols_v(const uint32_t *p, unsigned long long pol) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p), "l"(pol));
  return r;
}
__device__ __forceinline__ uint4 ldv(const uint4 *p) {
  uint4 r;
  asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}
__device__ __forceinline__ long long ldv(const long long *p) { long long r; asm volatile("ld.global.cg.b64 %0, [%1];" : "=l"(r) : "l"(p)); return r; }
__device__ __forceinline__ unsigned long long ldv(const unsigned long long *p) { unsigned long long r; asm volatile("ld.global.cg.b64 %0, [%1];" : "=l"(r) : "l"(p)); return r; }
__device__ __forceinline__ float ldv(const float *p) { float r; asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(r) : "l"(p)); return r; }
__device__ __forceinline__ uint16_t ldv(const uint16_t *p) { uint16_t r; asm volatile("ld.global.cg.u16 %0, [%1];" : "=h"(r) : "l"(p)); return r; }

// The zero behind the block's copy (one thread, before a block barrier; see gather_runs).
__device__ __forceinline__ void hot_zero(uint32_t at) {
  asm volatile("st.shared.b64 [%0], %1;" ::"r"(at), "l"(0ull) : "memory");
}

// The block's copy of the hot contributions: eight bulk copies issued by one thread (blocks
// start at different pieces), completion on the block's mbarrier.  The contributions were written by other SMs through the generic proxy.
__device__ __forceinline__ void stage_hot(const void *Cin, uint32_t bytes, uint32_t sbase, uint32_t bar) {
  asm volatile("fence.proxy.async;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
  const uint32_t piece = ((bytes >> 3) + 15u) & ~15u;
  for (uint32_t k = 0; k < 8; k++) {
    const uint32_t at = ((k + blockIdx.x) & 7u) * piece;
    if (at >= bytes) continue;
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(sbase + at),
                 "l"((const char *)Cin + at), "r"(min(piece, bytes - at)), "r"(bar)
                 : "memory");
  }
}

// The rounds of a pass that a block's warps take (in shared memory, set by thread 0 before a
// pass): tier t's round k of the block is round first[t] + k * stride of the tier (32 items, 4
// items, 1 chunk), while below rounds[t]; the tier's items start at base[t] and are items[t].
struct Rounds {
  uint32_t base[3], first[3], rounds[3], items[3], stride;
  uint32_t next[3];  // rounds taken so far
  uint32_t hfirst, hot;  // vertices [hfirst, hfirst + hot) have their contributions in shared memory
  uint32_t grew;         // compacted iterations: some vertex of the block's expanded for the first time
};

// All rounds of a single graph, dealt to the blocks in turn, starting after the block that took
// the last round of the tier before (with few rounds no block gets one more of every tier).
__device__ __forceinline__ void deal_rounds(Rounds &r, uint32_t n0, uint32_t n1, uint32_t n2, uint32_t off1,
                                            uint32_t off2, uint32_t hot) {
  const uint32_t nblk = gridDim.x, b = blockIdx.x;
  const uint32_t r0 = (uint32_t)(((uint64_t)n0 + 31) >> 5), r1 = (uint32_t)(((uint64_t)n1 + 3) >> 2);
  const uint32_t d1 = r0 % nblk, d2 = (uint32_t)(((uint64_t)r0 + r1) % nblk);
  r.base[0] = 0;
  r.base[1] = off1;
  r.base[2] = off2;
  r.first[0] = b;
  r.first[1] = b >= d1 ? b - d1 : b + nblk - d1;
  r.first[2] = b >= d2 ? b - d2 : b + nblk - d2;
  r.rounds[0] = r0;
  r.rounds[1] = r1;
  r.rounds[2] = n2;
  r.items[0] = n0;
  r.items[1] = n1;
  r.items[2] = n2;
  r.stride = nblk;
  r.next[0] = r.next[1] = r.next[2] = 0;
  r.hfirst = 0;
  r.hot = hot;
  r.grew = 0;
}

// What a pass over sweep items needs beside the handle's arguments and its rounds, and what it
// leaves.
template <bool F32>
struct Pass {
  uint32_t it;
  bool expand, pulling, erec;
  bool every;                  // batched: every vertex, no stamps
  uint32_t cap_end;
  uint32_t sbase;
  Rounds *r;
  typename Store<F32>::R base;  // batched: (1 - alpha) / n of the graph the rounds belong to
  typename Num<F32>::B my_max;
  uint32_t my_v, my_e, xloc, jloc;
};

// The block's part of one iteration of Eq. 1 over sweep items.  MODE 0: every vertex (Static,
// Naive-dynamic).  MODE 1: a dense Dynamic Frontier iteration over every item, vertices not
// affected skipped; when pulling, a tier-0/1 vertex not yet affected first checks its in-row
// against the previous iteration's change flags and joins if one is set (tier-2 rows were
// decided by the prologue).  MODE 2: a dense iteration over the compacted items of the
// affected vertices.  MODE 3: a batched handle, as MODE 1 (or MODE 0: io.every) for rounds of
// one graph at a time; first expansions are only counted (its frontier grows by pulls alone).
// Dynamic Frontier modes record change flags when asked, and first
// expansions (changes above tau_f of vertices whose out-row was never marked from; the
// stamp's top bit then caches that it was).  Per-vertex sums are taken exactly as in the
// persistent kernel's sweeps: thread rows in runs of eight, 8-lane groups, chunk-edge
// chunks added in chunk order.
template <bool F32, int MODE>
__device__ __forceinline__ void sweep_pass(const SweepArgs<F32> &a, Pass<F32> &io) {
  constexpr bool CMP = MODE == 2, MULTI = MODE == 3, ALL = MODE == 1 || MULTI;
  using S = Store<F32>;
  using R = typename S::R;
  using C = typename S::C;
  using A = typename S::A;
  using B = typename Num<F32>::B;
  RankCtl *ctl = a.ctl;
  const uint32_t tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
  Rounds &rr = *io.r;
  const uint32_t it = io.it, hot = rr.hot, hfirst = MULTI ? rr.hfirst : 0u, sbase = io.sbase;
  const int par = it & 1;
  const R *Rin = par ? a.R1 : a.R0;
  const C *Cin = par ? a.C1 : a.C0;
  R *Rout = par ? a.R0 : a.R1;
  C *Cout = par ? a.C0 : a.C1;
  const uint4 *T = CMP ? a.items_cmp : a.items;  // (tiers 1 and 2: from rr.base on)
  const bool every = MULTI && io.every;
  const bool expand = io.expand, pulling = io.pulling, erec = io.erec;
  const uint32_t cap_end = io.cap_end;
  bool xfull = false;
  uint32_t xloc = 0, jloc = 0;
  const uint8_t *Eprev = a.emap + (size_t)((it - 1) & 1) * a.n;  // read only when pulling (it > 0)
  uint8_t *Ecur = a.emap + (size_t)(it & 1) * a.n;
  const uint16_t itk = (uint16_t)it;
  const unsigned long long pol_cols = l2_evict_first(), pol_c = l2_evict_last();
  B my_max = 0;
  uint32_t my_v = 0, my_e = 0;

  // new rank and contribution of v; returns the change as delta bits
  auto finish = [&](uint32_t v, C sum, R rold, A ad) -> B {
    const R r = (MULTI ? io.base : a.base) + sum;
    Rout[v] = r;
    st_keep(Cout + v, S::contrib(r, ad), pol_c);
    const B dr = Num<F32>::delta(r, rold);
    my_max = dr > my_max ? dr : my_max;
    return dr;
  };
  // a vertex that joins by pull: stamp and affected bit (counted, not listed: the
  // writeback lists the affected set from the stamps)
  auto join_now = [&](uint32_t v) {
    a.stamp[v] = itk;
    if (!MULTI) atomicOr(a.bitmap + (v >> 5), 1u << (v & 31));
    jloc++;
  };
  // All-item iterations, after v's change dr: change flag (iterations that record them),
  // first-expansion test; true where v's out-row is to be marked from for the first time.
  // st = v's stamp as read and xw its word of the bitmap of out-rows the marking launch
  // scanned (a joined vertex's stamp is it and it never expanded)
  auto book = [&](uint32_t v, B dr, uint16_t st, bool joined, uint32_t xw) -> bool {
    if (!expand) return false;
    const bool big = dr > a.ftol;
    if (erec) Ecur[v] = big ? 1 : 0;
    if (!big || (st & kStampExp)) return false;
    const bool was = !joined && ((xw >> (v & 31)) & 1u);
    a.stamp[v] = (uint16_t)(st | kStampExp);
    return !was;
  };
  // A block's warps take its rounds as they get free, one ahead of the
  // round they work on, so that the next round's items are on their way.  (Dealt to the warps
  // beforehand, they waited 13% of an iteration for the slowest: 0.303 ms against 0.238.)
  auto take = [&](int t) -> uint32_t {  // the warp's next round of tier t
    uint32_t k = 0;
    if (lane == 0) k = atomicAdd(&rr.next[t], 1u);
    return rr.first[t] + __shfl_sync(kFull, k, 0) * rr.stride;
  };

  // tier 0: one thread per vertex, 32 consecutive items per warp.  In all-item iterations
  // the stamp, the expanded word, the rank, the factor and the first eight columns are
  // loaded together (the row's loads do not wait for the stamp; a vertex not affected
  // wastes them).  These launches serve self-loop mode only, where a one-entry row is the
  // vertex's own self-loop.
  //
  // Every tier has the items of its next round on the way while it works on the current
  // one, so a round's row loads wait for no item.
  const uint4 zero4 = make_uint4(0, 0, 0, 0), none4 = make_uint4(kNoCol, kNoCol, kNoCol, kNoCol);
  // A row's loads.  (Issued a round ahead they save nothing that the registers they need do not
  // cost: full sweep of scale 22 0.233 ms against 0.229, 1.3 M vertices FP32 0.061 against 0.0625,
  // 256 graphs batched 0.555 against 0.529.)
  struct Row {
    uint4 q[2];
    R rold;
    A ad;
    uint32_t xw;
    uint16_t st;
  };
  auto load0 = [&](const uint4 &item) -> Row {  // item.z == 0: none
    Row r{{none4, none4}, (R)0, (A)0, 0u, 0};
    if (item.z) {
      const uint32_t v = item.x;
      if (ALL) {
        if (!every) r.st = ldv(a.stamp + v);
        if (expand) r.xw = __ldcg(a.xbits + (v >> 5));
      }
      r.rold = ldv(Rin + v);
      r.ad = ldv(a.adeg + v);
      if (item.z > 1) {  // a one-entry row is v's self-loop: no column needed
        r.q[0] = ld_cols_v(a.in_col + item.y, pol_cols);
        if (item.z > 4) r.q[1] = ld_cols_v(a.in_col + item.y + 4, pol_cols);
      }
    }
    return r;
  };
  auto row0 = [&](const uint4 &item, Row &r, uint32_t i) {
    bool act = false, join = false, push = false;
    if (item.z) {
      act = !ALL || every || (r.st & kStampIt) <= itk;
      if (ALL && !act && pulling && item.z > 1) {
        if (item.z <= 8) {
          const uint32_t w[8] = {r.q[0].x, r.q[0].y, r.q[0].z, r.q[0].w, r.q[1].x, r.q[1].y, r.q[1].z, r.q[1].w};
          uint32_t any = 0;  // every flag load issued at once (no chain of dependent loads)
#pragma unroll
          for (uint32_t j = 0; j < 8; j++) any |= j < item.z ? (uint32_t)__ldcg(Eprev + w[j]) : 0u;
          join = any != 0;
        } else {
          for (uint32_t j = 0; j < item.z && !join; j++) join = __ldcg(Eprev + __ldg(a.in_col + item.y + j)) != 0;
        }
        if (join) join_now(item.x);
      }
    }
    if (act || join) {
      const uint32_t v = item.x;
      C sum = (C)0;
      if (item.z == 1) {
        // self-loop mode: the row is v's self-loop, and C[v] is contrib(R[v], A[v]) (stored
        // that way by the previous iteration), so it is recomputed from the values in hand
        sum += S::contrib(r.rold, r.ad);
      } else {
        // runs of eight columns, the first one in hand
        for (uint32_t j0 = 0;;) {
          sum = gather_runs<2, MULTI && F32>(sum, Cin, r.q, sbase, hfirst, hot, pol_c);
          if (item.z <= 8) break;
          if ((j0 += 8) >= item.z) break;
          r.q[0] = ld_cols(a.in_col + item.y + j0, pol_cols);
          r.q[1] = item.z - j0 > 4 ? ld_cols(a.in_col + item.y + j0 + 4, pol_cols) : none4;
        }
      }
      const B dr = finish(v, sum, r.rold, r.ad);
      if constexpr (ALL) push = book(v, dr, join ? itk : r.st, join, r.xw);
      if constexpr (CMP) {
        if (expand && dr > a.ftol && !item.w)
          expand_cmp(ctl, a.stamp, a.xbits, a.xlist, a.items_cmp, a.out_rd, v, i, true, &rr.grew);
      }
      if constexpr (ALL) {
        my_v++;
        my_e += item.z;
      }
    }
    if constexpr (MULTI) xloc += push ? 1u : 0u;
    else if constexpr (ALL) note_expansion(ctl, a.xlist, push, item.x, lane, cap_end, xfull, xloc);
  };
  auto tier0 = [&]() {
    const uint32_t r0 = rr.rounds[0], n0 = rr.items[0];
    if constexpr (MULTI) T = a.items + rr.base[0];
    auto item_at = [&](uint32_t k) -> uint4 { return k < r0 && k * 32 + lane < n0 ? ldv(T + k * 32 + lane) : zero4; };
    uint32_t k = take(0);
    uint4 item = item_at(k);
    while (k < r0) {
      const uint32_t now = k;
      const uint4 cur = item;
      k = take(0);
      item = item_at(k);
      Row r = load0(cur);
      row0(cur, r, now * 32 + lane);
    }
  };

  // tier 1: rows of lo < len <= group_max (<= kGroupMax) by 8-lane groups, four vertices per warp
  const uint32_t grp = lane >> 3, gl = lane & 7;
  auto load1 = [&](const uint4 &item) -> Row {
    Row r{{none4, none4}, (R)0, (A)0, 0u, 0};
    if (item.z) {
      if (ALL && !every) r.st = ldv(a.stamp + item.x);
      if (gl == 0) {
        r.rold = ldv(Rin + item.x);
        r.ad = ldv(a.adeg + item.x);
        if (ALL && expand) r.xw = __ldcg(a.xbits + (item.x >> 5));
      }
#pragma unroll
      for (int k = 0; k < 2; k++) {
        const uint32_t j = 4 * (gl + 8 * k);
        if (j < item.z) r.q[k] = ld_cols_v(a.in_col + item.y + j, pol_cols);
      }
    }
    return r;
  };
  auto row1 = [&](const uint4 &item, Row &r, uint32_t i) {  // i: the item's index
    const bool act = item.z && (!ALL || every || (r.st & kStampIt) <= itk);
    bool join = false;
    if (ALL && pulling) {
      bool h = false;
      if (item.z && !act) {
#pragma unroll
        for (int k = 0; k < 2; k++) {
          const uint32_t j = 4 * (gl + 8 * k);
          const uint32_t w[4] = {r.q[k].x, r.q[k].y, r.q[k].z, r.q[k].w};
#pragma unroll
          for (uint32_t k2 = 0; k2 < 4; k2++) h |= j + k2 < item.z && __ldcg(Eprev + w[k2]) != 0;
        }
      }
      join = ((__ballot_sync(kFull, h) >> (grp * 8)) & 0xFFu) != 0;
      if (join && gl == 0) join_now(item.x);
    }
    C sum = (C)0;
    if (act || join) sum = gather_runs<2, MULTI && F32>(sum, Cin, r.q, sbase, hfirst, hot, pol_c);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
    bool push = false;
    if ((act || join) && gl == 0) {
      const B dr = finish(item.x, sum, r.rold, r.ad);
      if constexpr (ALL) push = book(item.x, dr, join ? itk : r.st, join, r.xw);
      if constexpr (CMP) {
        if (expand && dr > a.ftol && !item.w)
          expand_cmp(ctl, a.stamp, a.xbits, a.xlist, a.items_cmp, a.out_rd, item.x, i, true, &rr.grew);
      }
      if constexpr (ALL) {
        my_v++;
        my_e += item.z;
      }
    }
    if constexpr (MULTI) xloc += push ? 1u : 0u;
    else if constexpr (ALL) note_expansion(ctl, a.xlist, push, item.x, lane, cap_end, xfull, xloc);
  };
  auto tier1 = [&]() {
    const uint32_t r1 = rr.rounds[1], n1 = rr.items[1], off1 = rr.base[1];
    if constexpr (MULTI) T = a.items;
    auto item_at = [&](uint32_t k) -> uint4 {
      return k < r1 && k * 4 + grp < n1 ? ldv(T + off1 + k * 4 + grp) : zero4;
    };
    uint32_t k = take(1);
    uint4 item = item_at(k);
    while (k < r1) {
      const uint32_t now = k;
      const uint4 cur = item;
      k = take(1);
      item = item_at(k);
      Row r = load1(cur);
      row1(cur, r, off1 + now * 4 + grp);
    }
  };

  // tier 2: chunks of at most kChunk edges dealt round-robin to warps; a row split into several chunks
  // is finished by the warp that completes its last chunk, which adds the partial sums in
  // chunk order
  C *part = a.partials;
  auto tier2 = [&]() {
    const uint32_t n2 = rr.rounds[2], off2 = rr.base[2];
    if constexpr (MULTI) T = a.items;
    uint32_t k = take(2);
    uint4 item_nx = k < n2 ? ldcg(T + off2 + k) : zero4;
    while (k < n2) {
      const uint4 ch = item_nx;
      k = take(2);
      if (k < n2) item_nx = ldcg(T + off2 + k);
      const uint32_t v = ch.x;
      uint16_t st = 0;
      if (ALL && !every) st = ldcg(a.stamp + v);
      const uint32_t len = ch.z & 0x3FFu;
      const bool several = (ch.z >> 31) != 0;
      R rold = (R)0;
      A ad = (A)0;
      uint32_t deg = len, xw = 0;
      if (lane == 0) {
        rold = ldcg(Rin + v);
        ad = __ldg(a.adeg + v);
        if (several) deg = __ldg(&a.in_rd[v]).y;
        if (ALL && expand) xw = __ldcg(a.xbits + (v >> 5));
        if (CMP && expand) st = ldcg(a.stamp + v);
      }
      const uint32_t *cols = a.in_col + ch.y;
      uint4 q[4] = {none4, none4, none4, none4};
#pragma unroll
      for (int r = 0; r < 4; r++) {
        const uint32_t j = 4 * (lane + 32 * r);
        if (j < len) q[r] = ld_cols(cols + j, pol_cols);
      }
      if (ALL && !every && (st & kStampIt) > itk) continue;  // warp-uniform: not affected
      // two runs at a time: all four in flight together need 16 more registers (0.238 ms a full
      // sweep of scale 22 against 0.235)
      C sum = gather_runs<2, MULTI && F32>((C)0, Cin, q, sbase, hfirst, hot, pol_c);
      if (len > 256) sum = gather_runs<2, MULTI && F32>(sum, Cin, q + 2, sbase, hfirst, hot, pol_c);
      sum = warp_sum(sum);
      bool fin = true;
      if (several) {
        const uint32_t nch = (__shfl_sync(kFull, deg, 0) + a.chunk - 1) / a.chunk;
        uint32_t old = 0;
        if (lane == 0) {
          part[ch.w] = sum;
          __threadfence();
          old = atomicAdd(&a.chunk_done[v], 1u);
        }
        old = __shfl_sync(kFull, old, 0);
        fin = old == nch - 1;
        if (fin) {
          __threadfence();
          const uint32_t first = ch.w - ((ch.z >> 10) & 0x1FFFFFu);
          C tot = (C)0;
          for (uint32_t c = lane; c < nch; c += 32) tot += ldcg(part + first + c);
          sum = warp_sum(tot);
          if (lane == 0) a.chunk_done[v] = 0;
        }
      }
      bool push = false;
      if (fin && lane == 0) {
        const B dr = finish(v, sum, rold, ad);
        // chunks have no cache bit: the stamp and the word read with the row decide
        if constexpr (ALL) push = book(v, dr, st, false, xw);
        if constexpr (CMP) {
          if (expand && dr > a.ftol && !(st & kStampExp))
            expand_cmp(ctl, a.stamp, a.xbits, a.xlist, a.items_cmp, a.out_rd, v, 0, false, &rr.grew);
        }
        if constexpr (ALL) {
          my_v++;
          my_e += deg;
        }
      }
      if constexpr (MULTI) xloc += push ? 1u : 0u;
      else if constexpr (ALL) note_expansion(ctl, a.xlist, push, v, lane, cap_end, xfull, xloc);
    }
  };

  // Three warps of four take the long rows first: their gathers, bound by the rate of random
  // loads, then overlap the latency-bound short rows of the fourth.  Full sweep of scale 22:
  // 0.223 ms; one warp of two 0.228, one of four 0.234, all 0.238, none 0.244.
  if (wib & 3) {
    tier2();
    tier0();
    tier1();
  } else {
    tier0();
    tier1();
    tier2();
  }
  io.my_max = my_max;
  io.my_v = my_v;
  io.my_e = my_e;
  io.xloc = xloc;
  io.jloc = jloc;
}

__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long k) {
  const uint32_t hi = (uint32_t)(k >> 32), top = __reduce_max_sync(kFull, hi);
  return (unsigned long long)top << 32 | __reduce_max_sync(kFull, hi == top ? (uint32_t)k : 0u);
}

// The L-inf change of an iteration from the threads' maxima: one atomic per block.  Called
// by the whole block; s_key is free after the next block barrier.  Returns the block's key in
// warp 0.
template <bool F32>
__device__ __forceinline__ unsigned long long block_max(typename Num<F32>::B my_max, unsigned long long *dR,
                                                        unsigned long long *s_key) {
  unsigned long long m = warp_max_key(Num<F32>::key(my_max));
  if ((threadIdx.x & 31) == 0) s_key[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = warp_max_key(threadIdx.x < kSweepWarps ? s_key[threadIdx.x] : 0ull);
    if (threadIdx.x == 0 && m) atomicMax(dR, m);
  }
  return m;
}

// RankCtl::tally: a run's grid barrier whose counter also says what the iteration left: blocks
// that have arrived (low bits), those with a change above the tolerance, those with first
// expansions, an error.  Two counters take turns, so that none is added to before every block
// has read it.
constexpr int kTallyAbove = 24, kTallyGrew = 43;
constexpr unsigned long long kTallyErr = 1ull << 63, kTallyOnes = (1ull << 19) - 1;

// A wait for the block's hot contributions that ran out ends the call (error 2); the copies
// in flight are waited for once more, bounded, before the block gives up its shared memory.
__device__ __forceinline__ bool hot_landed(RankCtl *ctl, uint32_t bar, uint32_t parity) {
  if (__all_sync(kFull, mbar_wait(bar, parity, kStageTimeoutNs))) return true;  // the same in the whole warp
  atomicOr(&ctl->err, 2u);
  atomicOr(&ctl->lbar, kBarErr);  // a run's barriers end too
  for (int k = 0; k < 2; k++) atomicOr(&ctl->tally[k], kTallyErr);
  mbar_wait(bar, parity, kStageTimeoutNs);
  return false;
}

// Grid barrier between the iterations of a persistent launch, its wait bounded; false in every
// thread of the block once the call has an error. 
__device__ __forceinline__ bool run_barrier(RankCtl *ctl, uint32_t &epoch, uint32_t *s_err) {
  __syncthreads();
  epoch++;
  if (threadIdx.x == 0) {
    asm volatile("fence.proxy.async;" ::: "memory");  // the next hot copies read what was written
    *s_err = bar_wait(ctl, &ctl->lbar, epoch) ? 0u : 1u;
  }
  __syncthreads();
  return *s_err == 0;
}

// The barrier between the iterations of a run: `above` and `grew` (thread 0's) are set to
// whether any block had them set.  seen: the two counters as last read, thread 0's.  The
// decision comes with the arrivals; reading the iteration's L-inf change and expansions after
// the barrier was one more round trip to L2.  (With the block's maximum by two reductions
// instead of ten shuffles, an iteration of a run over an R-MAT graph of 16,384 vertices takes
// 6.5 us instead of 6.9, and one over 1.3 M vertices 61.5 instead of 63.)
__device__ __forceinline__ bool run_tally(RankCtl *ctl, uint32_t &epoch, uint32_t *s_err, uint32_t *s_left,
                                          bool above, bool grew, unsigned long long (&seen)[2]) {
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("fence.proxy.async;" ::: "memory");  // the next hot copies read what was written
    unsigned long long *bar = &ctl->tally[epoch & 1u];
    red_release_add_u64(bar, 1ull | (unsigned long long)above << kTallyAbove | (unsigned long long)grew << kTallyGrew);
    const uint32_t target = (epoch / 2 + 1) * gridDim.x;
    const unsigned long long lim = *(volatile unsigned long long *)&ctl->bar_limit_ns;
    const uint32_t every = lim ? 0u : 127u;
    unsigned long long t0 = 0, x;
    for (uint32_t spins = 1;; spins++) {
      x = ld_acquire_u64(bar);
      if ((uint32_t)x % (1u << kTallyAbove) >= target || x >= kTallyErr) break;
      if ((spins & every) == 0) {
        const unsigned long long t = globaltimer_ns();
        if (t0 == 0) {
          t0 = t;
        } else if (t - t0 > (lim ? lim : kBarrierTimeoutNs)) {
          atomicExch(&ctl->err_where, epoch + 1);
          atomicOr(&ctl->err, 1u);
          for (int k = 0; k < 2; k++) atomicOr(&ctl->tally[k], kTallyErr);
          x = kTallyErr;
          break;
        }
      }
    }
    const unsigned long long old = seen[0];
    seen[0] = seen[1];
    seen[1] = x;
    *s_left = (((x >> kTallyAbove) & kTallyOnes) != ((old >> kTallyAbove) & kTallyOnes) ? 1u : 0u) |
              (((x >> kTallyGrew) & kTallyOnes) != ((old >> kTallyGrew) & kTallyOnes) ? 2u : 0u);
    *s_err = x >= kTallyErr ? 1u : 0u;
  }
  epoch++;
  __syncthreads();
  return *s_err == 0;
}

// Host side: a handle's sweep arguments (async: both parities aliased, and no copy in shared
// memory: contributions are written while the others' copies of them would still be read, and
// a copy taken at the start of an iteration would hide what the iteration has updated since).
template <bool F32>
SweepArgs<F32> sweep_args(const Graph *g, bool async) {
  using S = Store<F32>;
  SweepArgs<F32> a{};
  a.R0 = (typename S::R *)g->R[0];
  a.R1 = (typename S::R *)(async ? g->R[0] : g->R[1]);
  a.C0 = (typename S::C *)g->C[0];
  a.C1 = (typename S::C *)(async ? g->C[0] : g->C[1]);
  a.adeg = (const typename S::A *)g->adeg;
  a.in_col = g->in.col;
  a.in_rd = g->in.rd;
  a.items = g->items;
  a.items_cmp = g->items_cmp;
  a.partials = (typename S::C *)g->partials;
  a.chunk_done = g->chunk_done;
  a.stamp = g->stamp;
  a.bitmap = g->bitmap;
  a.list0 = g->list[0];
  a.xbits = g->xbits;
  a.xlist = g->xlist;
  a.emap = g->emap;
  a.out_rd = g->out.rd;
  a.ctl = g->ctl;
  a.hot = async ? 0u : g->hot;
  const double n = (double)g->n;
  if constexpr (F32) {
    a.base = (float)((1.0 - g->p.alpha) / n);
    float ft = (float)g->p.frontier_tol;
    std::memcpy(&a.ftol, &ft, 4);
    double tl = g->p.tol;
    std::memcpy(&a.tol_key, &tl, 8);
  } else {
    const double one = 4611686018427387904.0;  // 2^62
    a.base = std::llrint((1.0 - g->p.alpha) / n * one);
    a.ftol = (unsigned long long)std::floor(std::min(g->p.frontier_tol * one, 9.0e18));
    a.tol_key = (unsigned long long)std::floor(std::min(g->p.tol * one, 9.0e18));
  }
  a.n = g->n;
  a.chunk = g->chunk_len;
  a.max_iter = g->p.max_iter;
  return a;
}

}  // namespace prdf
