// sweep.cu - the rank iterations of single-graph handles in self-loop mode.
//
// Static and Naive-dynamic PageRank (Section 3.1, Section 3.3.1) and the dense iterations
// of Dynamic Frontier (Algorithm 1), its asynchronous form (Section 4.2) and Dynamic
// Traversal (Section 3.3.2) run here.  An iteration of Eq. 1 is one pass over sweep items
// (sweep_pass).  Iterations that need nothing from other kernels in between (all of Static
// and Naive-dynamic, the settled iterations of a dense Dynamic Frontier call) follow one
// another in one persistent cooperative launch (k_loop), a grid barrier apart; the
// iterations of a growing Dynamic Frontier set are a launch each (k_sweep).  A CUDA graph with
// conditional nodes strings these launches together on the device; the host is not
// involved between iterations.
//
// The dense iterations of a Dynamic Frontier call grow the affected set in one of two
// ways, which give the same set: Algorithm 1 marks the out-neighbours of every vertex
// whose rank changed by more than tau_f, so a vertex joins iteration i + 1 exactly when
// one of its in-neighbours in G^t changed by more than tau_f in iteration i.
//   pull  every sweep item is visited; a prologue finds the vertices not yet affected
//         that have such an in-neighbour (per-vertex change flags of iteration i, kept in
//         two parities) and they join; the sweep skips vertices not affected.
//   push  the prologue scans the out-rows of the vertices whose change exceeded tau_f
//         for the first time in iteration i (as the marking launch does; later changes
//         of a vertex mark nothing new), and appends the sweep items of every newly
//         marked vertex to the compacted items, which the sweep then visits alone.
// After an iteration with many first expansions the next one pulls (its cost is about a
// full sweep, while pushing millions of out-rows costs several); otherwise it pushes (a
// few expansions without long out-rows by a plain launch, the rest by a cooperative one).
// Leaving pull for push rebuilds the compacted items, as does a set that grew by more
// than 1/16 since they were last rebuilt.  The settled compacted iterations, which need
// no prologue, stay in one k_loop launch.  Sums are taken per vertex exactly as in the
// persistent kernel's dense sweeps, so results equal a single marking launch bit for bit.
#include <cstring>
#include <vector>

#include "sweep_dev.cuh"

namespace prdf {

constexpr uint32_t kPullDiv = 256;  // more than n / kPullDiv first expansions: the next iteration pulls
constexpr uint32_t kPullMin = 64;   // and at least this many
// A handle in a server: in-edges (of the whole graph) of a run's iterations at most, about 2 ms.  A
// block of a run holds its SM's registers, so other requests' launches wait for its end.  Eight R-MAT
// graphs of 2^18 to 2^24 vertices, 2 slots, 50 requests/s: 3 in 100 of the four smallest graphs'
// requests take more than 21 to 27 ms (23 to 30 with unbounded runs), of the largest's 54 (49);
// at saturation no difference, nor between 2^27 and 2^31.
constexpr uint64_t kRunEdges = 1ull << 29;
// ... and a graph of fewer edges than this runs on half of the device: its iterations are bound by
// latency, so two side by side end sooner than in turns.  Five graphs of 2^16 to 2^20 vertices, 2
// slots, all requests at once: 16.8 ms with those of up to 2^24 edges on half of the device, 17.2 of 2^22,
// 17.4 none, 18.2 of 2^25; 16.1 with their prologues (k_df_push) on half of it too.
constexpr uint64_t kShareEdges = 1ull << 24;
constexpr uint32_t kLightPush = 16384;  // at most this many first expansions: the light push may mark them

// End of an all-item iteration, or of a run of compacted iterations it_first ... it, by one
// thread of the last block to finish: L-inf test, the next iteration's way of marking, trace,
// loop condition.
template <bool F32>
__device__ void sweep_decide(const SweepArgs<F32> &a, uint32_t it_first, uint32_t it, bool all_items) {
  RankCtl *ctl = a.ctl;
  const unsigned long long dR = __ldcg(&ctl->dR_bits[it]);
  const uint32_t iters = it + 1;
  const bool conv = dR <= a.tol_key;
  // a prologue whose grid barrier timed out recorded an error: the loop ends
  const bool cont = !conv && (int)iters < a.max_iter && __ldcg(&ctl->err) == 0;
  ctl->iterations = iters;
  ctl->converged = conv ? 1u : 0u;
  ctl->last_key = dR;
  ctl->it_cur = iters;
  ctl->ticket = 0;
  ctl->bar = 0;  // a prologue's grid barriers count from zero, and so do a run's
  ctl->tally[0] = ctl->tally[1] = 0;
  ctl->launches += 1;
  uint32_t total = 0;
  for (int b = 0; b < 3; b++) {  // only the first iteration of a run has marks of its own
    const uint32_t d = __ldcg(&ctl->dcnt[b]) + __ldcg(&ctl->tail[it_first][b]);
    ctl->dcnt[b] = d;
    ctl->final_cnt[b] = d;
    total += d;
  }
  const uint32_t jt = __ldcg(&ctl->jtotal) + __ldcg(&ctl->tail[it_first][3]);
  ctl->jtotal = jt;
  total += jt;
  if (all_items) {
    ctl->t_ns[it + 2] = globaltimer_ns();
  } else {
    // compacted iterations swept exactly the compacted items (counted here, not by the
    // sweep: its loops keep the registers of a full sweep)
    const unsigned long long runs = it - it_first + 1;
    ctl->vproc += runs * (__ldcg(&ctl->cmp_total) + __ldcg(&ctl->app_since));
    ctl->eproc += runs * __ldcg(&ctl->cmp_edges);
  }
  ctl->eprev = __ldcg(&ctl->eproc);
  for (uint32_t k = it_first; k <= it; k++) {
    ctl->it_aff[k] = total;
    ctl->it_kind[k] = (uint8_t)(k == it_first ? __ldcg(&ctl->kind_cur) : 5u);
  }
  uint32_t pro = 0, all = 1;
  if (!cont && __ldcg(&ctl->dexpand)) {
    // the loop ends: this iteration's first expansions still mark their out-neighbours
    // (the affected set of Algorithm 1 includes the last iteration's marks), by a pull
    // over every tier when the change flags were recorded and the list may be partial,
    // by a push otherwise
    const uint32_t xend = __ldcg(&ctl->xcnt), lo = __ldcg(&ctl->xdone);
    const uint32_t x = xend - lo;
    const bool recorded = __ldcg(&ctl->erec) != 0;
    const uint32_t pull_at = max(kPullMin, a.n / kPullDiv);
    ctl->xdone = xend;
    ctl->compact_now = 0;
    ctl->push_items = 0;
    uint32_t fin = 0;
    if (x && recorded && (x > pull_at || x > __ldcg(&ctl->xcap))) {
      ctl->pull_check = 1;
      ctl->pull_all = 1;
      fin = 1;
    } else if (x) {
      ctl->push_lo = lo;
      ctl->push_n = x;
      fin = 2;
    }
    cudaGraphSetConditional(a.h_fin, fin);
  }
  if (cont) {
    const uint32_t xend = __ldcg(&ctl->xcnt), lo = __ldcg(&ctl->xdone);
    const uint32_t x = __ldcg(&ctl->dexpand) ? xend - lo : 0u;
    const bool recorded = __ldcg(&ctl->erec) != 0;
    const uint32_t pull_at = max(kPullMin, a.n / kPullDiv);
    ctl->xdone = xend;
    ctl->pull_check = 0;
    ctl->erec = 0;
    ctl->push_lo = lo;
    ctl->push_n = 0;
    ctl->compact_now = 0;
    ctl->push_items = 0;
    ctl->xcap = 0xFFFFFFFFu;
    const bool x_long = __ldcg(&ctl->x_long) != 0;
    ctl->x_long = 0;
    if (all_items && recorded && x > pull_at) {
      // many first expansions after an iteration that recorded its change flags: the next
      // iteration pulls (tiers 0 and 1 inline, tier-2 rows in a prologue); its own first
      // expansions are listed only while few enough to be pushed
      ctl->pull_check = 1;
      ctl->erec = 1;
      ctl->xcap = pull_at + 1;
      ctl->kind_cur = 7;
      pro = 1;
    } else {
      // otherwise the compacted items of the affected vertices (rebuilt when this
      // iteration swept every item: its joins are not among them), with pushed marks
      // appending their items
      ctl->push_n = x;
      ctl->compact_now = all_items ? 1u : 0u;
      ctl->push_items = all_items ? 0u : 1u;
      ctl->kind_cur = all_items ? 8u : 5u;
      pro = (x || all_items) ? 2u : 0u;
      // a few first expansions after a compacted iteration, none with a long out-row:
      // the light push (no grid barrier) marks them
      if (!all_items && x && x <= kLightPush && !x_long) pro = 3u;
      all = 0;
    }
  }
  cudaGraphSetConditional(a.h_pro, pro);
  cudaGraphSetConditional(a.h_mode, all);
  if (!cont) ctl->status = kStatusDone;
  cudaGraphSetConditional(a.h_loop, cont ? 1u : 0u);
}

// End of an iteration over every vertex that is a launch of its own.
template <bool F32>
__device__ void sweep_decide_every(const SweepArgs<F32> &a, uint32_t it) {
  RankCtl *ctl = a.ctl;
  const unsigned long long dR = __ldcg(&ctl->dR_bits[it]);
  const uint32_t iters = it + 1;
  const bool conv = dR <= a.tol_key;
  const bool cont = !conv && (int)iters < a.max_iter && __ldcg(&ctl->err) == 0;
  ctl->iterations = iters;
  ctl->converged = conv ? 1u : 0u;
  ctl->last_key = dR;
  ctl->it_cur = iters;
  ctl->ticket = 0;
  ctl->launches += 1;
  ctl->t_ns[it + 2] = globaltimer_ns();
  ctl->it_aff[it] = a.n;
  ctl->it_kind[it] = 3;
  ctl->vproc += a.n;
  ctl->eproc += __ldcg(&ctl->m_cur);
  if (!cont) ctl->status = kStatusDone;
  cudaGraphSetConditional(a.h_loop, cont ? 1u : 0u);
}

// One iteration: over every item of a dense Dynamic Frontier call (MODE 1), or over every
// vertex (MODE 0).  The last block to finish decides how the call goes on.
template <bool F32, int MODE>
__global__ void __launch_bounds__(kSweepBlock, 1) k_sweep(const SweepArgs<F32> a) {
  using C = typename Store<F32>::C;
  __shared__ unsigned long long s_key[kSweepWarps];
  __shared__ __align__(8) unsigned long long s_bar;
  __shared__ Rounds s_rounds;
  extern __shared__ __align__(128) unsigned char s_hot[];
  RankCtl *ctl = a.ctl;
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  const uint32_t it = __ldcg(&ctl->it_cur), bar = smem_addr(&s_bar), bytes = a.hot * (uint32_t)sizeof(C);
  Pass<F32> io{};
  io.sbase = smem_addr(s_hot);
  io.r = &s_rounds;
  if (tid == 0) {
    if (bytes) {
      mbar_init1(bar);
      stage_hot(it & 1 ? a.C1 : a.C0, bytes, io.sbase, bar);
    }
    deal_rounds(s_rounds, __ldcg(&ctl->sw_all[0]), __ldcg(&ctl->sw_all[1]), __ldcg(&ctl->sw_all[2]),
                __ldcg(&ctl->sw_off[0]), __ldcg(&ctl->sw_off[1]), a.hot);
  }
  __syncthreads();
  io.it = it;
  io.expand = __ldcg(&ctl->dexpand) != 0;
  io.pulling = __ldcg(&ctl->pull_check) != 0;
  io.erec = __ldcg(&ctl->erec) != 0;
  const uint32_t x0 = __ldcg(&ctl->xdone), xc = __ldcg(&ctl->xcap);
  io.cap_end = xc > 0xFFFFFFFFu - x0 ? 0xFFFFFFFFu : x0 + xc;
  if (!bytes || hot_landed(ctl, bar, 0)) sweep_pass<F32, MODE>(a, io);
  if constexpr (MODE == 0) {
    block_max<F32>(io.my_max, &ctl->dR_bits[it], s_key);
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      if (atomicAdd(&ctl->ticket, 1u) == gridDim.x - 1) {
        __threadfence();
        sweep_decide_every<F32>(a, it);
      }
    }
    return;
  }
  const unsigned long long vs = warp_sum((unsigned long long)io.my_v), es = warp_sum((unsigned long long)io.my_e);
  const uint32_t js = warp_sum(io.jloc);
  if (lane == 0) {
    if (vs) {
      atomicAdd(&ctl->vproc, vs);
      atomicAdd(&ctl->eproc, es);
    }
    if (io.xloc) atomicAdd(&ctl->xcnt, io.xloc);  // the same in every lane
    if (js) atomicAdd(&ctl->tail[it][3], js);
  }
  block_max<F32>(io.my_max, &ctl->dR_bits[it], s_key);
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    const uint32_t t = atomicAdd(&ctl->ticket, 1u);
    if (t == gridDim.x - 1) {
      __threadfence();
      sweep_decide<F32>(a, it, it, true);
    }
  }
}

// A run of iterations in one persistent cooperative launch, one grid barrier apart: all
// iterations of Static and Naive-dynamic (every vertex, from the first to the stop), or
// compacted Dynamic Frontier iterations until the stop or until a vertex expands for the
// first time.  One launch per iteration cost about 20 us beside the sweep itself (conditional
// node, launch, one thread's decision after the last block): 26 us a compacted iteration of
// an R-MAT graph of 16,384 vertices and 136,000 edges, 7.2 us in a run.
template <bool F32>
struct LoopArgs {
  SweepArgs<F32> a;
  // every-vertex runs: sizes and start
  uint32_t n0, n1, n2, m, is_static;
  typename Store<F32>::R init;
};

template <bool F32, bool CMP>
__global__ void __launch_bounds__(kSweepBlock, 1) k_loop(const LoopArgs<F32> p) {
  using S = Store<F32>;
  using R = typename S::R;
  using C = typename S::C;
  __shared__ unsigned long long s_key[kSweepWarps];
  __shared__ __align__(8) unsigned long long s_bar;
  __shared__ uint32_t s_left, s_err;
  __shared__ Rounds s_rounds;
  extern __shared__ __align__(128) unsigned char s_hot[];
  const SweepArgs<F32> &a = p.a;
  RankCtl *ctl = a.ctl;
  const uint32_t tid = threadIdx.x;
  const uint32_t gtid = blockIdx.x * kSweepBlock + tid, nthreads = gridDim.x * kSweepBlock;
  const uint32_t bar = smem_addr(&s_bar), bytes = a.hot * (uint32_t)sizeof(C);
  if (bytes && tid == 0) mbar_init1(bar);
  Pass<F32> io{};
  io.sbase = smem_addr(s_hot);
  io.r = &s_rounds;
  uint32_t it = 0, epoch = 0, it_cap = 0xFFFFFFFFu;  // it_cap: a bounded run ends with the iteration before
  unsigned long long seen[2] = {0, 0};
  // an error ends the device-side loop: nothing else would
  auto give_up = [&]() {
    if (CMP && tid == 0) {
      cudaGraphSetConditional(a.h_pro, 0u);
      cudaGraphSetConditional(a.h_fin, 0u);
      cudaGraphSetConditional(a.h_loop, 0u);
    }
  };
  if constexpr (CMP) {
    it = __ldcg(&ctl->it_cur);
    if (const uint32_t cap = __ldcg(&ctl->run_cap)) it_cap = it + cap;
    if (tid == 0)
      deal_rounds(s_rounds, __ldcg(&ctl->cmp_cur[0]), __ldcg(&ctl->cmp_cur[1]), __ldcg(&ctl->cmp_cur[2]),
                  __ldcg(&ctl->sw_off[0]), __ldcg(&ctl->sw_off[1]), a.hot);
    io.expand = __ldcg(&ctl->dexpand) != 0;
  } else {
    if (gtid == 0 && ctl->t_ns[0] == 0) ctl->t_ns[0] = globaltimer_ns();  // unless a marking launch ran first
    if (tid == 0) deal_rounds(s_rounds, p.n0, p.n1, p.n2, p.n0, p.n0 + p.n1, a.hot);
    if (p.is_static) {  // ranks restart at 1/n, in both parities
      for (uint32_t v = gtid; v < a.n; v += nthreads) {
        const C c = S::contrib(p.init, __ldg(a.adeg + v));
        a.R0[v] = p.init;
        a.R1[v] = p.init;
        a.C0[v] = c;
        a.C1[v] = c;
      }
      if (!run_tally(ctl, epoch, &s_err, &s_left, false, false, seen)) return;
    }
    if (gtid == 0) {
      ctl->t_ns[1] = globaltimer_ns();
      ctl->status = kStatusDone;
    }
    if (a.max_iter <= 0) return;
  }
  const uint32_t it_first = it;
  __syncthreads();  // the rounds are set, the block's mbarrier initialised
  for (;; it++) {
    if (bytes && tid == 0) stage_hot(it & 1 ? a.C1 : a.C0, bytes, io.sbase, bar);
    io.it = it;
    if (!bytes || hot_landed(ctl, bar, (it - it_first) & 1u)) sweep_pass<F32, CMP ? 2 : 0>(a, io);
    // (a block barrier: every warp has taken its last round)
    const unsigned long long key = block_max<F32>(io.my_max, &ctl->dR_bits[it], s_key);
    bool grew = false;
    if (tid == 0) {
      grew = CMP && s_rounds.grew;
      s_rounds.next[0] = s_rounds.next[1] = s_rounds.next[2] = s_rounds.grew = 0;
    }
    if (!run_tally(ctl, epoch, &s_err, &s_left, key > a.tol_key, grew, seen)) {
      give_up();
      return;
    }
    if (gtid == 0) {
      ctl->t_ns[it + 2] = globaltimer_ns();
      if (!CMP) {
        ctl->it_aff[it] = a.n;
        ctl->it_kind[it] = 3;
      }
    }
    if (s_left != 1u || (int)it + 1 >= a.max_iter || it + 1 >= it_cap) break;  // (nothing above the tolerance, or first expansions)
  }
  if constexpr (CMP) {
    if (tid == 0) {
      __threadfence();
      if (atomicAdd(&ctl->ticket, 1u) == gridDim.x - 1) {
        __threadfence();
        sweep_decide<F32>(a, it_first, it, false);
      }
    }
  } else {
    // both parities take the final values
    const uint32_t k = it + 1;
    const bool fp = k & 1;
    const R *Rf = fp ? a.R1 : a.R0;
    const C *Cf = fp ? a.C1 : a.C0;
    R *Ro = fp ? a.R0 : a.R1;
    C *Co = fp ? a.C0 : a.C1;
    for (uint32_t v = gtid; v < a.n; v += nthreads) {
      Ro[v] = ldcg(Rf + v);
      Co[v] = ldcg(Cf + v);
    }
    if (gtid == 0) {
      ctl->iterations = k;
      const unsigned long long dR = __ldcg(&ctl->dR_bits[it]);
      ctl->converged = dR <= a.tol_key ? 1u : 0u;
      ctl->last_key = dR;
      ctl->vproc += (unsigned long long)k * a.n;
      ctl->eproc += (unsigned long long)k * p.m;
    }
  }
}

// Handles tuned with df_split = 0 keep one launch per iteration for Static and Naive-dynamic
// (k_sweep<F32, 0> between these two).  Before the first iteration: Static starts from 1/n (both parities); the
// per-call sizes go to the control block, and the loop runs if max_iter > 0.
template <bool F32>
struct FullInit {
  using S = Store<F32>;
  typename S::R *R0, *R1;
  typename S::C *C0, *C1;
  const typename S::A *adeg;
  RankCtl *ctl;
  typename S::R init;
  uint32_t n, m, is_static;
  uint32_t sw_all[3], sw_off[2];
  int max_iter;
  cudaGraphConditionalHandle h_loop;
};

template <bool F32>
__global__ void k_full_init(const FullInit<F32> p) {
  using S = Store<F32>;
  const uint32_t nthreads = gridDim.x * blockDim.x, gtid = blockIdx.x * blockDim.x + threadIdx.x;
  if (gtid == 0 && p.ctl->t_ns[0] == 0) p.ctl->t_ns[0] = globaltimer_ns();  // unless a marking launch ran first
  if (p.is_static) {
    for (uint32_t v = gtid; v < p.n; v += nthreads) {
      const typename S::C c = S::contrib(p.init, __ldg(p.adeg + v));
      p.R0[v] = p.init;
      p.R1[v] = p.init;
      p.C0[v] = c;
      p.C1[v] = c;
    }
  }
  if (gtid == 0) {
    RankCtl *ctl = p.ctl;
    ctl->it_cur = 0;
    ctl->ticket = 0;
    for (int t = 0; t < 3; t++) ctl->sw_all[t] = p.sw_all[t];
    ctl->sw_off[0] = p.sw_off[0];
    ctl->sw_off[1] = p.sw_off[1];
    ctl->m_cur = p.m;
    ctl->status = kStatusDone;
    ctl->t_ns[1] = globaltimer_ns();
    cudaGraphSetConditional(p.h_loop, p.max_iter > 0 ? 1u : 0u);
  }
}

// After the last full-sweep iteration: both parities take the final values.
template <bool F32>
__global__ void k_full_finish(typename Store<F32>::R *R0, typename Store<F32>::R *R1, typename Store<F32>::C *C0,
                              typename Store<F32>::C *C1, uint32_t n, const RankCtl *ctl) {
  const uint32_t k = __ldcg(&ctl->iterations);
  if (k == 0) return;
  const bool fp = k & 1;
  const typename Store<F32>::R *Rf = fp ? R1 : R0;
  const typename Store<F32>::C *Cf = fp ? C1 : C0;
  typename Store<F32>::R *Ro = fp ? R0 : R1;
  typename Store<F32>::C *Co = fp ? C0 : C1;
  const uint32_t nthreads = gridDim.x * blockDim.x;
  for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += nthreads) {
    Ro[v] = Rf[v];
    Co[v] = Cf[v];
  }
}

// Before the first dense iteration of a Dynamic Frontier (or Traversal) call: the marking
// launch left the list lengths (save_cnt, including the marks that join at next_it) and
// the iteration.  The first iteration sweeps every item with the stamp check (the marks
// for it are in place), so it needs no prologue; Dynamic Traversal records no changes and
// compacts its fixed set before the second.
struct DenseInit {
  RankCtl *ctl;
  uint32_t sw_all[3], sw_off[2];
  uint32_t n, m;
  uint32_t traversal;
  uint32_t run_cap;
  int max_iter;
  cudaGraphConditionalHandle h_loop, h_pro, h_mode, h_fin;
};

__global__ void k_dense_init(const DenseInit p) {
  RankCtl *ctl = p.ctl;
  const uint32_t it0 = ctl->next_it;
  // per-iteration slots from it0 on start empty (a traversal's search used them for its
  // rounds; the marking launch's last marks are in save_cnt)
  for (uint32_t k = it0 + threadIdx.x; k < (uint32_t)kMaxIterLimit + 1; k += blockDim.x) {
    for (int t = 0; t < 4; t++) {
      ctl->tail[k][t] = 0;
      ctl->cmp[k][t] = 0;
    }
    ctl->hubq[k] = 0;
  }
  if (threadIdx.x == 0) {
    ctl->tail[kMaxIterLimit + 1][0] = ctl->tail[kMaxIterLimit + 1][1] = ctl->tail[kMaxIterLimit + 1][2] = 0;
    ctl->hubq[kMaxIterLimit + 1] = 0;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  ctl->it_cur = it0;
  ctl->ticket = 0;
  ctl->bar = 0;
  ctl->tally[0] = ctl->tally[1] = 0;
  for (int t = 0; t < 3; t++) {
    ctl->sw_all[t] = p.sw_all[t];
    ctl->dcnt[t] = ctl->save_cnt[t];
    ctl->final_cnt[t] = ctl->save_cnt[t];
    ctl->cmp_cur[t] = 0;
  }
  ctl->sw_off[0] = p.sw_off[0];
  ctl->sw_off[1] = p.sw_off[1];
  ctl->m_cur = p.m;
  ctl->run_cap = p.run_cap;
  ctl->xdone = ctl->xcnt;
  ctl->xcap = max(kPullMin, p.n / kPullDiv) + 1;  // first iteration: a pull may follow
  ctl->x_long = 0;
  ctl->jtotal = 0;
  ctl->eprev = ctl->eproc;
  ctl->dense_ran = 1;
  ctl->aff_total = 0;
  ctl->cmp_total = 0;
  ctl->app_since = 0;
  ctl->push_n = 0;  // pull_check: set by a marking launch that deferred its marks to a pull
  ctl->push_items = 0;
  ctl->compact_now = 0;
  ctl->dexpand = p.traversal ? 0u : 1u;
  ctl->erec = p.traversal ? 0u : 1u;
  ctl->kind_cur = ctl->pull_check ? 7u : 6u;
  ctl->status = kStatusDone;
  cudaGraphSetConditional(p.h_pro, 0u);
  cudaGraphSetConditional(p.h_mode, 1u);
  if (ctl->fin_only) {
    // the marking launch ran the last iteration (recording its change flags): only its
    // marks remain, by a pull over every tier
    ctl->pull_all = 1;
    cudaGraphSetConditional(p.h_fin, 1u);
    cudaGraphSetConditional(p.h_loop, 0u);
  } else {
    ctl->iterations = it0;
    cudaGraphSetConditional(p.h_fin, 0u);
    cudaGraphSetConditional(p.h_loop, (int)it0 < p.max_iter ? 1u : 0u);
  }
}

// Prologue of a pull iteration: tier-2 rows decide their joins before the sweep.
// After the last iteration (pull_all) tier-0/1 rows pull here too, as the sweep would have.
template <bool F32>
__global__ void __launch_bounds__(kRankBlock) k_df_pull(const RankArgs<F32> a) {
  RankCtl *ctl = a.ctl;
  const uint32_t it = ldcg_u32(&ctl->it_cur);
  const uint32_t cnt0 = ldcg_u32(&ctl->dcnt[0]);
  uint32_t joined = pull_tier2(a, it, cnt0, ldcg_u32(&ctl->sw_all[2]), ldcg_u32(&ctl->sw_off[1]));
  if (ldcg_u32(&ctl->pull_all)) {
    // tier 0 and 1 rows (items before the tier-2 chunks), one thread per row
    const uint8_t *E = a.emap + (size_t)((it - 1) & 1) * a.n;
    const uint32_t n01 = ldcg_u32(&ctl->sw_off[1]), lane = threadIdx.x & 31;
    const uint32_t nthreads = gridDim.x * blockDim.x;
    for (uint32_t b0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; b0 < n01; b0 += nthreads) {
      const uint32_t i = b0 + lane;
      bool join = false;
      uint32_t v = 0;
      if (i < n01) {
        const uint4 item = __ldg(a.items + i);
        v = item.x;
        if (item.z > 1 && ldcg(a.stamp + v) == kNoStamp)
          for (uint32_t j = 0; j < item.z && !join; j++) join = __ldcg(E + __ldg(a.in_col + item.y + j)) != 0;
      }
      joined += pull_join(a, join, v, it, cnt0, lane);
    }
  }
  const unsigned long long s0 = warp_sum((unsigned long long)joined);
  if ((threadIdx.x & 31) == 0 && s0) atomicAdd(&ctl->appended, s0);
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&ctl->launches, 1u);
}

// Prologue of a push iteration (cooperative): the out-rows of the previous iteration's
// first expansions are marked from (the marking launch's code; long rows by the whole grid
// after a barrier), newly marked vertices appending their items to the compacted items
// when the iteration sweeps those; then, if asked or if the set grew by more than 1/16
// since, the compacted items are rebuilt from the stamps, each item's cache bit taken from
// the expanded bitmap.
template <bool F32>
__global__ void __launch_bounds__(kRankBlock, 2) k_df_push(const RankArgs<F32> a) {
  __shared__ uint32_t s_err;
  __shared__ uint32_t s_mbuf[kWarps][4 * kMarkBuf];
  RankCtl *ctl = a.ctl;
  const uint32_t tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
  const uint32_t nthreads = gridDim.x * kRankBlock, gtid = blockIdx.x * kRankBlock + tid;
  const uint32_t nwarps = nthreads >> 5, gwarp = gtid >> 5;
  const uint32_t it = ldcg_u32(&ctl->it_cur);
  uint32_t epoch = 0;
  if (blockIdx.x == 0 && tid == 0) atomicAdd(&ctl->launches, 1u);
  uint32_t cnt[3];
#pragma unroll
  for (int b = 0; b < 3; b++) cnt[b] = ldcg_u32(&ctl->dcnt[b]);
  unsigned long long app = 0, xv = 0, xe = 0;
  bool compact = ldcg_u32(&ctl->compact_now) != 0;
  const bool items = ldcg_u32(&ctl->push_items) != 0;
  const uint32_t pn = ldcg_u32(&ctl->push_n);
  if (pn) {
    const uint32_t lo = ldcg_u32(&ctl->push_lo);
    WarpBuf wb{s_mbuf[wib], {0u, 0u, 0u, 0u}, false, it, items && !compact};
    const uint32_t per = warp_share(pn, nwarps);
    for (uint32_t k0 = (wib * gridDim.x + blockIdx.x) * per; k0 < pn; k0 += nwarps * per) {
      const bool p = lane < per && k0 + lane < pn;
      const uint32_t x = p ? ldcg_u32(a.xlist + lo + k0 + lane) : 0u;
      const ExpandOut o = expand_lanes(a, p ? 1 : 0, x, it, cnt[0], cnt[1], cnt[2], &wb);
      app += o.app;
      xv += o.xv;
      xe += o.xe;
    }
    flush_marks(a, it, cnt, lane, wb);
    if (!grid_sync(ctl, epoch, &s_err)) return;
    if (__ldcg(&ctl->hubq[it]) != 0) {
      app += hub_pass(a, it, cnt, lane, gwarp, nwarps, wb);
      flush_marks(a, it, cnt, lane, wb);
      if (!grid_sync(ctl, epoch, &s_err)) return;
    }
    if (items && !compact && ldcg_u32(&ctl->app_since) > ldcg_u32(&ctl->cmp_total) / 16) compact = true;
  }
  if (compact) {
    // keep the items of vertices stamped <= it, one pass: a block takes rounds of 2048
    // items (eight per thread, each a coalesced warp-wide load), counts the kept ones per
    // (load, warp), reserves their places with one atomic per round and writes them in the
    // round's item order (rounds land in the order of their atomics); the stamp also sets
    // each tier-0/1 item's cache bit
    __shared__ uint32_t s_cnt[8][kWarps], s_base;
    const uint32_t seg[3][2] = {{0u, ldcg_u32(&ctl->sw_all[0])},
                                {ldcg_u32(&ctl->sw_off[0]), ldcg_u32(&ctl->sw_all[1])},
                                {ldcg_u32(&ctl->sw_off[1]), ldcg_u32(&ctl->sw_all[2])}};
    const uint32_t slot = it + 1;
    // (cmp[slot][3] sums the in-edges of the kept vertices: a chunk item's length is its
    // share of the row)
    auto kept = [&](uint32_t t, uint32_t idx, uint4 &item) -> bool {
      item = __ldg(a.items + seg[t][0] + idx);
      const uint16_t st = ldcg(a.stamp + item.x);
      const bool keep = (st & kStampIt) <= (uint16_t)it;
      if (keep && t < 2)
        item.w = ((st & kStampExp) || (__ldcg(a.xbits + (item.x >> 5)) >> (item.x & 31)) & 1u) ? 1u : 0u;
      return keep;
    };
    constexpr uint32_t kRound = 8 * kRankBlock;
    for (uint32_t t = 0; t < 3; t++) {
      const uint32_t cntt = seg[t][1];
      uint32_t e = 0;
      for (uint32_t r0 = blockIdx.x * kRound; r0 < cntt; r0 += gridDim.x * kRound) {
        uint4 item[8];
        uint32_t keepm = 0;
#pragma unroll
        for (uint32_t j = 0; j < 8; j++) {
          const uint32_t idx = r0 + j * kRankBlock + tid;
          item[j] = make_uint4(0, 0, 0, 0);
          if (idx < cntt && kept(t, idx, item[j])) {
            keepm |= 1u << j;
            e += t < 2 ? item[j].z : (item[j].z & 0x3FFu);
          }
        }
#pragma unroll
        for (uint32_t j = 0; j < 8; j++) {
          const uint32_t m = __ballot_sync(kFull, (keepm >> j) & 1u);
          if (lane == 0) s_cnt[j][wib] = __popc(m);
        }
        __syncthreads();
        if (tid == 0) {
          uint32_t tot = 0;
          for (int j = 0; j < 8; j++)
            for (int w = 0; w < kWarps; w++) {
              const uint32_t c = s_cnt[j][w];
              s_cnt[j][w] = tot;
              tot += c;
            }
          s_base = tot ? atomicAdd(&ctl->cmp[slot][t], tot) : 0u;
        }
        __syncthreads();
        const uint32_t base = s_base;
#pragma unroll
        for (uint32_t j = 0; j < 8; j++) {
          const bool k = (keepm >> j) & 1u;
          const uint32_t m = __ballot_sync(kFull, k);
          if (k) a.items_cmp[seg[t][0] + base + s_cnt[j][wib] + __popc(m & lanemask_lt())] = item[j];
        }
        __syncthreads();  // s_cnt and s_base are reused by the next round
      }
      e = warp_sum(e);
      if (lane == 0 && e) atomicAdd(&ctl->cmp[slot][3], e);
    }
    if (!grid_sync(ctl, epoch, &s_err)) return;
    if (blockIdx.x == 0 && tid == 0) {
      uint32_t total = 0;
      for (int t = 0; t < 3; t++) {
        ctl->cmp_cur[t] = __ldcg(&ctl->cmp[slot][t]);
        total += cnt[t] + __ldcg(&ctl->tail[it][t]);
      }
      ctl->cmp_total = total + __ldcg(&ctl->jtotal);
      ctl->app_since = 0;
      ctl->cmp_edges = __ldcg(&ctl->cmp[slot][3]);
      ctl->kind_cur = 8;
    }
  }
  const unsigned long long s0 = warp_sum(app), s1 = warp_sum(xv), s2 = warp_sum(xe);
  if (lane == 0) {
    if (s0) atomicAdd(&ctl->appended, s0);
    if (s1) atomicAdd(&ctl->expv, s1);
    if (s2) atomicAdd(&ctl->expe, s2);
  }
}

// Prologue of a compacted iteration after which a few vertices expanded for the first time,
// none of them with an out-row longer than kInlineOut: the warps that read them from the
// expansion list mark their out-rows and append the items of the newly marked vertices,
// with no grid barrier (the hub queue is not needed), so it costs a plain launch instead
// of a cooperative one with barriers.
template <bool F32>
__global__ void __launch_bounds__(kRankBlock, 2) k_df_push_light(const RankArgs<F32> a) {
  __shared__ uint32_t s_mbuf[kWarps][4 * kMarkBuf];
  RankCtl *ctl = a.ctl;
  const uint32_t tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
  const uint32_t nwarps = (gridDim.x * kRankBlock) >> 5;
  const uint32_t it = ldcg_u32(&ctl->it_cur);
  if (blockIdx.x == 0 && tid == 0) atomicAdd(&ctl->launches, 1u);
  uint32_t cnt[3];
#pragma unroll
  for (int b = 0; b < 3; b++) cnt[b] = ldcg_u32(&ctl->dcnt[b]);
  const uint32_t pn = ldcg_u32(&ctl->push_n), lo = ldcg_u32(&ctl->push_lo);
  WarpBuf wb{s_mbuf[wib], {0u, 0u, 0u, 0u}, false, it, true};
  unsigned long long app = 0, xv = 0, xe = 0;
  const uint32_t per = warp_share(pn, nwarps);
  for (uint32_t k0 = (wib * gridDim.x + blockIdx.x) * per; k0 < pn; k0 += nwarps * per) {
    const bool p = lane < per && k0 + lane < pn;
    const uint32_t x = p ? ldcg_u32(a.xlist + lo + k0 + lane) : 0u;
    const ExpandOut o = expand_lanes(a, p ? 1 : 0, x, it, cnt[0], cnt[1], cnt[2], &wb);
    app += o.app;
    xv += o.xv;
    xe += o.xe;
  }
  flush_marks(a, it, cnt, lane, wb);
  const unsigned long long s0 = warp_sum(app), s1 = warp_sum(xv), s2 = warp_sum(xe);
  if (lane == 0) {
    if (s0) atomicAdd(&ctl->appended, s0);
    if (s1) atomicAdd(&ctl->expv, s1);
    if (s2) atomicAdd(&ctl->expe, s2);
  }
}

// Writeback of a dense Dynamic Frontier call: every affected vertex (stamp set) gets its
// final values in both parities (parity iterations & 1), its per-call marks and change
// flags are cleared, and it is listed in list 0 (each block lists its own range of
// vertices after one atomic for its offset), which is then the call's affected set.
template <bool F32>
__global__ void __launch_bounds__(256) k_df_finish(const RankArgs<F32> a) {
  using S = Store<F32>;
  using R = typename S::R;
  using C = typename S::C;
  __shared__ uint32_t s_w[8], s_base;
  RankCtl *ctl = a.ctl;
  const uint32_t tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
  const bool fp = __ldcg(&ctl->iterations) & 1;
  const R *Rf = fp ? a.R1 : a.R0;
  const C *Cf = fp ? a.C1 : a.C0;
  R *Ro = fp ? a.R0 : a.R1;
  C *Co = fp ? a.C0 : a.C1;
  const uint32_t per = ((a.n + gridDim.x - 1) / gridDim.x + 255) & ~255u;
  const uint32_t lo = min(a.n, blockIdx.x * per), hi = min(a.n, lo + per);
  uint32_t c = 0;
  for (uint32_t v = lo + tid; v < hi; v += 256) c += ldcg(a.stamp + v) != kNoStamp ? 1u : 0u;
  c = warp_sum(c);
  if (lane == 0) s_w[wib] = c;
  __syncthreads();
  if (tid == 0) {
    uint32_t t = 0;
    for (int w = 0; w < 8; w++) t += s_w[w];
    s_base = t ? atomicAdd(&ctl->aff_total, t) : 0u;
  }
  __syncthreads();
  uint32_t at = s_base;
  for (uint32_t v0 = lo; v0 < hi; v0 += 256) {
    const uint32_t v = v0 + tid;
    const bool f = v < hi && ldcg(a.stamp + v) != kNoStamp;
    const uint32_t mask = __ballot_sync(kFull, f);
    __syncthreads();  // s_w free again
    if (lane == 0) s_w[wib] = __popc(mask);
    __syncthreads();
    uint32_t before = 0, all = 0;
    for (int w = 0; w < 8; w++) {
      before += w < (int)wib ? s_w[w] : 0u;
      all += s_w[w];
    }
    if (f) {
      a.list0[at + before + __popc(mask & lanemask_lt())] = v;
      Ro[v] = __ldcg(Rf + v);
      Co[v] = __ldcg(Cf + v);
      a.bitmap[v >> 5] = 0u;
      a.xbits[v >> 5] = 0u;
      a.stamp[v] = kNoStamp;
      a.emap[v] = 0;
      a.emap[a.n + v] = 0;
    }
    at += all;
  }
}

// ------------------------------------------------------------------ host side ---

namespace {

struct LoopGraph {
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaGraphNode_t init = nullptr;
  cudaGraphConditionalHandle h_loop = 0, h_pro = 0, h_mode = 0, h_fin = 0;
  std::vector<unsigned char> key;
  void release() {
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    exec = nullptr;
    graph = nullptr;
    init = nullptr;
    key.clear();
  }
};

struct Loops {
  LoopGraph full;      // one launch per iteration (df_split = 0)
  LoopGraph dense[2];  // synchronous, asynchronous (aliased parities)
};

template <class T>
void append_key(std::vector<unsigned char> &k, const T &x) {
  const unsigned char *p = reinterpret_cast<const unsigned char *>(&x);
  k.insert(k.end(), p, p + sizeof(T));
}

#define CKG(call)                                           \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) return cuda_fail(g, e_, #call);  \
  } while (0)

cudaError_t add_kernel(cudaGraphNode_t *node, cudaGraph_t graph, const cudaGraphNode_t *dep, size_t ndep,
                       const void *fn, dim3 grid, dim3 block, void **args, bool coop, size_t smem = 0) {
  cudaKernelNodeParams kp{};
  kp.func = const_cast<void *>(fn);
  kp.gridDim = grid;
  kp.blockDim = block;
  kp.sharedMemBytes = (unsigned)smem;
  kp.kernelParams = args;
  cudaError_t e = cudaGraphAddKernelNode(node, graph, dep, ndep, &kp);
  if (e == cudaSuccess && coop) {
    cudaLaunchAttributeValue v{};
    v.cooperative = 1;
    e = cudaGraphKernelNodeSetAttribute(*node, cudaLaunchAttributeCooperative, &v);
  }
  return e;
}

cudaError_t add_conditional(cudaGraphNode_t *node, cudaGraph_t graph, const cudaGraphNode_t *dep, size_t ndep,
                            cudaGraphConditionalHandle h, cudaGraphConditionalNodeType type, cudaGraph_t *body,
                            unsigned size = 1) {
  cudaGraphNodeParams np{};
  np.type = cudaGraphNodeTypeConditional;
  np.conditional.handle = h;
  np.conditional.type = type;
  np.conditional.size = size;
  cudaError_t e = cudaGraphAddNode(node, graph, dep, nullptr, ndep, &np);
  if (e == cudaSuccess)
    for (unsigned k = 0; k < size; k++) body[k] = np.conditional.phGraph_out[k];
  return e;
}

}  // namespace

// A control-block reset and one cooperative kernel as a CUDA graph: built once per kind of call,
// later calls replace the kernel's arguments and replay.
pr_status graph_replay(Graph *g, int kind, const cudaKernelNodeParams &kp) {
  if (g->cg_exec && g->cg_kind != kind) {
    cudaGraphExecDestroy(g->cg_exec);
    g->cg_exec = nullptr;
  }
  if (!g->cg_exec) {
    if (g->cg) cudaGraphDestroy(g->cg);
    g->cg = nullptr;
    CKG(cudaGraphCreate(&g->cg, 0));
    cudaGraphNode_t reset = nullptr;
    cudaMemsetParams mp{};
    mp.dst = g->ctl;
    mp.value = 0;
    mp.elementSize = 1;
    mp.width = sizeof(RankCtl);
    mp.height = 1;
    mp.pitch = sizeof(RankCtl);
    CKG(cudaGraphAddMemsetNode(&reset, g->cg, nullptr, 0, &mp));
    CKG(add_kernel(&g->cg_kernel, g->cg, &reset, 1, kp.func, kp.gridDim, kp.blockDim, kp.kernelParams, true,
                   kp.sharedMemBytes));
    CKG(cudaGraphInstantiate(&g->cg_exec, g->cg, 0));
    g->cg_kind = kind;
  } else {
    CKG(cudaGraphExecKernelNodeSetParams(g->cg_exec, g->cg_kernel, &kp));
  }
  CKG(cudaGraphLaunch(g->cg_exec, g->st));
  count_launch();
  return PR_OK;
}

namespace {

template <bool F32>
size_t hot_bytes(const SweepArgs<F32> &a) { return (size_t)a.hot * sizeof(typename Store<F32>::C); }

template <bool F32>
pr_status full_impl(Graph *g, bool from_init) {
  LoopArgs<F32> p{};
  p.a = sweep_args<F32>(g, false);
  p.n0 = g->item_cnt[0];
  p.n1 = g->item_cnt[1];
  p.n2 = g->item_cnt[2];
  p.m = (uint32_t)g->m;
  p.is_static = from_init ? 1u : 0u;
  if constexpr (F32) p.init = (float)(1.0 / (double)g->n);
  else p.init = std::llrint(1.0 / (double)g->n * 4611686018427387904.0);
  void *args[] = {(void *)&p};
  if (g->use_graph) {
    cudaKernelNodeParams kp{};
    kp.func = (void *)k_loop<F32, false>;
    kp.gridDim = dim3(g->loop_grid);
    kp.blockDim = dim3(kSweepBlock);
    kp.sharedMemBytes = (unsigned)hot_bytes(p.a);
    kp.kernelParams = args;
    return graph_replay(g, kGraphEvery, kp);
  }
  CKG(cudaLaunchCooperativeKernel((const void *)k_loop<F32, false>, dim3(g->loop_grid), dim3(kSweepBlock), args,
                                  hot_bytes(p.a), g->st));
  count_launch();
  return PR_OK;
}

template <bool F32>
pr_status full_steps_impl(Graph *g, bool from_init) {
  using S = Store<F32>;
  Loops *L = (Loops *)g->loops;
  LoopGraph &lg = L->full;
  SweepArgs<F32> a = sweep_args<F32>(g, false);
  std::vector<unsigned char> key;
  append_key(key, a);
  if (lg.exec && key != lg.key) lg.release();
  FullInit<F32> ip{};
  ip.R0 = (typename S::R *)g->R[0];
  ip.R1 = (typename S::R *)g->R[1];
  ip.C0 = (typename S::C *)g->C[0];
  ip.C1 = (typename S::C *)g->C[1];
  ip.adeg = (const typename S::A *)g->adeg;
  ip.ctl = g->ctl;
  if constexpr (F32) ip.init = (float)(1.0 / (double)g->n);
  else ip.init = std::llrint(1.0 / (double)g->n * 4611686018427387904.0);
  ip.n = g->n;
  ip.m = (uint32_t)g->m;
  ip.is_static = from_init ? 1u : 0u;
  for (int t = 0; t < 3; t++) ip.sw_all[t] = g->item_cnt[t];
  ip.sw_off[0] = g->item_cnt[0];
  ip.sw_off[1] = g->item_cnt[0] + g->item_cnt[1];
  ip.max_iter = g->p.max_iter;
  const dim3 init_grid(std::max(1, g->sm_count * 4)), init_block(256);
  if (!lg.exec) {
    lg.release();  // what a failed call may have left of one
    CKG(cudaGraphCreate(&lg.graph, 0));
    CKG(cudaGraphConditionalHandleCreate(&lg.h_loop, lg.graph, 0, 0));
    ip.h_loop = lg.h_loop;
    a.h_loop = lg.h_loop;
    void *iargs[] = {(void *)&ip};
    CKG(add_kernel(&lg.init, lg.graph, nullptr, 0, (const void *)k_full_init<F32>, init_grid, init_block, iargs, false));
    cudaGraphNode_t wnode = nullptr, snode = nullptr, fnode = nullptr;
    cudaGraph_t body = nullptr;
    CKG(add_conditional(&wnode, lg.graph, &lg.init, 1, lg.h_loop, cudaGraphCondTypeWhile, &body));
    void *sargs[] = {(void *)&a};
    CKG(add_kernel(&snode, body, nullptr, 0, (const void *)k_sweep<F32, 0>, dim3(g->sm_count), dim3(kSweepBlock), sargs,
                   false, hot_bytes(a)));
    typename S::R *R0 = ip.R0, *R1 = ip.R1;
    typename S::C *C0 = ip.C0, *C1 = ip.C1;
    uint32_t n = g->n;
    const RankCtl *ctl = g->ctl;
    void *fargs[] = {(void *)&R0, (void *)&R1, (void *)&C0, (void *)&C1, (void *)&n, (void *)&ctl};
    CKG(add_kernel(&fnode, lg.graph, &wnode, 1, (const void *)k_full_finish<F32>, init_grid, init_block, fargs,
                   false));
    CKG(cudaGraphInstantiate(&lg.exec, lg.graph, 0));
    lg.key = key;
  } else {
    ip.h_loop = lg.h_loop;
    cudaKernelNodeParams kp{};
    void *iargs[] = {(void *)&ip};
    kp.func = (void *)k_full_init<F32>;
    kp.gridDim = init_grid;
    kp.blockDim = init_block;
    kp.kernelParams = iargs;
    CKG(cudaGraphExecKernelNodeSetParams(lg.exec, lg.init, &kp));
  }
  CKG(cudaGraphLaunch(lg.exec, g->st));
  count_launches(2);  // init and writeback; the loop's launches are counted on the device
  return PR_OK;
}

int run_grid(const Graph *g) { return g->bounded_runs && g->m < kShareEdges ? g->share_grid : g->sm_count; }
int push_grid(const Graph *g) { return std::max(1, g->pro_grid * run_grid(g) / g->sm_count); }

template <bool F32>
pr_status dense_impl(Graph *g, RankMode mode, const RankArgs<F32> &ra_in) {
  const bool async = mode == kModeDFAsync;
  Loops *L = (Loops *)g->loops;
  LoopGraph &lg = L->dense[async ? 1 : 0];
  SweepArgs<F32> a = sweep_args<F32>(g, async);
  // the prologue's arguments without the per-call fields it does not read (copied byte for
  // byte: the cache key below compares bytes, padding included, and the caller's
  // value-initialised struct has zero padding)
  RankArgs<F32> ra;
  std::memcpy(&ra, &ra_in, sizeof ra);
  ra.it_c0 = ra.it_c1 = ra.it_c2 = 0;
  ra.n_pend_src = ra.n_pend_tgt = 0;
  ra.pend_src = ra.pend_tgt = nullptr;
  ra.n_dead = 0;
  ra.D_ref_n = 0;
  ra.D_ref_d = 0.0;
  ra.mode = 0;
  ra.start_full = 0;
  ra.split = 0;
  ra.defer_at = 0;  // depends on the edge count, which changes with every batch
  std::vector<unsigned char> key;
  append_key(key, a);
  append_key(key, ra);
  append_key(key, run_grid(g));
  if (lg.exec && key != lg.key) lg.release();
  DenseInit ip{};
  ip.ctl = g->ctl;
  for (int t = 0; t < 3; t++) ip.sw_all[t] = g->item_cnt[t];
  ip.sw_off[0] = g->item_cnt[0];
  ip.sw_off[1] = g->item_cnt[0] + g->item_cnt[1];
  ip.traversal = mode == kModeDT ? 1u : 0u;
  if (g->bounded_runs) ip.run_cap = (uint32_t)std::max<uint64_t>(1, kRunEdges / std::max<uint64_t>(1, g->m));
  ip.max_iter = g->p.max_iter;
  ip.n = g->n;
  ip.m = (uint32_t)g->m;
  if (!lg.exec) {
    lg.release();  // what a failed call may have left of one
    CKG(cudaGraphCreate(&lg.graph, 0));
    CKG(cudaGraphConditionalHandleCreate(&lg.h_loop, lg.graph, 0, 0));
    CKG(cudaGraphConditionalHandleCreate(&lg.h_fin, lg.graph, 0, 0));
    ip.h_fin = lg.h_fin;
    a.h_fin = lg.h_fin;
    cudaGraphNode_t wnode = nullptr, inode = nullptr, pnode = nullptr, fnode = nullptr;
    cudaGraph_t body = nullptr;
    ip.h_loop = lg.h_loop;
    // the WHILE node and its body first: the prologue's handle belongs to the body, and the
    // init node (added after it, then made its predecessor) sets it
    CKG(add_conditional(&wnode, lg.graph, nullptr, 0, lg.h_loop, cudaGraphCondTypeWhile, &body));
    CKG(cudaGraphConditionalHandleCreate(&lg.h_pro, body, 0, 0));
    CKG(cudaGraphConditionalHandleCreate(&lg.h_mode, body, 1, 0));
    ip.h_pro = lg.h_pro;
    ip.h_mode = lg.h_mode;
    a.h_loop = lg.h_loop;
    a.h_pro = lg.h_pro;
    a.h_mode = lg.h_mode;
    // SWITCH on the prologue: 0 = none, 1 = tier-2 pull, 2 = push (and compaction), 3 = light push
    cudaGraph_t pb[4] = {nullptr, nullptr, nullptr, nullptr};
    CKG(add_conditional(&inode, body, nullptr, 0, lg.h_pro, cudaGraphCondTypeSwitch, pb, 4));
    cudaGraphNode_t enode = nullptr, pull_node = nullptr;
    CKG(cudaGraphAddEmptyNode(&enode, pb[0], nullptr, 0));
    void *pargs[] = {(void *)&ra};
    CKG(add_kernel(&pull_node, pb[1], nullptr, 0, (const void *)k_df_pull<F32>, dim3(std::max(1, g->sm_count * 8)),
                   dim3(kRankBlock), pargs, false));
    CKG(add_kernel(&pnode, pb[2], nullptr, 0, (const void *)k_df_push<F32>, dim3(push_grid(g)), dim3(kRankBlock), pargs,
                   true));
    cudaGraphNode_t lnode = nullptr;
    CKG(add_kernel(&lnode, pb[3], nullptr, 0, (const void *)k_df_push_light<F32>, dim3(std::max(1, g->sm_count)),
                   dim3(kRankBlock), pargs, false));
    // SWITCH on what follows: 0 = a run of compacted iterations, 1 = one iteration over every item
    cudaGraph_t sw[2] = {nullptr, nullptr};
    cudaGraphNode_t swnode = nullptr, s0 = nullptr, s1 = nullptr;
    CKG(add_conditional(&swnode, body, &inode, 1, lg.h_mode, cudaGraphCondTypeSwitch, sw, 2));
    LoopArgs<F32> la{};
    la.a = a;
    void *largs[] = {(void *)&la};
    CKG(add_kernel(&s0, sw[0], nullptr, 0, (const void *)k_loop<F32, true>, dim3(run_grid(g)), dim3(kSweepBlock), largs,
                   true, hot_bytes(a)));
    void *sargs[] = {(void *)&a};
    CKG(add_kernel(&s1, sw[1], nullptr, 0, (const void *)k_sweep<F32, 1>, dim3(g->sm_count),
                   dim3(kSweepBlock), sargs, false, hot_bytes(a)));
    void *iargs[] = {(void *)&ip};
    CKG(add_kernel(&lg.init, lg.graph, nullptr, 0, (const void *)k_dense_init, dim3(1), dim3(32), iargs, false));
    cudaGraphEdgeData ed{};
    CKG(cudaGraphAddDependencies(lg.graph, &lg.init, &wnode, &ed, 1));
    // the marks of the last iteration: 0 = none, 1 = pull over every tier, 2 = push
    cudaGraph_t fb[3] = {nullptr, nullptr, nullptr};
    cudaGraphNode_t fsw = nullptr, fe = nullptr, fpull = nullptr, fpush = nullptr;
    CKG(add_conditional(&fsw, lg.graph, &wnode, 1, lg.h_fin, cudaGraphCondTypeSwitch, fb, 3));
    CKG(cudaGraphAddEmptyNode(&fe, fb[0], nullptr, 0));
    CKG(add_kernel(&fpull, fb[1], nullptr, 0, (const void *)k_df_pull<F32>, dim3(std::max(1, g->sm_count * 8)),
                   dim3(kRankBlock), pargs, false));
    CKG(add_kernel(&fpush, fb[2], nullptr, 0, (const void *)k_df_push<F32>, dim3(push_grid(g)), dim3(kRankBlock),
                   pargs, true));
    void *fargs[] = {(void *)&ra};
    CKG(add_kernel(&fnode, lg.graph, &fsw, 1, (const void *)k_df_finish<F32>, dim3(std::max(1, g->sm_count * 4)),
                   dim3(256), fargs, false));
    CKG(cudaGraphInstantiate(&lg.exec, lg.graph, 0));
    lg.key = key;
  } else {
    ip.h_loop = lg.h_loop;
    ip.h_pro = lg.h_pro;
    ip.h_mode = lg.h_mode;
    ip.h_fin = lg.h_fin;
    cudaKernelNodeParams kp{};
    void *iargs[] = {(void *)&ip};
    kp.func = (void *)k_dense_init;
    kp.gridDim = dim3(1);
    kp.blockDim = dim3(32);
    kp.kernelParams = iargs;
    CKG(cudaGraphExecKernelNodeSetParams(lg.exec, lg.init, &kp));
  }
  CKG(cudaGraphLaunch(lg.exec, g->st));
  count_launches(2);  // init and writeback; the loop's launches are counted on the device
  return PR_OK;
}

}  // namespace

// (a batched handle's copies are widened to 16-byte pieces at both ends)
uint32_t hot_limit(bool f32) { return kHotBytes / (f32 ? 4 : 8) - 8; }

pr_status sweep_setup(Graph *g) {
  const void *fns[4] = {g->f32 ? (const void *)k_loop<true, false> : (const void *)k_loop<false, false>,
                        g->f32 ? (const void *)k_loop<true, true> : (const void *)k_loop<false, true>,
                        g->f32 ? (const void *)k_sweep<true, 1> : (const void *)k_sweep<false, 1>,
                        g->f32 ? (const void *)k_sweep<true, 0> : (const void *)k_sweep<false, 0>};
  for (const void *fn : fns) CKG(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHotBytes));
  g->loop_grid = g->share_grid = g->sm_count;
  int per_sm_pro = 0;
  CKG(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &per_sm_pro, g->f32 ? (const void *)k_df_push<true> : (const void *)k_df_push<false>, kRankBlock, 0));
  g->pro_grid = std::max(1, std::min(per_sm_pro, 4)) * g->sm_count;
  if (!g->loops) g->loops = new Loops();
  return PR_OK;
}

void sweep_share(Graph *g, int slots) {
  g->loop_grid = std::max(1, g->sm_count / slots);
  g->share_grid = std::max(1, g->sm_count / std::min(slots, 2));
  g->bounded_runs = slots > 1;
}

bool sweep_eligible(const Graph *g, bool marking) {
  return g->ncomp == 1 && !g->teleport && g->loops != nullptr && (!g->use_graph || (!marking && g->split_df));
}

pr_status sweep_full(Graph *g, bool from_init) {
  if (!g->split_df) return g->f32 ? full_steps_impl<true>(g, from_init) : full_steps_impl<false>(g, from_init);
  return g->f32 ? full_impl<true>(g, from_init) : full_impl<false>(g, from_init);
}

pr_status sweep_dense(Graph *g, RankMode mode, const void *rank_args) {
  return g->f32 ? dense_impl<true>(g, mode, *(const RankArgs<true> *)rank_args)
                : dense_impl<false>(g, mode, *(const RankArgs<false> *)rank_args);
}

void sweep_free(Graph *g) {
  Loops *L = (Loops *)g->loops;
  if (L) {
    L->full.release();
    L->dense[0].release();
    L->dense[1].release();
    delete L;
    g->loops = nullptr;
  }
}

}  // namespace prdf
