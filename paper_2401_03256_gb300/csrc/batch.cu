// batch.cu - the iterations of a batched handle (many independent graphs) in one persistent
// cooperative launch.
//
// Static and Naive-dynamic calls run here from the first iteration; a Dynamic Frontier or
// Dynamic Traversal call after the marking launch (k_rank: initial marking, the search, and
// iterations while the affected set is small) has handed over.  Each graph iterates as it
// would alone: its own (1 - alpha)/n, L-inf test and iteration count; a graph that has
// stopped is left out of the following iterations.
//
// What bounds it: random gathers, as for one graph (sweep_dev.cuh), but the contributions of
// one of these graphs mostly fit an SM's shared memory.  So the work is dealt by graph: the
// rounds of all graphs still iterating, laid end to end and weighted, are cut into one equal
// run per block, and a block sweeps its run one graph at a time, first copying that
// graph's hot contributions (all of them up to 32 K vertices in FP32, 16 K in 64-bit mode;
// the vertices of largest out-degree of a larger graph) to shared memory.  The cut is
// renewed when graphs stop.
//
// Affected sets grow by pulls alone: an iteration records change flags per vertex, and where
// it met first expansions in a graph, the graph's vertices not yet affected test their
// in-neighbours' flags in the next one (rows of more than group_max in-edges before the
// sweep, a grid barrier apart, because several blocks sweep their chunks).  A graph that
// stops with first expansions still makes those marks (Algorithm 1 marks in its last iteration too).
//
// 256 R-MAT graphs of scales 10 to 18 (14.8 M vertices, 128 M edges), FP32, Dynamic
// Frontier: 36 ms a call (93 iterations of 0.53 ms while all graphs iterate); in the general
// persistent kernel (k_rank, df_split 0) 70 ms (0.94 ms, and a recompaction of all items
// whenever a graph stopped).  An iteration moves about 1.5 GB, 42% of the HBM rate: without any gather
// it still takes 60% of the time, so it waits on the loads of the short rows, one behind
// another (item, row, columns) with 32 warps a SM.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sweep_dev.cuh"

namespace prdf {

namespace {

constexpr uint8_t kDead = 0, kLive = 1, kLastMarks = 2;
// Work of a round of each tier, in gathers: 32 rows of a few entries, 4 rows of 9 to 64, a chunk
// of up to 512 (130 on average on R-MAT graphs).
__device__ __forceinline__ uint32_t round_work(int t) { return t < 2 ? 100u : 130u; }

template <bool F32>
struct BatchArgs {
  using S = Store<F32>;
  SweepArgs<F32> a;
  uint32_t nc;
  const uint16_t *comp;          // graph of each vertex
  const uint32_t *first;         // [nc + 1] first vertex of each graph
  const uint32_t *hot;           // [nc] vertices from first on whose contributions are copied
  const uint32_t *item_first;    // [3][nc + 1] first sweep item of each graph, by tier
  const typename S::R *base, *init;  // [nc] (1 - alpha) / n_c, 1 / n_c
  unsigned long long *dRc;       // [3][nc] L-inf keys by iteration modulo 3
  uint32_t *xc;                  // [3][nc] first expansions by iteration modulo 3
  uint32_t *comp_out;            // [nc][4] iterations, converged, affected
  unsigned long long *comp_last; // [nc] last L-inf key
  uint32_t marking;              // after a marking launch; 0: every vertex from iteration 0
  uint32_t traversal;            // Dynamic Traversal: nothing is marked any more
  uint32_t is_static;
};

size_t state_bytes(uint32_t nc) { return 16 + 8ull * (nc + 1) + 12ull * (nc + 1) + 4ull * nc + 64; }

template <bool F32>
__global__ void __launch_bounds__(kSweepBlock, 1) k_batch(const BatchArgs<F32> p) {
  using S = Store<F32>;
  using R = typename S::R;
  using C = typename S::C;
  constexpr uint32_t kAlign = 16 / sizeof(C);  // entries of a 16-byte piece
  __shared__ unsigned long long s_key[kSweepWarps];
  __shared__ __align__(8) unsigned long long s_bar;
  __shared__ uint32_t s_err, s_cnt[kSweepWarps], s_at;
  __shared__ Rounds s_rounds;
  extern __shared__ __align__(128) unsigned char s_dyn[];
  const SweepArgs<F32> &a = p.a;
  RankCtl *ctl = a.ctl;
  const uint32_t nc = p.nc, tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
  const uint32_t gtid = blockIdx.x * kSweepBlock + tid, nthreads = gridDim.x * kSweepBlock;
  unsigned long long *s_pref = reinterpret_cast<unsigned long long *>(s_dyn + kHotBytes + 16);  // [nc + 1] work before a graph
  uint32_t *s_item = reinterpret_cast<uint32_t *>(s_pref + nc + 1);                        // [3][nc + 1]
  uint16_t *s_iters = reinterpret_cast<uint16_t *>(s_item + 3 * (nc + 1));                 // [nc]
  uint8_t *s_state = reinterpret_cast<uint8_t *>(s_iters + nc), *s_pull = s_state + nc;    // [nc] each
  const uint32_t bar = smem_addr(&s_bar);
  uint32_t epoch = 0;

  uint32_t it = 0;
  bool every = !p.marking, pre_pulled = false;
  if (p.marking) {
    const uint32_t status = __ldcg(&ctl->status);
    if (__ldcg(&ctl->err) || status == kStatusDone) return;  // the marking launch finished the call
    every = status == kStatusFull;                           // a search that reached its depth limit
    if (!every) {
      it = __ldcg(&ctl->next_it);
      pre_pulled = __ldcg(&ctl->pull_check) != 0;  // its last iteration left its marks to a pull (long rows done)
    }
  } else if (gtid == 0) {
    ctl->t_ns[0] = globaltimer_ns();
  }
  const bool expand = p.marking && !every && !p.traversal;
  if (tid == 0) mbar_init1(bar);
  for (uint32_t k = tid; k < 3 * (nc + 1); k += kSweepBlock) s_item[k] = p.item_first[k];
  for (uint32_t c = tid; c < nc; c += kSweepBlock) {
    const uint32_t k = every ? 0u : __ldcg(&p.comp_out[4 * c]);  // iterations of a graph that stopped before
    s_iters[c] = (uint16_t)k;
    s_state[c] = k == 0 ? kLive : (pre_pulled && k == it ? kLastMarks : kDead);
    s_pull[c] = pre_pulled ? 1 : 0;
  }
  if (blockIdx.x == 0)  // a marking launch left its own iterations' values in the other slots
    for (uint32_t c = tid; c < nc; c += kSweepBlock) p.dRc[(uint64_t)((it + 1) % 3) * nc + c] = 0;
  if (p.is_static) {
    for (uint32_t v = gtid; v < a.n; v += nthreads) {
      const R r = p.init[__ldg(p.comp + v)];
      const C c = S::contrib(r, __ldg(a.adeg + v));
      a.R0[v] = r;
      a.R1[v] = r;
      a.C0[v] = c;
      a.C1[v] = c;
    }
    if (!run_barrier(ctl, epoch, &s_err)) return;
  }
  if (gtid == 0 && !p.marking) ctl->t_ns[1] = globaltimer_ns();

  // s_pref from the states (called by the whole block after they changed): 1024 graphs at most,
  // one per thread
  auto cut = [&]() {
    __syncthreads();
    unsigned long long w = 0;
    if (tid < nc && s_state[tid] != kDead) {
      for (int t = 0; t < 3; t++) {
        const uint32_t k = s_item[t * (nc + 1) + tid + 1] - s_item[t * (nc + 1) + tid];
        w += (unsigned long long)round_work(t) * (t == 0 ? (k + 31) / 32 : t == 1 ? (k + 3) / 4 : k);
      }
    }
    unsigned long long incl = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(kFull, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    if (lane == 31) s_key[wib] = incl;
    __syncthreads();
    for (uint32_t k = 0; k < wib; k++) incl += s_key[k];
    if (tid < nc) s_pref[tid + 1] = incl;
    if (tid == 0) s_pref[0] = 0;
    __syncthreads();
  };
  // f(c, a0, a1, w) for every graph of this block's run: its work from a0 to a1 of w
  auto segments = [&](auto &&f) {
    const unsigned long long total = s_pref[nc];
    const unsigned long long x0 = total * blockIdx.x / gridDim.x, x1 = total * (blockIdx.x + 1) / gridDim.x;
    uint32_t lo = 0, hi = nc;  // last c with s_pref[c] <= x0
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (s_pref[mid] <= x0) lo = mid; else hi = mid;
    }
    for (uint32_t c = lo; c < nc && s_pref[c] < x1; c++) {
      const unsigned long long b = s_pref[c], w = s_pref[c + 1] - b;
      if (w == 0 || b + w <= x0) continue;
      f(c, x0 > b ? x0 - b : 0ull, (x1 < b + w ? x1 : b + w) - b, w);
    }
  };
  // thread 0: the rounds of graph c's work a0 .. a1 of w
  auto set_rounds = [&](uint32_t c, unsigned long long a0, unsigned long long a1, unsigned long long w) {
    for (int t = 0; t < 3; t++) {
      const uint32_t b = s_item[t * (nc + 1) + c], k = s_item[t * (nc + 1) + c + 1] - b;
      const uint32_t r = t == 0 ? (k + 31) / 32 : t == 1 ? (k + 3) / 4 : k;
      s_rounds.base[t] = b;
      s_rounds.items[t] = k;
      s_rounds.first[t] = (uint32_t)(r * a0 / w);
      s_rounds.rounds[t] = (uint32_t)(r * a1 / w);
      s_rounds.next[t] = 0;
    }
    s_rounds.stride = 1;
    // the copied vertices, widened to 16-byte pieces of the contribution array
    const uint32_t f = p.first[c], lo = f & ~(kAlign - 1);
    const uint32_t end = min((f + p.hot[c] + kAlign - 1) & ~(kAlign - 1), a.n & ~(kAlign - 1));
    s_rounds.hfirst = lo;
    s_rounds.hot = end > lo && p.hot[c] ? end - lo : 0u;
  };

  unsigned long long tot_v = 0, tot_e = 0;
  uint32_t phase = 0, joined = 0;
  Pass<F32> io{};
  io.sbase = smem_addr(s_dyn);
  io.r = &s_rounds;
  io.expand = expand;
  io.erec = expand;
  io.every = every;

  // Marks by pull for iteration `to` among the long rows of graph c (rounds set): the warp of a
  // row's first chunk decides.
  auto pull_long = [&](uint32_t to) {
    const uint8_t *E = a.emap + (size_t)((to - 1) & 1) * a.n;
    for (;;) {
      uint32_t k = 0;
      if (lane == 0) k = atomicAdd(&s_rounds.next[2], 1u);
      k = s_rounds.first[2] + __shfl_sync(kFull, k, 0);
      if (k >= s_rounds.rounds[2]) break;
      const uint4 ch = ldcg(a.items + s_rounds.base[2] + k);
      if (((ch.z >> 10) & 0x1FFFFFu) != 0 || ldcg(a.stamp + ch.x) != kNoStamp) continue;  // warp-uniform
      const uint2 d = __ldg(&a.in_rd[ch.x]);
      bool any = false;
      for (uint32_t j0 = 0; j0 < d.y && !any; j0 += 32) {
        const uint32_t j = j0 + lane;
        any = __any_sync(kFull, j < d.y && __ldcg(E + __ldg(a.in_col + d.x + j)) != 0);
      }
      if (any && lane == 0) {
        a.stamp[ch.x] = (uint16_t)to;
        joined++;
      }
    }
  };
  // ... and among its other rows, one thread a row (graphs that have stopped: the sweep does
  // it for the others)
  auto pull_short = [&](uint32_t to) {
    const uint8_t *E = a.emap + (size_t)((to - 1) & 1) * a.n;
    for (int t = 0; t < 2; t++) {
      const uint32_t per = t == 0 ? 32u : 4u;
      const uint32_t lo = s_rounds.first[t] * per, hi = min(s_rounds.rounds[t] * per, s_rounds.items[t]);
      for (uint32_t i = lo + tid; i < hi; i += kSweepBlock) {
        const uint4 item = ldcg(a.items + s_rounds.base[t] + i);
        if (item.z <= 1 || ldcg(a.stamp + item.x) != kNoStamp) continue;
        bool join = false;
        for (uint32_t j = 0; j < item.z && !join; j++) join = __ldcg(E + __ldg(a.in_col + item.y + j)) != 0;
        if (join) {
          a.stamp[item.x] = (uint16_t)to;
          joined++;
        }
      }
    }
  };

  cut();
  bool live = __syncthreads_or(tid < nc && s_state[tid] == kLive) != 0;
  live = live && (int)it < a.max_iter;
  uint32_t iters = it;
  for (;;) {
    // graphs with marks to pull: their long rows first
    const bool pulls = __syncthreads_or(tid < nc && s_state[tid] != kDead && s_pull[tid]) != 0;
    if (!live && !pulls) break;
    if (pulls && !pre_pulled) {
      segments([&](uint32_t c, unsigned long long a0, unsigned long long a1, unsigned long long w) {
        if (!s_pull[c]) return;
        if (tid == 0) set_rounds(c, a0, a1, w);
        __syncthreads();
        pull_long(it);
        __syncthreads();
      });
      if (!run_barrier(ctl, epoch, &s_err)) return;
    }
    pre_pulled = false;
    const C *Cin = it & 1 ? a.C1 : a.C0;
    bool ok = true;
    segments([&](uint32_t c, unsigned long long a0, unsigned long long a1, unsigned long long w) {
      if (tid == 0) {
        set_rounds(c, a0, a1, w);
        hot_zero(io.sbase + s_rounds.hot * (uint32_t)sizeof(C));
        if (s_state[c] == kLive && s_rounds.hot)
          stage_hot(Cin + s_rounds.hfirst, s_rounds.hot * (uint32_t)sizeof(C), io.sbase, bar);
      }
      __syncthreads();
      if (s_state[c] == kLastMarks) {
        pull_short(it);
      } else {
        if (s_rounds.hot) {
          ok = hot_landed(ctl, bar, phase & 1u) && ok;
          phase++;
        }
        io.it = it;
        io.pulling = s_pull[c] != 0;
        io.base = p.base[c];
        if (ok) sweep_pass<F32, 3>(a, io);
        tot_v += io.my_v;
        tot_e += io.my_e;
        joined += io.jloc;
        const uint32_t x = warp_sum(io.xloc);
        if (lane == 0 && x) atomicAdd(&p.xc[(it % 3) * nc + c], x);
        block_max<F32>(io.my_max, &p.dRc[(uint64_t)(it % 3) * nc + c], s_key);
      }
      __syncthreads();  // the rounds, the copy and s_key are free again
    });
    if (expand) {
      const uint32_t j = warp_sum(joined);
      joined = 0;
      if (lane == 0 && j) atomicAdd(&ctl->jtotal, j);
    }
    if (!run_barrier(ctl, epoch, &s_err)) return;
    if (!live) break;  // only the last marks were left
    // every block takes the same decisions
    int changed = 0;
    if (tid < nc) {
      if (s_state[tid] == kLastMarks) {
        s_state[tid] = kDead;
        changed = 1;
      } else if (s_state[tid] == kLive) {
        const unsigned long long key = __ldcg(&p.dRc[(uint64_t)(it % 3) * nc + tid]);
        const bool x = expand && __ldcg(&p.xc[(it % 3) * nc + tid]) != 0;
        const bool conv = key <= a.tol_key;
        s_iters[tid] = (uint16_t)(it + 1);
        s_pull[tid] = x ? 1 : 0;
        if (conv || (int)it + 1 >= a.max_iter) {
          s_state[tid] = x ? kLastMarks : kDead;
          changed = 1;
          if (blockIdx.x == 0) {
            p.comp_out[4 * tid + 0] = it + 1;
            p.comp_out[4 * tid + 1] = conv ? 1u : 0u;
            p.comp_last[tid] = key;
          }
        }
      }
      if (blockIdx.x == 0) {  // the slots of iteration it + 2, last read before this iteration's barrier
        p.dRc[(uint64_t)((it + 2) % 3) * nc + tid] = 0;
        p.xc[((it + 2) % 3) * nc + tid] = 0;
      }
    }
    if (gtid == 0) {
      ctl->t_ns[it + 2] = globaltimer_ns();
      ctl->it_kind[it] = every ? 3 : pulls ? 7 : 6;
      ctl->it_aff[it] =
          every ? a.n : ctl->save_cnt[0] + ctl->save_cnt[1] + ctl->save_cnt[2] + __ldcg(&ctl->jtotal);
    }
    it++;
    iters = it;
    if (__syncthreads_or(changed)) cut();
    live = __syncthreads_or(tid < nc && s_state[tid] == kLive) != 0;
  }

  // A call without iterations (max_iter 0) has passed no barrier: no block may write its status
  // before every block has read the marking launch's
  if (epoch == 0 && !run_barrier(ctl, epoch, &s_err)) return;

  // both parities take a graph's final values, which are in parity (its iterations) & 1; the
  // affected vertices are listed (list 0) and counted per graph, their per-call marks cleared
  auto copy_final = [&](uint32_t v, uint32_t c) {
    const bool fp = s_iters[c] & 1;
    (fp ? a.R0 : a.R1)[v] = ldcg((fp ? a.R1 : a.R0) + v);
    (fp ? a.C0 : a.C1)[v] = ldcg((fp ? a.C1 : a.C0) + v);
  };
  if (every) {
    for (uint32_t v = gtid; v < a.n; v += nthreads) copy_final(v, __ldg(p.comp + v));
  } else {
    uint32_t *s_aff = s_item;  // (the item ranges are not needed any more)
    __syncthreads();
    for (uint32_t c = tid; c < nc; c += kSweepBlock) s_aff[c] = 0;
    const uint32_t per = ((a.n + gridDim.x - 1) / gridDim.x + kSweepBlock - 1) / kSweepBlock * kSweepBlock;
    const uint32_t lo = (uint32_t)min((uint64_t)a.n, (uint64_t)blockIdx.x * per), hi = min(a.n, lo + per);
    uint32_t k = 0;
    for (uint32_t v = lo + tid; v < hi; v += kSweepBlock) k += ldcg(a.stamp + v) != kNoStamp ? 1u : 0u;
    k = warp_sum(k);
    if (lane == 0) s_cnt[wib] = k;
    __syncthreads();
    if (tid == 0) {
      uint32_t t = 0;
      for (int w = 0; w < kSweepWarps; w++) t += s_cnt[w];
      s_at = t ? atomicAdd(&ctl->aff_total, t) : 0u;
    }
    __syncthreads();
    uint32_t at = s_at;
    for (uint32_t v0 = lo; v0 < hi; v0 += kSweepBlock) {
      const uint32_t v = v0 + tid;
      const bool f = v < hi && ldcg(a.stamp + v) != kNoStamp;
      const uint32_t mask = __ballot_sync(kFull, f);
      __syncthreads();  // s_cnt free again
      if (lane == 0) s_cnt[wib] = __popc(mask);
      __syncthreads();
      uint32_t before = 0, all = 0;
      for (uint32_t w = 0; w < (uint32_t)kSweepWarps; w++) {
        before += w < wib ? s_cnt[w] : 0u;
        all += s_cnt[w];
      }
      if (f) {
        const uint32_t c = __ldg(p.comp + v);
        a.list0[at + before + __popc(mask & lanemask_lt())] = v;
        copy_final(v, c);
        atomicAdd(&s_aff[c], 1u);
        a.bitmap[v >> 5] = 0u;
        a.xbits[v >> 5] = 0u;
        a.stamp[v] = kNoStamp;
        a.emap[v] = 0;
        a.emap[a.n + v] = 0;
      }
      at += all;
    }
    __syncthreads();
    for (uint32_t c = tid; c < nc; c += kSweepBlock)
      if (s_aff[c]) atomicAdd(&p.comp_out[4 * c + 2], s_aff[c]);
  }
  tot_v = warp_sum(tot_v);
  tot_e = warp_sum(tot_e);
  if (lane == 0 && tot_v) {
    atomicAdd(&ctl->vproc, tot_v);
    atomicAdd(&ctl->eproc, tot_e);
  }
  if (gtid == 0) {
    ctl->iterations = iters;
    ctl->converged = 1;  // (per graph: comp_out)
    ctl->last_key = 0;
    ctl->status = kStatusDone;
    ctl->dense_ran = every ? 0u : 1u;
  }
}

#define CKG(call)                                           \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) return cuda_fail(g, e_, #call);  \
  } while (0)

template <bool F32>
BatchArgs<F32> batch_args(const Graph *g, RankMode mode, bool marking) {
  using S = Store<F32>;
  BatchArgs<F32> p{};
  p.a = sweep_args<F32>(g, false);
  p.nc = g->ncomp;
  p.comp = g->comp;
  p.first = g->comp_first_d;
  p.hot = g->comp_hot;
  p.item_first = g->comp_item;
  p.base = (const typename S::R *)g->comp_base;
  p.init = (const typename S::R *)g->comp_init;
  p.dRc = g->dRc;
  p.xc = g->comp_x;
  p.comp_out = g->comp_out;
  p.comp_last = g->comp_last;
  p.marking = marking ? 1u : 0u;
  p.traversal = mode == kModeDT ? 1u : 0u;
  p.is_static = mode == kModeStatic ? 1u : 0u;
  return p;
}

template <bool F32>
pr_status run_impl(Graph *g, RankMode mode, bool marking, const void *rank_args) {
  BatchArgs<F32> p = batch_args<F32>(g, mode, marking);
  void *bargs[] = {(void *)&p}, *margs[] = {const_cast<void *>(rank_args)};
  const void *bfn = (const void *)k_batch<F32>, *mfn = marking_kernel(F32);
  const size_t bsm = kHotBytes + state_bytes(g->ncomp), msm = marking_smem(g);
  if (!g->use_graph) {
    if (marking) {
      CKG(cudaLaunchCooperativeKernel(mfn, dim3(g->rank_grid), dim3(kRankBlock), margs, msm, g->st));
      count_launch();
    }
    CKG(cudaLaunchCooperativeKernel(bfn, dim3(g->loop_grid), dim3(kSweepBlock), bargs, bsm, g->st));
    count_launch();
    return PR_OK;
  }
  // CUDA-graph launch: control-block reset, marking launch and iterations, built once per kind
  // of call; later calls only replace the kernels' arguments and replay
  cudaKernelNodeParams bk{}, mk{};
  bk.func = const_cast<void *>(bfn);
  bk.gridDim = dim3(g->loop_grid);
  bk.blockDim = dim3(kSweepBlock);
  bk.sharedMemBytes = (unsigned)bsm;
  bk.kernelParams = bargs;
  mk.func = const_cast<void *>(mfn);
  mk.gridDim = dim3(g->rank_grid);
  mk.blockDim = dim3(kRankBlock);
  mk.sharedMemBytes = (unsigned)msm;
  mk.kernelParams = margs;
  const int kind = marking ? kGraphBatchMarking : kGraphBatchEvery;
  if (g->cg_exec && g->cg_kind != kind) {
    cudaGraphExecDestroy(g->cg_exec);
    cudaGraphDestroy(g->cg);
    g->cg_exec = nullptr;
    g->cg = nullptr;
  }
  if (!g->cg_exec) {
    cudaGraphNode_t reset = nullptr, dep;
    cudaMemsetParams mp{};
    mp.dst = g->ctl;
    mp.value = 0;
    mp.elementSize = 1;
    mp.width = sizeof(RankCtl);
    mp.height = 1;
    mp.pitch = sizeof(RankCtl);
    cudaLaunchAttributeValue coop{};
    coop.cooperative = 1;
    if (g->cg) cudaGraphDestroy(g->cg);
    g->cg = nullptr;
    CKG(cudaGraphCreate(&g->cg, 0));
    CKG(cudaGraphAddMemsetNode(&reset, g->cg, nullptr, 0, &mp));
    dep = reset;
    if (marking) {
      CKG(cudaGraphAddKernelNode(&g->cg_kernel, g->cg, &dep, 1, &mk));
      CKG(cudaGraphKernelNodeSetAttribute(g->cg_kernel, cudaLaunchAttributeCooperative, &coop));
      dep = g->cg_kernel;
    }
    CKG(cudaGraphAddKernelNode(&g->cg_kernel2, g->cg, &dep, 1, &bk));
    CKG(cudaGraphKernelNodeSetAttribute(g->cg_kernel2, cudaLaunchAttributeCooperative, &coop));
    CKG(cudaGraphInstantiate(&g->cg_exec, g->cg, 0));
    g->cg_kind = kind;
  } else {
    if (marking) CKG(cudaGraphExecKernelNodeSetParams(g->cg_exec, g->cg_kernel, &mk));
    CKG(cudaGraphExecKernelNodeSetParams(g->cg_exec, g->cg_kernel2, &bk));
  }
  CKG(cudaGraphLaunch(g->cg_exec, g->st));
  count_launches(marking ? 2 : 1);
  return PR_OK;
}

// First item of every graph in every tier: items are in vertex order within a tier.
__global__ void k_comp_items(const uint4 *items, uint32_t n0, uint32_t n1, uint32_t n2, const uint32_t *first,
                             uint32_t nc, uint32_t *item_first) {
  const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= 3 * (nc + 1)) return;
  const uint32_t t = k / (nc + 1), v = first[k % (nc + 1)];
  const uint32_t b = t == 0 ? 0u : t == 1 ? n0 : n0 + n1;
  uint32_t lo = 0, hi = t == 0 ? n0 : t == 1 ? n1 : n2;
  while (lo < hi) {
    const uint32_t mid = lo + (hi - lo) / 2;
    if (items[b + mid].x < v) lo = mid + 1; else hi = mid;
  }
  item_first[k] = b + lo;
}

}  // namespace

// Where this launch is ahead of the one persistent launch (k_rank).  An iteration here sweeps a block's
// graphs one after another and starts a copy for each; there all rows are dealt to all warps, at
// the general kernel's rate.  Calls over every vertex, R-MAT graphs of equal size (edge factor 8), us
// an iteration here and there: 1024 graphs of 32 vertices 47 and 9, 512 of 1024 49.5 and 30, of 2048 69
// and 56 (FP32 53 and 52), 128 of 4096 34 and 34 (27 and 36), 8 of 2^14 (1.1 M edges) 19 and 14 (17 and
// 15), 32 of 2^14 (4.4 M) 33 and 36 (27 and 37), 2 of 2^18 (4.6 M) 34 and 33 (28 and 34), 32 of 2^16 92 and
// 138 (70 and 124): from 4 M edges (FP32 2 M) in graphs of 4096 (2048) vertices on average.
// Marking calls gain from the cheaper growth of the frontier too (time here over there mostly 0.55
// to 0.95), except where a block has several small graphs: 512 graphs of 1024 vertices 1.76 at
// 1e-5 of the edges and 1.00 at 1e-3, of 256 0.93 and 1.26, of 32 0.95 and 1.49; 128 of 32 0.96 and 1.25,
// of 256 0.94 and 0.94, of 1024 0.93 and 0.85.
bool batch_eligible(const Graph *g, bool marking) {
  if (g->ncomp <= 1 || !g->split_df) return false;
  const uint64_t mean = g->n / g->ncomp;
  if (marking) return mean >= 2048 || g->ncomp <= std::min<uint64_t>((uint64_t)g->sm_count, 2 * mean);
  return g->f32 ? g->m >= (2u << 20) && mean >= 2048 : g->m >= (4u << 20) && mean >= 4096;
}

pr_status batch_setup(Graph *g) {
  // the limit belongs to the function: the same for every handle, whatever its number of graphs
  CKG(cudaFuncSetAttribute(g->f32 ? (const void *)k_batch<true> : (const void *)k_batch<false>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kHotBytes + state_bytes(kMaxComponents))));
  return batch_items(g);
}

pr_status batch_items(Graph *g) {
  const uint32_t k = 3 * (g->ncomp + 1);
  k_comp_items<<<(k + 255) / 256, 256, 0, g->st>>>(g->items, g->item_cnt[0], g->item_cnt[1], g->item_cnt[2],
                                                    g->comp_first_d, g->ncomp, g->comp_item);
  count_launch();
  CKG(cudaGetLastError());
  return PR_OK;
}

pr_status batch_run(Graph *g, RankMode mode, bool marking, const void *rank_args) {
  return g->f32 ? run_impl<true>(g, mode, marking, rank_args) : run_impl<false>(g, mode, marking, rank_args);
}

}  // namespace prdf
