// noalloc.cu - Static PageRank over a caller's device CSR without any device allocation.
//
// The library's graph handles own their device memory (cudaMalloc at creation and on
// growth).  Some callers cannot allow that: code whose device memory all comes from a host
// application's own pool or budget, code on latency-critical paths where the implicit
// device-wide synchronisation of cudaMalloc / cudaFree would stall other streams, and
// plugins that are handed device buffers but no right to allocate.  pr_static_noalloc
// serves them: the caller passes the graph and the output ranks in device memory, and the
// only working memory is the fixed array below, a file-scope __device__ array that exists
// on every device that loads this library, from module load until the process exits.
//
// Host code never names that array as an address: in host code its name is a host-side
// stand-in.  The device address is fetched once per device with cudaGetSymbolAddress, with
// that device current, on the first call on the device, and passed to the kernels.
//
// Every call uses the same array, and a call leaves its contents behind: the control words
// and out-degree counters are cleared at the start of each call.  Calls whose work overlaps
// on the GPU (two host threads, or two streams of one device) race on the array.
#include <algorithm>
#include <mutex>

#include "prdf_common.cuh"
#include "../../include/prdf.h"

namespace {

constexpr uint32_t kMaxN = PR_NOALLOC_MAX_VERTICES;
constexpr int kThreads = 256;
constexpr int kMaxDevices = 64;

struct NaCtl {
  unsigned long long dmax[3];  // max |Delta R| by iteration modulo 3 (bits of a double >= 0)
  uint32_t arrived;         // arrivals at the grid barrier (monotonic)
  uint32_t timeout;         // 1 once a barrier wait ran out
  uint32_t done;            // 1 once an iteration's max change was <= tol
  uint32_t bad;             // 1 malformed offsets, 2 column id >= n, 4 vertex without out-edges
  int32_t iterations;
  double last_delta;
};

// Layout: control block (256 bytes), out-degrees [kMaxN], contributions c0 [kMaxN], c1 [kMaxN].
constexpr size_t kCtlBytes = 256;
constexpr size_t kDegBytes = sizeof(uint32_t) * kMaxN;
constexpr size_t kContribBytes = sizeof(double) * kMaxN;
constexpr size_t kScratchBytes = kCtlBytes + kDegBytes + 2 * kContribBytes;
static_assert(sizeof(NaCtl) <= kCtlBytes, "control block");
static_assert(kScratchBytes == PR_NOALLOC_SCRATCH_BYTES, "scratch size stated in prdf.h");

__device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

std::mutex g_addr_mu;
unsigned char *g_addr[kMaxDevices] = {};
int g_sms[kMaxDevices] = {};  // multiprocessors of each device, read with the address

// off must be non-decreasing from 0 to m.
__global__ void k_na_offsets(const uint64_t *off, uint32_t n, uint64_t m, NaCtl *ctl) {
  uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v > n) return;
  bool ok = v == 0 ? off[0] == 0 : off[v - 1] <= off[v];
  if (v == n) ok = ok && off[n] == m;
  if (!ok) atomicOr(&ctl->bad, 1u);
}

// Out-degree of u = its appearances as a source in the in-edge rows.
__global__ void k_na_degree(const uint32_t *col, uint64_t m, uint32_t n, uint32_t *deg, NaCtl *ctl) {
  uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m) return;
  uint32_t u = col[e];
  if (u >= n) atomicOr(&ctl->bad, 2u);
  else atomicAdd(&deg[u], 1u);
}

__global__ void k_na_check_deg(const uint32_t *deg, uint32_t n, NaCtl *ctl) {
  uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n && deg[v] == 0) atomicOr(&ctl->bad, 4u);
}

// The iterations: one persistent cooperative launch, one block of kLoopThreads threads per SM.
//
// What bounds it: latency (an iteration's gathers hit L2; 60 K rows are about 1 M of them) and
// the FP64 rate (2 adds per clock and SM), so lanes are kept full wherever FP64 is issued.
// A block owns a run of consecutive rows holding 1/grid of the work (edges + kRowWeight a
// row, found by binary search in the offsets once).  Rows of at most kLaneRow edges take four
// lanes each; longer ones are listed once and cut into segments of kSegment edges, which take
// four lanes each too: a warp-wide tree costs five full FP64 instructions (16 clocks each) for
// every row.  The division is left to a pass with a thread per row, the sums meeting in
// shared memory.  Every row's sum has one fixed order of additions.
// On the 60,013-vertex R-MAT graph of 1 M edges: a thread per row 450 us an iteration (29.5 ms
// a call), because of its hub rows; segments of 512 edges summed by warps and finished by one
// lane 35 us (2.4 ms); this 20 us (1.47 ms).
//
// A block whose rows are alike gives each of them a thread, which needs no tree and finishes the row
// at once: most rows longer than kLaneRow (limit x 4 until at most one row in eight is above it; those
// are listed), or none and kShortRows edges on average.  262,144 vertices with 25 in-edges each 0.37 ms
// a call (four lanes, segments and warps for what the lists have no room for: 1.18), 131,072 with 81 each
// 0.42 (0.57), the same with 25 and 130 hubs of 5000 0.43 (0.69), a path of 200,000 0.94 (1.43), a grid of
// 250,000 0.70 (1.01).  With a mean of up to 10 for short rows nothing else changes.
//
// One Jacobi iteration of Eq. 1: R[v] = (1 - alpha) / n + alpha * sum over in-edges (u, v)
// of c_in[u]; c_out[v] = R[v] / |out(v)|.  The rank is updated in place (the sums read only
// c_in, through L2: other SMs wrote it during this launch).  After each iteration's barrier
// every block reads the same L-inf change and all stop together.
constexpr int kLoopThreads = 1024;
constexpr int kLoopWarps = kLoopThreads / 32;
constexpr uint32_t kRowWeight = 4;     // work of a row beside its edges, in edges
constexpr uint32_t kLaneRow = 16;      // edges of a row summed by four lanes at once
constexpr uint32_t kSegment = 64;      // edges of a segment of a longer row
constexpr uint32_t kThreadRow = 16384; // edges of a row summed by one thread at most
constexpr uint32_t kShortRows = 6;     // mean edges of rows that are short enough for a thread each
constexpr uint32_t kMaxSegs = 1024;    // segments of one row at most (more edges each for huge rows)
constexpr uint32_t kLongCap = 1024, kSegCap = 2048;  // listed rows and their segments per block
constexpr uint32_t kTile = 2048;       // rows whose sums are in shared memory together
constexpr unsigned long long kBarrierNs = 4000000000ull;  // a barrier wait gives up after 4 s

__device__ __forceinline__ double na_warp_sum(double s) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// Sum of c_in over columns [s, e) by a whole warp, eight gathers a lane in flight.
__device__ __forceinline__ double na_warp_row(const uint32_t *col, const double *c_in, uint64_t s, uint64_t e,
                                              uint32_t lane) {
  double t = 0.0;
  for (uint64_t j0 = s; j0 < e; j0 += 256) {
    double x[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint64_t j = j0 + 32u * k + lane;
      x[k] = j < e ? __ldcg(c_in + __ldg(col + j)) : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 8; k += 2)
      if (j0 + 32u * k < e) t += x[k] + x[k + 1];  // the same in every lane
  }
  return na_warp_sum(t);
}

__global__ void __launch_bounds__(kLoopThreads, 1)
    k_na_loop(uint32_t n, uint64_t m, const uint64_t *off, const uint32_t *col, const uint32_t *deg, double base,
              double alpha, double tol, double *c0, double *c1, double *R, NaCtl *ctl, int32_t max_iter) {
  __shared__ double s_sum[kTile], s_part[kSegCap], s_max[kLoopWarps];
  __shared__ uint32_t s_long[kLongCap], s_first[kLongCap + 1], s_seglen[kLongCap], s_nlong, s_list_end;
  __shared__ uint32_t s_range[2], s_cnt[kLoopWarps];
  __shared__ int s_stop;
  const uint32_t tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
  const uint32_t gtid = blockIdx.x * kLoopThreads + tid, nthreads = gridDim.x * kLoopThreads;
  if (*(volatile uint32_t *)&ctl->bad) return;  // the CSR failed its checks: ranks stay untouched
  // this block's rows: the first v with off[v] + kRowWeight v at or above its share
  if (tid < 2) {
    const uint64_t total = m + (uint64_t)kRowWeight * n, share = (total + gridDim.x - 1) / gridDim.x;
    const uint64_t at = share * (blockIdx.x + tid);
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
      const uint32_t mid = lo + (hi - lo) / 2;
      if (__ldg(off + mid) + (uint64_t)kRowWeight * mid < at) lo = mid + 1; else hi = mid;
    }
    s_range[tid] = lo;
  }
  const double r0 = 1.0 / (double)n;
  for (uint32_t v = gtid; v < n; v += nthreads) {  // R = 1/n, c = R / |out(u)|
    R[v] = r0;
    c0[v] = r0 / (double)deg[v];
  }
  __syncthreads();
  const uint32_t lo = s_range[0], hi = s_range[1], rows = hi - lo;
  uint32_t listed_rows = 0;  // rows longer than the limit so far, in row order
  auto list_rows = [&](uint32_t limit) {
    listed_rows = 0;
    for (uint32_t b0 = lo; b0 < hi; b0 += kLoopThreads) {
      const uint32_t v = b0 + tid;
      const bool f = v < hi && __ldg(off + v + 1) - __ldg(off + v) > limit;
      const uint32_t mask = __ballot_sync(0xffffffffu, f);
      if (lane == 0) s_cnt[wib] = __popc(mask);
      __syncthreads();
      uint32_t at = listed_rows + __popc(mask & prdf::lanemask_lt());
      for (uint32_t w = 0; w < (uint32_t)kLoopWarps; w++) {
        at += w < wib ? s_cnt[w] : 0u;
        listed_rows += s_cnt[w];
      }
      if (f && at < kLongCap) s_long[at] = v;
      __syncthreads();
    }
  };
  // how this block takes its rows (see above): four lanes each, or a thread each up to `limit` edges
  uint32_t limit = kLaneRow;
  list_rows(limit);
  bool by_thread = listed_rows == 0 && rows && __ldg(off + hi) - __ldg(off + lo) <= (uint64_t)kShortRows * rows;
  if (listed_rows * 2 > rows) {
    by_thread = true;
    while (listed_rows * 8 > rows && limit < kThreadRow) list_rows(limit *= 4);
  }
  if (tid == 0) {
    // segments of the listed rows; rows from s_list_end on, which the lists have no room for,
    // are summed by the warps that meet them
    const uint32_t nl = listed_rows < kLongCap ? listed_rows : kLongCap;
    uint32_t at = 0, k = 0;
    for (; k < nl; k++) {
      const uint64_t len = off[s_long[k] + 1] - off[s_long[k]];
      uint64_t sl = kSegment;
      if (len > (uint64_t)kMaxSegs * sl) sl = ((len + kMaxSegs - 1) / kMaxSegs + 31) / 32 * 32;
      const uint32_t ns = sl > 0xFFFFFFFFull ? kSegCap + 1 : (uint32_t)((len + sl - 1) / sl);
      if (at + ns > kSegCap) break;
      s_first[k] = at;
      s_seglen[k] = (uint32_t)sl;
      at += ns;
    }
    s_list_end = k == listed_rows ? hi : (k ? s_long[k - 1] + 1 : lo);
    s_nlong = k;
    s_first[k] = at;
  }
  uint32_t bar = 0;
  auto grid_barrier = [&]() -> bool {  // false after a wait that ran out (here or in another block)
    __syncthreads();
    bar++;
    if (tid == 0) {
      __threadfence();
      prdf::red_release_add_u32(&ctl->arrived, 1u);
      const uint32_t want = bar * gridDim.x;
      unsigned long long t0 = 0;
      for (uint32_t spins = 0; prdf::ld_acquire_u32(&ctl->arrived) < want; spins++) {
        if (*(volatile uint32_t *)&ctl->timeout) break;
        if ((spins & 255u) == 255u) {
          const unsigned long long t = prdf::globaltimer_ns();
          if (t0 == 0) t0 = t;
          else if (t - t0 > kBarrierNs) atomicExch(&ctl->timeout, 1u);
        }
      }
      __threadfence();
      s_stop = *(volatile uint32_t *)&ctl->timeout != 0;
    }
    __syncthreads();
    return s_stop == 0;
  };
  if (!grid_barrier()) return;
  const uint32_t nlong = s_nlong, nseg = s_first[nlong];
  const uint32_t list_end = s_list_end;
  for (int32_t it = 0; it < max_iter; it++) {
    const double *c_in = it & 1 ? c1 : c0;
    double *c_out = it & 1 ? c0 : c1;
    double lmax = 0.0;
    auto finish = [&](uint32_t v, double sum) {
      const double r = base + alpha * sum;
      lmax = fmax(lmax, fabs(r - R[v]));
      R[v] = r;
      c_out[v] = r / (double)__ldg(deg + v);
    };
    // segments of the listed rows, eight a warp
    for (uint32_t k0 = wib * 8; k0 < nseg; k0 += kLoopWarps * 8) {
      const uint32_t k = k0 + (lane >> 2), gl = lane & 3;
      uint64_t s = 0, e = 0;
      if (k < nseg) {
        uint32_t a = 0, b = nlong;  // the row: last with s_first <= k
        while (b - a > 1) {
          const uint32_t mid = (a + b) >> 1;
          if (s_first[mid] <= k) a = mid; else b = mid;
        }
        const uint32_t v = s_long[a];
        s = __ldg(off + v) + (uint64_t)(k - s_first[a]) * s_seglen[a];
        e = __ldg(off + v + 1);
        if (s + s_seglen[a] < e) e = s + s_seglen[a];
      }
      const uint32_t len = (uint32_t)(e - s), longest = __reduce_max_sync(0xffffffffu, len);
      double t = 0.0;
      for (uint32_t j0 = 0; j0 < longest; j0 += 32) {
        double x[8];
#pragma unroll
        for (int q = 0; q < 8; q++) {
          const uint32_t j = j0 + 4u * q + gl;
          x[q] = j < len ? __ldcg(c_in + __ldg(col + s + j)) : 0.0;
        }
#pragma unroll
        for (int q = 0; q < 8; q += 2)
          if (j0 + 4u * q < longest) t += x[q] + x[q + 1];
      }
      t += __shfl_xor_sync(0xffffffffu, t, 1);
      t += __shfl_xor_sync(0xffffffffu, t, 2);
      if (gl == 0 && k < nseg) s_part[k] = t;
    }
    if (by_thread) {
      // a row a lane, eight gathers in flight, the next columns on their way meanwhile
      for (uint32_t b0 = lo + wib * 32; b0 < hi; b0 += kLoopThreads) {
        const uint32_t v = b0 + lane;
        uint64_t s = 0, e = 0;
        if (v < hi) {
          s = __ldg(off + v);
          e = __ldg(off + v + 1);
        }
        const uint64_t len = e - s;
        const bool mine = v < hi && len <= limit;
        double t = 0.0;
        if (mine) {
          const uint32_t k = (uint32_t)len;
          const uint32_t *c = col + s;
          for (uint32_t j0 = 0; j0 < k; j0 += 8) {
            double x[8];
#pragma unroll
            for (int q = 0; q < 8; q++) x[q] = j0 + q < k ? __ldcg(c_in + __ldg(c + j0 + q)) : 0.0;
            const uint32_t left = k - j0;  // (no additions of zeros: the FP64 rate is the bound)
            double u = x[0];
            if (left > 1) u += x[1];
            if (left > 2) u += left > 3 ? x[2] + x[3] : x[2];
            if (left > 4) u += left > 6 ? (x[4] + x[5]) + (left > 7 ? x[6] + x[7] : x[6]) : (left > 5 ? x[4] + x[5] : x[4]);
            t += u;
          }
        }
        uint32_t more = __ballot_sync(0xffffffffu, v < hi && !mine && v >= list_end);
        const bool listed = v < hi && !mine && v < list_end;
        while (more) {
          const int src = __ffs(more) - 1;
          more &= more - 1;
          const uint64_t rs = __shfl_sync(0xffffffffu, s, src), re = __shfl_sync(0xffffffffu, e, src);
          const double x = na_warp_row(col, c_in, rs, re, lane);
          if ((int)lane == src) t = x;
        }
        if (v < hi && !listed) finish(v, t);
      }
      __syncthreads();  // the segments of the listed rows
    }
    for (uint32_t t0 = lo; t0 < hi && !by_thread; t0 += kTile) {
      const uint32_t t1 = hi - t0 < kTile ? hi : t0 + kTile;
      // eight rows a warp, four lanes a row
      for (uint32_t b0 = t0 + wib * 8; b0 < t1; b0 += kLoopWarps * 8) {
        const uint32_t v = b0 + (lane >> 2), gl = lane & 3;
        uint64_t s = 0, e = 0;
        if (v < t1) {
          s = __ldg(off + v);
          e = __ldg(off + v + 1);
        }
        const uint64_t len = e - s;
        const uint32_t mine = len <= kLaneRow ? (uint32_t)len : 0u;
        const uint32_t longest = __reduce_max_sync(0xffffffffu, mine);
        double t = 0.0, x[kLaneRow / 4];
#pragma unroll
        for (int k = 0; k < (int)kLaneRow / 4; k++) {
          const uint32_t j = 4u * k + gl;
          x[k] = j < mine ? __ldcg(c_in + __ldg(col + s + j)) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < (int)kLaneRow / 4; k += 2)
          if (4u * k < longest) t += x[k] + x[k + 1];
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        if (gl == 0 && v < t1 && len <= kLaneRow) s_sum[v - t0] = t;
        // longer rows among the eight that are not listed, the whole warp on each
        uint32_t more = __ballot_sync(0xffffffffu, gl == 0 && len > kLaneRow && v >= list_end);
        while (more) {
          const int src = __ffs(more) - 1;
          more &= more - 1;
          const uint64_t rs = __shfl_sync(0xffffffffu, s, src), re = __shfl_sync(0xffffffffu, e, src);
          const uint32_t rv = __shfl_sync(0xffffffffu, v, src);
          const double x = na_warp_row(col, c_in, rs, re, lane);
          if (lane == 0) s_sum[rv - t0] = x;
        }
      }
      __syncthreads();  // also after the segments of the long rows
      for (uint32_t v = t0 + tid; v < t1; v += kLoopThreads) {
        const bool listed = v < list_end && __ldg(off + v + 1) - __ldg(off + v) > kLaneRow;
        if (!listed) finish(v, s_sum[v - t0]);
      }
      __syncthreads();  // s_sum is free again
    }
    for (uint32_t k = tid; k < nlong; k += kLoopThreads) {
      double t = 0.0;
      for (uint32_t j = s_first[k]; j < s_first[k + 1]; j++) t += s_part[j];
      finish(s_long[k], t);
    }
    for (int o = 16; o > 0; o >>= 1) lmax = fmax(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
    if (lane == 0) s_max[wib] = lmax;
    __syncthreads();
    // the maximum of this iteration: three slots in turn, the next one cleared meanwhile (it was
    // last read two iterations ago, before the previous barrier)
    if (tid == 0) {
      double bmax = s_max[0];
      for (int w = 1; w < kLoopWarps; w++) bmax = fmax(bmax, s_max[w]);
      if (blockIdx.x == 0) ctl->dmax[(it + 1) % 3] = 0;
      atomicMax(&ctl->dmax[it % 3], (unsigned long long)__double_as_longlong(bmax));
    }
    if (!grid_barrier()) return;
    const double d = __longlong_as_double((long long)__ldcg(&ctl->dmax[it % 3]));
    if (gtid == 0) {
      ctl->last_delta = d;
      ctl->iterations = it + 1;
      ctl->done = d <= tol;
    }
    if (d <= tol) break;
  }
}

bool on_device(const void *p, int dev) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged) && at.device == dev;
}

inline unsigned blocks_for(uint64_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }

}  // namespace

extern "C" pr_status pr_static_noalloc(uint32_t n, int64_t m, const uint64_t *in_off, const uint32_t *in_col,
                                       const pr_params *params, void *cuda_stream, double *ranks, pr_stats *stats) {
  if (stats) *stats = pr_stats{};
  if (n > kMaxN) return PR_ERR_CAPACITY;  // more vertices than the fixed scratch holds
  pr_params p;
  if (params) p = *params; else pr_params_default(&p);
  if (n == 0 || m < 0 || !in_off || !ranks || (m > 0 && !in_col)) return PR_ERR_INVALID_ARG;
  if (!(p.alpha > 0.0 && p.alpha < 1.0) || !(p.tol >= 0.0) || p.max_iter < 0 || p.max_iter > prdf::kMaxIterLimit ||
      p.precision != PR_F64 || p.dead_end != PR_DEADEND_SELFLOOP)
    return PR_ERR_INVALID_ARG;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return PR_ERR_CUDA;
  }
  if (!on_device(in_off, dev) || !on_device(ranks, dev) || (m > 0 && !on_device(in_col, dev)))
    return PR_ERR_INVALID_ARG;
  unsigned char *base_ptr = nullptr;
  int sm_count = 0;
  {
    std::lock_guard<std::mutex> lk(g_addr_mu);
    if (!g_addr[dev]) {
      void *a = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&a, g_noalloc_scratch);
      if (e != cudaSuccess || !a) {
        cudaGetLastError();
        return PR_ERR_CUDA;
      }
      int sms = 0;
      if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) {
        cudaGetLastError();
        return PR_ERR_CUDA;
      }
      g_sms[dev] = sms;
      g_addr[dev] = (unsigned char *)a;
    }
    base_ptr = g_addr[dev];
    sm_count = g_sms[dev];
  }
  NaCtl *ctl = (NaCtl *)base_ptr;
  uint32_t *deg = (uint32_t *)(base_ptr + kCtlBytes);
  double *c[2] = {(double *)(base_ptr + kCtlBytes + kDegBytes),
                  (double *)(base_ptr + kCtlBytes + kDegBytes + kContribBytes)};
  cudaStream_t st = (cudaStream_t)cuda_stream;

  // checks of the caller's CSR first: nothing is written to ranks unless it is well formed
  cudaError_t e = cudaMemsetAsync(ctl, 0, sizeof(NaCtl), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(deg, 0, sizeof(uint32_t) * n, st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return PR_ERR_CUDA;
  }
  k_na_offsets<<<blocks_for((uint64_t)n + 1), kThreads, 0, st>>>(in_off, n, (uint64_t)m, ctl);
  prdf::count_launch();
  if (m > 0) {
    k_na_degree<<<blocks_for((uint64_t)m), kThreads, 0, st>>>(in_col, (uint64_t)m, n, deg, ctl);
    prdf::count_launch();
  }
  k_na_check_deg<<<blocks_for(n), kThreads, 0, st>>>(deg, n, ctl);
  prdf::count_launch();
  // the iterations are queued behind the checks and return at once if one failed: one launch
  // and one synchronisation a call
  const double base = (1.0 - p.alpha) / (double)n;
  const uint64_t share = 4096;  // edges and row weights a block is worth launching for
  const uint64_t want = ((uint64_t)m + (uint64_t)kRowWeight * n + share - 1) / share;
  const unsigned grid = (unsigned)std::min<uint64_t>(std::max<uint64_t>(want, 1), (uint64_t)sm_count);
  uint64_t m_u = (uint64_t)m;
  double alpha = p.alpha, tol = p.tol, *c0 = c[0], *c1 = c[1];
  int32_t max_iter = p.max_iter;
  void *args[] = {&n, &m_u, (void *)&in_off, (void *)&in_col, &deg, (void *)&base, &alpha, &tol, &c0, &c1, &ranks,
                  &ctl, &max_iter};
  e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaLaunchCooperativeKernel((const void *)k_na_loop, dim3(grid), dim3(kLoopThreads), args, 0, st);
  prdf::count_launch();
  NaCtl h{};
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, ctl, sizeof(NaCtl), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return PR_ERR_CUDA;
  }
  if (h.bad & 2u) return PR_ERR_VERTEX_RANGE;
  if (h.bad) return PR_ERR_INVALID_ARG;  // malformed offsets, or a vertex without out-edges
  if (h.timeout) return PR_ERR_DEVICE_TIMEOUT;
  if (stats) {
    stats->iterations = h.iterations;
    stats->converged = h.done ? 1 : 0;
    stats->affected_final = n;
    stats->vertices_processed = (int64_t)h.iterations * n;
    stats->edges_processed = (int64_t)h.iterations * m;
    stats->bytes_algorithmic = (double)h.iterations * (12.0 * (double)m + 36.0 * (double)n);
    stats->last_delta = h.last_delta;
  }
  return PR_OK;
}
