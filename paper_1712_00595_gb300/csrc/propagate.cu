// Offset score propagation: the cumulative power iteration of Algorithm 1,
//   x(i) = (1-c) B~^T x(i-1),  r += x(i),  until ||x(i)||_1 <= eps,
// run as one persistent cooperative kernel per call.
//
// The kernel keeps the gather vector y(i) = (1-c) x(i) / d (the scale is
// applied once per source node, so a step is a plain sum over in-edges) and
// moves between two step kinds:
//   push: x(i) is sparse. Each frontier node u scatters y(i-1)[u] to its
//         out-neighbours (atomic adds into xacc, first touch appends to the
//         next frontier); an epilogue over the new frontier adds x(i) into r,
//         forms y(i) and sums |x(i)|.
//   pull: x(i) is dense. Each node v sums y(i-1) over its in-list and the
//         same pass adds x(i) into r, writes y(i) and sums |x(i)|. Warps take
//         tasks of consecutive nodes (about equal edges + nodes) from a
//         shared counter; long lists are summed in pieces by all warps.
// The step switches to pull once the frontier's out-edges exceed m / alpha or
// its size exceeds n / beta, and stays there. Between steps a grid barrier
// (bounded wait) reduces the per-CTA |x| partials in a fixed order and takes
// the do-while stopping decision on the device, so a whole call needs no
// host round trip.
#include <type_traits>

#include "common.cuh"
#include "gridbar.cuh"
#include "kernels.h"

namespace osp {
namespace {

// What every CTA knows of the call between two grid barriers (its own copy in
// shared memory; the copies are equal because each CTA sums the same partials
// in the same order). CTA 0 writes its copy back at the end.
struct CallState {
  int iter, mode, stop, ok;
  int q_cur, q_next;  // sizes of the current frontier and of the one being built
  int n_big;          // pieces of long rows listed by the push step
  int push_iters, pull_used, noconv;
  long long ef, visited, push_f, push_r;
};

// One grid barrier, run by warp 0 between two __syncthreads (the caller's):
// arrive, wait, and true if the call goes on. All lanes return the same value
// and see what lane 0's wait has acquired (the shuffle alone orders no memory).
__device__ __forceinline__ bool warp0_barrier(const Dev& d, unsigned target) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) ok = grid_wait(d.bar, target, d.ctl);
  __syncwarp();
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// Barrier without a decision, inside a push step. *count: the pieces listed so
// far, *queued: the next frontier's size, both read after the barrier.
__device__ __forceinline__ bool mid_barrier(const Dev& d, unsigned target, CallState& cs, int* count,
                                            int* queued) {
  __syncthreads();
  if (threadIdx.x < 32) {
    bool ok = warp0_barrier(d, target);
    if (threadIdx.x == 0) {
      const int st = *(volatile int*)&d.ctl->status;
      cs.n_big = *(volatile int*)count;
      cs.q_next = *(volatile int*)queued;
      cs.ok = ok && st == 0;
    }
  }
  __syncthreads();
  return cs.ok;
}

// Barrier at the end of a step: per-CTA partials of ||x||_1 and of the
// frontier's out-edges, arrival, and the stopping / step-kind decision
// (Algorithm 1 loop test, do-while form), which every CTA takes for itself
// from all partials summed in one fixed order. Against one CTA deciding for
// all this saves the release hop and the re-read of its verdict, and one CTA
// per SM quarters the arrivals: a step of a 10,000-node graph in double went
// from 17.8 to 14.9 us, and to 9.6 us with the cheaper double sums of stream_lists.
__device__ bool step_barrier(const Dev& d, const PropParams& pp, int step_mode, int n, long long m,
                             double l1, long long ef, unsigned target, CallState& cs, double* s_red,
                             double* s_l1, long long* s_ef) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  Ctl* ctl = d.ctl;
  const int it = step_mode < 0 ? 0 : cs.iter + 1;  // the step that ends here
  if (step_mode != kPull) ef = warp_sum(ef);
  if (lane == 0) s_ef[w] = ef;
  // the CTA's |x|: 36 warp-wide double additions against 165 with a warp
  // reduction in each warp (16 cycles of the SM apiece)
  s_red[threadIdx.x] = l1;
  __syncthreads();
  if (w < 4) {
    double a = s_red[threadIdx.x];
#pragma unroll
    for (int j = 1; j < 8; ++j) a += s_red[threadIdx.x + 128 * j];
    if (w > 0) s_red[threadIdx.x] = a;
    else l1 = a;
  }
  __syncthreads();
  if (w == 0) {
    const int par = (it & 1) * kMaxGrid;  // a slow CTA may still read the last step's partials
    double a = warp_sum((l1 + s_red[lane + 32]) + (s_red[lane + 64] + s_red[lane + 96]));
    long long b = step_mode != kPull ? warp_sum(s_ef[lane]) : 0;
    if (lane == 0) {
      d.part_l1[par + blockIdx.x] = a;
      d.part_ef[par + blockIdx.x] = b;
    }
    const bool ok = warp0_barrier(d, target);
    a = 0.0;
    b = 0;
    for (int i = lane; i < (int)gridDim.x; i += 32) {
      a += __ldcg(d.part_l1 + par + i);
      if (step_mode != kPull) b += __ldcg(d.part_ef + par + i);
    }
    const int st = *(volatile int*)&ctl->status;
    const int queued = step_mode != kPull ? *(volatile int*)&ctl->q_size[it & 1] : 0;
    a = warp_sum(a);
    if (step_mode != kPull) b = warp_sum(b);
    if (lane == 0) {
      s_l1[0] = a;
      cs.ok = ok && st == 0;
      cs.ef = b;
      cs.q_next = queued;
    }
  }
  if (pp.det && step_mode == kPull) {  // the long in-lists' |x|, in a fixed order too
    __syncthreads();
    double a = 0.0;
    const int nh = ctl->n_hubs;
    const double* hub_l1 = d.hub_l1[it & 1];  // by parity like the partials
    for (int i = threadIdx.x; i < nh; i += blockDim.x) a += __ldcg(hub_l1 + i);
    a = warp_sum(a);
    if (lane == 0 && w > 0) s_l1[w] = a;
    __syncthreads();
    if (threadIdx.x == 0)
      for (int i = 0; i < kOneWarps; ++i) s_l1[0] += i ? s_l1[i] : a;
  }
  if (threadIdx.x == 0) {
    const double L1 = s_l1[0];
    if (blockIdx.x == 0 && it < kMaxHist) {
      d.l1_hist[it] = L1;
      d.step_ns[it + 1] = global_ns();
    }
    cs.iter = it;
    int stop = 0;  // at least one step always runs
    if (step_mode >= 0) {
      if (step_mode == kPush) {
        cs.push_iters += 1;
        cs.push_f += cs.q_cur;
        cs.push_r += cs.q_next;
      } else {
        cs.visited += m;
        cs.pull_used = 1;
      }
      stop = pp.force_iters > 0 ? it >= pp.force_iters : L1 <= pp.eps;
      if (!stop && it >= pp.max_iter) {
        stop = 1;
        cs.noconv = 1;
      }
    }
    cs.stop = stop;
    cs.q_cur = cs.q_next;
    cs.mode = kPull;
    if (step_mode != kPull && !pp.det &&
        !((double)cs.ef > (double)m / pp.alpha || (double)cs.q_cur > (double)n / pp.beta)) {
      cs.mode = kPush;
      if (!stop) cs.visited += cs.ef;  // the next step reads these edges
    }
  }
  __syncthreads();
  return cs.ok;
}

// y(u) * out-edges of up to 32 * R positions of a warp's stream of rows: lane
// l's R targets v (ok: a real one) get val added in xacc; a target met first in
// this step (its stamp) joins the next frontier, one queue reservation per call.
template <int R>
__device__ __forceinline__ void push_targets(const Dev& d, const int (&v)[R], const bool (&ok)[R],
                                             const double (&val)[R], int* qdst, int* qdst_size, int ep) {
  const int lane = threadIdx.x & 31;
  int old[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    old[r] = ep;
    if (ok[r]) {
      atomicAdd(&d.xacc[v[r]], val[r]);
      old[r] = atomicExch(&d.mark[v[r]], ep);
    }
  }
  unsigned bm[R];
  int tot = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    bm[r] = __ballot_sync(0xffffffffu, old[r] != ep);
    tot += __popc(bm[r]);
  }
  if (!tot) return;
  int at = 0;
  if (lane == 0) at = atomicAdd(qdst_size, tot);
  at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (old[r] != ep) qdst[at + __popc(bm[r] & lanemask_lt())] = v[r];
    at += __popc(bm[r]);
  }
}

// Push step, scatter. A warp takes `per` consecutive frontier nodes (as few as
// leave every warp some, at most 32) and walks their rows as one stream of
// edges, R rounds of 32 with their loads and atomics in flight; rows above
// kPushPiece entries are listed in pieces for all warps. Bound by the latency
// of its atomics, hence as many as possible at once: the push step after one
// edge of a 100,003-node, 1.2 M-edge graph takes 31 us (380 us with 32 frontier
// nodes and rows of up to 1,024 entries to a warp, one round in flight).
template <typename T>
__device__ void push_scatter(const Dev& d, const int* qsrc, int qs, T* ys, int* qdst, int* qdst_size,
                             int ep, int* big_count) {
  constexpr int R = 4;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  const int per = min(32, (qs + nw - 1) / nw);
  for (int i0 = gw * per; i0 < qs; i0 += nw * per) {
    const int i = i0 + lane;
    const bool valid = lane < per && i < qs;
    int u = valid ? __ldcg(qsrc + i) : 0;
    if (!OSP_GUARD(d.ctl, u >= 0 && u < d.nc, "push frontier id", i, u, qs)) u = 0;
    T val = (T)0;
    unsigned o = 0;
    int len = 0;
    if (valid) {
      val = __ldcg(ys + u);
      ys[u] = (T)0;
      o = __ldg(d.off_r + u);
      len = __ldg(d.len_r + u);
      if (val == (T)0) len = 0;
    }
    // long rows: one list entry per piece
    unsigned bigs = __ballot_sync(0xffffffffu, len > kPushPiece);
    while (bigs) {
      const int l = __ffs(bigs) - 1;
      bigs &= bigs - 1;
      const unsigned ho = __shfl_sync(0xffffffffu, o, l);
      const int hl = __shfl_sync(0xffffffffu, len, l);
      const double hv = (double)__shfl_sync(0xffffffffu, val, l);
      const int np = (hl + kPushPiece - 1) / kPushPiece;
      int at = 0;
      if (lane == 0) at = atomicAdd(big_count, np);
      at = __shfl_sync(0xffffffffu, at, 0);
      for (int q = lane; q < np; q += 32) {
        d.big_off[at + q] = ho + (unsigned)(q * kPushPiece);
        d.big_len[at + q] = min(kPushPiece, hl - q * kPushPiece);
        d.big_y[at + q] = hv;
      }
    }
    const int ll = len > kPushPiece ? 0 : len;
    int P = ll;  // exclusive prefix of the stream
#pragma unroll
    for (int q = 1; q < 32; q <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, P, q);
      if (lane >= q) P += y;
    }
    const int total = __shfl_sync(0xffffffffu, P, 31);
    P -= ll;
    for (int eb = 0; eb < total; eb += 32 * R) {
      int v[R];
      bool ok[R];
      double x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int e = eb + 32 * r + lane;
        int lo = 0;  // the row of position e: the last lane with P <= e
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) {
          const int pm = __shfl_sync(0xffffffffu, P, lo + q);
          if (pm <= e) lo += q;
        }
        const unsigned ob = __shfl_sync(0xffffffffu, o, lo);
        const int pb = __shfl_sync(0xffffffffu, P, lo);
        x[r] = (double)__shfl_sync(0xffffffffu, val, lo);
        ok[r] = e < total;
        v[r] = ok[r] ? __ldg(d.pool_r + ob + (unsigned)(e - pb)) : 0;
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (ok[r]) ok[r] = OSP_GUARD(d.ctl, v[r] >= 0 && v[r] < d.nc, "push target", eb, r, v[r]);
      push_targets<R>(d, v, ok, x, qdst, qdst_size, ep);
    }
  }
}

// Pieces of the push rows longer than kPushPiece, spread over all warps.
__device__ void push_big_rows(const Dev& d, int nb, int* qdst, int* qdst_size, int ep) {
  constexpr int R = kPushPiece / 32;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int b = gw; b < nb; b += nw) {
    const int* row = d.pool_r + __ldcg(d.big_off + b);
    const int len = __ldcg(d.big_len + b);
    const double val = __ldcg(d.big_y + b);
    int v[R];
    bool ok[R];
    double x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      ok[r] = 32 * r + lane < len;
      v[r] = ok[r] ? __ldg(row + 32 * r + lane) : 0;
      x[r] = val;
      if (ok[r]) ok[r] = OSP_GUARD(d.ctl, v[r] >= 0 && v[r] < d.nc, "push big target", b, r, v[r]);
    }
    push_targets<R>(d, v, ok, x, qdst, qdst_size, ep);
  }
}

__device__ __forceinline__ void finish_node(const Dev& d, int v, double x, void* yd, bool fp32,
                                            double& l1) {
  if (!OSP_GUARD(d.ctl, v >= 0 && v < d.nc, "finish node", v, 0, 0)) return;
  if (x != 0.0) d.r[v] += x;  // an empty in-list leaves r as it is
  l1 += fabs(x);
  if (fp32) ((float*)yd)[v] = (float)x * __ldg(d.scale_f + v);
  else ((double*)yd)[v] = x * __ldg(d.scale_d + v);
}

// ---------------------------------------------------------------------------
// The short in-lists of up to 32 consecutive nodes as one stream of edges, 32
// positions a round, with coalesced id loads and the gathers of several rounds
// in flight. Which list a position belongs to comes from a bit mask of list
// starts per round: its rank among the nonempty lists = starts up to it.
// How the values are added depends on the type, because this chip adds 32
// doubles in about 16 cycles per SM and 32 floats in a quarter cycle:
//   float   a segmented warp scan per round.
//   double  a batch of K <= 8 rounds goes through shared memory and lane l adds
//           positions [K l, K l + K) one after the other: K - 1 serial
//           additions and one scan per batch instead of a scan per round
//           (300,007 nodes, 3 M edges: 52 -> 29 us a step; floats gain nothing
//           from it, 42 against 41 us a step at 2^19 nodes and 2^23 edges).
// ---------------------------------------------------------------------------
// Longest list that joins the stream; longer ones are summed by the whole warp.
template <typename T>
constexpr int kStreamMax = std::is_same<T, float>::value ? 32 : 128;

template <typename T>
struct WarpStream {
  static constexpr bool kF32 = std::is_same<T, float>::value;
  static constexpr int kRounds = kF32 ? 4 : 8;  // rounds in flight
  static constexpr int kVals = kF32 ? 1 : 32 * 8 + 16;
  T val[kVals];                     // double: the batch, one padding element per 16
  T sum[32];                        // per nonempty list of the chunk
  unsigned delta[32];               // pool offset of the list minus its first position
  unsigned starts[2][kRounds];      // double: list starts by round, two batches
  int before[2][kRounds];           // double: nonempty lists started before the round
};

// Lane j holds node j's list (length ll, 0 to leave it out, at pool offset o):
// first position P and rank of the list; returns the stream's length.
template <typename T>
__device__ __forceinline__ int stream_begin(int ll, unsigned o, WarpStream<T>& W, int& P, int& rank) {
  const int lane = threadIdx.x & 31;
  P = ll;
#pragma unroll
  for (int q = 1; q < 32; q <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, P, q);
    if (lane >= q) P += y;
  }
  const int total = __shfl_sync(0xffffffffu, P, 31);
  P -= ll;
  rank = __popc(__ballot_sync(0xffffffffu, ll > 0) & lanemask_lt());
  __syncwarp();  // the last chunk's sums have been read
  W.sum[lane] = (T)0;
  if (ll > 0) W.delta[rank] = o - (unsigned)P;
  __syncwarp();
  return total;
}

// List starts among positions [eb, eb + 32), bit by bit.
__device__ __forceinline__ unsigned stream_starts(int ll, int P, int eb) {
  const unsigned at = (unsigned)(P - eb);
  return __reduce_or_sync(0xffffffffu, ll > 0 && at < 32u ? 1u << at : 0u);
}

// Sums of the lists of a chunk; returns lane j's.
__device__ __forceinline__ float stream_lists(const Dev& d, const float* ys, int ll, unsigned o,
                                              WarpStream<float>& W) {
  constexpr int R = WarpStream<float>::kRounds;
  const int lane = threadIdx.x & 31;
  const unsigned le = lanemask_lt() | (1u << lane);
  int P, rank;
  const int total = stream_begin(ll, o, W, P, rank);
  int started = -1;  // rank of the list that runs into the round
  for (int eb = 0; eb < total; eb += 32 * R) {
    unsigned hm[R];
    int k[R], id[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      hm[r] = stream_starts(ll, P, eb + 32 * r);
      const int e = eb + 32 * r + lane;
      k[r] = started + __popc(hm[r] & le);
      // the sum wraps back
      id[r] = e < total ? list_id(d, __ldg(d.pool_c + (W.delta[k[r]] + (unsigned)e)), e) : -1;
      started += __popc(hm[r]);
    }
    float v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = id[r] >= 0 ? ys[id[r]] : 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int seg0 = 31 - __clz((hm[r] | 1u) & le);
      float x = v[r];
#pragma unroll
      for (int q = 1; q < 32; q <<= 1) {
        const float t = __shfl_up_sync(0xffffffffu, x, q);
        if (lane - q >= seg0) x += t;
      }
      // the last lane of a list's run in this round holds its sum
      if (id[r] >= 0 && (lane == 31 || ((hm[r] >> lane) & 2u) || eb + 32 * r + lane == total - 1))
        W.sum[k[r]] += x;
      __syncwarp();
    }
  }
  return ll > 0 ? W.sum[rank] : 0.f;
}

__device__ __forceinline__ double stream_lists(const Dev& d, const double* ys, int ll, unsigned o,
                                               WarpStream<double>& W) {
  constexpr int R = WarpStream<double>::kRounds;
  const int lane = threadIdx.x & 31;
  int P, rank;
  const int total = stream_begin(ll, o, W, P, rank);
  const int longest = __reduce_max_sync(0xffffffffu, ll);
  int started = 0;  // lists started before the round whose ids load next
  int id[R];
  auto load_ids = [&](int eb, int buf) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      id[r] = -1;
      if (eb + 32 * r >= total) continue;  // warp-uniform
      const unsigned hm = stream_starts(ll, P, eb + 32 * r);
      if (lane == r) {
        W.starts[buf][r] = hm;
        W.before[buf][r] = started;
      }
      const int e = eb + 32 * r + lane;
      const int k = started + __popc(hm & (lanemask_lt() | (1u << lane))) - 1;
      if (e < total) id[r] = list_id(d, __ldg(d.pool_c + (W.delta[k] + (unsigned)e)), e);  // wraps back
      started += __popc(hm);
    }
  };
  load_ids(0, 0);
  for (int eb = 0, buf = 0; eb < total; eb += 32 * R, buf ^= 1) {
    const int left = total - eb;
    const int K = min(R, (left + 31) >> 5);
    double v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = id[r] >= 0 ? ys[id[r]] : 0.0;
    if (left > 32 * R) load_ids(eb + 32 * R, buf ^ 1);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int q = 32 * r + lane;
      if (r < K) W.val[q + (q >> 4)] = v[r];
    }
    __syncwarp();
    // this lane's K positions: starts among them, list of the first one
    const int p0 = lane * K, w0 = p0 >> 5;
    const unsigned m0 = W.starts[buf][w0];
    const unsigned m1 = w0 + 1 < K ? W.starts[buf][w0 + 1] : 0u;
    unsigned bits = __funnelshift_r(m0, m1, p0 & 31);
    int cur = W.before[buf][w0] + __popc(m0 & ((1u << (p0 & 31)) - 1u)) - 1;
    const int cur0 = cur;
    bool any = bits & 1u;
    double acc = W.val[p0 + (p0 >> 4)], first = 0.0;
    cur += any;
    for (int k = 1; k < K; ++k) {
      const int q = p0 + k;
      const double x = W.val[q + (q >> 4)];
      bits >>= 1;
      if (bits & 1u) {
        if (any) W.sum[cur] = acc;  // began and ended in this lane
        else first = acc;
        any = true;
        ++cur;
        acc = x;
      } else {
        acc += x;
      }
    }
    // acc: the part of list `cur` that ends this lane; join it with the lanes
    // before, as far back as the longest list reaches
    const unsigned heads = __ballot_sync(0xffffffffu, any) | 1u;
    const int seg0 = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
    const int span = (longest + K - 1) / K;  // lanes before its last one that a list can cover
#pragma unroll
    for (int q = 1; q < 32; q <<= 1) {
      if (q > span) break;  // warp-uniform
      const double t = __shfl_up_sync(0xffffffffu, acc, q);
      if (lane - q >= seg0) acc += t;
    }
    const double carry = __shfl_up_sync(0xffffffffu, acc, 1);
    // lists that began before this lane and end in it; the batch's last lane
    // with a position adds its own, which may go on in the next batch
    if (any && cur0 >= 0) W.sum[cur0] += lane ? first + carry : first;
    __syncwarp();
    if (lane == (min(left, 32 * K) - 1) / K) W.sum[cur] += acc;
    __syncwarp();
  }
  return ll > 0 ? W.sum[rank] : 0.0;
}

// Dense step. Warp tasks of about kTaskItems edges + nodes (planned per batch,
// lists never split) are taken 32 consecutive nodes at a time (stream_lists);
// a list above hub_thr is cut into pieces dealt to all warps before the tasks
// (the piece that completes a list finishes it).
template <typename T>
__device__ double pull_step(const Dev& d, const T* ys, T* yd, int n_hubs, int n_pieces,
                            int n_tasks, WarpStream<T>& W, int* grab, int hub_thr, int hub_piece,
                            bool det, double* hub_l1) {
  constexpr bool kF32 = std::is_same<T, float>::value;
  double l1 = 0.0;
  const int lane = threadIdx.x & 31;
  // Work items 0 .. n_pieces-1 are pieces of the long in-lists, the rest the
  // warp tasks; each warp takes the next item from a grid-wide counter, so the
  // long lists go first and warps that finish early take more of the rest.
  const int n_items = n_pieces + n_tasks;
  // Tasks are taken in a scrambled order, t -> t * P mod n_tasks (P prime and
  // coprime to n_tasks), so that the warps busy at any moment hold a mix of
  // list lengths rather than one run of neighbouring (similar) nodes.
  long long P = 7919;
  if (n_tasks % 7919 == 0) P = 7907;
  if (n_tasks % P == 0) P = 1;
  // Deterministic mode: warp gw takes items gw, gw + nw, ... instead, so every
  // lane sums its |x| terms in the same order on every run.
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int k = 0;; ++k) {
    // the first item is the warp's own number, so a graph with no more items
    // than warps needs no counter
    int t = gw + k * nw;
    if (!det && k > 0) {
      if (n_items <= nw) break;
      if (lane == 0) t = nw + atomicAdd(grab, 1);
      t = __shfl_sync(0xffffffffu, t, 0);
    }
    if (t >= n_items) break;
    if (t < n_pieces) {
      const int h = __ldg(d.piece_hub + t);  // the long list this piece belongs to
      const int v = __ldg(d.hubs + h);
      const int piece = t - __ldg(d.hub_pstart + h);
      const int full = __ldg(d.len_c + v);
      const int* p = d.pool_c + __ldg(d.off_c + v) + (unsigned)(piece * hub_piece);
      const int L = min(hub_piece, full - piece * hub_piece);
      T acc = (T)0;
      int j = lane;
      for (; j + 96 < L; j += 128) {
        const int a0 = list_id(d, __ldg(p + j), j), a1 = list_id(d, __ldg(p + j + 32), j),
                  a2 = list_id(d, __ldg(p + j + 64), j), a3 = list_id(d, __ldg(p + j + 96), j);
        acc += (ys[a0] + ys[a1]) + (ys[a2] + ys[a3]);
      }
      for (; j < L; j += 32) acc += ys[list_id(d, __ldg(p + j), j)];
      acc = warp_sum(acc);
      if (lane == 0) {
        const int np = (full + hub_piece - 1) / hub_piece;
        if (det) {
          // pieces leave their sums in slots; the last one adds them up in
          // piece order and parks |x_v| for the step's fixed-order norm sum
          d.piece_part[t] = (double)acc;
          __threadfence();
          if (atomicAdd(&d.hub_cnt[h], 1) == np - 1) {
            __threadfence();
            const double* slots = d.piece_part + (t - piece);
            double x = 0.0;
            for (int q = 0; q < np; ++q) x += __ldcg(slots + q);
            d.hub_cnt[h] = 0;
            double hl = 0.0;
            finish_node(d, v, x, yd, kF32, hl);
            hub_l1[h] = hl;
          }
        } else {
          atomicAdd(&d.hub_acc[h], (double)acc);
          __threadfence();
          if (atomicAdd(&d.hub_cnt[h], 1) == np - 1) {
            __threadfence();
            const double x = __longlong_as_double(
                (long long)atomicExch((unsigned long long*)&d.hub_acc[h], 0ull));
            d.hub_cnt[h] = 0;
            finish_node(d, v, x, yd, kF32, l1);
          }
        }
      }
      continue;
    }
    const int task = (int)(((long long)(t - n_pieces) * P) % n_tasks);
    const int c0 = __ldg(d.task_first + task), c1 = __ldg(d.task_first + task + 1);
    for (int vb = c0; vb < c1; vb += 32) {
      const int v = vb + lane;
      const bool valid = v < c1;
      unsigned o = 0;
      int len = 0;
      if (valid) {
        o = __ldg(d.off_c + v);
        len = __ldg(d.len_c + v);
      }
      const bool hub = len > hub_thr;
      const bool light = len <= kStreamMax<T>;
      T s = stream_lists(d, ys, light ? len : 0, o, W);
      // longer lists: the whole warp, blocks of 256 entries (eight coalesced id
      // loads and gathers per lane); the ids of the next block (of this list or
      // the next one) load while the current block's gathers are in flight
      unsigned hm = __ballot_sync(0xffffffffu, !light && !hub);
      if (hm) {
        int l = __ffs(hm) - 1;
        hm &= hm - 1;
        const int* p = d.pool_c + __shfl_sync(0xffffffffu, o, l);
        int hl = __shfl_sync(0xffffffffu, len, l);
        int jb = 0;
        int a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          a[q] = 32 * q + lane < hl ? list_id(d, __ldg(p + 32 * q + lane), q) : -1;
        T acc = (T)0;
        for (;;) {
          T t[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) t[q] = a[q] >= 0 ? ys[a[q]] : (T)0;
          const int left = hl - jb;
          // the next block: the rest of this list, else the next long list
          const bool same = left > 256;
          int nl = l, nhl = hl, njb = jb + 256;
          const int* np = p;
          if (!same && hm) {
            nl = __ffs(hm) - 1;
            nhl = __shfl_sync(0xffffffffu, len, nl);
            np = d.pool_c + __shfl_sync(0xffffffffu, o, nl);
            njb = 0;
          }
          const bool more = same || hm != 0;
          if (more) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const int j = njb + 32 * q + lane;
              a[q] = j < nhl ? list_id(d, __ldg(np + j), j) : -1;
            }
          }
          if (kF32) {
            acc += ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
          } else {  // double additions are dear: none for rounds past the end (warp-uniform)
            T x = t[0];
#pragma unroll
            for (int q = 1; q < 8; ++q)
              if (left > 32 * q) x += t[q];
            acc += x;
          }
          if (!same) {  // list l is complete
            const T tot = warp_sum(acc);
            if (lane == l) s = tot;
            acc = (T)0;
            if (!hm) break;
            hm &= hm - 1;
          }
          l = nl;
          hl = nhl;
          p = np;
          jb = njb;
        }
      }
      if (valid && !hub) finish_node(d, v, (double)s, yd, kF32, l1);
    }
  }
  return l1;
}

}  // namespace

template <typename T>
__global__ void __launch_bounds__(kOneThreads, 1) k_propagate(Dev d, PropParams pp) {
  __shared__ CallState cs;
  __shared__ double s_red[kOneThreads];  // the threads' |x| (apart from dsm, which slower warps still use)
  __shared__ double s_l1[kOneWarps];
  __shared__ long long s_ef[kOneWarps];
  extern __shared__ __align__(16) unsigned char dsm[];  // the warps' stream buffers
  __shared__ int s_qw[kOneWarps];    // dense x(0) scan: queue offsets of the warps
  __shared__ int s_qbase;
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  const int n = ctl->n;
  const long long m = ctl->m;
  const int epoch = ctl->epoch;
  const int n_hubs = ctl->n_hubs;
  const int n_pieces = ctl->n_pieces;
  const int n_tasks = ctl->n_tasks;
  const int hub_thr = ctl->hub_thr, hub_piece = ctl->hub_piece;
  T* yb[2] = {(T*)d.y0, (T*)d.y1};
  int* qb[2] = {d.q0, d.q1};
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  const int nthreads = gridDim.x * blockDim.x;
  if (tid == 0) d.step_ns[0] = global_ns();
  if (threadIdx.x == 0) cs = CallState{};  // read after the first barrier
  unsigned target = 0;  // arrivals that open the next grid barrier

  // x(0) (the offset vector, or c e_s for CPI) sits in xacc over queue 0
  {
    double l1 = 0.0;
    long long ef = 0;
    const int qs = *(volatile int*)&ctl->q_size[0];
    if (!OSP_GUARD(ctl, qs >= 0 && qs <= d.nc, "first frontier size", qs, 0, 0)) return;
    if (pp.det) {
      // Deterministic mode: every step pulls, so no frontier queue is kept; a
      // fixed pass over all nodes collects x(0) from xacc and from the merge's
      // fixed-point accumulator (exact integer sums, so their order is moot).
      for (int v = tid; v < n; v += nthreads) {
        double x = __ldcg(d.xacc + v);
        const long long q = (long long)__ldcg(d.xfix + v);
        if (q != 0) {
          x += (double)q * 0x1p-62;
          d.xfix[v] = 0ull;
        }
        if (x != 0.0) {
          d.xacc[v] = 0.0;
          d.r[v] += x;
          l1 += fabs(x);
          yb[0][v] = (T)(x * __ldg(d.scale_d + v));
          ef += __ldg(d.len_r + v);
        }
      }
    } else if (*(volatile int*)&ctl->dense0) {
      // The merge reached more than n/beta nodes and queued none of them: one
      // coalesced pass over all nodes collects x(0) (xacc is zero off its
      // support) and builds the frontier queue of its nonzero entries.
      // One queue reservation per CTA tile of 4 x blockDim.x nodes, whose x
      // values load together (the loop is uniform over the CTA).
      const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
      for (int base = blockIdx.x * 4 * blockDim.x; base < n; base += 4 * nthreads) {
        double xs[4];
        int vs[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          vs[k] = base + k * blockDim.x + threadIdx.x;
          xs[k] = vs[k] < n ? __ldcg(d.xacc + vs[k]) : 0.0;
        }
        int cnt = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (xs[k] != 0.0) {
            const int v = vs[k];
            d.xacc[v] = 0.0;
            d.r[v] += xs[k];
            l1 += fabs(xs[k]);
            yb[0][v] = (T)(xs[k] * __ldg(d.scale_d + v));
            ef += __ldg(d.len_r + v);
            ++cnt;
          }
        }
        int inc = cnt;  // inclusive warp scan of the counts
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += y;
        }
        if (lane == 31) s_qw[w] = inc;
        __syncthreads();
        if (threadIdx.x == 0) {
          int t = 0;
          for (int i = 0; i < kOneWarps; ++i) {
            const int c = s_qw[i];
            s_qw[i] = t;
            t += c;
          }
          s_qbase = t ? atomicAdd(&ctl->q_size[0], t) : 0;
        }
        __syncthreads();
        int pos = s_qbase + s_qw[w] + inc - cnt;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (xs[k] != 0.0) d.q0[pos++] = vs[k];
        __syncthreads();
      }
    } else {
      for (int k = tid; k < qs; k += nthreads) {
        const int v = __ldcg(d.q0 + k);
        if (!OSP_GUARD(ctl, v >= 0 && v < d.nc, "first frontier id", k, v, qs)) continue;
        const double x = __ldcg(d.xacc + v);
        d.xacc[v] = 0.0;
        d.r[v] += x;
        l1 += fabs(x);
        yb[0][v] = (T)(x * __ldg(d.scale_d + v));
        ef += __ldg(d.len_r + v);
      }
    }
    target += gridDim.x;
    if (!step_barrier(d, pp, -1, n, m, l1, ef, target, cs, s_red, s_l1, s_ef)) return;
  }

  int it = 0;
  while (!cs.stop) {
    ++it;
    const int mode = cs.mode;
    const int src = (it - 1) & 1, dst = it & 1;
    double l1 = 0.0;
    long long ef = 0;
    // nobody uses the work counter of two steps on before the next barrier
    if (tid == 0) ctl->ctr[(it + 2) & 3] = 0;
    if (mode == kPush) {
      int* qn_p = &ctl->q_size[dst];
      push_scatter<T>(d, qb[src], cs.q_cur, yb[src], qb[dst], qn_p, epoch + it, &ctl->n_big);
      target += gridDim.x;
      if (!mid_barrier(d, target, cs, &ctl->n_big, qn_p)) return;
      if (cs.n_big > 0) {  // uniform: every CTA read the same count after the barrier
        push_big_rows(d, cs.n_big, qb[dst], qn_p, epoch + it);
        target += gridDim.x;
        if (!mid_barrier(d, target, cs, &ctl->n_big, qn_p)) return;
      }
      const int qn = cs.q_next;
      if (tid == 0) {  // both are read again only after the next barrier
        ctl->q_size[src] = 0;
        ctl->n_big = 0;
      }
      T* yd = yb[dst];
      for (int k = tid; k < qn; k += nthreads) {
        const int v = __ldcg(qb[dst] + k);
        if (!OSP_GUARD(ctl, v >= 0 && v < d.nc && qn <= d.nc, "frontier id", k, v, qn)) continue;
        const double x = __ldcg(d.xacc + v);
        d.xacc[v] = 0.0;
        d.r[v] += x;
        l1 += fabs(x);
        yd[v] = (T)(x * __ldg(d.scale_d + v));
        ef += __ldg(d.len_r + v);
      }
    } else {
      l1 = pull_step<T>(d, yb[src], yb[dst], n_hubs, n_pieces, n_tasks,
                        reinterpret_cast<WarpStream<T>*>(dsm)[threadIdx.x >> 5],
                        &ctl->ctr[it & 3], hub_thr, hub_piece,
                        pp.det != 0, d.hub_l1[it & 1]);
    }
    target += gridDim.x;
    if (!step_barrier(d, pp, mode, n, m, l1, ef, target, cs, s_red, s_l1, s_ef)) return;
  }

  // leave both gather vectors all-zero for the next call
  const int k_last = cs.iter;
  if (cs.pull_used) {
    T* a = yb[0];
    T* b = yb[1];
    for (int v = tid; v < n; v += nthreads) {
      a[v] = (T)0;
      b[v] = (T)0;
    }
  } else {
    const int last = k_last & 1;
    const int qs = cs.q_cur;
    for (int k = tid; k < qs; k += nthreads) yb[last][__ldcg(qb[last] + k)] = (T)0;
  }
  if (tid == 0) {
    ctl->epoch = epoch + k_last + 1;
    ctl->iter = k_last;
    ctl->push_iters = cs.push_iters;
    ctl->pull_used = cs.pull_used;
    ctl->noconv = cs.noconv;
    ctl->visited = cs.visited;
    ctl->push_f = cs.push_f;
    ctl->push_r = cs.push_r;
  }
}

template __global__ void k_propagate<double>(Dev, PropParams);
template __global__ void k_propagate<float>(Dev, PropParams);

namespace {
template <typename T>
constexpr int one_smem() { return kOneWarps * (int)sizeof(WarpStream<T>); }
}  // namespace

int propagate_grid(int fp32, int num_sms) {
  const void* fn = fp32 ? (const void*)k_propagate<float> : (const void*)k_propagate<double>;
  const int smem = fp32 ? one_smem<float>() : one_smem<double>();
  int bps = 0;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, fn, kOneThreads, smem) != cudaSuccess ||
      bps <= 0)
    return 0;
  return num_sms > kMaxGrid ? kMaxGrid : num_sms;
}

cudaError_t launch_propagate(const Dev& d, const PropParams& pp, int grid, cudaStream_t s) {
  Dev dd = d;
  PropParams p = pp;
  void* args[] = {&dd, &p};
  const void* fn = pp.fp32 ? (const void*)k_propagate<float> : (const void*)k_propagate<double>;
  const int smem = pp.fp32 ? one_smem<float>() : one_smem<double>();
  return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kOneThreads), args, (size_t)smem, s);
}

}  // namespace osp
