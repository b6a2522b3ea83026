// Delta-merge of the slotted graph store, fused with the offset vector.
//
// Every changed list (out-list row u, or in-list column v) is cut into pieces
// of kPiece old entries, and independent warps handle the pieces in three
// passes, so a hub list costs no more latency than a short one:
//   count  survivors of each piece (an entry goes if the batch deletes it or
//          its other end is a node deleted by the batch); for out-lists the
//          removed entries contribute q_offset[v] += (1-c) r_old[u] (0 - 1/d_u)
//   plan   per list: exclusive scan of its pieces' survivor counts, new length
//          d' = survivors + insertions, fresh pool space, new slot and (for
//          out-lists) the new (1-c)/d'
//   write  survivors go to rank + (insertions below them); each insertion goes
//          to its index + (survivors below it); for out-lists survivors
//          contribute (1-c) r_old[u] (1/d'_u - 1/d_u) and insertions
//          (1-c) r_old[u] / d'_u.
// The contributions add up to q_offset = (1-c) (B~^T - A~^T) r_old over the
// rows where B~ differs from A~ (Sec. 3.1, Algorithm 1 first step; Sec. 3.3:
// only the modified rows contribute). Every node that receives a contribution
// joins the first frontier.
#include "common.cuh"
#include "kernels.h"

namespace osp {
namespace {

// Adds val to the offset of the targets a[r] of this lane whose bit of want[r] is
// set. queue == false: the batch may touch more than n/beta nodes, and x(0) will
// be found by a dense scan of xacc, so no mark or queue entry is made here.
// All rounds of a piece at once: each mark exchange and each append to the queue
// returns a value, and one after the other for eight rounds they were the time
// of the kernels that form the offset (one edge at a hub of 100,003 nodes: 20 ->
// 11 us to write the lists; 1,000 ops at 2^20 nodes: 21 -> 13 us to count them).
template <int R>
__device__ __forceinline__ void offset_add(const Dev& d, const unsigned (&want)[R], int (&a)[R],
                                           double val, int epoch, bool queue) {
  const int lane = threadIdx.x & 31;
  unsigned mine = 0;  // bit r: a[r] is wanted
#pragma unroll
  for (int r = 0; r < R; ++r)
    mine |= (OSP_GUARD(d.ctl, !((want[r] >> lane) & 1u) || (a[r] >= 0 && a[r] < d.nc), "offset target",
                       a[r], 0, 0)
                 ? (want[r] >> lane) & 1u
                 : 0u)
            << r;
  if (d.xfix) {
    // deterministic mode: exact integer sums in units of 2^-62 (|q_offset_v| <=
    // (1-c) ||r_old||_1 < 2, and two's-complement wrap-around leaves partial
    // sums harmless), collected by the x(0) scan, so no queue either
    const unsigned long long q = (unsigned long long)__double2ll_rn(val * 0x1p62);
#pragma unroll
    for (int r = 0; r < R; ++r)
      if ((mine >> r) & 1u) atomicAdd(d.xfix + a[r], q);
    return;
  }
#pragma unroll
  for (int r = 0; r < R; ++r)
    if ((mine >> r) & 1u) atomicAdd(&d.xacc[a[r]], val);
  if (!queue) return;
  int old[R];
#pragma unroll
  for (int r = 0; r < R; ++r) old[r] = (mine >> r) & 1u ? d.mark[a[r]] : epoch;
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (old[r] != epoch) old[r] = atomicExch(&d.mark[a[r]], epoch);
  int total = 0, at[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const unsigned b = __ballot_sync(0xffffffffu, old[r] != epoch);
    at[r] = total + __popc(b & lanemask_lt());
    total += __popc(b);
  }
  if (!total) return;
  int base = 0;
  if (lane == 0) base = atomicAdd(&d.ctl->q_size[0], total);
  base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (old[r] != epoch) d.q0[base + at[r]] = a[r];
}

// One changed list, seen through the combined record index c (out-lists first).
struct ListRec {
  bool rows;
  int node, is, ic, ds, dc;
  const int* ins;
  const int* del;
  int* pool;
};

__device__ __forceinline__ ListRec list_rec(const Dev& d, int c, int n_rows) {
  ListRec L;
  L.rows = c < n_rows;
  const int k = L.rows ? c : c - n_rows;
  if (L.rows) {
    L.node = d.rec_r_node[k];
    L.is = d.rec_r_is[k];
    L.ic = d.rec_r_ic[k];
    L.ds = d.rec_r_ds[k];
    L.dc = d.rec_r_dc[k];
    L.ins = d.ins_r;
    L.del = d.del_r;
    L.pool = d.pool_r;
  } else {
    L.node = d.rec_c_node[k];
    L.is = d.rec_c_is[k];
    L.ic = d.rec_c_ic[k];
    L.ds = d.rec_c_ds[k];
    L.dc = d.rec_c_dc[k];
    L.ins = d.ins_c;
    L.del = d.del_c;
    L.pool = d.pool_c;
  }
  return L;
}

// Old entries of a list go in pieces of kPiece; an empty list has one piece.
__device__ __forceinline__ int pieces_of(int len) { return max(1, (len + kPiece - 1) / kPiece); }

}  // namespace

// List each changed list's pieces and remember its old slot: 1,024 lists a CTA at a
// time, whose pieces get the next places of the table (their order does not
// matter). The CTA that finishes last bounds the offset's support. In one CTA
// 30,000 lists took 34 us, 7 so.
__global__ void __launch_bounds__(1024) k_merge_pieces(Dev d, double beta) {
  __shared__ int s_w[32];
  __shared__ long long s_b[32];
  __shared__ int s_base;
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  const int nr = ctl->n_rec_r;
  const int R = nr + ctl->n_rec_c;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool alone = gridDim.x == 1;  // small batches: no atomics to wait for
  int listed = 0;                     // thread 31: pieces of this CTA
  long long touch = 0;                // out-list entries old and new of the changed rows
  for (int c0 = blockIdx.x * 1024; c0 < R; c0 += gridDim.x * 1024) {
    const int c = c0 + tid;
    int L = 0;
    unsigned o = 0;
    if (c < nr) {
      const int node = d.rec_r_node[c];
      L = d.len_r[node];
      o = d.off_r[node];
      touch += L + d.rec_r_ic[c];
    } else if (c < R) {
      const int node = d.rec_c_node[c - nr];
      L = d.len_c[node];
      o = d.off_c[node];
    }
    const int np = c < R ? pieces_of(L) : 0;
    int x = np;
    for (int k = 1; k < 32; k <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, k);
      if (lane >= k) x += y;
    }
    if (lane == 31) s_w[w] = x;
    __syncthreads();
    if (w == 0) {
      int t = s_w[lane];
      for (int k = 1; k < 32; k <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, t, k);
        if (lane >= k) t += y;
      }
      s_w[lane] = t;
      if (lane == 31) {
        s_base = alone ? listed : atomicAdd(&ctl->n_mpieces, t);
        listed += t;
      }
    }
    __syncthreads();
    const int base = s_base + (w ? s_w[w - 1] : 0) + x - np;
    if (c < R) {
      d.rec_old_off[c] = o;
      d.rec_old_len[c] = L;
      d.rec_pstart[c] = base;
      for (int k = 0; k < np; ++k) d.piece_rec[base + k] = c;
    }
    __syncthreads();
  }
  touch = warp_sum(touch);
  if (lane == 0) s_b[w] = touch;
  if (alone && tid == 31) ctl->n_mpieces = listed;
  __syncthreads();
  if (tid == 0) {
    long long t = 0;
    for (int i = 0; i < 32; ++i) t += s_b[i];
    // the offset reaches at most `touch` nodes; above n/beta the first step is
    // dense anyway and x(0) is collected by a scan instead of a queue (sticky over
    // sub-batches)
    if (alone) {
      ctl->dense0 |= (double)t > (double)ctl->n / beta;
      return;
    }
    if (t) atomicAdd((unsigned long long*)&ctl->touch, (unsigned long long)t);
    __threadfence();
    if (atomicAdd(&ctl->plan_done, 1) == (int)gridDim.x - 1) {
      __threadfence();
      ctl->dense0 |= (double)*(volatile long long*)&ctl->touch > (double)ctl->n / beta;
    }
  }
}

// Survivors per piece; removed out-list entries contribute to q_offset. Four CTAs an SM,
// as many as are launched (built for six it spilled and took 0.3 us longer on 1,000 ops).
__global__ void __launch_bounds__(256, 4) k_merge_count(Dev d) {
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  const int np = ctl->n_mpieces, nr = ctl->n_rec_r;
  const double c1 = 1.0 - ctl->c;
  const int epoch = ctl->epoch;
  const bool queue = !ctl->dense0;
  const bool multi = ctl->multi;
  const bool any_dead = ctl->n_del > 0;  // only nodes deleted by this batch still have edges
  const bool any_clr = ctl->n_clr > 0;   // rows zeroed by this batch
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int p = gw; p < np; p += nw) {
    const int c = d.piece_rec[p];
    const ListRec R = list_rec(d, c, nr);
    const int q = p - d.rec_pstart[c];
    const unsigned o = d.rec_old_off[c];
    const int L = d.rec_old_len[c];
    const bool cleared =
        (any_dead && d.dead[R.node]) || (any_clr && R.rows && d.clr_pos[R.node] >= 0);
    const bool drop_clr = any_clr && !R.rows;  // in-lists drop sources whose row was zeroed
    const double ru = R.rows && !multi ? d.r[R.node] : 0.0;  // the seed block has its own offset kernel
    const bool contrib = R.rows && ru != 0.0;
    const double wa = L ? 1.0 / (double)L : 0.0;
    int cnt = 0, a[kPiece / 32];
    unsigned gone[kPiece / 32];
#pragma unroll
    for (int r = 0; r < kPiece / 32; ++r) {
      const int i = q * kPiece + r * 32 + lane;
      a[r] = i < L ? R.pool[o + i] : 0;
    }
#pragma unroll
    for (int r = 0; r < kPiece / 32; ++r) {
      const int i = q * kPiece + r * 32 + lane;
      const bool in = i < L;
      if (in && !OSP_GUARD(d.ctl, a[r] >= 0 && a[r] < d.nc, "merge count entry", c, i, a[r])) a[r] = 0;
      const bool keep = in && !cleared && !(any_dead && d.dead[a[r]]) &&
                        !(drop_clr && d.clr_pos[a[r]] >= 0) && !contains_i(R.del + R.ds, R.dc, a[r]);
      cnt += __popc(__ballot_sync(0xffffffffu, keep));
      gone[r] = __ballot_sync(0xffffffffu, in && !keep);
    }
    if (contrib && cnt != min(kPiece, L - q * kPiece))
      offset_add(d, gone, a, c1 * ru * (0.0 - wa), epoch, queue);
    if (lane == 0) d.piece_cnt[p] = cnt;
  }
}

// Per list: piece bases, new length, fresh pool space, new slot. Lane = list (the
// warp together for the lists of many pieces), one draw of pool space a warp: a warp
// and a draw per list took 20 us for 30,000 lists, 8 so.
__global__ void __launch_bounds__(256) k_merge_plan(Dev d) {
  constexpr int kAlone = 8;  // pieces that a lane adds up by itself
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  const int nr = ctl->n_rec_r;
  const int R = nr + ctl->n_rec_c;
  const double c1 = 1.0 - ctl->c;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  long long mdelta = 0;
  for (int b = gw * 32; b < R; b += nw * 32) {
    const int c = b + lane;
    const bool in = c < R;
    const bool rows = c < nr;
    int node = 0, ic = 0, p0 = 0, np = 0, old = 0;
    if (in) {
      node = rows ? d.rec_r_node[c] : d.rec_c_node[c - nr];
      ic = rows ? d.rec_r_ic[c] : d.rec_c_ic[c - nr];
      p0 = d.rec_pstart[c];
      old = d.rec_old_len[c];
      np = pieces_of(old);
    }
    int run = 0;
    if (np <= kAlone) {
      for (int k = 0; k < np; ++k) {
        const int v = d.piece_cnt[p0 + k];
        d.piece_base[p0 + k] = run;
        run += v;
      }
    }
    for (unsigned m = __ballot_sync(0xffffffffu, np > kAlone); m; m &= m - 1) {
      const int j = __ffs(m) - 1;
      const int q0 = __shfl_sync(0xffffffffu, p0, j), q1 = q0 + __shfl_sync(0xffffffffu, np, j);
      int sum = 0;
      for (int q = q0; q < q1; q += 32) {  // exclusive scan of the piece counts
        const int p = q + lane;
        const int v = p < q1 ? d.piece_cnt[p] : 0;
        int x = v;
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x += y;
        }
        if (p < q1) d.piece_base[p] = sum + x - v;
        sum += __shfl_sync(0xffffffffu, x, 31);
      }
      if (lane == j) run = sum;
    }
    const int dp = in ? run + ic : 0;
    unsigned long long fb = 0;
#pragma unroll
    for (int kind = 0; kind < 2; ++kind) {  // out-lists, in-lists
      const bool mine = in && rows == (kind == 0);
      long long x = mine ? dp : 0;
      if (!__any_sync(0xffffffffu, x > 0)) continue;
      for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      unsigned long long base = 0;
      if (lane == 31)
        base = atomicAdd(kind == 0 ? &ctl->pool_top_r : &ctl->pool_top_c, (unsigned long long)x);
      base = __shfl_sync(0xffffffffu, base, 31);
      if (mine && dp > 0) fb = base + (unsigned long long)(x - dp);
    }
    if (__any_sync(0xffffffffu,
                   in && fb + (unsigned long long)dp > (rows ? ctl->pool_cap_r : ctl->pool_cap_c))) {
      if (lane == 0) atomicCAS(&ctl->status, 0, (int)OSP_ENOMEM);
      return;
    }
    if (!in) continue;
    d.rec_fbase[c] = (unsigned)fb;
    d.rec_dp[c] = dp;
    if (rows) {
      d.off_r[node] = (unsigned)fb;
      d.len_r[node] = dp;
      const double s = dp ? c1 / (double)dp : 0.0;
      d.scale_d[node] = s;
      d.scale_f[node] = (float)s;
      mdelta += dp - old;
      d.rflag[node] = 0;
    } else {
      d.off_c[node] = (unsigned)fb;
      d.len_c[node] = dp;
      d.cflag[node] = 0;
    }
  }
  mdelta = warp_sum(mdelta);
  if (lane == 0 && mdelta) atomicAdd((unsigned long long*)&ctl->m_delta, (unsigned long long)mdelta);
}

// Survivors and insertions to their final positions; out-list contributions. Four
// CTAs an SM, as many as are launched (an update phase of 1,000 ops at 2^20 nodes
// 131 -> 126 us against the compiler's own three).
__global__ void __launch_bounds__(256, 4) k_merge_write(Dev d) {
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  const int np = ctl->n_mpieces, nr = ctl->n_rec_r;
  const double c1 = 1.0 - ctl->c;
  const int epoch = ctl->epoch;
  const bool queue = !ctl->dense0;
  const bool multi = ctl->multi;
  const bool any_dead = ctl->n_del > 0;
  const bool any_clr = ctl->n_clr > 0;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int p = gw; p < np; p += nw) {
    const int c = d.piece_rec[p];
    const ListRec R = list_rec(d, c, nr);
    const int q = p - d.rec_pstart[c];
    const unsigned o = d.rec_old_off[c];
    const int L = d.rec_old_len[c];
    const int npieces = pieces_of(L);
    const int dp = d.rec_dp[c];
    int* F = R.pool + d.rec_fbase[c];
    const int base = d.piece_base[p];
    const int* I = R.ins + R.is;
    const int ic = R.ic;
    const bool cleared =
        (any_dead && d.dead[R.node]) || (any_clr && R.rows && d.clr_pos[R.node] >= 0);
    const bool drop_clr = any_clr && !R.rows;  // in-lists drop sources whose row was zeroed
    const double ru = R.rows && !multi ? d.r[R.node] : 0.0;  // the seed block has its own offset kernel
    const bool contrib = R.rows && ru != 0.0;
    const double wa = L ? 1.0 / (double)L : 0.0;
    const double wb = dp ? 1.0 / (double)dp : 0.0;
    const bool shift = contrib && dp != L;
    unsigned masks[kPiece / 32];
    int run = 0, a[kPiece / 32];
#pragma unroll
    for (int r = 0; r < kPiece / 32; ++r) {
      const int i = q * kPiece + r * 32 + lane;
      a[r] = i < L ? R.pool[o + i] : 0;
    }
#pragma unroll
    for (int r = 0; r < kPiece / 32; ++r) {
      const int i = q * kPiece + r * 32 + lane;
      const bool in = i < L;
      if (in && !OSP_GUARD(d.ctl, a[r] >= 0 && a[r] < d.nc, "merge write entry", c, i, a[r])) a[r] = 0;
      const bool keep = in && !cleared && !(any_dead && d.dead[a[r]]) &&
                        !(drop_clr && d.clr_pos[a[r]] >= 0) && !contains_i(R.del + R.ds, R.dc, a[r]);
      const unsigned m = __ballot_sync(0xffffffffu, keep);
      masks[r] = m;
      if (keep) {
        const int pos = base + run + __popc(m & lanemask_lt()) + lower_bound_i(I, ic, a[r]);
        if (OSP_GUARD(d.ctl, pos >= 0 && pos < dp, "merge write position", c, pos, dp)) F[pos] = a[r];
      }
      run += __popc(m);
    }
    if (shift && run) offset_add(d, masks, a, c1 * ru * (wb - wa), epoch, queue);
    // insertions that fall inside this piece of the old list
    if (ic > 0) {
      const int* A = R.pool + o;
      const int a0 = q * kPiece;
      const int a1 = min(L, a0 + kPiece);
      const int jlo = q == 0 ? 0 : lower_bound_i(I, ic, A[a0 - 1] + 1);
      // piece q takes the insertions above the old entry before it, up to its own last
      // one (the last piece also those above every old entry): an insertion can equal
      // an old entry of a row that was zeroed before it
      const int jhi = q == npieces - 1 ? ic : lower_bound_i(I, ic, A[a1 - 1] + 1);
      for (int jb = jlo; jb < jhi; jb += 32) {
        const int j = jb + lane;
        const bool in = j < jhi;
        const int e = in ? I[j] : 0;
        if (in) {
          const int t = lower_bound_i(A + a0, a1 - a0, e);  // old entries of this piece below e
          int kept = 0;
#pragma unroll
          for (int r = 0; r < kPiece / 32; ++r) {
            const int lo_r = r * 32;
            if (t >= lo_r + 32) kept += __popc(masks[r]);
            else if (t > lo_r) kept += __popc(masks[r] & ((1u << (t - lo_r)) - 1u));
          }
          if (OSP_GUARD(d.ctl, j + base + kept < dp, "merge insert position", c, j + base + kept, dp))
            F[j + base + kept] = e;
        }
        if (contrib) {
          const unsigned want[1] = {__ballot_sync(0xffffffffu, in)};
          int to[1] = {e};
          offset_add(d, want, to, c1 * ru * (wb - 0.0), epoch, queue);
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Pull-step plan. Warp task t starts at the first node v with
// f(v) = (in-list entries below v) + node_w v >= t task_items (so a task holds
// about task_items items, an edge counting 1 and a node node_w, and never
// splits a list); in-lists longer than hub_thr are listed and cut into pieces.
// Two launches, a range of consecutive nodes a CTA: sums of the ranges,
// then every CTA scans its own range from the sum of those before it. A prefix
// over all nodes in memory, the task starts from it and the pieces were six
// launches, with two 64-bit divisions a node; an update phase of 1,000 edge ops
// at 2^20 nodes took 142 us with them and 126 so, of 100 at 10,000 nodes 85 and
// 73 (with the offset above).
// ---------------------------------------------------------------------------
namespace {
constexpr int kPlanThreads = 1024;

// Nodes [lo, hi) of this CTA: a multiple of four each, but for the last.
__device__ __forceinline__ void plan_range(int n, int& lo, int& hi) {
  const long long per = (((long long)n + gridDim.x - 1) / gridDim.x + 3) & ~3ll;
  lo = (int)min((long long)n, per * blockIdx.x);
  hi = (int)min((long long)n, per * (blockIdx.x + 1));
}

// a[v .. v + 4), zero from hi on (v a multiple of four)
__device__ __forceinline__ int4 load4(const int* a, int v, int hi) {
  if (v + 4 <= hi) return *reinterpret_cast<const int4*>(a + v);
  return make_int4(v < hi ? a[v] : 0, v + 1 < hi ? a[v + 1] : 0, v + 2 < hi ? a[v + 2] : 0, 0);
}
}  // namespace

// In-list entries of each CTA's nodes; nodes with a nonempty list of either kind
// (byte accounting). Folds the batch's edge-count change into m.
__global__ void __launch_bounds__(kPlanThreads) k_plan_sums(Dev d, unsigned* part) {
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ctl->m += ctl->m_delta;
    ctl->m_delta = 0;
    ctl->n_hubs = 0;
    ctl->plan_done = 0;
    // a dense first frontier is rebuilt by the x(0) scan: drop entries queued by
    // earlier sub-batches of the same batch
    if (ctl->dense0) ctl->q_size[0] = 0;
  }
  int lo, hi;
  plan_range(ctl->n, lo, hi);
  unsigned sum = 0, nd = 0, ns = 0;
  for (int v = lo + 4 * (int)threadIdx.x; v < hi; v += 4 * kPlanThreads) {
    const int4 a = load4(d.len_c, v, hi), b = load4(d.len_r, v, hi);
    sum += (unsigned)a.x + (unsigned)a.y + (unsigned)a.z + (unsigned)a.w;
    nd += (a.x > 0) + (a.y > 0) + (a.z > 0) + (a.w > 0);
    ns += (b.x > 0) + (b.y > 0) + (b.z > 0) + (b.w > 0);
  }
  __shared__ unsigned s_sum[3];
  if (threadIdx.x < 3) s_sum[threadIdx.x] = 0;
  __syncthreads();
  sum = __reduce_add_sync(0xffffffffu, sum);
  nd = __reduce_add_sync(0xffffffffu, nd);
  ns = __reduce_add_sync(0xffffffffu, ns);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&s_sum[0], sum);
    atomicAdd(&s_sum[1], nd);
    atomicAdd(&s_sum[2], ns);
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  part[blockIdx.x] = s_sum[0];
  if (s_sum[1]) atomicAdd((unsigned long long*)&ctl->n_dst_nz, (unsigned long long)s_sum[1]);
  if (s_sum[2]) atomicAdd((unsigned long long*)&ctl->n_src_nz, (unsigned long long)s_sum[2]);
}

// Task starts and long lists of each CTA's nodes; the CTA that finishes last cuts
// the long lists into pieces. Small graphs get shorter tasks, down to task_min
// items, so that `want` warps have one each.
// det: the long lists, listed in whatever order the CTAs ran, are rebuilt in
// ascending node order (one ordered compaction over all nodes), so that the
// pieces and the per-list norm slots have the same positions on every run.
__global__ void __launch_bounds__(kPlanThreads)
    k_pull_plan(Dev d, const unsigned* __restrict__ part, int hub_thr, int hub_piece, int node_w,
                int task_items, int task_min, int want, int det) {
  __shared__ int s_w[32];
  __shared__ int s_base;
  __shared__ long long s_f;
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  {
    const int n = ctl->n;
    const long long W = (long long)node_w * n + ctl->m;
    task_items = (int)min((long long)task_items, max((long long)task_min, (W + want - 1) / want));
    const int nt = (int)((W + task_items - 1) / task_items);
    if (blockIdx.x == 0 && tid == 0) {
      ctl->n_tasks = nt;
      ctl->hub_thr = hub_thr;
      ctl->hub_piece = hub_piece;
      d.task_first[0] = 0;
      d.task_first[nt] = n;
    }
    int lo, hi;
    plan_range(n, lo, hi);
    unsigned before = 0;
    for (int b = tid; b < (int)blockIdx.x; b += kPlanThreads) before += part[b];
    int4 a = load4(d.len_c, lo + 4 * tid, hi);
    if (tid == 0) s_f = (long long)node_w * lo;
    __syncthreads();
    before = __reduce_add_sync(0xffffffffu, before);
    if (before && lane == 0) atomicAdd((unsigned long long*)&s_f, (unsigned long long)before);
    for (int v0 = lo; v0 < hi; v0 += 4 * kPlanThreads) {
      const int v = v0 + 4 * tid;
      if (v0 > lo) a = load4(d.len_c, v, hi);
      const int len[4] = {a.x, a.y, a.z, a.w};
      const unsigned mine = (unsigned)a.x + (unsigned)a.y + (unsigned)a.z + (unsigned)a.w;
      unsigned x = mine;
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) s_w[w] = (int)x;
      __syncthreads();
      if (w == 0) {
        unsigned t = (unsigned)s_w[lane];
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned y = __shfl_up_sync(0xffffffffu, t, o);
          if (lane >= o) t += y;
        }
        s_w[lane] = (int)t;
      }
      __syncthreads();
      // f at this thread's first node; the nodes of the tile before it count node_w each
      long long f = s_f + (w ? (unsigned)s_w[w - 1] : 0u) + (x - mine) + (long long)node_w * (4 * tid);
      const unsigned total = (unsigned)s_w[31];
      if (v < hi) {
        // boundaries t task_items in (f(u), f(u + 1)] start at node u + 1
        long long t = W <= 0xffffffffll ? (long long)((unsigned)f / (unsigned)task_items) : f / task_items;
        long long at = (t + 1) * task_items;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (v + q >= hi) break;
          f += len[q] + node_w;
          for (; at <= f && t + 1 < nt; at += task_items) d.task_first[++t] = v + q + 1;
          if (len[q] > hub_thr) d.hubs[atomicAdd(&ctl->n_hubs, 1)] = v + q;
        }
      }
      if (v0 + 4 * kPlanThreads >= hi) break;
      __syncthreads();
      if (tid == 0) s_f += total + (long long)node_w * (4 * kPlanThreads);
      __syncthreads();
    }
  }
  // the last CTA has every long list
  __threadfence();
  __syncthreads();
  if (tid == 0) s_base = atomicAdd(&ctl->plan_done, 1);
  __syncthreads();
  if (s_base != (int)gridDim.x - 1) return;
  __threadfence();
  __syncthreads();
  if (det) {
    const int n = ctl->n;
    if (tid == 0) s_base = 0;
    __syncthreads();
    for (int b0 = 0; b0 < n; b0 += 1024) {
      const int v = b0 + tid;
      const bool h = v < n && d.len_c[v] > hub_thr;
      const unsigned bm = __ballot_sync(0xffffffffu, h);
      if (lane == 0) s_w[w] = __popc(bm);
      __syncthreads();
      if (w == 0) {
        int x = s_w[lane];
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x += y;
        }
        s_w[lane] = x;
      }
      __syncthreads();
      if (h) d.hubs[s_base + (w ? s_w[w - 1] : 0) + __popc(bm & lanemask_lt())] = v;
      __syncthreads();
      if (tid == 0) s_base += s_w[31];
      __syncthreads();
    }
  }
  const int nh = *(volatile int*)&ctl->n_hubs;
  const int per = (nh + 1023) / 1024;
  const int lo = min(nh, tid * per), hi = min(nh, lo + per);
  int mine = 0;
  for (int h = lo; h < hi; ++h) mine += (d.len_c[d.hubs[h]] + hub_piece - 1) / hub_piece;
  int x = mine;
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[w] = x;
  __syncthreads();
  if (w == 0) {
    int t = s_w[lane];
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    s_w[lane] = t;
  }
  __syncthreads();
  int base = (w ? s_w[w - 1] : 0) + x - mine;
  for (int h = lo; h < hi; ++h) {
    d.hub_pstart[h] = base;
    const int np = (d.len_c[d.hubs[h]] + hub_piece - 1) / hub_piece;
    for (int q = 0; q < np; ++q) d.piece_hub[base + q] = h;  // a piece finds its list in one load
    base += np;
    d.hub_acc[h] = 0.0;
    d.hub_cnt[h] = 0;
  }
  if (tid == 0) {
    d.hub_pstart[nh] = s_w[31];
    ctl->n_pieces = s_w[31];
  }
}

// (1-c) / d_u for every node (0 for dead-ends).
__global__ void k_set_scale(Dev d, int n, double c) {
  for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
    const int l = d.len_r[u];
    const double s = l ? (1.0 - c) / (double)l : 0.0;
    d.scale_d[u] = s;
    d.scale_f[u] = (float)s;
  }
}

// ---------------------------------------------------------------------------
// Compaction: exclusive scan of list lengths, then one warp per list copies it.
// ---------------------------------------------------------------------------
constexpr int kScanPer = 4;
constexpr int kScanTile = 1024 * kScanPer;

__global__ void __launch_bounds__(1024) k_scan_local(const int* __restrict__ len, unsigned* out,
                                                     unsigned* bsum, int n) {
  __shared__ unsigned s_w[32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int base = blockIdx.x * kScanTile + tid * kScanPer;
  unsigned v[kScanPer];
  unsigned mine = 0;
#pragma unroll
  for (int k = 0; k < kScanPer; ++k) {
    v[k] = base + k < n ? (unsigned)len[base + k] : 0u;
    mine += v[k];
  }
  unsigned x = mine;
  for (int o = 1; o < 32; o <<= 1) {
    unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[w] = x;
  __syncthreads();
  if (w == 0) {
    unsigned t = s_w[lane];
    for (int o = 1; o < 32; o <<= 1) {
      unsigned y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    s_w[lane] = t;
  }
  __syncthreads();
  unsigned run = (w ? s_w[w - 1] : 0u) + x - mine;
#pragma unroll
  for (int k = 0; k < kScanPer; ++k) {
    if (base + k < n) out[base + k] = run;
    run += v[k];
  }
  if (tid == 0) bsum[blockIdx.x] = s_w[31];
}

__global__ void __launch_bounds__(1024) k_scan_top(unsigned* bsum, int nb) {
  __shared__ unsigned s_w[32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int per = (nb + 1023) / 1024;
  const int lo = min(nb, tid * per), hi = min(nb, lo + per);
  unsigned mine = 0;
  for (int i = lo; i < hi; ++i) mine += bsum[i];
  unsigned x = mine;
  for (int o = 1; o < 32; o <<= 1) {
    unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[w] = x;
  __syncthreads();
  if (w == 0) {
    unsigned t = s_w[lane];
    for (int o = 1; o < 32; o <<= 1) {
      unsigned y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    s_w[lane] = t;
  }
  __syncthreads();
  unsigned run = (w ? s_w[w - 1] : 0u) + x - mine;
  for (int i = lo; i < hi; ++i) {
    unsigned t = bsum[i];
    bsum[i] = run;
    run += t;
  }
}

__global__ void k_scan_add(unsigned* out, const unsigned* __restrict__ bsum, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] += bsum[i / kScanTile];
}

// A warp copies kCopyChunk entries of the new pool, whichever lists they belong
// to (a warp per list had the longest list's copy as its time: 225 us for 3 M
// entries): the first list by binary search, then 32 lists at a time as one
// stream of entries, four rounds of 32 in flight.
constexpr int kCopyChunk = 1024;
__global__ void __launch_bounds__(256) k_compact_copy(const unsigned* __restrict__ off_old,
                                                      const int* __restrict__ len,
                                                      const int* __restrict__ pool_old,
                                                      const unsigned* __restrict__ off_new,
                                                      int* pool_new, int n) {
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  const unsigned m = off_new[n - 1] + (unsigned)len[n - 1];
  for (long long c0 = (long long)gw * kCopyChunk; c0 < (long long)m; c0 += (long long)nw * kCopyChunk) {
    const unsigned p0 = (unsigned)c0, p1 = min(m, p0 + kCopyChunk);
    int lo = 0, hi = n - 1;  // the last list that starts at or before p0
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (off_new[mid] <= p0) lo = mid;
      else hi = mid - 1;
    }
    unsigned p = p0;
    for (int u0 = lo; p < p1; u0 += 32) {
      const int u = u0 + lane;
      const unsigned b = u < n ? off_new[u] : m;       // ascending over the lanes
      const unsigned a = u < n ? off_old[u] : 0u;
      const unsigned end = min(p1, u0 + 32 < n ? off_new[u0 + 32] : m);
      for (; p < end; p += 128) {
        unsigned from[4];
        int v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const unsigned e = p + 32 * r + lane;
          int l = 0;  // the last lane whose list starts at or before e
#pragma unroll
          for (int q = 16; q > 0; q >>= 1) {
            const unsigned bm = __shfl_sync(0xffffffffu, b, l + q);
            if (bm <= e) l += q;
          }
          from[r] = __shfl_sync(0xffffffffu, a, l) + (e - __shfl_sync(0xffffffffu, b, l));
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = p + 32 * r + lane < end ? pool_old[from[r]] : 0;
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (p + 32 * r + lane < end) pool_new[p + 32 * r + lane] = v[r];
      }
      p = end;
    }
  }
}

// ||r||_1 and r / ||r||_1. With parts == nullptr the per-CTA partials are
// added atomically into *out (cleared by the caller); otherwise each CTA
// stores its partial in parts[blockIdx.x] and the last CTA to finish adds them
// in index order into *out, so the norm has the same bits on every run.
// parts[kAbsParts] (as an unsigned int) counts finished CTAs; the grid must
// not exceed kAbsParts, and the last CTA resets the count.
__global__ void k_abs_sum(const double* __restrict__ r, int n, double* out, double* parts) {
  double s = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    s += fabs(r[i]);
  s = warp_sum(s);
  __shared__ double sw[32];
  __shared__ bool s_last;
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = threadIdx.x < (blockDim.x >> 5) ? sw[threadIdx.x] : 0.0;
    t = warp_sum(t);
    if (threadIdx.x == 0) {
      if (!parts) {
        atomicAdd(out, t);
      } else {
        parts[blockIdx.x] = t;
        __threadfence();
        unsigned* cnt = (unsigned*)(parts + kAbsParts);
        s_last = atomicAdd(cnt, 1u) == gridDim.x - 1;
      }
    }
  }
  if (!parts) return;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (threadIdx.x < 32) {
    double t = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += 32) t += __ldcg(parts + i);
    t = warp_sum(t);
    if (threadIdx.x == 0) {
      *out = t;
      *(unsigned*)(parts + kAbsParts) = 0u;
    }
  }
}

// Scores in caller order: out[x] = r[ext2int[x]].
__global__ void k_gather_ext(const double* __restrict__ r, const int* __restrict__ ext2int, int n,
                             double* out) {
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += gridDim.x * blockDim.x)
    out[x] = r[ext2int[x]];
}

__global__ void k_scale_copy(const double* r, int n, const double* __restrict__ sum, double* out) {
  const double s = *sum;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = s > 0.0 ? r[i] / s : 0.0;
}

}  // namespace osp
