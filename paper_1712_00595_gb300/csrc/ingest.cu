// Batch ingest: validation, canonical ordering and net edits (one CTA up to kIngestOne
// ops, many above), then the expansion of node deletions to the rows and columns they
// touch.
//
// Semantics (osp.h): ops apply in order; the net effect on an edge (u,v) is
// the last edge op naming it, unless u or v is deleted by the batch, in which
// case the edge is gone. Delta A (Algorithm 1) is therefore "rows after the
// whole batch minus rows before it" (Sec. 3.1, Sec. 3.4.1).
#include "common.cuh"
#include "kernels.h"

namespace osp {
namespace {

constexpr unsigned long long kNoKey = ~0ull;
constexpr int kIngestThreads = 1024;

// Exclusive scan over a 1024-thread block. Returns the prefix; *total gets the sum.
__device__ int block_exscan(int v, int* total) {
  __shared__ int s_w[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[w] = x;
  __syncthreads();
  if (w == 0) {
    int t = s_w[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    s_w[lane] = t;
  }
  __syncthreads();
  int res = (w ? s_w[w - 1] : 0) + x - v;
  *total = s_w[31];
  __syncthreads();
  return res;
}

// In-place ascending bitonic sort of N (a power of two) keys in shared memory.
__device__ void bitonic_sort(unsigned long long* a, int N) {
  for (int k = 2; k <= N; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < (N >> 1); t += blockDim.x) {
        int lo = ((t & ~(j - 1)) << 1) | (t & (j - 1));
        int hi = lo | j;
        bool asc = (lo & k) == 0;
        unsigned long long x = a[lo], y = a[hi];
        if ((x > y) == asc) {
          a[lo] = y;
          a[hi] = x;
        }
      }
      __syncthreads();
    }
  }
}

// An op with its node ids mapped to the engine's internal order. The map is a
// permutation of the loaded ids and the identity above them, so an id is in
// range before the mapping exactly when it is in range after it.
__device__ __forceinline__ osp_update load_op(const osp_update* ops, int p, const Dev& d) {
  osp_update o = ops[p];
  if (o.u >= 0 && o.u < d.nc) o.u = d.ext2int[o.u];
  if (o.v >= 0 && o.v < d.nc) o.v = d.ext2int[o.v];
  return o;
}

__device__ __forceinline__ int next_pow2(int x) {
  int p = 2;
  while (p < x) p <<= 1;
  return p;
}

// From N sorted keys whose per-position edit flags are known, write the
// insert / delete lists (ascending within each group) and one record per
// group that has at least one edit. group_of(key) gives the group node,
// member_of(key) the list value. flags[k] for k < per: bit0 insert, bit1 delete.
template <typename GroupF, typename MemberF>
__device__ void emit_groups(const unsigned long long* skey, int N, int per, int pi0,
                            const unsigned* flagbits, GroupF group_of, MemberF member_of,
                            int* ins_out, int* del_out, int* gi, int* gd, int* rec_node,
                            int* rec_is, int* rec_ic, int* rec_ds, int* rec_dc, int* flag_arr,
                            int* n_rec_out, long long* n_ins_out, long long* n_del_out) {
  unsigned fb = *flagbits;
  int my_ins = 0, my_del = 0;
  for (int k = 0; k < per; ++k) {
    my_ins += (fb >> (2 * k)) & 1;
    my_del += (fb >> (2 * k + 1)) & 1;
  }
  int tot_ins, tot_del;
  int ib = block_exscan(my_ins, &tot_ins);
  int db = block_exscan(my_del, &tot_del);
  for (int k = 0; k < per; ++k) {
    int i = pi0 + k;
    if (i >= N) break;
    gi[i] = ib;
    gd[i] = db;
    unsigned long long key = skey[i];
    if ((fb >> (2 * k)) & 1) ins_out[ib++] = member_of(key);
    if ((fb >> (2 * k + 1)) & 1) del_out[db++] = member_of(key);
  }
  if (threadIdx.x == 0) {
    gi[N] = tot_ins;
    gd[N] = tot_del;
  }
  __syncthreads();
  // one record per group (equal group node) holding at least one edit
  int my_rec = 0;
  for (int pass = 0; pass < 2; ++pass) {
    int rb = 0;
    if (pass == 1) {
      int tot_rec;
      rb = block_exscan(my_rec, &tot_rec);
      if (threadIdx.x == 0) *n_rec_out = tot_rec;
    }
    for (int k = 0; k < per; ++k) {
      int i = pi0 + k;
      if (i >= N) break;
      unsigned long long key = skey[i];
      if (key == kNoKey) break;
      int g = group_of(key);
      if (i > 0 && group_of(skey[i - 1]) == g) continue;
      int j = i;
      while (j + 1 < N && skey[j + 1] != kNoKey && group_of(skey[j + 1]) == g) ++j;
      int ic = gi[j + 1] - gi[i], dc = gd[j + 1] - gd[i];
      if (ic + dc == 0) continue;
      if (pass == 0) {
        ++my_rec;
      } else {
        rec_node[rb] = g;
        rec_is[rb] = gi[i];
        rec_ic[rb] = ic;
        rec_ds[rb] = gd[i];
        rec_dc[rb] = dc;
        flag_arr[g] = 1;
        ++rb;
      }
    }
  }
  if (threadIdx.x == 0) {
    *n_ins_out = tot_ins;
    *n_del_out = tot_del;
  }
  __syncthreads();
}

}  // namespace

// cont != 0: a later sub-batch of one large batch. The offset accumulated so
// far (xacc, stamps, first frontier), the edge-count change and the edit
// counts carry over; only the per-sub-batch records restart.
__global__ void k_reset_batch(Dev d, int cont) {
  Ctl* c = d.ctl;
  // rows zeroed by the previous batch (merged by now) lose their mark
  for (int i = threadIdx.x; i < c->n_clr; i += blockDim.x) d.clr_pos[d.clr_nodes[i]] = -1;
  if (threadIdx.x != 0) return;
  c->ing_bad = kNoPos;
  c->ing_clr = 0;
  c->ing_reins = 0;
  c->status = 0;
  c->bad_op = -1;
  c->n_old = c->n;
  c->n_rec_r = 0;
  c->n_rec_c = 0;
  c->n_del = 0;
  c->n_mpieces = 0;
  c->plan_done = 0;
  c->touch = 0;
  if (cont) return;
  c->m_delta = 0;
  c->net_ins = 0;
  c->net_del = 0;
  c->n_rec_r = 0;
  c->n_rec_c = 0;
  c->n_del = 0;
  c->q_size[0] = 0;
  c->q_size[1] = 0;
  c->dense0 = 0;
  c->n_dst_nz = 0;
  c->n_src_nz = 0;
  for (int i = 0; i < 4; ++i) c->ctr[i] = 0;
  c->n_big = 0;
  c->bar_count = 0;
  d.bar[0] = 0;
  c->iter = 0;
  c->mode = kPush;
  c->push_iters = 0;
  c->stop = 0;
  c->pull_used = 0;
  c->noconv = 0;
  c->visited = 0;
  c->ef = 0;
  c->push_f = 0;
  c->push_r = 0;
}

// CPI start (Sec. 2.2): x(0) = c e_s, r = 0 before the propagation adds x(0).
// CPI start with the uniform restart vector q = 1/n0 over nodes 0..n0-1
// (PageRank mode): x(0) = c q, collected by the dense x(0) scan.
__global__ void k_cpi_begin_uniform(Dev d, int n0) {
  Ctl* c = d.ctl;
  const double x = c->c / (double)n0;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n0; v += gridDim.x * blockDim.x)
    d.xacc[v] = x;
  if (blockIdx.x == 0 && threadIdx.x == 0) c->dense0 = 1;
}

__global__ void k_cpi_begin(Dev d) {
  Ctl* c = d.ctl;
  int s = c->seed;
  d.xacc[s] = c->c;
  d.mark[s] = c->epoch;
  d.q0[0] = s;
  c->q_size[0] = 1;
}

// At most kIngestOne ops: one a thread.
static_assert(kIngestOne <= kIngestThreads, "k_ingest's keys and flags");
__global__ void __launch_bounds__(kIngestThreads) k_ingest(Dev d, const osp_update* __restrict__ ops,
                                                           int U) {
  extern __shared__ unsigned long long skey[];
  __shared__ int s_bad, s_ndel, s_nclr, s_anyclr;
  __shared__ long long s_reins;
  __shared__ unsigned s_flags[kIngestThreads];
  Ctl* ctl = d.ctl;
  if (U < 0) U = ctl->batch_U;  // replayed from a CUDA graph: the size is set per call
  const int tid = threadIdx.x;
  const int n_old = ctl->n;
  if (tid == 0) {
    s_bad = kNoPos;
    s_ndel = 0;
    s_nclr = 0;
    s_anyclr = 0;
    s_reins = 0;
  }
  __syncthreads();

  // ---- validation (sequential rules checked in parallel) ----
  const int per_op = (U + kIngestThreads - 1) / kIngestThreads;
  const int lo = min(U, tid * per_op), hi = min(U, lo + per_op);
  int adds = 0;
  for (int p = lo; p < hi; ++p) adds += ops[p].op == OSP_OP_ADD_NODE;
  int tot_adds;
  const int add_base = block_exscan(adds, &tot_adds);
  int run = add_base;
  for (int p = lo; p < hi; ++p) {
    osp_update o = load_op(ops, p, d);
    if (o.op == OSP_OP_ADD_NODE) {
      ++run;
    } else if (o.op == OSP_OP_DELETE_NODE) {
      const int na = n_old + run;
      const int w = o.u;
      if (w >= 0 && w < na && !d.dead[w] && !d.seedflag[w]) atomicMin(&d.del_pos[w], p);
      else atomicMin(&s_bad, p);
    } else if (o.op == OSP_OP_ZERO_ROW) {
      // the last zeroing of a row in the batch voids the row's earlier edge ops
      s_anyclr = 1;
      if (o.u >= 0 && o.u < n_old + run) atomicMax(&d.clr_pos[o.u], p);
      else atomicMin(&s_bad, p);
    }
  }
  __syncthreads();
  run = add_base;
  for (int p = lo; p < hi; ++p) {
    osp_update o = load_op(ops, p, d);
    const int na = n_old + run;
    bool ok;
    if (o.op == OSP_OP_INSERT_EDGE || o.op == OSP_OP_DELETE_EDGE) {
      ok = o.u >= 0 && o.u < na && o.v >= 0 && o.v < na && !d.dead[o.u] && !d.dead[o.v] &&
           d.del_pos[o.u] > p && d.del_pos[o.v] > p;
    } else if (o.op == OSP_OP_ADD_NODE) {
      ok = true;
      ++run;
    } else if (o.op == OSP_OP_DELETE_NODE) {
      ok = o.u >= 0 && o.u < na && !d.dead[o.u] && !d.seedflag[o.u] && d.del_pos[o.u] == p;
    } else if (o.op == OSP_OP_ZERO_ROW) {
      ok = o.u >= 0 && o.u < na && !d.dead[o.u] && d.del_pos[o.u] > p;
    } else {
      ok = false;
    }
    if (!ok) atomicMin(&s_bad, p);
  }
  __syncthreads();
  if (s_bad != kNoPos) {
    for (int p = lo; p < hi; ++p) {
      const int op = ops[p].op;
      if (op == OSP_OP_DELETE_NODE || op == OSP_OP_ZERO_ROW) {
        const osp_update o = load_op(ops, p, d);
        if (o.u >= 0 && o.u < d.nc) {
          if (op == OSP_OP_DELETE_NODE) d.del_pos[o.u] = kNoPos;
          else d.clr_pos[o.u] = -1;
        }
      }
    }
    if (tid == 0) {
      ctl->status = OSP_EINVAL;
      ctl->bad_op = s_bad;
      ctl->n_clr = 0;
    }
    return;
  }

  // ---- canonical order: sort edge ops by (u, v, position) ----
  const int N = next_pow2(U);
  for (int p = lo; p < hi; ++p) {
    osp_update o = load_op(ops, p, d);
    unsigned long long key = kNoKey;
    if ((o.op == OSP_OP_INSERT_EDGE || o.op == OSP_OP_DELETE_EDGE) && d.del_pos[o.u] == kNoPos &&
        d.del_pos[o.v] == kNoPos && (!s_anyclr || d.clr_pos[o.u] < p))
      key = ((unsigned long long)o.u << 39) | ((unsigned long long)o.v << 14) | (unsigned)p;
    skey[p] = key;
  }
  for (int i = U + tid; i < N; i += kIngestThreads) skey[i] = kNoKey;
  __syncthreads();
  bitonic_sort(skey, N);

  // ---- net edits: the last op of each (u, v) against the current row ----
  const int per = max(1, N / kIngestThreads);
  const int pi0 = tid * per;
  unsigned fb = 0;
  int reins = 0;
  for (int k = 0; k < per; ++k) {
    int i = pi0 + k;
    if (i >= N) break;
    unsigned long long key = skey[i];
    if (key == kNoKey) break;
    bool last = (i == N - 1) || ((skey[i + 1] >> 14) != (key >> 14));
    if (!last) continue;
    int p = (int)(key & 0x3FFF);
    int u = (int)(key >> 39);
    int v = (int)((key >> 14) & 0x1FFFFFF);
    bool present_after = ops[p].op == OSP_OP_INSERT_EDGE;
    bool present_before = false;
    if (u < n_old && v < n_old) {
      // u -> v exists iff v is in u's out-list, or u in v's in-list: search the shorter
      const int lr = d.len_r[u], lc = d.len_c[v];
      present_before = lr <= lc ? contains_i(d.pool_r + d.off_r[u], lr, v)
                                : contains_i(d.pool_c + d.off_c[v], lc, u);
    }
    if (s_anyclr && d.clr_pos[u] >= 0) {
      // u's row was zeroed before this op: the merge drops every old entry of
      // the row (and u from the old in-lists), so a surviving edge is written
      // again as an insertion, but it is not a new edge
      reins += present_after && present_before;
      present_before = false;
    }
    if (present_after && !present_before) fb |= 1u << (2 * k);
    if (!present_after && present_before) fb |= 2u << (2 * k);
  }
  s_flags[tid] = fb;
  if (reins) atomicAdd((unsigned long long*)&s_reins, (unsigned long long)reins);
  long long n_ins = 0, n_del = 0;
  emit_groups(
      skey, N, per, pi0, &s_flags[tid], [](unsigned long long k) { return (int)(k >> 39); },
      [](unsigned long long k) { return (int)((k >> 14) & 0x1FFFFFF); }, d.ins_r, d.del_r, d.gi,
      d.gd, d.rec_r_node, d.rec_r_is, d.rec_r_ic, d.rec_r_ds, d.rec_r_dc, d.rflag, &ctl->n_rec_r,
      &n_ins, &n_del);
  if (tid == 0) {  // summed over the sub-batches of a large batch
    ctl->net_ins += n_ins - s_reins;
    ctl->net_del += n_del;
  }

  // ---- the same edits keyed (v, u) for the in-lists ----
  // edit e of row u (in row order) -> key (v << 32) | (u << 1) | is_delete
  unsigned long long my_keys[16];
  int my_nk = 0;
  for (int k = 0; k < per && k < 16; ++k) {
    int i = pi0 + k;
    if (i >= N) break;
    if (!((fb >> (2 * k)) & 3)) continue;
    unsigned long long key = skey[i];
    unsigned long long u = key >> 39, v = (key >> 14) & 0x1FFFFFF;
    my_keys[my_nk++] = (v << 32) | (u << 1) | ((fb >> (2 * k + 1)) & 1);
  }
  int tot_e;
  const int ebase = block_exscan(my_nk, &tot_e);  // also orders the reads of skey above
  for (int t = 0; t < my_nk; ++t) skey[ebase + t] = my_keys[t];
  const int N2 = next_pow2(tot_e);
  for (int i = tot_e + tid; i < N2; i += kIngestThreads) skey[i] = kNoKey;
  __syncthreads();
  bitonic_sort(skey, N2);
  const int per2 = max(1, N2 / kIngestThreads);
  const int pj0 = tid * per2;
  unsigned fb2 = 0;
  for (int k = 0; k < per2; ++k) {
    int i = pj0 + k;
    if (i >= N2) break;
    unsigned long long key = skey[i];
    if (key == kNoKey) break;
    fb2 |= ((key & 1) ? 2u : 1u) << (2 * k);
  }
  s_flags[tid] = fb2;
  __syncthreads();
  long long c_ins = 0, c_del = 0;
  emit_groups(
      skey, N2, per2, pj0, &s_flags[tid], [](unsigned long long k) { return (int)(k >> 32); },
      [](unsigned long long k) { return (int)((unsigned)k >> 1); }, d.ins_c, d.del_c, d.gi, d.gd,
      d.rec_c_node, d.rec_c_is, d.rec_c_ic, d.rec_c_ds, d.rec_c_dc, d.cflag, &ctl->n_rec_c, &c_ins,
      &c_del);

  // ---- node deletions and additions ----
  for (int p = lo; p < hi; ++p) {
    if (ops[p].op == OSP_OP_DELETE_NODE) d.del_nodes[atomicAdd(&s_ndel, 1)] = load_op(ops, p, d).u;
    if (s_anyclr && ops[p].op == OSP_OP_ZERO_ROW) {
      const int u = load_op(ops, p, d).u;
      if (d.clr_pos[u] == p) d.clr_nodes[atomicAdd(&s_nclr, 1)] = u;  // once per row
    }
  }
  __syncthreads();
  for (int p = lo; p < hi; ++p)
    if (ops[p].op == OSP_OP_DELETE_NODE) d.del_pos[load_op(ops, p, d).u] = kNoPos;
  if (tid == 0) {
    ctl->n_del = s_ndel;
    ctl->n_clr = s_nclr;
    ctl->n = n_old + tot_adds;
  }
}

// ---------------------------------------------------------------------------
// Larger batches (more than kIngestOne ops): the same steps over many CTAs. One
// CTA spent 760 us on 10,001 ops and 867 us on 15,000: two bitonic sorts (105
// passes of 16,384 keys through shared memory each), the existence searches
// (some 14 scattered loads an op from one SM) and 16 ops a thread one after the
// other. Here all but the emission runs one op a thread, and two CTAs emit the
// lists, one sorting the edits for the columns by stable 8-bit radix passes over the
// bits in use.
//   k_ingest_scan   node count before each op; first deletion, last zeroing
//   k_ingest_keys   validation; sort keys (u, v, position)
//   k_ingest_rank   their order (or the report of the first invalid op)
//   k_ingest_edits  last op of each pair against the current row: net edits
//   k_ingest_emit   edit lists and records of rows, the same sorted for columns
// ---------------------------------------------------------------------------
namespace {

constexpr int kSortRows = kMaxBatch / kIngestThreads;  // keys a thread
constexpr unsigned long long kLastKeys = ~0ull << 14;    // ops without an edge, by position

// Bits of a node id among n nodes, so that no id has all of them set.
__device__ __forceinline__ int id_bits(int n) { return 32 - __clz(n); }

// Stable radix sort of `per` * 1024 keys by bits [lo, hi), eight a pass. Thread
// (warp w, lane l) holds keys w per 32 + 32 r + l, r < per, before and after.
// s_key: the keys' buffer; s_cnt: 32 x 256 counts.
__device__ void radix_sort(unsigned long long (&key)[kSortRows], int per, int lo, int hi,
                           unsigned long long* s_key, int* s_cnt) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int sh = lo; sh < hi; sh += 8) {
    const unsigned mask = (1u << min(8, hi - sh)) - 1u;
    for (int i = tid; i < 32 * 256; i += kIngestThreads) s_cnt[i] = 0;
    __syncthreads();
    unsigned rank[kSortRows / 2];  // two 16-bit ranks a register
#pragma unroll
    for (int r = 0; r < kSortRows; ++r) {
      if (r >= per) break;
      const unsigned dg = (unsigned)(key[r] >> sh) & mask;
      unsigned peers = 0xffffffffu;  // lanes with this digit, a ballot a bit
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        const unsigned v = __ballot_sync(0xffffffffu, (dg >> b) & 1u);
        peers &= (dg >> b) & 1u ? v : ~v;
      }
      const int leader = __ffs(peers) - 1;
      int old = 0;
      if (lane == leader) {
        old = s_cnt[w * 256 + dg];
        s_cnt[w * 256 + dg] = old + __popc(peers);
      }
      __syncwarp();
      const unsigned rk = __shfl_sync(0xffffffffu, old, leader) + __popc(peers & lanemask_lt());
      rank[r / 2] = r & 1 ? rank[r / 2] | rk << 16 : rk;
    }
    __syncthreads();
    // exclusive scan, digits first, then warps: thread t owns warps 8 (t % 4) ..
    // of digit t / 4
    {
      const int dg = tid >> 2, w0 = 8 * (tid & 3);
      int c[8], sum = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        c[q] = s_cnt[(w0 + q) * 256 + dg];
        sum += c[q];
      }
      int tot;
      int base = block_exscan(sum, &tot);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        s_cnt[(w0 + q) * 256 + dg] = base;
        base += c[q];
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortRows; ++r) {
      if (r >= per) break;
      const int at = s_cnt[w * 256 + ((unsigned)(key[r] >> sh) & mask)] +
                     (int)(r & 1 ? rank[r / 2] >> 16 : rank[r / 2] & 0xFFFFu);
      s_key[at] = key[r];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortRows; ++r) {
      if (r >= per) break;
      key[r] = s_key[(w * per + r) * 32 + lane];
    }
    __syncthreads();
  }
}

// Edit lists and records of one direction from `per` * 1024 sorted edits (key[r]
// as in radix_sort; kind 0 none, 1 insert, 2 delete; group_of(key) the list's
// node, member_of(key) the entry). s_key: the keys, and once the groups' heads are
// known the counts before each group (2 (1024 per + 1) ints, the buffer is longer).
template <typename GroupF, typename MemberF>
__device__ void emit_edits(const unsigned long long (&key)[kSortRows], const int (&kind)[kSortRows],
                           int per, unsigned long long* s_key, GroupF group_of, MemberF member_of, int* ins_out, int* del_out, int* rec_node, int* rec_is,
                           int* rec_ic, int* rec_ds, int* rec_dc, int* flag_arr, int* n_rec,
                           int* n_ins, int* n_del) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  int* s_a = reinterpret_cast<int*>(s_key);
  int* s_b = s_a + per * kIngestThreads + 1;
  // the three running counts (insertions, deletions, groups) by warp: a warp's
  // keys are consecutive
  __shared__ int s_heads;
  int ci = 0, cd = 0, ch = 0;
  unsigned bi[kSortRows], bd[kSortRows], bh[kSortRows];
#pragma unroll
  for (int r = 0; r < kSortRows; ++r) {
    bi[r] = bd[r] = bh[r] = 0;
    if (r >= per) continue;
    const int i = (w * per + r) * 32 + lane;
    const bool real = key[r] != kNoKey;
    const bool head = real && (i == 0 || group_of(s_key[i - 1]) != group_of(key[r]));
    bi[r] = __ballot_sync(0xffffffffu, kind[r] == 1);
    bd[r] = __ballot_sync(0xffffffffu, kind[r] == 2);
    bh[r] = __ballot_sync(0xffffffffu, head);
    ci += __popc(bi[r]);
    cd += __popc(bd[r]);
    ch += __popc(bh[r]);
  }
  int ti, td, th;
  const int one = lane == 0;
  int pi = block_exscan(one ? ci : 0, &ti), pd = block_exscan(one ? cd : 0, &td),
      ph = block_exscan(one ? ch : 0, &th);
  pi = __shfl_sync(0xffffffffu, pi, 0);
  pd = __shfl_sync(0xffffffffu, pd, 0);
  ph = __shfl_sync(0xffffffffu, ph, 0);
  // edits out; for group g: counts before its first edit (s_a, s_b)
  int* head_at = rec_node;  // scratch until the records are written: the groups' nodes
#pragma unroll
  for (int r = 0; r < kSortRows; ++r) {
    if (r >= per) break;
    const unsigned lt = lanemask_lt();
    const int ai = pi + __popc(bi[r] & lt), ad = pd + __popc(bd[r] & lt);
    if (kind[r] == 1) ins_out[ai] = member_of(key[r]);
    if (kind[r] == 2) del_out[ad] = member_of(key[r]);
    if ((bh[r] >> lane) & 1u) {
      const int g = ph + __popc(bh[r] & lt);
      s_a[g] = ai;
      s_b[g] = ad;
      head_at[g] = group_of(key[r]);
    }
    pi += __popc(bi[r]);
    pd += __popc(bd[r]);
    ph += __popc(bh[r]);
  }
  if (tid == 0) {
    s_a[th] = ti;
    s_b[th] = td;
    s_heads = 0;
  }
  __syncthreads();
  // groups with an edit, in order
  for (int b = 0; b < th; b += kIngestThreads) {
    const int g = b + tid;
    int node = 0, is = 0, ic = 0, ds = 0, dc = 0;
    if (g < th) {
      node = head_at[g];
      is = s_a[g];
      ic = s_a[g + 1] - is;
      ds = s_b[g];
      dc = s_b[g + 1] - ds;
    }
    int tot;
    const int at = s_heads + block_exscan(ic + dc > 0, &tot);
    if (ic + dc > 0) {  // at <= g: the nodes still to be read lie at or above it
      rec_node[at] = node;
      rec_is[at] = is;
      rec_ic[at] = ic;
      rec_ds[at] = ds;
      rec_dc[at] = dc;
      flag_arr[node] = 1;
    }
    __syncthreads();
    if (tid == 0) s_heads += tot;
    __syncthreads();
  }
  if (tid == 0) {
    *n_rec = s_heads;
    *n_ins = ti;
    *n_del = td;
  }
  __syncthreads();
}

__device__ __forceinline__ int batch_size(const Dev& d, int U) { return U < 0 ? d.ctl->batch_U : U; }

// Keys a thread for a batch of U: whole rows of 1024.
__device__ __forceinline__ int sort_rows(int U) { return max(1, (U + kIngestThreads - 1) / kIngestThreads); }

}  // namespace

__global__ void __launch_bounds__(256) k_ingest_scan(Dev d, const osp_update* __restrict__ ops, int U) {
  __shared__ int s_w[8];
  Ctl* ctl = d.ctl;
  U = batch_size(d, U);
  const int b0 = blockIdx.x * 256;
  if (b0 >= U && blockIdx.x) return;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  // node additions before this CTA's ops, then before each of them
  int before = 0;
  for (int i = tid; i < b0; i += 256) before += ops[i].op == OSP_OP_ADD_NODE;
  before = warp_sum(before);
  if (lane == 0) s_w[w] = before;
  __syncthreads();
  int base = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) base += s_w[q];
  __syncthreads();
  const int p = b0 + tid;
  const bool add = p < U && ops[p].op == OSP_OP_ADD_NODE;
  const unsigned m = __ballot_sync(0xffffffffu, add);
  if (lane == 0) s_w[w] = __popc(m);
  __syncthreads();
  for (int q = 0; q < w; ++q) base += s_w[q];
  const int run = base + __popc(m & lanemask_lt());
  if (p == U - 1) ctl->ing_adds = run + add;
  if (U == 0 && tid == 0) ctl->ing_adds = 0;
  if (p >= U) return;
  const int na = ctl->n + run;
  d.ing_na[p] = na;
  const osp_update o = load_op(ops, p, d);
  if (o.op == OSP_OP_DELETE_NODE) {
    if (o.u >= 0 && o.u < na && !d.dead[o.u] && !d.seedflag[o.u]) atomicMin(&d.del_pos[o.u], p);
    else atomicMin(&ctl->ing_bad, p);
  } else if (o.op == OSP_OP_ZERO_ROW) {
    // the last zeroing of a row in the batch voids the row's earlier edge ops
    ctl->ing_clr = 1;
    if (o.u >= 0 && o.u < na) atomicMax(&d.clr_pos[o.u], p);
    else atomicMin(&ctl->ing_bad, p);
  }
}

__global__ void __launch_bounds__(256) k_ingest_keys(Dev d, const osp_update* __restrict__ ops, int U) {
  Ctl* ctl = d.ctl;
  U = batch_size(d, U);
  const int p = blockIdx.x * 256 + threadIdx.x;
  if (p >= U) return;
  const osp_update o = load_op(ops, p, d);
  const int na = d.ing_na[p];
  const int bits = id_bits(ctl->n + ctl->ing_adds);
  bool ok = false;
  unsigned long long key = kLastKeys | (unsigned)p;
  if (o.op == OSP_OP_INSERT_EDGE || o.op == OSP_OP_DELETE_EDGE) {
    if (o.u >= 0 && o.u < na && o.v >= 0 && o.v < na) {
      const int du = d.del_pos[o.u], dv = d.del_pos[o.v];
      ok = !d.dead[o.u] && !d.dead[o.v] && du > p && dv > p;
      if (du == kNoPos && dv == kNoPos && (!ctl->ing_clr || d.clr_pos[o.u] < p))
        key = ((unsigned long long)o.u << (14 + bits)) | ((unsigned long long)o.v << 14) | (unsigned)p;
    }
  } else if (o.op == OSP_OP_ADD_NODE) {
    ok = true;
  } else if (o.op == OSP_OP_DELETE_NODE) {
    ok = o.u >= 0 && o.u < na && !d.dead[o.u] && !d.seedflag[o.u] && d.del_pos[o.u] == p;
  } else if (o.op == OSP_OP_ZERO_ROW) {
    ok = o.u >= 0 && o.u < na && !d.dead[o.u] && d.del_pos[o.u] > p;
  }
  if (!ok) atomicMin(&ctl->ing_bad, p);
  d.ing_key[p] = key;
}

// n -= a < b: the borrow of a - b, three instructions.
__device__ __forceinline__ void sub_borrow(int& n, unsigned long long a, unsigned long long b) {
  asm("{\n.reg .u32 t;\nsub.cc.u32 t, %1, %3;\nsubc.cc.u32 t, %2, %4;\nsubc.u32 %0, %0, 0;\n}"
      : "+r"(n)
      : "r"((unsigned)a), "r"((unsigned)(a >> 32)), "r"((unsigned)b), "r"((unsigned)(b >> 32)));
}

// Sorted place of each key = how many keys are smaller (they differ in the position;
// ops without a key sort last), or the report of the first invalid op. Lane = key,
// a warp an eighth of the others, which all lanes read together. U^2 comparisons
// over the whole chip are less than five radix passes in one CTA (15,000 keys 62 ->
// 52 us, 10,000 46 -> 34).
__global__ void __launch_bounds__(256) k_ingest_rank(Dev d, const osp_update* __restrict__ ops, int U) {
  __shared__ int s_cnt[8][32];
  __shared__ ulonglong2 s_key[8][32];
  Ctl* ctl = d.ctl;
  U = batch_size(d, U);
  const int i0 = blockIdx.x * 32;
  if (i0 >= U && blockIdx.x) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = i0 + lane;
  const int bad = ctl->ing_bad;
  if (bad != kNoPos) {
    if (w == 0 && i < U) {
      const int op = ops[i].op;
      if (op == OSP_OP_DELETE_NODE || op == OSP_OP_ZERO_ROW) {
        const osp_update o = load_op(ops, i, d);
        if (o.u >= 0 && o.u < d.nc) {
          if (op == OSP_OP_DELETE_NODE) d.del_pos[o.u] = kNoPos;
          else d.clr_pos[o.u] = -1;
        }
      }
    }
    if (i0 == 0 && threadIdx.x == 0) {
      ctl->status = OSP_EINVAL;
      ctl->bad_op = bad;
      ctl->n_clr = 0;
    }
    return;
  }
  const unsigned long long key = i < U ? d.ing_key[i] : kNoKey;
  // 64 keys at a time, a pair a lane, through shared memory; the next ones load
  // meanwhile
  const int pairs = U >> 1;
  const int lo = (int)((long long)pairs * w >> 3), hi = (int)((long long)pairs * (w + 1) >> 3);
  const ulonglong2* all = reinterpret_cast<const ulonglong2*>(d.ing_key);
  const ulonglong2 none = make_ulonglong2(~0ull, ~0ull);  // below no key
  int cnt = 0;
  ulonglong2 next = lo + lane < hi ? __ldg(all + lo + lane) : none;
  for (int b = lo; b < hi; b += 32) {
    __syncwarp();
    s_key[w][lane] = next;
    __syncwarp();
    next = b + 32 + lane < hi ? __ldg(all + b + 32 + lane) : none;
#pragma unroll 16
    for (int q = 0; q < 32; ++q) {
      const ulonglong2 k = s_key[w][q];
      sub_borrow(cnt, k.x, key);
      sub_borrow(cnt, k.y, key);
    }
  }
  cnt = -cnt;
  if (w == 0 && (U & 1)) cnt += d.ing_key[U - 1] < key;
  s_cnt[w][lane] = cnt;
  __syncthreads();
  if (w != 0 || i >= U) return;
#pragma unroll
  for (int q = 1; q < 8; ++q) cnt += s_cnt[q][lane];
  d.ing_sorted[cnt] = key >= kLastKeys ? kNoKey : key;
}

// One thread per sorted op: the last op of each (u, v) against the current row.
__global__ void __launch_bounds__(256) k_ingest_edits(Dev d, const osp_update* __restrict__ ops, int U) {
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  U = batch_size(d, U);
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= U) return;
  const unsigned long long key = d.ing_sorted[i];
  const int n_old = ctl->n;
  const int bits = id_bits(n_old + ctl->ing_adds);
  int kind = 0;
  if (key != kNoKey && (i == U - 1 || (d.ing_sorted[i + 1] >> 14) != (key >> 14))) {
    const int p = (int)(key & 0x3FFF);
    const int u = (int)(key >> (14 + bits));
    const int v = (int)((key >> 14) & ((1ull << bits) - 1));
    const bool after = ops[p].op == OSP_OP_INSERT_EDGE;
    bool before = false;
    if (u < n_old && v < n_old) {
      // u -> v exists iff v is in u's out-list, or u in v's in-list: search the shorter
      const int lr = d.len_r[u], lc = d.len_c[v];
      before = lr <= lc ? contains_i(d.pool_r + d.off_r[u], lr, v)
                        : contains_i(d.pool_c + d.off_c[v], lc, u);
    }
    if (ctl->ing_clr && d.clr_pos[u] >= 0) {
      // u's row was zeroed before this op: the merge drops every old entry of
      // the row (and u from the old in-lists), so a surviving edge is written
      // again as an insertion, but it is not a new edge
      if (after && before) atomicAdd((unsigned long long*)&ctl->ing_reins, 1ull);
      before = false;
    }
    kind = after && !before ? 1 : !after && before ? 2 : 0;
  }
  d.ing_na[i] = kind;
}

// A cluster of two CTAs: rows, node deletions and zeroed rows in the first, the
// columns (with their sort) in the second; one after the other in one CTA they took
// 98 us for 15,000 ops, 59 so. Both read the keys that the columns' edits
// replace, so nothing is written before both have them in registers.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kIngestThreads)
    k_ingest_emit(Dev d, const osp_update* __restrict__ ops, int U) {
  extern __shared__ unsigned long long skey[];
  __shared__ int s_ndel, s_nclr;
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  U = batch_size(d, U);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int per = sort_rows(U);
  const int adds = ctl->ing_adds;
  const int bits = id_bits(ctl->n + adds);
  const bool columns = blockIdx.x == 1;
  int* s_cnt = reinterpret_cast<int*>(skey + per * kIngestThreads);  // 32 x 256 ints
  unsigned long long key[kSortRows];
  int kind[kSortRows];
#pragma unroll
  for (int r = 0; r < kSortRows; ++r) {
    const int i = (w * per + r) * 32 + lane;
    key[r] = r < per && i < U ? d.ing_sorted[i] : kNoKey;
    kind[r] = r < per && i < U ? d.ing_na[i] : 0;
    if (r < per) skey[i] = key[r];
  }
  if (tid == 0) s_ndel = s_nclr = 0;
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  int n_ins = 0, n_del = 0;
  if (!columns) {
    emit_edits(
        key, kind, per, skey, [&](unsigned long long k) { return (int)(k >> (14 + bits)); },
        [&](unsigned long long k) { return (int)((k >> 14) & ((1ull << bits) - 1)); }, d.ins_r, d.del_r,
        d.rec_r_node, d.rec_r_is, d.rec_r_ic, d.rec_r_ds, d.rec_r_dc, d.rflag, &ctl->n_rec_r, &n_ins,
        &n_del);
    if (tid == 0) {  // summed over the sub-batches of a large batch
      ctl->net_ins += n_ins - ctl->ing_reins;
      ctl->net_del += n_del;
    }
    // node deletions and zeroed rows
    for (int p = tid; p < U; p += kIngestThreads) {
      const int op = ops[p].op;
      if (op == OSP_OP_DELETE_NODE) {
        const int u = load_op(ops, p, d).u;
        d.del_nodes[atomicAdd(&s_ndel, 1)] = u;
        d.del_pos[u] = kNoPos;
      } else if (op == OSP_OP_ZERO_ROW) {
        const int u = load_op(ops, p, d).u;
        if (d.clr_pos[u] == p) d.clr_nodes[atomicAdd(&s_nclr, 1)] = u;  // once per row
      }
    }
    __syncthreads();
    if (tid == 0) {
      ctl->n_del = s_ndel;
      ctl->n_clr = s_nclr;
      ctl->n += adds;
    }
    return;
  }
  // the same edits by (v, u): they come by u, so a stable sort by v is enough
#pragma unroll
  for (int r = 0; r < kSortRows; ++r) {
    if (kind[r]) {
      const unsigned long long u = key[r] >> (14 + bits), v = (key[r] >> 14) & ((1ull << bits) - 1);
      key[r] = (v << (bits + 1)) | (u << 1) | (kind[r] == 2);
    } else {
      key[r] = kNoKey;
    }
  }
  __syncthreads();
  radix_sort(key, per, bits + 1, 2 * bits + 1, skey, s_cnt);
#pragma unroll
  for (int r = 0; r < kSortRows; ++r) {
    if (r < per) skey[(w * per + r) * 32 + lane] = key[r];
    kind[r] = r >= per || key[r] == kNoKey ? 0 : key[r] & 1 ? 2 : 1;
  }
  __syncthreads();
  emit_edits(
      key, kind, per, skey, [&](unsigned long long k) { return (int)(k >> (bits + 1)); },
      [&](unsigned long long k) { return (int)((k >> 1) & ((1ull << bits) - 1)); }, d.ins_c, d.del_c,
      d.rec_c_node, d.rec_c_is, d.rec_c_ic, d.rec_c_ds, d.rec_c_dc, d.cflag, &ctl->n_rec_c, &n_ins,
      &n_del);
}

// Node deletions: the deleted node's own row and column are cleared, and every
// row / column holding it as a neighbour is re-written without it. A zeroed
// row (OSP_OP_ZERO_ROW) is re-written empty but for its insertions after the
// op, and so is every in-list holding it.
__global__ void k_expand(Dev d) {
  Ctl* ctl = d.ctl;
  if (*(volatile int*)&ctl->status) return;
  const int nd = ctl->n_del;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int k = gw; k < nd; k += nw) {
    const int w = d.del_nodes[k];
    if (lane == 0) {
      d.dead[w] = 1;
      if (atomicExch(&d.rflag[w], 1) == 0) {
        int at = atomicAdd(&ctl->n_rec_r, 1);
        d.rec_r_node[at] = w;
        d.rec_r_is[at] = d.rec_r_ic[at] = d.rec_r_ds[at] = d.rec_r_dc[at] = 0;
      }
      if (atomicExch(&d.cflag[w], 1) == 0) {
        int at = atomicAdd(&ctl->n_rec_c, 1);
        d.rec_c_node[at] = w;
        d.rec_c_is[at] = d.rec_c_ic[at] = d.rec_c_ds[at] = d.rec_c_dc[at] = 0;
      }
    }
    // out-neighbours x of w: column x loses source w
    const unsigned orow = d.off_r[w];
    const int lrow = d.len_r[w];
    for (int j = lane; j < lrow; j += 32) {
      int x = d.pool_r[orow + j];
      if (atomicExch(&d.cflag[x], 1) == 0) {
        int at = atomicAdd(&ctl->n_rec_c, 1);
        d.rec_c_node[at] = x;
        d.rec_c_is[at] = d.rec_c_ic[at] = d.rec_c_ds[at] = d.rec_c_dc[at] = 0;
      }
    }
    // in-neighbours x of w: row x loses target w
    const unsigned ocol = d.off_c[w];
    const int lcol = d.len_c[w];
    for (int j = lane; j < lcol; j += 32) {
      int x = d.pool_c[ocol + j];
      if (atomicExch(&d.rflag[x], 1) == 0) {
        int at = atomicAdd(&ctl->n_rec_r, 1);
        d.rec_r_node[at] = x;
        d.rec_r_is[at] = d.rec_r_ic[at] = d.rec_r_ds[at] = d.rec_r_dc[at] = 0;
      }
    }
  }
  const int nz = ctl->n_clr;
  for (int k = gw; k < nz; k += nw) {
    const int w = d.clr_nodes[k];
    if (lane == 0 && atomicExch(&d.rflag[w], 1) == 0) {
      int at = atomicAdd(&ctl->n_rec_r, 1);
      d.rec_r_node[at] = w;
      d.rec_r_is[at] = d.rec_r_ic[at] = d.rec_r_ds[at] = d.rec_r_dc[at] = 0;
    }
    // old out-neighbours x of w: column x loses source w (re-inserted if kept)
    const unsigned orow = d.off_r[w];
    const int lrow = d.len_r[w];
    for (int j = lane; j < lrow; j += 32) {
      int x = d.pool_r[orow + j];
      if (atomicExch(&d.cflag[x], 1) == 0) {
        int at = atomicAdd(&ctl->n_rec_c, 1);
        d.rec_c_node[at] = x;
        d.rec_c_is[at] = d.rec_c_ic[at] = d.rec_c_ds[at] = d.rec_c_dc[at] = 0;
      }
    }
  }
}

}  // namespace osp
